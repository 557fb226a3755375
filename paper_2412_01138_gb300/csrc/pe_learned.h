// Internal declarations of the learned coarse correction (pe_learned.cu).
#pragma once
#include "pe_internal.h"
#include "pe_phi.cuh"

#define PE_MLP_WIDTH 64
#define PE_LEARNED_BANDS 4096

struct pe_mlp {
  float* params = nullptr;    // float32 master weights (training)
  void* params16 = nullptr;   // float16 copy used for inference
  float* grad = nullptr;
  float* adam_m = nullptr;
  float* adam_v = nullptr;
  float* loss_dev = nullptr;
  float* partial = nullptr;   // per-CTA partial gradients of the training kernel [CTAs][NPARAM + 1]
  int partial_cap = 0;        // CTAs partial has room for
  unsigned* sync = nullptr;   // grid barrier of the training kernel: arrival count, unused, error flag
  int64_t step = 0;
};

struct Nodes8 {
  double c[PE_MAX_S];
};

// per source term: sine kind flag, frequency, phase, amplitude
struct TermsW {
  int R;
  int is_sin[PE_MAX_TERMS];
  double omega[PE_MAX_TERMS];
  double phase[PE_MAX_TERMS];
  double amp[PE_MAX_TERMS];
};

// The band table of the attached network: K^(lam, w_r) (Ktab [R][NB][re, im], null: no network), NB
// bands log-spaced from loglo by logstep in log(lam dT).  The learned term of slice n is
// sum_r P amp Im(e^{i(w T_n + phi)} K^), which is K^'s real part on the sine column of the term and
// its imaginary part on the cosine column: it joins the column weights of the coarse step.
struct LearnedTerms {
  int NB;
  double loglo, logstep, dT;
  const double* Ktab;
};

// Band table of the attached network (one launch); fills *L.
pe_status launch_learned_tables(pe_ctx* c, LearnedTerms* L);
