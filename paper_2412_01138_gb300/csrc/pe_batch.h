// Internal layout of the batched solver (pe_batch): per-problem records,
// work items and arenas.  Not part of the ABI.
#pragma once
#include <mutex>
#include <vector>

#include "pe_forcing_common.cuh"
#include "pe_internal.h"

// One problem of the batch, as the kernels see it (offsets index the arenas).
struct BProb {
  Geom g;
  int N, M, q, p, R, Ru;   // slices, substeps, fine/coarse stages, forcing / u0 terms
  int K;                   // source columns (one per exponential, two per sinusoid)
  int tf, tu;              // first forcing / u0 term in the terms array
  double D, t0, dT, dt;
  double lo[PE_MAX_D], h[PE_MAX_D];
  double cF[PE_MAX_S], cG[PE_MAX_S];
  double lagF[PE_MAX_S][PE_MAX_S], lagG[PE_MAX_S][PE_MAX_S];
  int64_t oU;    // U arena: (N+1)*ndof
  int64_t oCF;   // coefF / coefF32 arenas: (q+2)*ndof
  int64_t oCG;   // coefG arena: (p+1)*ndof
  int64_t oAx;   // axisF / axisF32: R*nsum
  int64_t oAxU;  // axisU0: Ru*nsum
  int64_t oY;    // Y: column values, N*K (float: N * 2 * roundup(K, 4), high and low rows, at oY32)
  int64_t oY32;
  int64_t oV;    // V, G: column weights, K*ndof
  int64_t oZ;    // ZF, ZG: shifts of the fine nodes, q*K, then of the coarse ones, p*K
  int64_t oCh;   // chain powers of the terms, [steps][R][4] (float: (hi, lo) pairs at twice the offset)
  int64_t oXs;   // chain scales of the terms, R (float: pairs at twice the offset)
  int64_t oCol;  // column map: K entries, (term << 1) | kind
  int64_t oFirst;  // first column of each term, R entries
  int64_t oMu;   // muM / ratio / rows: nsum
  int64_t oItems;  // first residual slot of this problem
  // learned coarse correction (pe_batch_set_learned): band table K^[r][band] (re, im) at oKt,
  // bands log-spaced in log(lam dT) from lloglo by lstep
  int64_t oKt;
  double lloglo, lstep;
};

struct ModeItem {
  int p;
  int pad;
  int64_t J0;
};

// Walk item: `threads` consecutive modes of a problem, every slice of it; its residual sums go to
// partials[slot].
struct WalkItem {
  int p;
  int slot;
  int64_t J0;
};

struct FactorJob {
  int p, axis, r, u0;
};

// Walk items of one CTA size, longest (most slices) first.
struct WalkItems {
  WalkItem* d_items = nullptr;
  int n = 0;
};

struct pe_batch {
  int P = 0;
  int precision = PE_MIXED;
  int quad_pts = 3;
  int sm_count = 152;
  cudaStream_t stream = nullptr;   // owned, non-blocking (graph capture needs one)
  cudaStream_t user_stream = nullptr;
  std::vector<BProb> probs;
  BProb* d_probs = nullptr;
  std::vector<pe_term> terms;
  pe_term* d_terms = nullptr;
  Gauss gauss;
  int nmax = 1;
  // items
  ModeItem* d_mode_items = nullptr;
  int n_mode_items = 0;
  WalkItems walk128, walk256;
  int Kmax = 1;            // largest column count of a problem
  FactorJob* d_factor_jobs = nullptr;
  int n_factor_jobs = 0;
  int64_t* d_mu_prefix = nullptr;
  int64_t mu_total = 0;
  int64_t* d_tt_prefix = nullptr;
  int64_t tt_total = 0;
  // arenas
  double *muM = nullptr, *ratio = nullptr;
  double* rows = nullptr;     // per axis: sqrt(2/(n+1)) sin(pi m/(n+1)), m = 1..n (the transforms' sine rows)
  double* scratch = nullptr;  // two nodal fields of the largest problem (get_solution)
  int64_t ndof_max = 1;
  double *coefF = nullptr, *coefG = nullptr;
  float *coefF32 = nullptr, *coefG32 = nullptr;
  double* U = nullptr;
  size_t u_total = 0;         // its length
  double *axisF = nullptr, *axisU0 = nullptr;
  float* axisF32 = nullptr;
  // time tables and column weights (pe_contract.cuh); float forms in the mixed form
  double *Y = nullptr, *Z = nullptr, *chain = nullptr, *xs = nullptr;
  float *Y32 = nullptr, *Z32 = nullptr, *chain32 = nullptr, *xs32 = nullptr;
  double *V = nullptr, *G = nullptr;
  float *V32 = nullptr, *G32 = nullptr;
  short* d_first = nullptr;
  short* d_cols = nullptr;
  double* partials = nullptr;
  // per-problem iteration state
  int *active = nullptr, *kcount = nullptr;
  double* resid = nullptr;
  int* counter = nullptr;
  int* dflags = nullptr;   // [0] active problems after the last iteration, [1] non-finite seen
  int* n_active = nullptr;
  int* nonfinite = nullptr;
  int* h_flags = nullptr;  // pinned copy of dflags
  // one graph for the first iteration (which makes the coarse iterates), one for the others
  cudaGraphExec_t graph_exec[2] = {};
  double graph_tol = -1.0;
  int graph_threads = 0, graph_ctas = 0;
  // learned coarse correction (pe_batch_set_learned)
  const struct pe_mlp* mlp = nullptr;
  double* Kt = nullptr;       // band tables of every problem
  int64_t* d_kt_prefix = nullptr;  // per problem: first band-table job (R * bands)
  int64_t kt_jobs = 0;
  int fine_engine = PE_FINE_SIMT;  // (both run the same kernels)
  // launch shape of the persistent walk kernel
  int tune_threads = 128, tune_ctas = 4;
  cudaEvent_t ev[3] = {};          // timing of a solve
  cudaEvent_t ev_order = nullptr;  // between the caller's stream and the batch's
  std::mutex fetch;                // one fetch at a time: it owns scratch until it has waited
  bool have_problem = false;
  int64_t launches = 0;
  uint64_t signature = 0;
};

// pe_batch.cu
pe_status batch_set_attributes(pe_batch* b);
pe_status batch_launch_axis_tables(pe_batch* b);
pe_status batch_launch_coef_tables(pe_batch* b);
pe_status batch_launch_prepare(pe_batch* b);
pe_status batch_enqueue_iteration(pe_batch* b, cudaStream_t st, double tol, bool first);
pe_status batch_time_walk(pe_batch* b, int threads, int ctas, float* ms);
// pe_learned.cu: band tables of the learned correction for every problem of a batch
constexpr int kBatchLearnedBands = 2048;
pe_status batch_learned_tables(pe_batch* b, cudaStream_t st);
