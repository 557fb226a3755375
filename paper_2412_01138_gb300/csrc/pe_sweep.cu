// Coarse sweep, fine sweep, correction and residual of Algorithm 1 (PEIFE-linear).
//
// In mode space every step of Eq. (1-7) is  c <- E c + sum_i (tau b_i) ghat(t_i).  Modes are
// independent, so one thread owns one mode and walks the slices n = 0..N-1 sequentially (the
// "sequential" parts of Algorithm 1 are sequential in n only).
//
//   coarse sweep   U^{n+1,(0)} = G(U^{n,(0)}) = E_G U^n + gG_n.
//   fine sweep     F^M(U^{n,(k)}) = E_F^M U^{n,(k)} + F^M(0)_n, the step being affine in its
//                  argument; F^M(0)_n and gG_n are sums over the K columns of the source
//                  (pe_contract.cuh), evaluated anew in every sweep.
//   correction     U^{n+1,(k+1)} = G(U^{n,(k+1)}) + F^M(U^{n,(k)}) - G(U^{n,(k)}).  G is affine too
//                  (a learned correction adds a term that does not depend on the argument), so
//                  the update is evaluated as
//                    U^{n+1,(k+1)} = F^M(U^{n,(k)}) + E_G (U^{n,(k+1)} - U^{n,(k)}):
//                  the same value, without G(U^{n,(k)}) stored between iterations and
//                  without the cancellation of the two G terms.
//                  Float64 sums  sum mu^M_J (U^{new} - U^{old})^2, sum mu^M_J (U^{new})^2
//                  (per-CTA partial sums, added by the last CTA to finish).
#include <algorithm>

#include "pe_contract.cuh"
#include "pe_internal.h"

namespace {

// Stopping decision of a device-resident loop, run by one thread after the residual sums are
// complete: r_k appended to the history, k advanced, and the graph's while condition set to
// continue while r > tol and k < max_iter (a non-finite sum stops the loop and is flagged).
__device__ void loop_decide(LoopCtl* L, unsigned long long handle, double num, double den, bool first, double tol) {
  const bool finite = isfinite(num) && isfinite(den);
  const double r = den > 0.0 ? sqrt(num) / sqrt(den) : sqrt(num);
  const int k = first ? 0 : L->k;
  if (k < L->hist_cap) L->hist[k] = r;
  L->k = k + 1;
  // the host reads k, r and the flag from its mapped mirror after the solve's one wait
  volatile LoopCtl* H = L->host;
  H->k = k + 1;
  H->r = r;
  if (!finite) H->nonfinite = 1;
  __threadfence_system();
  cudaGraphSetConditional((cudaGraphConditionalHandle)handle,
                          (finite && r > tol && k + 1 < L->max_iter) ? 1u : 0u);
}

// The walk: one thread per mode, the slices in order.  MODE kCoarse makes the coarse iterate, MODE
// kIterate one iteration from the iterate in U, MODE kFirst both in one pass (the coarse value of
// a slice stays in a register; pe_solve).  With o the old and d = U^{new} - U^{old} (0 at n = 0),
//   F = fma(E_F^M, o, F^M(0)_n),  U^{n+1} = fma(E_G, d, F),  d <- U^{n+1} - o',
// o' the old value of slice n + 1 (kFirst: fma(E_G, o, gG_n)), and the residual terms fma(d, d, sd),
// fma(U, U, su): five float64 operations per mode and slice (kFirst: six).
//
// The forced parts come from memory (SRC = 0: the float64 and the general path, made by a kernel
// before) or, in the mixed form (SRC = 1), from the K float32 weights of the mode in registers and
// the float32 columns of the slices in shared memory, read as float4 broadcasts: 2 KB,
// KB = roundup(K, 4), FMAs per part on the float32 pipe, under the float64 operations, of which GB300 does two per
// SM and clock; the sums enter the float64 recurrence through widen_f32.  F^M(0) never exists in
// memory and U is read and written once.  At 255^2 x
// 32 slices, K = 17: 34 us for the coarse sweep and first iteration in one pass, 30 us for a further
// iteration (float64 rate alone: 20 and 17 us), against 17 us (coarse) and 62 + 26 us per iteration
// with every substep taken on the tensor cores; 127^3 x 64, K = 33: 1.57 and 1.37 ms (1.25 and
// 1.04 ms by the float64 rate) against 0.50 and 3.3 + 1.06 ms.
//
// Loads are issued kPF slices ahead (one thread per mode leaves too few threads to cover HBM
// latency with one slice in flight).
constexpr int kCoarse = 0, kIterate = 1, kFirst = 2;
constexpr int kPF = 8;

struct WalkArgs {
  Geom g;
  int N, K, SL;             // SL: slices of columns staged at a time (a multiple of kPF)
  const float *V, *G, *Y;   // SRC = 1: column weights [K][ndof], columns [N][2 KB]
  const double *f, *gG;     // SRC = 0: forced parts [N][ndof]
  const double *EG, *EM;    // e^{-lam dT} of the coarse step, e^{-lam M dt}
  const double* muM_axis;
  double *U, *partials, *red;  // red: mapped host memory
  unsigned int* done;
  LoopCtl* loop;
  const LoopCtl* loop_host;    // its mapped mirror, whose tol the host sets before every solve
  unsigned long long handle;
};

// Threads per CTA: as many as 65536 registers allow with the weights in registers.
__host__ __device__ constexpr int walk_cap(int SRC, int KB, int MODE) {
  return SRC == 0 || (MODE == kIterate ? KB <= 40 : KB <= 28) ? 512 : 256;
}

template <int SRC, int KB, int MODE>
__global__ void __launch_bounds__(walk_cap(SRC, KB, MODE)) walk_kernel(WalkArgs a) {
  extern __shared__ __align__(16) float sY[];  // [SL][2 KB]
  __shared__ double sh[32];
  __shared__ bool s_last;
  const int64_t J = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nd = a.g.ndof;
  const int N = a.N;
  const bool on = J < nd;
  constexpr bool kOld = MODE == kIterate, kF = MODE != kCoarse, kG = MODE != kIterate;
  float V[SRC && kF ? KB : 1], G[SRC && kG ? KB : 1];
  if constexpr (SRC) {
#pragma unroll
    for (int k = 0; k < KB; ++k) {
      if constexpr (kF) V[k] = on && k < a.K ? a.V[(int64_t)k * nd + J] : 0.f;
      if constexpr (kG) G[k] = on && k < a.K ? a.G[(int64_t)k * nd + J] : 0.f;
    }
  }
  double E = 0.0, EM = 0.0, o = 0.0, d = 0.0, sd = 0.0, su = 0.0, w = 0.0;
  // the tolerance of this solve, fetched now so that the last CTA's decision does not wait for it
  double tol = 0.0;
  if (MODE != kCoarse && a.loop && threadIdx.x == 0) tol = reinterpret_cast<const volatile LoopCtl*>(a.loop_host)->tol;
  double* U = a.U + J;
  if (on) {
    E = a.EG[J];
    o = U[0];
    if constexpr (kF) {
      EM = a.EM[J];
      int j[PE_MAX_D];
      unflatten(a.g, J, j);
      w = a.muM_axis[a.g.off[0] + j[0]];
#pragma unroll
      for (int x = 1; x < PE_MAX_D; ++x) if (x < a.g.d) w *= a.muM_axis[a.g.off[x] + j[x]];
    }
  }
  // the next kPF slices' old values and forced parts
  double on1[kOld ? kPF : 1], f1[!SRC && kF ? kPF : 1], g1[!SRC && kG ? kPF : 1];
  auto fetch = [&](int n0) {
#pragma unroll
    for (int e = 0; e < kPF; ++e) {
      const int64_t n = n0 + e;
      const bool in = on && n < N;
      if constexpr (kOld) on1[e] = in ? U[(n + 1) * nd] : 0.0;
      if constexpr (!SRC && kF) f1[e] = in ? a.f[n * nd + J] : 0.0;
      if constexpr (!SRC && kG) g1[e] = in ? a.gG[n * nd + J] : 0.0;
    }
  };
  fetch(0);
  for (int c0 = 0; c0 < N; c0 += a.SL) {
    const int c1 = min(N, c0 + a.SL);
    if constexpr (SRC) {
      __syncthreads();  // the previous chunk's reads are done
      // rows past N (up to a whole group of kPF) are zero
      const int rows = (c1 - c0 + kPF - 1) / kPF * kPF;
      const float4* src = reinterpret_cast<const float4*>(a.Y + (int64_t)c0 * 2 * KB);
      for (int e = threadIdx.x; e < rows * (KB / 2); e += blockDim.x)
        reinterpret_cast<float4*>(sY)[e] = e < (c1 - c0) * (KB / 2) ? src[e] : make_float4(0.f, 0.f, 0.f, 0.f);
      __syncthreads();
    }
    if (on) {
      for (int n0 = c0; n0 < c1; n0 += kPF) {
        double o1[kOld ? kPF : 1], f[!SRC && kF ? kPF : 1], gg[!SRC && kG ? kPF : 1];
#pragma unroll
        for (int e = 0; e < kPF; ++e) {
          if constexpr (kOld) o1[e] = on1[e];
          if constexpr (!SRC && kF) f[e] = f1[e];
          if constexpr (!SRC && kG) gg[e] = g1[e];
        }
        if constexpr (kOld || !SRC) fetch(n0 + kPF);
#pragma unroll
        for (int e = 0; e < kPF; ++e) {
          const int n = n0 + e;
          double fn = 0.0, gn = 0.0;
          if constexpr (SRC) {
            const float* y = sY + (n - c0) * 2 * KB;
            if constexpr (kF) fn = widen_f32(column_dot<KB>(y, V));
            if constexpr (kG) gn = widen_f32(column_dot<KB>(y, G));
          } else {
            if constexpr (kF) fn = f[e];
            if constexpr (kG) gn = gg[e];
          }
          if (n < N) {
            if constexpr (MODE == kCoarse) {
              o = fma(E, o, gn);
              U[(int64_t)(n + 1) * nd] = o;
            } else {
              const double un = fma(E, d, fma(EM, o, fn));
              U[(int64_t)(n + 1) * nd] = un;
              if constexpr (MODE == kFirst) o = fma(E, o, gn);
              else o = o1[e];
              d = un - o;
              sd = fma(d, d, sd);
              su = fma(un, un, su);
            }
          }
        }
      }
    }
  }
  if constexpr (kF) {
    // the weight mu^M_J is the same for every slice of the mode: applied once
    sd = block_sum(sd * w, sh);
    su = block_sum(su * w, sh);
    // the last CTA to finish adds the per-CTA partial sums (in CTA order) and re-arms the counter
    if (threadIdx.x == 0) {
      a.partials[2 * blockIdx.x] = sd;
      a.partials[2 * blockIdx.x + 1] = su;
      __threadfence();
      s_last = atomicAdd(a.done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (s_last) {
      __threadfence();
      double td = 0.0, tu = 0.0;
      for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) {
        td += __ldcg(a.partials + 2 * b);
        tu += __ldcg(a.partials + 2 * b + 1);
      }
      td = block_sum(td, sh);
      tu = block_sum(tu, sh);
      if (threadIdx.x == 0) {
        reinterpret_cast<volatile double*>(a.red)[0] = td;
        reinterpret_cast<volatile double*>(a.red)[1] = tu;
        *a.done = 0u;
        if (a.loop) loop_decide(a.loop, a.handle, td, tu, MODE == kFirst, tol);
      }
    }
  }
}

// F^M(0) of every slice from the float32 weights, stored as float64 (cache_forced and the general path of
// the mixed form; the same sums as the walk makes): a CTA takes 256 modes and SL slices.
template <int KB>
__global__ void __launch_bounds__(256) forced_f32_kernel(int64_t ndof, int N, int K, int SL,
                                                         const float* __restrict__ Y, const float* __restrict__ V,
                                                         double* __restrict__ out) {
  pdl_wait();
  extern __shared__ __align__(16) float sY[];
  const int n0 = blockIdx.y * SL, n1 = min(N, n0 + SL);
  for (int e = threadIdx.x; e < (n1 - n0) * 2 * KB; e += blockDim.x) sY[e] = Y[(int64_t)n0 * 2 * KB + e];
  __syncthreads();
  const int64_t J = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (J >= ndof) return;
  float w[KB];
#pragma unroll
  for (int k = 0; k < KB; ++k) w[k] = k < K ? V[(int64_t)k * ndof + J] : 0.f;
  for (int n = n0; n < n1; ++n) out[(int64_t)n * ndof + J] = (double)column_dot<KB>(sY + (n - n0) * 2 * KB, w);
}

template <int SRC, int KB, int MODE>
pe_status walk_launch(pe_ctx* c, WalkArgs a) {
  const int threads = per_mode_block(c->g.ndof, c->sms, walk_cap(SRC, KB, MODE));
  const int64_t blocks = (c->g.ndof + threads - 1) / threads;
  if (blocks > (int64_t)c->max_blocks) return pe_fail(PE_EINVAL, "walk: partials buffer too small");
  size_t smem = 0;
  a.SL = c->N;
  if (SRC) {
    const int most = (40 * 1024) / (int)(sizeof(float) * 2 * KB) / kPF * kPF;
    a.SL = std::min((c->N + kPF - 1) / kPF * kPF, most);
    smem = sizeof(float) * 2 * (size_t)a.SL * KB;
  }
  // a plain launch (no early start beside the kernel before): one CTA per SM is the even share that
  // per_mode_block chose (200 x 117 nodes: 8 us of a 277 us solve)
  walk_kernel<SRC, KB, MODE><<<(unsigned)blocks, threads, smem, c->stream>>>(a);
  PE_CUDA_TRY(cudaGetLastError());
  c->launches += 1;
  return PE_OK;
}

template <int MODE>
pe_status walk_columns(pe_ctx* c, const WalkArgs& a) {
  switch ((c->K + 3) / 4) {
#define PE_W(X) \
  case X:       \
    return walk_launch<1, 4 * X, MODE>(c, a);
    PE_W(1) PE_W(2) PE_W(3) PE_W(4) PE_W(5) PE_W(6) PE_W(7) PE_W(8) PE_W(9) PE_W(10) PE_W(11) PE_W(12) PE_W(13)
    PE_W(14) PE_W(15) PE_W(16)
#undef PE_W
  }
  return pe_fail(PE_EINVAL, "source columns must be in 1..64");
}

pe_status forced_f32(pe_ctx* c, double* out) {
  const int KB = (c->K + 3) / 4 * 4, threads = 256;
  const int SL = std::min(c->N, std::max(1, (16 * 1024) / (int)(sizeof(float) * 2 * KB)));
  const dim3 grid((unsigned)((c->g.ndof + threads - 1) / threads), (unsigned)((c->N + SL - 1) / SL));
  const size_t smem = sizeof(float) * 2 * (size_t)SL * KB;
  switch (KB / 4) {
#define PE_F(X)                                                                                                    \
  case X:                                                                                                          \
    PE_CUDA_TRY(launch_pdl(forced_f32_kernel<4 * X>, grid, dim3(threads), smem, c->stream, c->g.ndof, c->N, c->K, \
                           SL, (const float*)c->tab.Y32, (const float*)c->V32, out));                              \
    break;
    PE_F(1) PE_F(2) PE_F(3) PE_F(4) PE_F(5) PE_F(6) PE_F(7) PE_F(8) PE_F(9) PE_F(10) PE_F(11) PE_F(12) PE_F(13)
    PE_F(14) PE_F(15) PE_F(16)
#undef PE_F
    default:
      return pe_fail(PE_EINVAL, "source columns must be in 1..64");
  }
  c->launches += 1;
  return PE_OK;
}

WalkArgs walk_args(pe_ctx* c, LoopCtl* loop, unsigned long long handle) {
  WalkArgs a{};
  a.g = c->g;
  a.N = c->N;
  a.K = c->K;
  a.V = c->V32;
  a.G = c->G32;
  a.Y = c->tab.Y32;
  a.f = c->Fbar;
  a.gG = c->gG;
  a.EG = c->coefG;
  a.EM = c->coefF + (int64_t)(c->q + 1) * c->g.ndof;
  a.muM_axis = c->muM_axis;
  a.U = c->U;
  a.partials = c->partials;
  a.red = c->red;
  a.done = c->done_ctr;
  a.loop = loop;
  a.loop_host = c->h_loop_dev;
  a.handle = handle;
  return a;
}

// The walk makes the forced parts itself: the mixed form, every term a sum over columns.
bool mixed_columns(const pe_ctx* c, int precision) {
  return precision == PE_MIXED && c->forcing_path == PE_FORCING_SEPARABLE;
}

// Forced parts in memory: F^M(0) into f, the coarse forcing (float64 here in either form) into gG,
// where not null.
pe_status forced_parts(pe_ctx* c, int precision, double* f, double* gG) {
  // Without a fixed source there are no column sums and the moving terms store theirs (the moving hat on a line
  // of 1023, set-up and four iterations, mixed: one kernel an iteration and six of the set-up fewer, 492 to 460 us)
  if (c->only_moving) {
  } else if (precision == PE_MIXED) {
    if (f) PE_TRY(forced_f32(c, f));
    if (gG) PE_TRY(launch_forced_f64(c, nullptr, gG));
  } else {
    if (f) PE_TRY(launch_column_weights_f64(c));
    PE_TRY(launch_forced_f64(c, f, gG));
  }
  if (gG) PE_TRY(general_add_coarse(c));
  if (f) PE_TRY(general_add_fine(c, precision));
  return PE_OK;
}

}  // namespace

bool first_fused(const pe_ctx* c) { return !c->cache_forced; }

pe_status launch_coarse_sweep(pe_ctx* c) {
  const WalkArgs a = walk_args(c, nullptr, 0ull);
  if (mixed_columns(c, c->precision)) return walk_columns<kCoarse>(c, a);
  PE_TRY(forced_parts(c, c->precision, nullptr, c->gG));
  return walk_launch<0, 4, kCoarse>(c, a);
}

pe_status launch_iteration(pe_ctx* c, int precision, bool first, LoopCtl* loop, unsigned long long handle,
                           cudaEvent_t mid) {
  WalkArgs a = walk_args(c, loop, handle);
  if (mixed_columns(c, precision) && !c->cache_forced) {
    c->sweeps += 1;
    PE_TRY(first ? walk_columns<kFirst>(c, a) : walk_columns<kIterate>(c, a));
    if (mid) PE_CUDA_TRY(cudaEventRecord(mid, c->stream));
    return PE_OK;
  }
  if (c->cache_forced) {
    // one sweep per problem and precision, its forced part kept
    if (c->fz_prec != precision) {
      PE_TRY(forced_parts(c, precision, c->Fz, nullptr));
      c->fz_prec = precision;
      c->sweeps += 1;
    }
    a.f = c->Fz;
  } else {
    if (!c->Fbar && cudaMalloc((void**)&c->Fbar, sizeof(double) * (size_t)c->N * c->g.ndof) != cudaSuccess) {
      cudaGetLastError();
      c->Fbar = nullptr;
      return pe_fail(PE_ENOMEM, "pe_refine: allocation of the forced parts failed");
    }
    a.f = c->Fbar;
    c->sweeps += 1;
    PE_TRY(forced_parts(c, precision, c->Fbar, first ? c->gG : nullptr));
  }
  if (mid) PE_CUDA_TRY(cudaEventRecord(mid, c->stream));
  return first ? walk_launch<0, 4, kFirst>(c, a) : walk_launch<0, 4, kIterate>(c, a);
}

pe_status read_sums(pe_ctx* c, double* num, double* den, cudaEvent_t after) {
  if (after) PE_CUDA_TRY(cudaEventRecord(after, c->stream));
  PE_CUDA_TRY(cudaStreamSynchronize(c->stream));
  const volatile double* h = c->h_red;  // the walk's last CTA wrote the sums here
  *num = h[0];
  *den = h[1];
  return PE_OK;
}
