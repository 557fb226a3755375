// The forced parts of the float64 form: F^M(0)_n = sum_k Y_k(T_n) V_k and the coarse forcing
// gG_n = sum_k Y_k(T_n) G_k of every slice (pe_contract.cuh).
//
// Bound by the float64 FMA rate (K per mode, slice and part; GB300 has two float64 lanes per SM),
// so the parts are made by their own kernel, in parallel over modes and slices, rather than inside
// the walk over the slices, whose one thread per mode would leave most SMs idle on small grids
// and spread unevenly over their schedulers on others.  A CTA takes 256 modes and SL slices of one
// part: its weights sit in registers (K is a template parameter, no padded columns), the slices'
// columns in shared memory as broadcasts.  255^2 x 32 slices, K = 17: 128 us for both parts (0.88 of
// the measured float64 rate), 65 us for one; a sweep of 64 substeps taken one by one was 3.9 ms.
#include <algorithm>
#include <utility>

#include "pe_internal.h"

namespace {

template <int K>
__global__ void __launch_bounds__(256) forced_f64_kernel(int64_t ndof, int N, int SL, const double* __restrict__ Y,
                                                         const double* __restrict__ V, const double* __restrict__ G,
                                                         double* __restrict__ f, double* __restrict__ gG) {
  pdl_wait();
  extern __shared__ __align__(16) double sYd[];
  const int n0 = blockIdx.y * SL, n1 = min(N, n0 + SL);
  for (int e = threadIdx.x; e < (n1 - n0) * K; e += blockDim.x) sYd[e] = Y[(int64_t)n0 * K + e];
  __syncthreads();
  const int64_t J = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (J >= ndof) return;
  const bool fine = f != nullptr && blockIdx.z == 0;
  const double* src = fine ? V : G;
  double* out = fine ? f : gG;
  double w[K];
#pragma unroll
  for (int k = 0; k < K; ++k) w[k] = src[(int64_t)k * ndof + J];
#pragma unroll 2
  for (int n = n0; n < n1; ++n) {
    const double* y = sYd + (n - n0) * K;
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < K; ++k) acc = fma(y[k], w[k], acc);
    out[(int64_t)n * ndof + J] = acc;
  }
}

template <int K>
pe_status run(pe_ctx* c, double* f, double* gG) {
  const int threads = 256, parts = (f ? 1 : 0) + (gG ? 1 : 0);
  const int64_t tiles = (c->g.ndof + threads - 1) / threads;
  // slices per CTA: about eight CTAs per SM, so that the last wave is a small part of the run
  const int64_t chunks = std::max<int64_t>(1, (8 * (int64_t)std::max(c->sms, 1) + tiles * parts - 1) / (tiles * parts));
  int SL = (int)std::max<int64_t>(1, (c->N + chunks - 1) / chunks);
  SL = std::min(SL, (48 * 1024) / (int)(sizeof(double) * K));
  const dim3 grid((unsigned)tiles, (unsigned)((c->N + SL - 1) / SL), (unsigned)parts);
  PE_CUDA_TRY(launch_pdl(forced_f64_kernel<K>, grid, dim3(threads), sizeof(double) * (size_t)SL * K, c->stream,
                         c->g.ndof, c->N, SL, (const double*)c->tab.Y, (const double*)c->V64, (const double*)c->G64,
                         f, gG));
  c->launches += 1;
  return PE_OK;
}

template <int... I>
pe_status dispatch(int K, pe_ctx* c, double* f, double* gG, std::integer_sequence<int, I...>) {
  pe_status st = PE_EINVAL;
  const bool hit = ((K == I + 1 ? (st = run<I + 1>(c, f, gG), true) : false) || ...);
  return hit ? st : pe_fail(PE_EINVAL, "source columns must be in 1..64");
}

}  // namespace

pe_status launch_forced_f64(pe_ctx* c, double* f, double* gG) {
  return dispatch(c->K, c, f, gG, std::make_integer_sequence<int, 2 * PE_MAX_TERMS>{});
}
