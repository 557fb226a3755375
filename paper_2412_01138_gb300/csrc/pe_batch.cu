// Batched Parareal EIFE-linear: many independent problems in one set of launches.
//
// Each array kind (slice arrays, tables, forcing factors) lives in one arena; a
// device table of per-problem records (BProb) holds offsets into the arenas.
// Work is cut into items:
//   mode items  (problem, 256 consecutive modes)      coefficient tables, column weights, U^0
//   walk items  (problem, 128 or 256 modes)           the walk over the problem's slices: fine step,
//                                                     correction, residual terms (and, in the first
//                                                     iteration, the coarse iterate)
// The walk kernel is persistent: every CTA pulls items from an atomic counter, longest first.
// One Parareal iteration (reset of the counter, walk, per-problem residual + stop flags, readback
// of the number of active problems) is captured once as a CUDA graph and replayed.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <fstream>
#include <new>
#include <sstream>
#include <string>
#include <vector>

#include "pe_batch.h"
#include "pe_contract.cuh"
#include "pe_phi.cuh"

namespace {

__device__ __forceinline__ int find_prob(const int64_t* __restrict__ prefix, int P, int64_t idx) {
  int lo = 0, hi = P - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (prefix[mid] <= idx) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// ---------------------------------------------------------------------------
// setup kernels
// ---------------------------------------------------------------------------
__global__ void b_axis_tables_kernel(const BProb* __restrict__ probs, const int64_t* __restrict__ mu_prefix, int P,
                                     int64_t total, double* __restrict__ muM, double* __restrict__ ratio,
                                     double* __restrict__ rows) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= total) return;
  const int p = find_prob(mu_prefix, P, idx);
  const BProb& B = probs[p];
  const int local = (int)(idx - B.oMu);
  int a = 0;
  while (a + 1 < B.g.d && local >= B.g.off[a + 1]) ++a;
  const int j = local - B.g.off[a];
  const double h = B.h[a];
  const double np1 = (double)(B.g.n[a] + 1);
  const double cth = cospi((double)(j + 1) / np1);
  const double sh = sinpi((double)(j + 1) / (2.0 * np1));
  const double mM = (h / 3.0) * (2.0 + cth);
  const double mK = (4.0 / h) * (sh * sh);
  muM[idx] = mM;
  ratio[idx] = mK / mM;
  rows[idx] = sqrt(2.0 / np1) * sinpi((double)(j + 1) / np1);
}

__global__ void b_coef_tables_kernel(const BProb* __restrict__ probs, const ModeItem* __restrict__ items,
                                     int n_items, const double* __restrict__ ratio, double* __restrict__ coefF,
                                     double* __restrict__ coefG, float* __restrict__ coefF32,
                                     float* __restrict__ coefG32) {
  for (int it = blockIdx.x; it < n_items; it += gridDim.x) {
    const ModeItem m = items[it];
    const BProb& B = probs[m.p];
    const int64_t J = m.J0 + threadIdx.x;
    if (J >= B.g.ndof) continue;
    const int64_t nd = B.g.ndof;
    int j[PE_MAX_D];
    unflatten(B.g, J, j);
    double s = 0.0;
#pragma unroll
    for (int a = 0; a < PE_MAX_D; ++a) if (a < B.g.d) s += ratio[B.oMu + B.g.off[a] + j[a]];
    const double lam = B.D * s;
    Lag LF, LG;
    for (int i = 0; i < PE_MAX_S; ++i)
      for (int k = 0; k < PE_MAX_S; ++k) {
        LF.a[i][k] = B.lagF[i][k];
        LG.a[i][k] = B.lagG[i][k];
      }
    double b[PE_MAX_S];
    {
      const double z = -lam * B.dt;
      const double E = exp(z);
      b_weights(z, B.q, LF, b);
      double* cf = coefF + B.oCF;
      cf[J] = E;
      for (int i = 0; i < B.q; ++i) cf[(1 + i) * nd + J] = B.dt * b[i];
      cf[(B.q + 1) * nd + J] = exp(-lam * ((double)B.M * B.dt));
      if (coefF32) {
        float* c32 = coefF32 + B.oCF;
        const float ehi = (float)E;
        c32[J] = ehi;
        c32[nd + J] = (float)(E - (double)ehi);
        for (int i = 0; i < B.q; ++i) c32[(2 + i) * nd + J] = (float)(B.dt * b[i]);
      }
    }
    {
      const double z = -lam * B.dT;
      b_weights(z, B.p, LG, b);
      double* cg = coefG + B.oCG;
      cg[J] = exp(z);
      for (int i = 0; i < B.p; ++i) {
        cg[(1 + i) * nd + J] = B.dT * b[i];
        if (coefG32) coefG32[B.oCG + (1 + i) * nd + J] = (float)(B.dT * b[i]);
      }
    }
  }
}

// Time tables of every problem, one thread per entry, as the single-problem solver makes them
// (pe_forcing.cu): column values of every slice, shifts of the fine and coarse nodes, chain powers
// and scales of the terms.  Column k of a problem is cols[oCol + k] = (term << 1) | kind.
struct BTables {
  double *Y, *Z, *chain, *xs;
  float *Y32, *Z32, *chain32, *xs32;
};

__global__ void b_time_tables_kernel(const BProb* __restrict__ probs, const int64_t* __restrict__ tt_prefix, int P,
                                     int64_t total, const pe_term* __restrict__ terms,
                                     const short* __restrict__ cols, BTables D) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= total) return;
  const int p = find_prob(tt_prefix, P, idx);
  const BProb& B = probs[p];
  const int R = B.R, K = B.K, steps = chain_steps(B.M);
  int64_t e = idx - tt_prefix[p];
  if (e < (int64_t)B.N * K) {
    const int n = (int)(e / K), k = (int)(e - (int64_t)n * K);
    const int c = cols[B.oCol + k];
    const double v = column_value(terms[B.tf + (c >> 1)], c & 1, B.t0 + (double)n * B.dT, B.t0 + (double)(n + 1) * B.dT);
    if (!D.Y32) {
      D.Y[B.oY + e] = v;
    } else {
      const int KC = (K + 3) & ~3;
      float* row = D.Y32 + B.oY32 + (int64_t)n * 2 * KC;
      row[k] = (float)v;
      row[KC + k] = (float)(v - (double)(float)v);
      if (k == K - 1)
        for (int z = K; z < KC; ++z) row[z] = row[KC + z] = 0.f;
    }
    return;
  }
  e -= (int64_t)B.N * K;
  const int nf = B.q * K, ng = B.p * K;
  if (e < nf + ng) {
    const bool fine = e < nf;
    const int l = (int)(fine ? e : e - nf), i = l / K, k = l - i * K;
    const int c = cols[B.oCol + k];
    const double v = column_shift(terms[B.tf + (c >> 1)], c & 1, fine ? B.cF[i] : B.cG[i], fine ? B.dt : B.dT);
    if (D.Y32) D.Z32[B.oZ + e] = (float)v;
    else D.Z[B.oZ + e] = v;
    return;
  }
  e -= nf + ng;
  const int s = (int)(e / R) - 1, r = (int)(e - (int64_t)(s + 1) * R);
  const pe_term& T = terms[B.tf + r];
  if (s < 0) {
    const double v = chain_scale(T, B.dt);
    if (!D.Y32) {
      D.xs[B.oXs + r] = v;
    } else {
      D.xs32[2 * (B.oXs + r)] = (float)v;
      D.xs32[2 * (B.oXs + r) + 1] = (float)(v - (double)(float)v);
    }
    return;
  }
  double v[4];
  const int L = chain_length(B.M, steps, s);
  chain_power(T, L, B.dt, v[0], v[1]);
  chain_power(T, 2 * L, B.dt, v[2], v[3]);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t o = B.oCh + (int64_t)(s * R + r) * 4 + i;
    if (!D.Y32) {
      D.chain[o] = v[i];
    } else {
      D.chain32[2 * o] = (float)v[i];
      D.chain32[2 * o + 1] = (float)(v[i] - (double)(float)v[i]);
    }
  }
}

// The learned correction's band tables (Kt null: no network).
struct BLearn {
  const double* ratio;    // per-axis mu^K / mu^M (lam = D sum_a ratio)
  const double* Kt;
  const double* axisF64;
  int NB;
};

// Per-mode column weights V and G of every problem (column_weights_kernel of the single-problem
// solver over mode items).
template <typename T>
__global__ void __launch_bounds__(256) b_column_weights_kernel(const BProb* __restrict__ probs,
                                                               const ModeItem* __restrict__ items, int n_items,
                                                               const short* __restrict__ first,
                                                               const short* __restrict__ cols,
                                                               const T* __restrict__ axisF, const T* __restrict__ coefF,
                                                               const T* __restrict__ coefG, const T* __restrict__ Z,
                                                               const T* __restrict__ chain, const T* __restrict__ xs,
                                                               T* __restrict__ V, T* __restrict__ G, BLearn L) {
  constexpr bool F64 = sizeof(T) == 8;
  constexpr int kERows = F64 ? 1 : 2, kPair = F64 ? 1 : 2;
  for (int it = blockIdx.x; it < n_items; it += gridDim.x) {
    const ModeItem mi = items[it];
    const BProb& B = probs[mi.p];
    const int64_t J = mi.J0 + threadIdx.x;
    if (J >= B.g.ndof) continue;
    const int64_t nd = B.g.ndof;
    const int K = B.K, R = B.R, q = B.q, p = B.p, steps = chain_steps(B.M);
    int j[PE_MAX_D];
    unflatten(B.g, J, j);
    const T* cf = coefF + B.oCF;
    T b[PE_MAX_S], bg[PE_MAX_S];
#pragma unroll
    for (int i = 0; i < PE_MAX_S; ++i) {
      b[i] = i < q ? cf[(int64_t)(kERows + i) * nd + J] : T(0);
      bg[i] = i < p ? coefG[B.oCG + (int64_t)(1 + i) * nd + J] : T(0);
    }
    const T Eh = cf[J];
    T El = T(0);
    if constexpr (!F64) El = cf[nd + J];
    int band = 0;
    double bf = 0.0;
    if (L.Kt) {
      double sum = 0.0;
#pragma unroll
      for (int a = 0; a < PE_MAX_D; ++a) if (a < B.g.d) sum += L.ratio[B.oMu + B.g.off[a] + j[a]];
      double pos = (log(B.D * sum * B.dT) - B.lloglo) / B.lstep;
      pos = fmin(fmax(pos, 0.0), (double)(L.NB - 1) - 1e-9);
      band = (int)pos;
      bf = pos - (double)band;
    }
    const T* ax = axisF + B.oAx;
    const T* ZF = Z + B.oZ;
    const T* ZG = ZF + (int64_t)q * K;
    for (int r = 0; r < R; ++r) {
      const int k = first[B.oFirst + r];
      const bool two = k + 1 < K && (cols[B.oCol + k + 1] >> 1) == r;
      T P = ax[(int64_t)R * B.g.off[0] + (int64_t)r * B.g.n[0] + j[0]];
#pragma unroll
      for (int a = 1; a < PE_MAX_D; ++a) if (a < B.g.d) P *= ax[(int64_t)R * B.g.off[a] + (int64_t)r * B.g.n[a] + j[a]];
      T br = T(0), bi = T(0), gr = T(0), gi = T(0);
#pragma unroll
      for (int i = 0; i < PE_MAX_S; ++i)
        if (i < q) {
          br = fma(b[i], ZF[i * K + k], br);
          if (two) bi = fma(b[i], ZF[i * K + k + 1], bi);
        }
#pragma unroll
      for (int i = 0; i < PE_MAX_S; ++i)
        if (i < p) {
          gr = fma(bg[i], ZG[i * K + k], gr);
          if (two) gi = fma(bg[i], ZG[i * K + k + 1], gi);
        }
      gr *= P;
      gi *= P;
      if (L.Kt && two) {
        const double* ax64 = L.axisF64 + B.oAx;
        double Pd = ax64[(int64_t)R * B.g.off[0] + (int64_t)r * B.g.n[0] + j[0]];
#pragma unroll
        for (int a = 1; a < PE_MAX_D; ++a)
          if (a < B.g.d) Pd *= ax64[(int64_t)R * B.g.off[a] + (int64_t)r * B.g.n[a] + j[a]];
        const double* k0 = L.Kt + B.oKt + 2 * ((int64_t)r * L.NB + band);
        gr += (T)(Pd * ((1.0 - bf) * k0[0] + bf * k0[2]));
        gi += (T)(Pd * ((1.0 - bf) * k0[1] + bf * k0[3]));
      }
      T v0, v1;
      const T* ch = chain + kPair * (B.oCh + 4 * r);
      const T* x = xs + kPair * (B.oXs + r);
      if constexpr (F64) {
        double Sr, Si;
        chain_sum(Eh * x[0], B.M, steps, ch, 4 * R, Sr, Si);
        v0 = P * fma(br, Sr, -(bi * Si));
        v1 = P * fma(br, Si, bi * Sr);
      } else {
        F2 Sr, Si;
        chain_sum(f2_mul(F2{Eh, El}, F2{x[0], x[1]}), B.M, steps, ch, 8 * R, Sr, Si);
        const F2 br2{br, 0.f}, bi2{bi, 0.f};
        const F2 re = f2_add(f2_mul(br2, Sr), f2_neg(f2_mul(bi2, Si)));
        const F2 im = f2_add(f2_mul(br2, Si), f2_mul(bi2, Sr));
        v0 = fmaf(P, re.h, P * re.l);
        v1 = fmaf(P, im.h, P * im.l);
      }
      V[B.oV + (int64_t)k * nd + J] = v0;
      G[B.oV + (int64_t)k * nd + J] = gr;
      if (two) {
        V[B.oV + (int64_t)(k + 1) * nd + J] = v1;
        G[B.oV + (int64_t)(k + 1) * nd + J] = gi;
      }
    }
  }
}

// One CTA per (problem, axis, term): the 1D consistent load of the term's factor on that axis, its DST-I
// (sine table in shared memory) and the division by mu^M.  The transform is folded by its symmetry: even
// outputs from the sums of mirrored loads, odd ones from the differences, n/2 float64 FMAs per
// output, which bound the kernel.  Jobs are ordered longest axis first.  64 problems (1626 jobs): 179 us
// against 409 us unfolded.
__global__ void __launch_bounds__(256) b_axis_factor_kernel(const BProb* __restrict__ probs,
                                                            const FactorJob* __restrict__ jobs,
                                                            const pe_term* __restrict__ terms, Gauss G,
                                                            const double* __restrict__ muM,
                                                            double* __restrict__ axisF, float* __restrict__ axisF32,
                                                            double* __restrict__ axisU0) {
  extern __shared__ double sh[];
  const FactorJob job = jobs[blockIdx.x];
  const BProb& B = probs[job.p];
  const int a = job.axis;
  const int n = B.g.n[a], h = (n + 1) / 2;
  const int period = 2 * (n + 1);
  double* F = sh;             // [n]
  double* tab = sh + n;       // [period]: sin(pi m/(n+1))
  const pe_term& T = terms[job.u0 ? B.tu + job.r : B.tf + job.r];
  const double lo = B.lo[a], hx = B.h[a];
  for (int m = threadIdx.x; m <= n; m += blockDim.x) {
    const double s = sinpi((double)m / (double)(n + 1));
    tab[m] = s;
    tab[m + n + 1] = -s;
  }
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    double left = 0.0, right = 0.0;
    for (int qi = 0; qi < G.npts; ++qi) {
      const double xl = lo + ((double)k + G.s[qi]) * hx;
      const double xr = lo + ((double)(k + 1) + G.s[qi]) * hx;
      left += G.w[qi] * eval_space(T.skind[a], T.sp[a], xl) * G.s[qi];
      right += G.w[qi] * eval_space(T.skind[a], T.sp[a], xr) * (1.0 - G.s[qi]);
    }
    F[k] = hx * left + hx * right;
  }
  __syncthreads();
  // F[k] <- sum, F[n-1-k] <- difference of the mirrored loads (the middle one of an odd n stays)
  for (int k = threadIdx.x; k < n / 2; k += blockDim.x) {
    const double u = F[k], v = F[n - 1 - k];
    F[k] = u + v;
    F[n - 1 - k] = u - v;
  }
  __syncthreads();
  const double scale = sqrt(2.0 / (double)(n + 1));
  const int Rj = job.u0 ? B.Ru : B.R;
  const int64_t obase = (job.u0 ? B.oAxU : B.oAx) + (int64_t)Rj * B.g.off[a] + (int64_t)job.r * n;
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    double acc = 0.0;
    int idx = 0;
    const int step = j + 1;
    const bool odd = j & 1;
    const int cnt = odd ? n / 2 : h;
    const double* f = odd ? F + n - 1 : F;
    const int df = odd ? -1 : 1;
#pragma unroll 4
    for (int k = 0; k < cnt; ++k) {
      idx += step;
      if (idx >= period) idx -= period;
      acc = fma(tab[idx], *f, acc);
      f += df;
    }
    const double v = scale * acc / muM[B.oMu + B.g.off[a] + j];
    if (job.u0) {
      axisU0[obase + j] = v;
    } else {
      axisF[obase + j] = v;
      if (axisF32) axisF32[obase + j] = (float)v;
    }
  }
}

// U^0 = sum_t amp_t prod_a axisU0 (P_h of separable initial data)
__global__ void b_u0_kernel(const BProb* __restrict__ probs, const ModeItem* __restrict__ items, int n_items,
                            const pe_term* __restrict__ terms, const double* __restrict__ axisU0,
                            double* __restrict__ U) {
  for (int it = blockIdx.x; it < n_items; it += gridDim.x) {
    const ModeItem m = items[it];
    const BProb& B = probs[m.p];
    const int64_t J = m.J0 + threadIdx.x;
    if (J >= B.g.ndof) continue;
    int j[PE_MAX_D];
    unflatten(B.g, J, j);
    double acc = 0.0;
    for (int t = 0; t < B.Ru; ++t) {
      double v = axisU0[B.oAxU + (int64_t)B.Ru * B.g.off[0] + (int64_t)t * B.g.n[0] + j[0]];
#pragma unroll
      for (int a = 1; a < PE_MAX_D; ++a) if (a < B.g.d)
        v *= axisU0[B.oAxU + (int64_t)B.Ru * B.g.off[a] + (int64_t)t * B.g.n[a] + j[a]];
      acc += terms[B.tu + t].amp * v;
    }
    U[B.oU + J] = acc;
  }
}

// The walk of the single-problem solver (walk_kernel, pe_sweep.cu) over items of many problems: F =
// fma(E_F^M, o, F^M(0)_n), U^{n+1} = fma(E_G, d, F), d <- U^{n+1} - o'; FIRST makes the coarse
// iterate o' = fma(E_G, o, gG_n) on the way, else o' is the old U^{n+1}.
//
// T = float (mixed form): the item's K column weights in registers, KB = the batch's largest K rounded up
// to 8 (the float32 FMAs of the padding run under the five or six float64 operations per mode and slice
// that bound the kernel).  T = double: weights in shared memory with a runtime column count, since
// every padded column would cost a float64 operation, and one per operation is what two shared-memory
// reads hide under.  A batch has modes enough for one thread per mode, so that the float64 forced parts
// never go to memory either.  64 uneven 2D problems (1.6M modes, 16 to 64 slices, 9 to 33 columns), mixed: 0.89 ms for
// the coarse sweep and first iteration in one pass, 0.76 ms for a further one, against 0.94 ms (every substep on the
// tensor cores) + 0.49 ms (correction) per iteration beside the coarse sweep.
constexpr int kPF = 8;  // slices of loads in flight

template <typename T>
struct BWalkArgs {
  const BProb* probs;
  const WalkItem* items;
  int n_items, SL;       // SL: slices staged at a time (a multiple of kPF)
  const int* active;
  int* counter;
  const T *Y, *V, *G;
  const double *coefF, *coefG, *muM;
  double *U, *partials;
};

template <typename T, int KB, bool FIRST>
__global__ void __launch_bounds__(256) b_walk_kernel(BWalkArgs<T> a) {
  constexpr bool F64 = sizeof(T) == 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double sh[32];
  __shared__ int s_item;
  const int tid = threadIdx.x, B_ = blockDim.x;
  T* sY = reinterpret_cast<T*>(smem_raw);  // float: [SL][2 KB]; double: [SL][K]
  for (;;) {
    if (tid == 0) s_item = atomicAdd(a.counter, 1);
    __syncthreads();
    const int it = s_item;
    if (it >= a.n_items) return;
    const WalkItem mi = a.items[it];
    if (!a.active[mi.p]) {  // uniform over the CTA
      __syncthreads();
      continue;
    }
    const BProb& B = a.probs[mi.p];
    const int64_t J = mi.J0 + tid, nd = B.g.ndof;
    const int N = B.N, K = B.K;
    const bool on = J < nd;
    T* sV = sY + (F64 ? a.SL * K : 0);  // double: [K][threads], then G
    float V[F64 ? 1 : KB], G[!F64 && FIRST ? KB : 1];
    if constexpr (F64) {
      for (int k = 0; k < K; ++k) {
        sV[k * B_ + tid] = on ? a.V[B.oV + (int64_t)k * nd + J] : T(0);
        if constexpr (FIRST) sV[(K + k) * B_ + tid] = on ? a.G[B.oV + (int64_t)k * nd + J] : T(0);
      }
    } else {
#pragma unroll
      for (int k = 0; k < KB; ++k) {
        V[k] = on && k < K ? a.V[B.oV + (int64_t)k * nd + J] : 0.f;
        if constexpr (FIRST) G[k] = on && k < K ? a.G[B.oV + (int64_t)k * nd + J] : 0.f;
      }
    }
    double E = 0.0, EM = 0.0, o = 0.0, d = 0.0, sd = 0.0, su = 0.0, w = 0.0;
    double* U = a.U + B.oU + J;
    if (on) {
      E = a.coefG[B.oCG + J];
      EM = a.coefF[B.oCF + (int64_t)(B.q + 1) * nd + J];
      o = U[0];
      int j[PE_MAX_D];
      unflatten(B.g, J, j);
      w = a.muM[B.oMu + B.g.off[0] + j[0]];
#pragma unroll
      for (int x = 1; x < PE_MAX_D; ++x) if (x < B.g.d) w *= a.muM[B.oMu + B.g.off[x] + j[x]];
    }
    double on1[FIRST ? 1 : kPF];
    auto fetch = [&](int n0) {
      if constexpr (!FIRST) {
#pragma unroll
        for (int e = 0; e < kPF; ++e) on1[e] = on && n0 + e < N ? U[(int64_t)(n0 + e + 1) * nd] : 0.0;
      }
    };
    fetch(0);
    const int KC = F64 ? K : (K + 3) & ~3;
    for (int c0 = 0; c0 < N; c0 += a.SL) {
      const int c1 = min(N, c0 + a.SL), rows = (c1 - c0 + kPF - 1) / kPF * kPF;
      __syncthreads();  // the previous chunk's (or item's) reads are done
      if constexpr (F64) {
        const T* src = a.Y + B.oY + (int64_t)c0 * K;
        for (int e = tid; e < rows * K; e += B_) sY[e] = e < (c1 - c0) * K ? src[e] : T(0);
      } else {
        // rows of KC columns widened to KB with zeros, high and low parts
        const T* src = a.Y + B.oY32 + (int64_t)c0 * 2 * KC;
        for (int e = tid; e < rows * 2 * KB; e += B_) {
          const int row = e / KB, k = e - row * KB;
          sY[e] = row < 2 * (c1 - c0) && k < KC ? src[row * KC + k] : T(0);
        }
      }
      __syncthreads();
      if (on) {
        for (int n0 = c0; n0 < c1; n0 += kPF) {
          double o1[FIRST ? 1 : kPF];
          if constexpr (!FIRST) {
#pragma unroll
            for (int e = 0; e < kPF; ++e) o1[e] = on1[e];
            fetch(n0 + kPF);
          }
          double fv[F64 ? kPF : 1], gv[F64 && FIRST ? kPF : 1];
          if constexpr (F64) {
#pragma unroll
            for (int e = 0; e < kPF; ++e) {
              fv[e] = 0.0;
              if constexpr (FIRST) gv[e] = 0.0;
            }
            for (int k = 0; k < K; ++k) {
              const T v = sV[k * B_ + tid];
              T g = T(0);
              if constexpr (FIRST) g = sV[(K + k) * B_ + tid];
#pragma unroll
              for (int e = 0; e < kPF; ++e) {
                const T y = sY[(n0 - c0 + e) * K + k];
                fv[e] = fma(y, v, fv[e]);
                if constexpr (FIRST) gv[e] = fma(y, g, gv[e]);
              }
            }
          }
#pragma unroll
          for (int e = 0; e < kPF; ++e) {
            const int n = n0 + e;
            double fn, gn = 0.0;
            if constexpr (F64) {
              fn = fv[e];
              if constexpr (FIRST) gn = gv[e];
            } else {
              const float* y = reinterpret_cast<const float*>(sY) + (n - c0) * 2 * KB;
              fn = widen_f32(column_dot<KB>(y, V));
              if constexpr (FIRST) gn = widen_f32(column_dot<KB>(y, G));
            }
            if (n < N) {
              const double un = fma(E, d, fma(EM, o, fn));
              U[(int64_t)(n + 1) * nd] = un;
              if constexpr (FIRST) o = fma(E, o, gn);
              else o = o1[e];
              d = un - o;
              sd = fma(d, d, sd);
              su = fma(un, un, su);
            }
          }
        }
      }
    }
    sd = block_sum(sd * w, sh);
    su = block_sum(su * w, sh);
    if (tid == 0) {
      a.partials[2 * mi.slot] = sd;
      a.partials[2 * mi.slot + 1] = su;
    }
  }
}

// one CTA per problem: residual, iteration count, stop flag, active count
__global__ void b_reduce_kernel(const BProb* __restrict__ probs, int P, int item_modes,
                                const double* __restrict__ partials,
                                int* __restrict__ active, int* __restrict__ kcount, double* __restrict__ resid,
                                double tol, int* __restrict__ n_active, int* __restrict__ nonfinite) {
  __shared__ double sh[32];
  const int p = blockIdx.x;
  if (p >= P) return;
  const BProb& B = probs[p];
  if (!active[p]) return;  // uniform
  double sd = 0.0, su = 0.0;
  const int nItems = (int)((B.g.ndof + item_modes - 1) / item_modes);  // at slots oItems + i
  for (int i = threadIdx.x; i < nItems; i += blockDim.x) {
    sd += partials[2 * (B.oItems + i)];
    su += partials[2 * (B.oItems + i) + 1];
  }
  sd = block_sum(sd, sh);
  su = block_sum(su, sh);
  if (threadIdx.x == 0) {
    const double r = su > 0.0 ? sqrt(sd) / sqrt(su) : sqrt(sd);
    resid[p] = r;
    const int k = kcount[p] + 1;
    kcount[p] = k;
    if (!isfinite(r)) {
      atomicExch(nonfinite, 1);
      active[p] = 0;
    } else if (r <= tol || k >= B.N) {
      active[p] = 0;
    } else {
      atomicAdd(n_active, 1);
    }
  }
}

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
namespace {

// Dynamic shared memory of the walk and the slices it stages: float rows of 2 KB within 32 KB; double rows
// of Kmax beside the weights of `threads` modes.
template <typename T>
size_t walk_smem(const pe_batch* b, int threads, int KB, int* SL) {
  int Nmax = 1;
  for (const BProb& B : b->probs) Nmax = std::max(Nmax, B.N);
  const size_t row = sizeof(T) * (size_t)(sizeof(T) == 8 ? b->Kmax : 2 * KB);
  int sl = (int)((size_t)32 * 1024 / row) / kPF * kPF;
  sl = std::max(kPF, std::min(sl, (Nmax + kPF - 1) / kPF * kPF));
  *SL = sl;
  return row * sl + (sizeof(T) == 8 ? sizeof(T) * 2 * (size_t)b->Kmax * threads : 0);
}

template <typename T, int KB, bool FIRST>
pe_status walk_launch(pe_batch* b, cudaStream_t st, int threads, int ctas, bool set_attr) {
  int SL = 0;
  const size_t smem = walk_smem<T>(b, threads, KB, &SL);
  if (set_attr) {  // at set-up, outside any capture: the limit any batch may need (40 columns, 256 threads)
    if (sizeof(T) == 8)
      PE_CUDA_TRY(cudaFuncSetAttribute(b_walk_kernel<T, KB, FIRST>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       200 * 1024));
    return PE_OK;
  }
  const WalkItems& wi = threads == 128 ? b->walk128 : b->walk256;
  BWalkArgs<T> a{};
  a.probs = b->d_probs;
  a.items = wi.d_items;
  a.n_items = wi.n;
  a.SL = SL;
  a.active = b->active;
  a.counter = b->counter;
  if constexpr (sizeof(T) == 8) {
    a.Y = b->Y;
    a.V = b->V;
    a.G = b->G;
  } else {
    a.Y = b->Y32;
    a.V = b->V32;
    a.G = b->G32;
  }
  a.coefF = b->coefF;
  a.coefG = b->coefG;
  a.muM = b->muM;
  a.U = b->U;
  a.partials = b->partials;
  const int grid = std::min(b->sm_count * ctas, wi.n);
  b_walk_kernel<T, KB, FIRST><<<grid, threads, smem, st>>>(a);
  PE_CUDA_TRY(cudaGetLastError());
  return PE_OK;
}

pe_status launch_walk(pe_batch* b, cudaStream_t st, int threads, int ctas, bool first, bool set_attr = false) {
  if (b->precision != PE_MIXED)
    return first ? walk_launch<double, 8, true>(b, st, threads, ctas, set_attr)
                 : walk_launch<double, 8, false>(b, st, threads, ctas, set_attr);
  switch ((b->Kmax + 7) / 8) {
#define PE_BW(X)                                                                       \
  case X:                                                                              \
    return first ? walk_launch<float, 8 * X, true>(b, st, threads, ctas, set_attr)     \
                 : walk_launch<float, 8 * X, false>(b, st, threads, ctas, set_attr);
    PE_BW(1) PE_BW(2) PE_BW(3) PE_BW(4) PE_BW(5)
#undef PE_BW
  }
  return pe_fail(PE_EINVAL, "batch: source columns must be in 1..40");
}

}  // namespace

pe_status batch_set_attributes(pe_batch* b) {
  // the limit any batch may need (n_a <= 4096)
  PE_CUDA_TRY(cudaFuncSetAttribute(b_axis_factor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)sizeof(double) * (4096 + 2 * 4097)));
  for (int threads = 128; threads <= 256; threads += 128)
    for (int first = 0; first < 2; ++first) PE_TRY(launch_walk(b, b->stream, threads, 1, first != 0, true));
  return PE_OK;
}

pe_status batch_launch_axis_tables(pe_batch* b) {
  const int64_t total = b->mu_total;
  b_axis_tables_kernel<<<(unsigned)((total + 255) / 256), 256, 0, b->stream>>>(b->d_probs, b->d_mu_prefix, b->P,
                                                                              total, b->muM, b->ratio, b->rows);
  b->launches += 1;
  PE_CUDA_TRY(cudaGetLastError());
  return PE_OK;
}

// phi/b coefficient tables: a function of lam, the step sizes and the nodes only (made at set-up)
pe_status batch_launch_coef_tables(pe_batch* b) {
  b_coef_tables_kernel<<<b->sm_count * 8, 256, 0, b->stream>>>(b->d_probs, b->d_mode_items, b->n_mode_items,
                                                               b->ratio, b->coefF, b->coefG, b->coefF32,
                                                               b->coefG32);
  b->launches += 1;
  PE_CUDA_TRY(cudaGetLastError());
  return PE_OK;
}

pe_status batch_launch_prepare(pe_batch* b) {
  const int grid_items = b->sm_count * 8;
  // time tables
  const BTables D{b->Y, b->Z, b->chain, b->xs, b->Y32, b->Z32, b->chain32, b->xs32};
  b_time_tables_kernel<<<(unsigned)((b->tt_total + 127) / 128), 128, 0, b->stream>>>(
      b->d_probs, b->d_tt_prefix, b->P, b->tt_total, b->d_terms, b->d_cols, D);
  // per-axis factors of forcing and initial data
  const size_t smem = sizeof(double) * (size_t)(b->nmax + 2 * (b->nmax + 1));
  b_axis_factor_kernel<<<b->n_factor_jobs, 256, smem, b->stream>>>(b->d_probs, b->d_factor_jobs, b->d_terms,
                                                                   b->gauss, b->muM, b->axisF, b->axisF32,
                                                                   b->axisU0);
  // per-mode column weights, the learned correction's bands first
  BLearn L{};
  if (b->mlp) {
    PE_TRY(batch_learned_tables(b, b->stream));
    L.ratio = b->ratio;
    L.Kt = b->Kt;
    L.axisF64 = b->axisF;
    L.NB = kBatchLearnedBands;
  }
  if (b->precision == PE_MIXED)
    b_column_weights_kernel<float><<<b->n_mode_items, 256, 0, b->stream>>>(
        b->d_probs, b->d_mode_items, b->n_mode_items, b->d_first, b->d_cols, b->axisF32, b->coefF32, b->coefG32, b->Z32,
        b->chain32, b->xs32, b->V32, b->G32, L);
  else
    b_column_weights_kernel<double><<<b->n_mode_items, 256, 0, b->stream>>>(
        b->d_probs, b->d_mode_items, b->n_mode_items, b->d_first, b->d_cols, b->axisF, b->coefF, b->coefG, b->Z,
        b->chain, b->xs, b->V, b->G, L);
  b_u0_kernel<<<grid_items, 256, 0, b->stream>>>(b->d_probs, b->d_mode_items, b->n_mode_items, b->d_terms, b->axisU0,
                                                 b->U);
  b->launches += 4;
  PE_CUDA_TRY(cudaGetLastError());
  return PE_OK;
}

pe_status batch_enqueue_iteration(pe_batch* b, cudaStream_t st, double tol, bool first) {
  PE_CUDA_TRY(cudaMemsetAsync(b->counter, 0, sizeof(int), st));
  PE_CUDA_TRY(cudaMemsetAsync(b->n_active, 0, sizeof(int), st));
  PE_TRY(launch_walk(b, st, b->tune_threads, b->tune_ctas, first));
  b_reduce_kernel<<<b->P, 256, 0, st>>>(b->d_probs, b->P, b->tune_threads, b->partials, b->active, b->kcount,
                                        b->resid, tol, b->n_active, b->nonfinite);
  PE_CUDA_TRY(cudaMemcpyAsync(b->h_flags, b->n_active, 2 * sizeof(int), cudaMemcpyDeviceToHost, st));
  PE_CUDA_TRY(cudaGetLastError());
  return PE_OK;
}

pe_status batch_time_walk(pe_batch* b, int threads, int ctas, float* ms) {
  PE_CUDA_TRY(cudaMemsetAsync(b->counter, 0, sizeof(int), b->stream));
  PE_CUDA_TRY(cudaEventRecord(b->ev[0], b->stream));
  PE_TRY(launch_walk(b, b->stream, threads, ctas, false));
  PE_CUDA_TRY(cudaEventRecord(b->ev[1], b->stream));
  PE_CUDA_TRY(cudaEventSynchronize(b->ev[1]));
  PE_CUDA_TRY(cudaEventElapsedTime(ms, b->ev[0], b->ev[1]));
  b->launches += 1;
  return PE_OK;
}
