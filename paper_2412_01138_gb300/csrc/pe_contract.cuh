// The substep sum of a separable source, contracted over a whole slice.
//
// Every time factor of a separable source is shift invariant: A(t + s) = sum_k Y_k(t) Z_k(s), one
// column k for an exponential, two for a sinusoid (sin(w(t+s)+phi) = sin(wt+phi) cos(ws) +
// cos(wt+phi) sin(ws)).  The q stages of one substep therefore add up to sum_k Y_k(t_m) W_k with a
// per-mode weight W_k = P sum_i dt b_i Z_k(c_i dt), and the M substeps of a slice, each damped by
// the substeps after it, add up the same way:
//   F^M(0) = sum_m E^{M-1-m} sum_k Y_k(T_n + m dt) W_k = sum_k Y_k(T_n) V_k,
// where for the two columns of a sinusoid, as one complex number (sin column real),
//   V_0 + i V_1 = (W_0 + i W_1) S_M,   S_L = sum_{m<L} E^{L-1-m} z^m,  z = e^{i w dt},
// and for an exponential e^{at} the same with z = e^{a dt} real.  So the fine propagator of Eq.
// (1-7), all M substeps and q stages of it, costs K multiply-adds per mode and slice instead of
// M (K + 1), once the weights V are known; they are the same for every slice and iteration.
//
// S_M by doubling over the bits of M (S_{2L} = (E^L + z^L) S_L, S_{L+1} = E S_L + z^L): log2 M
// steps whose terms are all at most M in size (E <= 1, |z| <= 1), no division and no
// cancellation beyond that of the sum itself.  A growing exponential (a > 0) takes its value at
// the slice's end as its column and counts back from it, x = E e^{-a dt} in place of E and z = 1, so
// that no factor exceeds 1 there either.
//
// The powers z^L of the chain depend on the term alone and are tabulated: step s holds D = z^{L_s}
// (doubling) and, where the next bit of M is set, A = z^{2 L_s} (the step after it).
#pragma once
#include "pe_internal.h"

// Doubling steps of the chain for M substeps.
__host__ __device__ inline int chain_steps(int M) {
  int s = 0;
  while (M > 1) {
    M >>= 1;
    ++s;
  }
  return s;
}

// Step s of M (0 = the first doubling): the length before it, and whether one more is added.
__host__ __device__ inline int chain_length(int M, int steps, int s) { return M >> (steps - s); }
__host__ __device__ inline bool chain_adds(int M, int steps, int s) { return (M >> (steps - s - 1)) & 1; }

// S_M for x (= E, or E e^{-a dt}), float64.  tab: the term's entries, `stride` doubles per step.  The tables hold Re D, Im D,
// Re A, Im A of step s and term r at [(s * R + r) * 4 ..]; the float form (hi, lo) pairs of the same.
__device__ __forceinline__ void chain_sum(double x, int M, int steps, const double* __restrict__ tab, int stride,
                                          double& Sr, double& Si) {
  double xL = x;
  Sr = 1.0;
  Si = 0.0;
  for (int s = 0; s < steps; ++s) {
    const double* t = tab + (int64_t)s * stride;
    const double a = xL + t[0], c = t[1];
    const double r = fma(a, Sr, -(c * Si));
    Si = fma(a, Si, c * Sr);
    Sr = r;
    xL *= xL;
    if (chain_adds(M, steps, s)) {
      Sr = fma(x, Sr, t[2]);
      Si = fma(x, Si, t[3]);
      xL *= x;
    }
  }
}

// Pairs of float32 (an unevaluated sum hi + lo, about 48 bits): the mixed form runs the chain in
// them, so that the doubling does not add to the rounding of the float32 weights it ends in, and
// the float64 pipe (two lanes per SM) stays out of it.
struct F2 {
  float h, l;
};
__device__ __forceinline__ F2 f2_quick(float h, float l) {  // |h| >= |l| or h = 0
  const float s = h + l;
  return F2{s, l - (s - h)};
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
  const float s = a.h + b.h, t = s - a.h;
  const float e = (a.h - (s - t)) + (b.h - t);
  return f2_quick(s, e + (a.l + b.l));
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
  const float p = a.h * b.h;
  const float e = fmaf(a.h, b.h, -p);
  return f2_quick(p, fmaf(a.h, b.l, fmaf(a.l, b.h, e)));
}
__device__ __forceinline__ F2 f2_neg(F2 a) { return F2{-a.h, -a.l}; }

__device__ __forceinline__ void chain_sum(F2 x, int M, int steps, const float* __restrict__ tab, int stride, F2& Sr,
                                          F2& Si) {
  F2 xL = x;
  Sr = F2{1.f, 0.f};
  Si = F2{0.f, 0.f};
  for (int s = 0; s < steps; ++s) {
    const float* t = tab + (int64_t)s * stride;
    const F2 a = f2_add(xL, F2{t[0], t[1]}), c = F2{t[2], t[3]};
    const F2 r = f2_add(f2_mul(a, Sr), f2_neg(f2_mul(c, Si)));
    Si = f2_add(f2_mul(a, Si), f2_mul(c, Sr));
    Sr = r;
    xL = f2_mul(xL, xL);
    if (chain_adds(M, steps, s)) {
      Sr = f2_add(f2_mul(x, Sr), F2{t[4], t[5]});
      Si = f2_add(f2_mul(x, Si), F2{t[6], t[7]});
      xL = f2_mul(xL, x);
    }
  }
}

// Response tables.  The weight of a term's columns is P times a function of lam alone,
//   H_r(lam) = (sum_i dt b_i(-lam dt) Z(c_i dt)) S_M(lam)   (complex for a sinusoid),
// smooth over scales of lam itself: on an interval of relative width w the interpolation at n Chebyshev
// nodes is off by 2 (w/4)^n at most (in units of int e^{-lam s} ds times the term's size; a term that decays over a
// slice has a far smaller weight than that, and is left to the direct evaluation: response_exact).  Where a grid has many
// more modes than an interval table has nodes, H is tabulated per problem and a mode evaluates a
// polynomial instead of the q stages and the chain.  Intervals split each octave of lam evenly into 2^bits
// (index and local coordinate are bits of lam): float 16 per octave and 5 nodes (2e-9 of the scale, a
// thirtieth of a float's rounding), double 32 and 8 (3e-17).  One more interval, the last, is lam = 0.
template <typename T>
struct Resp;
template <>
struct Resp<float> {
  static constexpr int bits = 4, nodes = 5, comp = 6;  // c0 high, c0 low, c1 .. c4
};
template <>
struct Resp<double> {
  static constexpr int bits = 5, nodes = 8, comp = 8;
};
// interval index of lam >= 0 (base: the first interval's leading bits, T intervals and the zero one) and the local
// coordinate in [-1, 1)
__device__ __forceinline__ int resp_locate(double lam, int base, int T, float& x) {
  constexpr int B = Resp<float>::bits;
  const int hi = __double2hiint(lam), idx = (hi >> (20 - B)) - base;
  if (idx < 0) {  // lam = 0
    x = 0.f;
    return T;
  }
  const unsigned m = ((unsigned)(hi & ((1 << (20 - B)) - 1)) << (B + 4)) | ((unsigned)__double2loint(lam) >> (28 - B));
  x = fmaf((float)m, 0x1p-23f, -1.f);  // 24 bits below the interval's own: exact
  return min(idx, T - 1);
}
__device__ __forceinline__ int resp_locate(double lam, int base, int T, double& x) {
  constexpr int B = Resp<double>::bits;
  const int hi = __double2hiint(lam), idx = (hi >> (20 - B)) - base;
  if (idx < 0) {
    x = 0.0;
    return T;
  }
  // mantissa in [1, 2) less the interval's middle, times 2^(B+1): exact
  const double m = __hiloint2double((hi & 0xFFFFF) | 0x3FF00000, __double2loint(lam));
  const double mid = __hiloint2double((((hi & 0xFFFFF) >> (20 - B)) << (20 - B)) | (1 << (19 - B)) | 0x3FF00000, 0);
  x = (m - mid) * (double)(1 << (B + 1));
  return min(idx, T - 1);
}

// Time-table entries of one term (t: the term; dt, dT the fine and coarse steps).
// column value of slice n, kind 0 or 1 (the cosine partner of a sinusoid)
__device__ __forceinline__ bool grows(const pe_term& t) { return t.tkind != PE_T_SIN && t.tp[0] > 0.0; }

// Y_k of the slice [Ta, Tb]: the value at its start, of a growing exponential at its end
__device__ __forceinline__ double column_value(const pe_term& t, int kind, double Ta, double Tb) {
  if (t.tkind == PE_T_SIN) {
    const double th = t.tp[0] * Ta + t.tp[1];
    return t.amp * (kind == 1 ? cos(th) : sin(th));
  }
  return t.amp * exp(t.tp[0] * (grows(t) ? Tb : Ta));
}

// Z_k(c tau): the shift to node c of a step tau from the step's start (growing: from its end)
__device__ __forceinline__ double column_shift(const pe_term& t, int kind, double c, double tau) {
  if (t.tkind == PE_T_SIN) {
    const double s = t.tp[0] * (c * tau);
    return kind == 1 ? sin(s) : cos(s);
  }
  return exp(t.tp[0] * (grows(t) ? (c - 1.0) * tau : c * tau));
}

// z^L (re, im)
__device__ __forceinline__ void chain_power(const pe_term& t, int L, double dt, double& re, double& im) {
  im = 0.0;
  if (t.tkind == PE_T_SIN) sincos(t.tp[0] * ((double)L * dt), &im, &re);
  else re = grows(t) ? 1.0 : exp(t.tp[0] * ((double)L * dt));
}

// what x is of E: 1, or e^{-a dt} for a growing exponential
__device__ __forceinline__ double chain_scale(const pe_term& t, double dt) {
  return grows(t) ? exp(-t.tp[0] * dt) : 1.0;
}

// sum_k y_k w_k over a slice's staged columns, a row of KB high parts and one of KB low parts:
// rounding Y_k(T_n) to one float would be an error of the whole slice, which M separately rounded
// substeps average out
template <int KB>
__device__ __forceinline__ float column_dot(const float* y, const float (&w)[KB]) {
  float hi = 0.f, lo = 0.f;
#pragma unroll
  for (int k = 0; k < KB; k += 4) {
    const float4 v = *reinterpret_cast<const float4*>(y + k);
    const float4 l = *reinterpret_cast<const float4*>(y + KB + k);
    hi = fmaf(v.x, w[k], hi);
    lo = fmaf(l.x, w[k], lo);
    hi = fmaf(v.y, w[k + 1], hi);
    lo = fmaf(l.y, w[k + 1], lo);
    hi = fmaf(v.z, w[k + 2], hi);
    lo = fmaf(l.z, w[k + 2], lo);
    hi = fmaf(v.w, w[k + 3], hi);
    lo = fmaf(l.w, w[k + 3], lo);
  }
  return hi + lo;
}

template <typename T>
__device__ inline T block_sum(T v, T* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  T out = T(0);
  if (threadIdx.x < 32) {
    T x = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : T(0);
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    out = x;
  }
  __syncthreads();
  return out;
}
