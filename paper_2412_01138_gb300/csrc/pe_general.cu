// General forcing path: sources with spatial factors that move with t (the oscillating hat of
// Example 4 of Sec. 5).
//
// The modal factors of a moving term cannot be formed once.  At every stage time t of Eq. (1-7) this path
// (i) evaluates the consistent 1D loads of the term's moving axes by element Gauss-Legendre
// quadrature (a product of per-axis factors integrates as the product of 1D element integrals) and
// (ii) applies the DST-I along that axis: the tensor transform of a product is the product of the
// 1D transforms, so the d-D load is never assembled and no d-D transform is taken; what is
// transformed is one pencil per stage, term and moving axis.  The fine recurrence then reads, per mode and
// stage, one value of each moving axis; the term's other axes and Lambda_M^{-1} are a factor
// of the mode.  Terms that do not move, whatever path the problem asked for, are projected once and
// summed as columns (pe_contract.cuh).  The sweeps add both parts (pe_sweep.cu).
// In the mixed form the fine sweep's loads and transforms run in float32 (the coarse forcing,
// computed once per problem, stays float64).
//
// Bound: float64 FMA rate, q + 1 per mode, substep and moving term (float32 rate in the mixed form); the
// stage tables (stages x n_a) stay in L2.  255 x 127 nodes, 8 x 32 substeps, q = 4, one hat and four
// fixed terms, per sweep: 39 us loads, 15 us transforms, 82 us recurrence (66 us by the float64 rate), against 3.2 ms
// with the load of every term assembled and transformed on the whole grid at each of the 1024 stage times.
//
// Slices are processed in chunks so that the stage tables of a chunk fit a fixed device budget.
#include <math.h>

#include <algorithm>

#include "pe_forcing_common.cuh"
#include "pe_internal.h"

namespace {

// stage times of a chunk: fine (n0 + s / (M q), m, i) or coarse (s / p, i)
struct StageGen {
  int coarse;   // 0 fine, 1 coarse
  int n0;       // first slice of the chunk (fine)
  int M, s;     // substeps and nodes per step
  double t0, dT, dt;
  double c[PE_MAX_S];
};

__device__ inline double stage_time(const StageGen& G, int idx) {
  if (G.coarse) {
    const int n = idx / G.s, i = idx % G.s;
    const double Tn = G.t0 + (double)n * G.dT;
    return Tn + G.c[i] * G.dT;
  }
  const int per = G.M * G.s;
  const int n = G.n0 + idx / per, rem = idx % per;
  const int m = rem / G.s, i = rem % G.s;
  const double Tn = G.t0 + (double)n * G.dT;
  const double tl = Tn + (double)m * G.dt;
  return tl + G.c[i] * G.dt;
}

// The moving (term, axis) pairs, ordered by axis: pair e holds the rows [stages][n_a] of its loads
// (and of their transforms) at off[e] * stages.  The first moving axis of a term carries
// amp_r time_r(t).
constexpr int kMaxPairs = PE_MAX_TERMS * PE_MAX_D;
struct MovingPairs {
  int n;
  int64_t total;  // sum of n_a over the pairs
  signed char term[kMaxPairs], axis[kMaxPairs], lead[kMaxPairs];
  int off[kMaxPairs];
};

MovingPairs find_pairs(const pe_ctx* c) {
  MovingPairs P{};
  bool led[PE_MAX_TERMS] = {};
  for (int a = 0; a < c->g.d; ++a)
    for (int r = 0; r < c->Rm; ++r) {
      if (c->mterms[r].skind[a] != PE_S_MOVING_HAT) continue;
      const int e = P.n++;
      P.term[e] = (signed char)r;
      P.axis[e] = (signed char)a;
      P.lead[e] = led[r] ? 0 : 1;
      led[r] = true;
      P.off[e] = (int)P.total;
      P.total += c->g.n[a];
    }
  return P;
}

// L[off[e] * stages + st * n_a + k] = int g_{r,a}(x, t_st) phi_{k+1}(x) dx (grid: node blocks of 128, pairs,
// stages), times amp_r time_r(t_st) on the term's lead axis.  Element m = [lo + m h, lo + (m+1) h] contributes
// h int g s ds to its right node and h int g (1-s) ds to its left node; each element's
// quadrature is evaluated once (into shared memory) and node k sums the rising part of element
// k and the falling part of element k+1.  TL = float evaluates the factors in float32 (mixed
// precision).  Per block the factor's parameters, the moving hat's centre at t_st and the
// quadrature weights w_q s_q, w_q (1 - s_q) are converted once into shared memory; per element
// only the node positions are formed in float64 (lo + m h + s_q h).

// The moving hat at x from parameters already in TL (its centre in p[0]).
template <typename TL>
__device__ __forceinline__ TL eval_hat(const TL* p, TL x) {
  return fmax(TL(1) - fabs(x - p[0]) / p[1], TL(0));
}

template <typename TL>
__global__ void __launch_bounds__(128) gen_loads_kernel(TermsDev T, MovingPairs P, Geom g, double lo0, double lo1,
                                                        double lo2, double h0, double h1, double h2, Gauss Q,
                                                        StageGen SG, int64_t stages, TL* __restrict__ L) {
  pdl_wait();
  __shared__ TL rise[129], fall[129];
  __shared__ TL sp[2], samp, sws[8], sw1s[8];
  __shared__ double ssh[8];
  const int st = blockIdx.z, e = blockIdx.y;
  const int r = P.term[e], a = P.axis[e];
  const int n = g.n[a];
  const int k0 = blockIdx.x * 128;
  if (k0 >= n) return;  // uniform over the block
  const double lo = a == 0 ? lo0 : (a == 1 ? lo1 : lo2);
  const double h = a == 0 ? h0 : (a == 1 ? h1 : h2);
  const int nq = Q.npts;
  if (threadIdx.x == 0) {
    const pe_term& tm = T.t[r];
    const double t = stage_time(SG, st);
    sp[0] = (TL)(tm.sp[a][0] + tm.sp[a][1] * sinpi(2.0 * tm.sp[a][2] * t));
    sp[1] = (TL)tm.sp[a][3];
    samp = P.lead[e] ? (TL)(tm.amp * eval_time(tm, t)) : TL(1);
  } else if (threadIdx.x <= 8) {
    const int q = threadIdx.x - 1;
    if (q < nq) {
      sws[q] = (TL)(Q.w[q] * Q.s[q]);
      sw1s[q] = (TL)(Q.w[q] * (1.0 - Q.s[q]));
      ssh[q] = Q.s[q] * h;
    }
  }
  __syncthreads();
  // elements k0 .. k0 + 128 (the last one only for its falling part); on a periodic axis
  // node k's elements are k-1 and k, i.e. k0-1 .. k0+127 taken modulo n
  const bool per = g.per[a] != 0;
  for (int i = threadIdx.x; i <= 128; i += blockDim.x) {
    int m = per ? k0 - 1 + i : k0 + i;
    if (per) m = (m + n) % n;
    TL up = TL(0), dn = TL(0);
    if (per || m <= n) {
      const double xm = fma((double)m, h, lo);
      for (int qi = 0; qi < nq; ++qi) {
        const TL gv = eval_hat<TL>(sp, (TL)(xm + ssh[qi]));
        up += sws[qi] * gv;
        dn += sw1s[qi] * gv;
      }
    }
    rise[i] = up;
    fall[i] = dn;
  }
  __syncthreads();
  const int k = k0 + threadIdx.x;
  if (k < n)
    L[(int64_t)P.off[e] * stages + (int64_t)st * n + k] =
        samp * ((TL)h * rise[threadIdx.x] + (TL)h * fall[threadIdx.x + 1]);
}

// The factor of mode J that a moving term r does not change with t: its static axes' modal factors and
// 1 / mu^M of its moving axes.
__device__ __forceinline__ double static_factor(const Geom& g, const int* j, int r, int Rm, const pe_term& t,
                                                const double* __restrict__ axisM, const double* __restrict__ muM) {
  double C = 1.0;
#pragma unroll
  for (int a = 0; a < PE_MAX_D; ++a)
    if (a < g.d) {
      if (t.skind[a] == PE_S_MOVING_HAT) C /= muM[g.off[a] + j[a]];
      else C *= axisM[(int64_t)Rm * g.off[a] + (int64_t)r * g.n[a] + j[a]];
    }
  return C;
}

// The moving terms' part of F^M(0) (rows n0 .. of slices, blockIdx.y), added to Fbar:
// sum_r C_r(J) sum_m E^{M-1-m} sum_i dt b_i prod_{a moving} X_{r,a}[st][j_a].  T = float: the recurrence in
// float32 with E as hi + lo.  Q: the number of stages where it is at most 4 (the loads of several
// substeps are then in flight without predicates), else 0.
template <typename T, int Q>
__global__ void __launch_bounds__(256) gen_fine_kernel(TermsDev D, MovingPairs P, Geom g, int n0, int M, int q,
                                                       int64_t stages, const double* __restrict__ axisM,
                                                       const double* __restrict__ muM, const T* __restrict__ coef,
                                                       const T* __restrict__ X, double* __restrict__ Fbar, int add) {
  pdl_wait();
  constexpr bool F64 = sizeof(T) == 8;
  const int64_t nd = g.ndof;
  const int64_t J = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (J >= nd) return;
  int j[PE_MAX_D];
  unflatten(g, J, j);
  const T E = coef[J];
  T El = T(0);
  if constexpr (!F64) El = coef[nd + J];
  constexpr int QM = Q ? Q : PE_MAX_S;
  if (Q) q = Q;
  T b[QM];
#pragma unroll
  for (int i = 0; i < QM; ++i)
    if (i < q) b[i] = coef[(int64_t)((F64 ? 1 : 2) + i) * nd + J];
  const int64_t s0 = (int64_t)blockIdx.y * M * q;
  double sum = 0.0;
  for (int r = 0; r < D.n; ++r) {
    // the term's moving axes: rows of the tables, one value per stage each
    const T* x[PE_MAX_D];
    int stride[PE_MAX_D], nx = 0;
    for (int e = 0; e < P.n; ++e)
      if (P.term[e] == r) {
        const int a = P.axis[e];
        const int ja = a == 0 ? j[0] : (a == 1 ? j[1] : j[2]);
        const T* row = X + (int64_t)P.off[e] * stages + s0 * g.n[a] + ja;
        if (nx == 0) { x[0] = row; stride[0] = g.n[a]; }
        else if (nx == 1) { x[1] = row; stride[1] = g.n[a]; }
        else { x[2] = row; stride[2] = g.n[a]; }
        ++nx;
      }
    T c = T(0);
    if (nx == 1) {
      const T* x0 = x[0];
      const int s0r = stride[0];
#pragma unroll 4
      for (int m = 0; m < M; ++m) {
        T acc = T(0);
#pragma unroll
        for (int i = 0; i < QM; ++i)
          if (i < q) acc = fma(b[i], __ldg(x0 + (int64_t)i * s0r), acc);
        x0 += (int64_t)q * s0r;
        if constexpr (F64) c = fma(E, c, acc);
        else c = fmaf(E, c, fmaf(El, c, acc));
      }
    } else {
      for (int m = 0; m < M; ++m) {
        T acc = T(0);
#pragma unroll
        for (int i = 0; i < QM; ++i)
          if (i < q) {
            const int64_t st = m * q + i;
            T v = x[0][st * stride[0]] * x[1][st * stride[1]];
            if (nx == 3) v *= x[2][st * stride[2]];
            acc = fma(b[i], v, acc);
          }
        if constexpr (F64) c = fma(E, c, acc);
        else c = fmaf(E, c, fmaf(El, c, acc));
      }
    }
    sum = fma(static_factor(g, j, r, D.n, D.t[r], axisM, muM), (double)c, sum);
  }
  double* out = Fbar + (int64_t)(n0 + blockIdx.y) * nd + J;
  *out = add ? *out + sum : sum;
}

// The moving terms' part of the coarse forcing, added to gG: sum_r C_r sum_i dT b_i prod X_{r,a}[n p + i][j_a].
__global__ void __launch_bounds__(256) gen_coarse_kernel(TermsDev D, MovingPairs P, Geom g, int p, int64_t stages,
                                                         const double* __restrict__ axisM,
                                                         const double* __restrict__ muM,
                                                         const double* __restrict__ coefG,
                                                         const double* __restrict__ X, double* __restrict__ gG,
                                                         int add) {
  pdl_wait();
  const int64_t nd = g.ndof;
  const int64_t J = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int n = blockIdx.y;
  if (J >= nd) return;
  int j[PE_MAX_D];
  unflatten(g, J, j);
  double sum = 0.0;
  for (int r = 0; r < D.n; ++r) {
    double acc = 0.0;
    for (int i = 0; i < p; ++i) {
      double v = coefG[(int64_t)(1 + i) * nd + J];
      for (int e = 0; e < P.n; ++e)
        if (P.term[e] == r) {
          const int a = P.axis[e];
          const int ja = a == 0 ? j[0] : (a == 1 ? j[1] : j[2]);
          v *= X[(int64_t)P.off[e] * stages + ((int64_t)n * p + i) * g.n[a] + ja];
        }
      acc += v;
    }
    sum = fma(static_factor(g, j, r, D.n, D.t[r], axisM, muM), acc, sum);
  }
  double* out = gG + (int64_t)n * nd + J;
  *out = add ? *out + sum : sum;
}

StageGen make_gen(const pe_ctx* c, int coarse, int n0) {
  StageGen G{};
  G.coarse = coarse;
  G.n0 = n0;
  G.M = c->M;
  G.s = coarse ? c->p : c->q;
  G.t0 = c->t0;
  G.dT = c->dT;
  G.dt = c->dt;
  for (int i = 0; i < PE_MAX_S; ++i) G.c[i] = coarse ? c->cG[i] : c->cF[i];
  return G;
}

// slices per chunk: the chunk's two stage tables within 1 GiB, and at most 65535 stage times per
// chunk (grid dimension of the load kernel)
int slices_per_chunk(const pe_ctx* c, const MovingPairs& P) {
  const size_t per_slice = (size_t)c->M * c->q * (size_t)P.total * sizeof(double) * 2;
  int ns = (int)std::max<size_t>(1, ((size_t)1 << 30) / std::max<size_t>(per_slice, 1));
  ns = std::min(ns, std::max(1, 65535 / (c->M * c->q)));
  return std::min(ns, c->N);
}

// The moving pairs' loads of `stages` stage times and their transforms along their axes, in *X (element
// type T).  Pairs of one axis are consecutive: one transform per axis.
template <typename T>
pe_status stage_tables(pe_ctx* c, const MovingPairs& P, const StageGen& SG, int64_t stages, T** X) {
  const TermsDev TD = pack_terms(c->mterms, c->Rm);
  const Gauss Q = make_gauss(c->quad_pts);
  int nmax = 1;
  for (int a = 0; a < c->g.d; ++a) nmax = std::max(nmax, c->g.n[a]);
  T* L = reinterpret_cast<T*>(c->gen_L);
  *X = reinterpret_cast<T*>(c->gen_X);
  const dim3 grid((unsigned)((nmax + 127) / 128), (unsigned)P.n, (unsigned)stages);
  PE_CUDA_TRY(launch_pdl(gen_loads_kernel<T>, grid, dim3(128), 0, c->stream, TD, P, c->g, c->lo[0], c->lo[1], c->lo[2],
                         c->h[0], c->h[1], c->h[2], Q, SG, stages, L));
  c->launches += 1;
  for (int a = 0, e = 0; a < c->g.d; ++a) {
    int cnt = 0;
    while (e + cnt < P.n && P.axis[e + cnt] == a) ++cnt;
    if (cnt == 0) continue;
    const int64_t o = (int64_t)P.off[e] * stages;
    if constexpr (sizeof(T) == 8)
      PE_TRY(dst_axis_f64(c->S[a], L + o, *X + o, cnt * stages, c->g.n[a], 1, c->stream, c->g.per[a]));
    else
      PE_TRY(dst_axis_f32(c->S32[a], L + o, *X + o, cnt * stages, c->g.n[a], 1, c->stream, c->g.per[a]));
    c->launches += 1;
    e += cnt;
  }
  return PE_OK;
}

}  // namespace

// Buffers and static modal factors of the current problem's moving terms (c->mterms): made by
// pe_set_problem, after its own factors.
pe_status general_prepare(pe_ctx* c) {
  if (c->Rm == 0) return PE_OK;
  const MovingPairs P = find_pairs(c);
  const int64_t stages = std::max<int64_t>((int64_t)slices_per_chunk(c, P) * c->M * c->q, (int64_t)c->N * c->p);
  const size_t need = (size_t)stages * (size_t)P.total;
  if (need > c->gen_cap) {
    PE_CUDA_TRY(cudaStreamSynchronize(c->stream));
    if (c->gen_L) cudaFree(c->gen_L);
    if (c->gen_X) cudaFree(c->gen_X);
    c->gen_L = c->gen_X = nullptr;
    c->gen_cap = 0;
    if (cudaMalloc((void**)&c->gen_L, need * sizeof(double)) != cudaSuccess ||
        cudaMalloc((void**)&c->gen_X, need * sizeof(double)) != cudaSuccess) {
      cudaGetLastError();
      return pe_fail(PE_ENOMEM, "pe_set_problem: stage-table allocation failed");
    }
    c->gen_cap = need;
  }
  // (on a line every factor moves: none is static)
  return P.n == c->Rm * c->g.d ? PE_OK : launch_separable_factors(c, c->mterms, c->Rm, c->axisM, 1);
}

pe_status general_add_coarse(pe_ctx* c) {
  if (c->Rm == 0) return PE_OK;
  const MovingPairs P = find_pairs(c);
  const int64_t stages = (int64_t)c->N * c->p;
  double* X = nullptr;
  PE_TRY(stage_tables<double>(c, P, make_gen(c, 1, 0), stages, &X));
  PE_CUDA_TRY(launch_pdl(gen_coarse_kernel, dim3((unsigned)((c->g.ndof + 255) / 256), c->N), dim3(256), 0, c->stream,
                         pack_terms(c->mterms, c->Rm), P, c->g, c->p, stages, (const double*)c->axisM,
                         (const double*)c->muM_axis, (const double*)c->coefG, (const double*)X, c->gG,
                         c->only_moving ? 0 : 1));
  c->launches += 1;
  return PE_OK;
}

template <typename T>
static pe_status add_fine(pe_ctx* c, const T* coef) {
  const MovingPairs P = find_pairs(c);
  const TermsDev TD = pack_terms(c->mterms, c->Rm);
  const int chunk = slices_per_chunk(c, P);
  auto kern = gen_fine_kernel<T, 0>;
  if (c->q == 1) kern = gen_fine_kernel<T, 1>;
  else if (c->q == 2) kern = gen_fine_kernel<T, 2>;
  else if (c->q == 3) kern = gen_fine_kernel<T, 3>;
  else if (c->q == 4) kern = gen_fine_kernel<T, 4>;
  for (int n0 = 0; n0 < c->N; n0 += chunk) {
    const int ns = std::min(chunk, c->N - n0);
    const int64_t stages = (int64_t)ns * c->M * c->q;
    T* X = nullptr;
    PE_TRY(stage_tables<T>(c, P, make_gen(c, 0, n0), stages, &X));
    PE_CUDA_TRY(launch_pdl(kern, dim3((unsigned)((c->g.ndof + 255) / 256), ns), dim3(256), 0, c->stream, TD, P, c->g, n0,
                           c->M, c->q, stages, (const double*)c->axisM, (const double*)c->muM_axis, coef, (const T*)X,
                           c->Fbar, c->only_moving ? 0 : 1));
    c->launches += 1;
  }
  return PE_OK;
}

pe_status general_add_fine(pe_ctx* c, int precision) {
  if (c->Rm == 0) return PE_OK;
  return precision == PE_MIXED ? add_fine<float>(c, c->coefF32) : add_fine<double>(c, c->coefF);
}
