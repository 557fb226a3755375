// The load P_h f in mode space for separable sources, and the projection of u0.
//
// P_h is the L2 projection (Sec. 2.1, Eq. (3-11)); its modal coefficients are
// ghat = Lambda_M^{-1} V^T F with F_k = (f, phi_k) the consistent load.  For a
// separable term amp * time(t) * prod_a g_a(x_a) the load is the outer product
// of 1D loads F_a[k] = int g_a phi_k, so
//   ghat_J(t) = sum_r amp_r time_r(t) prod_a (S_a F_{r,a})_{j_a} / mu^M_a(j_a).
// 1D loads use a Gauss-Legendre rule with quad_pts points on each element.
// The per-axis modal factors, the time columns of every slice and the per-mode column weights of
// the fine propagator and the coarse step (pe_contract.cuh) are tabulated here; the sweeps
// multiply columns and weights together on the fly.
#include <math.h>
#include <string.h>

#include <algorithm>

#include "pe_contract.cuh"
#include "pe_forcing_common.cuh"
#include "pe_internal.h"
#include "pe_learned.h"
#include "pe_phi.cuh"

namespace {

// Time tables of one problem, one thread per entry (pe_contract.cuh): the columns Y_k of every
// slice, the shifts of the fine and coarse nodes, and per term the chain's powers and scale.
// Float copies (the mixed form): Y as a row of high and one of low parts, KC = roundup(K, 4) long
// with zeros past K, shifts rounded, chain powers and scales as (hi, lo) pairs.
__global__ void time_tables_kernel(TermsDev T, StageCols C, ColumnTables D, int N, int M, int q, int p, double t0,
                                   double dT, double dt, Nodes cF, Nodes cG) {
  pdl_wait();
  const int R = T.n, K = C.K, steps = chain_steps(M);
  const int ny = N * K, nf = q * K, ng = p * K;
  int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < ny) {
    const int n = e / K, k = e - n * K;
    const double v = column_value(T.t[C.term[k]], C.kind[k], t0 + (double)n * dT, t0 + (double)(n + 1) * dT);
    D.Y[e] = v;
    if (D.Y32) {
      const int KC = (K + 3) & ~3;
      float* row = D.Y32 + (int64_t)n * 2 * KC;
      row[k] = (float)v;
      row[KC + k] = (float)(v - (double)(float)v);
      if (k == K - 1)
        for (int z = K; z < KC; ++z) row[z] = row[KC + z] = 0.f;
    }
    return;
  }
  e -= ny;
  if (e < nf + ng) {
    const bool fine = e < nf;
    const int l = fine ? e : e - nf, i = l / K, k = l - i * K;
    const double v = column_shift(T.t[C.term[k]], C.kind[k], fine ? cF.c[i] : cG.c[i], fine ? dt : dT);
    (fine ? D.ZF : D.ZG)[l] = v;
    if (D.Y32) (fine ? D.ZF32 : D.ZG32)[l] = (float)v;
    return;
  }
  e -= nf + ng;
  if (e >= R * (steps + 1)) return;
  const int s = e / R - 1, r = e - (s + 1) * R;
  if (s < 0) {
    const double v = chain_scale(T.t[r], dt);
    D.xs[r] = v;
    if (D.Y32) {
      D.xs32[2 * r] = (float)v;
      D.xs32[2 * r + 1] = (float)(v - (double)(float)v);
    }
    return;
  }
  double v[4];
  const int L = chain_length(M, steps, s);
  chain_power(T.t[r], L, dt, v[0], v[1]);
  chain_power(T.t[r], 2 * L, dt, v[2], v[3]);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    D.chain[(s * R + r) * 4 + i] = v[i];
    if (D.Y32) {
      D.chain32[(s * R + r) * 8 + 2 * i] = (float)v[i];
      D.chain32[(s * R + r) * 8 + 2 * i + 1] = (float)(v[i] - (double)(float)v[i]);
    }
  }
}

// Per-mode column weights: V[k * ndof + J] of the fine propagator's slice sum and G[k * ndof + J]
// of the coarse step (sum_i dT b^G_i Z_k(c_i dT), plus the learned correction's P K^ on the
// columns of a sinusoid), P_{r,J} = prod_a axisF; V or G may be null.  A thread takes TPT
// consecutive terms of one mode.  T = float (mixed form): float32 weights from float32 factors, the chain in float pairs.
// coef: E (float: hi and lo rows), then the q rows dt b_i; coefG: the p rows dT b^G_i.
template <typename T>
__global__ void __launch_bounds__(256) column_weights_kernel(Geom g, StageCols C, ColumnTables D, int R, int M, int q,
                                                             int p, int tpt, const T* __restrict__ axisF,
                                                             const T* __restrict__ coef, const T* __restrict__ coefG,
                                                             T* __restrict__ V, T* __restrict__ G, LearnedTerms L,
                                                             const double* __restrict__ axisF64,
                                                             const double* __restrict__ lam) {
  pdl_wait();
  constexpr bool F64 = sizeof(T) == 8;
  const int64_t J = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (J >= g.ndof) return;
  const int64_t nd = g.ndof;
  const int K = C.K, steps = chain_steps(M);
  const T* ZF;
  const T* ZG;
  if constexpr (F64) {
    ZF = D.ZF;
    ZG = D.ZG;
  } else {
    ZF = D.ZF32;
    ZG = D.ZG32;
  }
  int j[PE_MAX_D];
  unflatten(g, J, j);
  T b[PE_MAX_S], bg[PE_MAX_S];
  constexpr int kERows = F64 ? 1 : 2;
#pragma unroll
  for (int i = 0; i < PE_MAX_S; ++i) {
    b[i] = i < q ? coef[(int64_t)(kERows + i) * nd + J] : T(0);
    bg[i] = G && i < p ? coefG[(int64_t)i * nd + J] : T(0);
  }
  const T Eh = coef[J];
  T El = T(0);
  if constexpr (!F64) El = coef[nd + J];
  int band = 0;
  double bf = 0.0;
  if (L.Ktab) {
    double pos = (log(lam[J] * L.dT) - L.loglo) / L.logstep;
    pos = fmin(fmax(pos, 0.0), (double)(L.NB - 1) - 1e-9);
    band = (int)pos;
    bf = pos - (double)band;
  }
  const int r1 = min(R, (int)(blockIdx.y + 1) * tpt);
  for (int r = blockIdx.y * tpt; r < r1; ++r) {
    const int k = C.first[r];
    const bool two = k + 1 < K && C.term[k + 1] == r;
    T P = axisF[(int64_t)R * g.off[0] + (int64_t)r * g.n[0] + j[0]];
#pragma unroll
    for (int a = 1; a < PE_MAX_D; ++a) if (a < g.d) P *= axisF[(int64_t)R * g.off[a] + (int64_t)r * g.n[a] + j[a]];
    T br = T(0), bi = T(0), gr = T(0), gi = T(0);
#pragma unroll
    for (int i = 0; i < PE_MAX_S; ++i)
      if (i < q) {
        br = fma(b[i], ZF[i * K + k], br);
        if (two) bi = fma(b[i], ZF[i * K + k + 1], bi);
      }
    if (G) {
#pragma unroll
      for (int i = 0; i < PE_MAX_S; ++i)
        if (i < p) {
          gr = fma(bg[i], ZG[i * K + k], gr);
          if (two) gi = fma(bg[i], ZG[i * K + k + 1], gi);
        }
      gr *= P;
      gi *= P;
      if (L.Ktab && two) {
        double Pd = axisF64[(int64_t)R * g.off[0] + (int64_t)r * g.n[0] + j[0]];
#pragma unroll
        for (int a = 1; a < PE_MAX_D; ++a) if (a < g.d)
          Pd *= axisF64[(int64_t)R * g.off[a] + (int64_t)r * g.n[a] + j[a]];
        const double* k0 = L.Ktab + 2 * ((int64_t)r * L.NB + band);
        gr += (T)(Pd * ((1.0 - bf) * k0[0] + bf * k0[2]));
        gi += (T)(Pd * ((1.0 - bf) * k0[1] + bf * k0[3]));
      }
      G[(int64_t)k * nd + J] = gr;
      if (two) G[(int64_t)(k + 1) * nd + J] = gi;
    }
    if (!V) continue;
    T v0, v1;
    if constexpr (F64) {
      double Sr, Si;
      chain_sum(Eh * D.xs[r], M, steps, D.chain + 4 * r, 4 * R, Sr, Si);
      v0 = P * fma(br, Sr, -(bi * Si));
      v1 = P * fma(br, Si, bi * Sr);
    } else {
      F2 Sr, Si;
      chain_sum(f2_mul(F2{Eh, El}, F2{D.xs32[2 * r], D.xs32[2 * r + 1]}), M, steps, D.chain32 + 8 * r, 8 * R, Sr, Si);
      const F2 B{br, 0.f}, C2{bi, 0.f};
      const F2 re = f2_add(f2_mul(B, Sr), f2_neg(f2_mul(C2, Si))), im = f2_add(f2_mul(B, Si), f2_mul(C2, Sr));
      v0 = fmaf(P, re.h, P * re.l);
      v1 = fmaf(P, im.h, P * im.l);
    }
    V[(int64_t)k * nd + J] = v0;
    if (two) V[(int64_t)(k + 1) * nd + J] = v1;
  }
}

// The same weights from the response table (pe_contract.cuh): per mode and term a polynomial of the
// mode's lam, whose interval and coordinate are found once.  Memory-bound (the weights written), where the direct
// evaluation is bound by its chain (60 float64 or 700 float32 operations per mode and sinusoid).  255^2 modes, 9 terms: 9.5 us after an 8.5 us table
// (beside the loads) against 24.7 us in float32, 31 after 13 against 91 us in float64; 127^3, 17 terms, float32: 208
// against 821 us.
template <typename T>
__global__ void __launch_bounds__(256) response_weights_kernel(Geom g, StageCols C, ColumnTables D, int R, int p, int tpt,
                                                               int base, int T_, const T* __restrict__ resp,
                                                               const T* __restrict__ axisF, const T* __restrict__ coefG,
                                                               T* __restrict__ V, T* __restrict__ G,
                                                               const double* __restrict__ lam) {
  pdl_wait();
  constexpr int CO = Resp<T>::comp;
  const int64_t J = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (J >= g.ndof) return;
  const int64_t nd = g.ndof;
  const int K = C.K;
  const T* ZG;
  if constexpr (sizeof(T) == 8) ZG = D.ZG;
  else ZG = D.ZG32;
  int j[PE_MAX_D];
  unflatten(g, J, j);
  T x;
  const int idx = resp_locate(lam[J], base, T_, x);
  T bg[PE_MAX_S];
#pragma unroll
  for (int i = 0; i < PE_MAX_S; ++i) bg[i] = G && i < p ? coefG[(int64_t)i * nd + J] : T(0);
  const int r1 = min(R, (int)(blockIdx.y + 1) * tpt);
  for (int r = blockIdx.y * tpt; r < r1; ++r) {
    const int k = C.first[r];
    const bool two = k + 1 < K && C.term[k + 1] == r;
    T P = axisF[(int64_t)R * g.off[0] + (int64_t)r * g.n[0] + j[0]];
#pragma unroll
    for (int a = 1; a < PE_MAX_D; ++a) if (a < g.d) P *= axisF[(int64_t)R * g.off[a] + (int64_t)r * g.n[a] + j[a]];
    const T* c = resp + ((int64_t)r * (T_ + 1) + idx) * 2 * CO;
    T v0, v1 = T(0);
    if constexpr (sizeof(T) == 4) {
      // 12 coefficients as three float4: c0 high and low, c1, c2 | c3, c4, then the second column's
      const float4 a0 = *reinterpret_cast<const float4*>(c), a1 = *reinterpret_cast<const float4*>(c + 4);
      v0 = a0.x + fmaf(x, fmaf(x, fmaf(x, fmaf(x, a1.y, a1.x), a0.w), a0.z), a0.y);
      if (two) {
        const float4 a2 = *reinterpret_cast<const float4*>(c + 8);
        v1 = a1.z + fmaf(x, fmaf(x, fmaf(x, fmaf(x, a2.w, a2.z), a2.y), a2.x), a1.w);
      }
    } else {
      v0 = c[CO - 1];
#pragma unroll
      for (int i = CO - 2; i >= 0; --i) v0 = fma(x, v0, c[i]);
      if (two) {
        v1 = c[2 * CO - 1];
#pragma unroll
        for (int i = CO - 2; i >= 0; --i) v1 = fma(x, v1, c[CO + i]);
      }
    }
    V[(int64_t)k * nd + J] = P * v0;
    if (two) V[(int64_t)(k + 1) * nd + J] = P * v1;
    if (G) {
      T gr = T(0), gi = T(0);
#pragma unroll
      for (int i = 0; i < PE_MAX_S; ++i)
        if (i < p) {
          gr = fma(bg[i], ZG[i * K + k], gr);
          if (two) gi = fma(bg[i], ZG[i * K + k + 1], gi);
        }
      G[(int64_t)k * nd + J] = P * gr;
      if (two) G[(int64_t)(k + 1) * nd + J] = P * gi;
    }
  }
}

// lam of node i of an interval (T: the zero interval)
__device__ __forceinline__ double resp_node(int base, int T, int t, int i, int bits, int nodes) {
  if (t == T) return 0.0;
  const double lo = __hiloint2double((base + t) << (20 - bits), 0), hi = __hiloint2double((base + t + 1) << (20 - bits), 0);
  return lo + (hi - lo) * (0.5 + 0.5 * cospi((2.0 * i + 1.0) / (2.0 * nodes)));
}

// E and dt b_1..q at every node: out[(t * nodes + i) * (1 + q)]
__global__ void response_nodes_kernel(int base, int T, int bits, int nodes, double dt, int q, Lag LF,
                                      double* __restrict__ out) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (T + 1) * nodes) return;
  const double lam = resp_node(base, T, e / nodes, e % nodes, bits, nodes);
  double b[PE_MAX_S];
  b_weights(-lam * dt, q, LF, b);
  out[(int64_t)e * (1 + q)] = exp(-lam * dt);
  for (int i = 0; i < q; ++i) out[(int64_t)e * (1 + q) + 1 + i] = dt * b[i];
}

// Polynomial coefficients of H_r on every interval (a CTA per interval; a thread per term and node, then per
// coefficient).  Minv: monomial coefficients from node values; applied to the differences from the middle
// node's value, which the interval makes small, so that its entries do not amplify their rounding.
struct RespInv {
  double m[8][8];
};
template <typename T>
__global__ void __launch_bounds__(256) response_kernel(StageCols C, ColumnTables D, int R, int M, int q, int T_,
                                                       RespInv I, const double* __restrict__ nodes,
                                                       T* __restrict__ resp) {
  pdl_wait();
  constexpr int NN = Resp<T>::nodes, CO = Resp<T>::comp;
  __shared__ double val[PE_MAX_TERMS * NN][2];
  const int t = blockIdx.x, K = C.K, steps = chain_steps(M);
  for (int e = threadIdx.x; e < R * NN; e += blockDim.x) {
    const int r = e / NN, i = e - r * NN;
    const double* nb = nodes + ((int64_t)t * NN + i) * (1 + q);
    const int k = C.first[r];
    const bool two = k + 1 < K && C.term[k + 1] == r;
    double br = 0.0, bi = 0.0;
    for (int s = 0; s < q; ++s) {
      br = fma(nb[1 + s], D.ZF[s * K + k], br);
      if (two) bi = fma(nb[1 + s], D.ZF[s * K + k + 1], bi);
    }
    double Sr, Si;
    chain_sum(nb[0] * D.xs[r], M, steps, D.chain + 4 * r, 4 * R, Sr, Si);
    val[e][0] = fma(br, Sr, -(bi * Si));
    val[e][1] = fma(br, Si, bi * Sr);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < R * 2 * NN; e += blockDim.x) {
    const int d = e % NN, rc = e / NN, r = rc >> 1, comp = rc & 1;
    const double mid = val[r * NN + NN / 2][comp];
    double c = 0.0;
#pragma unroll
    for (int i = 0; i < NN; ++i) c = fma(I.m[d][i], val[r * NN + i][comp] - mid, c);
    if (d == 0) c += mid;
    T* o = resp + (((int64_t)r * (T_ + 1) + t) * 2 + comp) * CO;
    if constexpr (sizeof(T) == 4) {
      if (d == 0) {
        o[0] = (float)c;
        o[1] = (float)(c - (double)(float)c);
      } else {
        o[1 + d] = (float)c;
      }
    } else {
      o[d] = c;
    }
  }
}

// 1D consistent loads of every (term, axis): out[R*off[a] + r*n_a + k] = int g_{r,a} phi_{k+1}.
// Eight lanes per node (blockDim = 8 x 32 nodes): lane s evaluates the quadrature points
// e = s, s + 8, ... of the node's 2 npts (its left element's points, then its right element's),
// and the eight partial sums are added by shuffles in a fixed order.  The float64 exponentials
// and sines of the factors thus spread over eight times more warps than a thread per node.
constexpr int kLoadLanes = 8;
__global__ void __launch_bounds__(256) loads_1d_kernel(TermsDev T, Geom g, double lo0, double lo1, double lo2,
                                                       double h0, double h1, double h2, Gauss G,
                                                       double* __restrict__ out) {
  pdl_wait();
  const int a = blockIdx.z;
  const int r = blockIdx.y;
  const int sub = threadIdx.x & (kLoadLanes - 1);
  const int k = blockIdx.x * (blockDim.x / kLoadLanes) + threadIdx.x / kLoadLanes;  // 0-based node
  if (a >= g.d || r >= T.n || k >= g.n[a]) return;  // whole groups of eight lanes leave together
  const double lo = a == 0 ? lo0 : (a == 1 ? lo1 : lo2);
  const double h = a == 0 ? h0 : (a == 1 ? h1 : h2);
  const pe_term& t = T.t[r];
  const int lk = T.lk[r][a];
  const unsigned grp = 0xFFu << (threadIdx.x & 24);  // this node's eight lanes of the warp
  if (lk != 0) {
    // lifting of Dirichlet data: the factor at full-grid nodes k, k+1, k+2 (x = lo + i h)
    if (sub == 0) {
      const double g0 = eval_space(t.skind[a], t.sp[a], lo + (double)k * h);
      const double g1 = eval_space(t.skind[a], t.sp[a], lo + (double)(k + 1) * h);
      const double g2 = eval_space(t.skind[a], t.sp[a], lo + (double)(k + 2) * h);
      double v = g1;
      if (lk == 1) v = (h / 6.0) * (g0 + 4.0 * g1 + g2);
      else if (lk == 2) v = (1.0 / h) * (2.0 * g1 - g0 - g2);
      out[(int64_t)T.n * g.off[a] + (int64_t)r * g.n[a] + k] = v;
    }
    return;
  }
  // Dirichlet: node k sits at lo + (k+1) h; element k ([lo + k h, lo + (k+1) h]) has it as
  // right vertex (shape s), element k+1 as left vertex (shape 1-s).  Periodic: node k sits
  // at lo + k h; the elements are k-1 (element n-1 for k = 0) and k.
  const int el = g.per[a] ? (k == 0 ? g.n[a] - 1 : k - 1) : k;
  const int er = g.per[a] ? k : k + 1;
  double part = 0.0;
  for (int e = sub; e < 2 * G.npts; e += kLoadLanes) {
    const bool left = e < G.npts;
    const int qi = left ? e : e - G.npts;
    const double x = lo + ((double)(left ? el : er) + G.s[qi]) * h;
    part += G.w[qi] * eval_space(t.skind[a], t.sp[a], x) * (left ? G.s[qi] : 1.0 - G.s[qi]);
  }
#pragma unroll
  for (int o = kLoadLanes / 2; o > 0; o >>= 1) part += __shfl_xor_sync(grp, part, o);
  if (sub == 0) out[(int64_t)T.n * g.off[a] + (int64_t)r * g.n[a] + k] = h * part;
}

// Per-axis source factors in matrix form, for grids whose axes are short: out[e],
// e = R off_a + r n_a + j (the layout of the per-axis tables), is sum_k S_a[j][k] L[R off_a + r
// n_a + k], times 1 / mu^M_a(j) when muInv is given.  A warp per output splits k (a row of the
// symmetric transform matrix and the term's loads, both contiguous: coalesced reads, all of a
// lane's loads in flight at once for n < 256, so a row read from HBM costs one latency); a shuffle
// sum in a fixed order.  The float64 work (n FMAs per output) spreads over every SM, where a
// half-length FFT per pencil pair runs one chain of dependent float64 latencies on a few SMs.
constexpr int kFactorLanes = 32;
// where the factors of one list of R terms go (muInv: 1 / mu^M, or null for none)
struct FactorOut {
  int R;
  double* fac;
  float* fac32;
  const double* muInv;
};
__global__ void __launch_bounds__(256) axis_factor_matrix_kernel(Geom g, int R, const double* __restrict__ S0,
                                                                 const double* __restrict__ S1,
                                                                 const double* __restrict__ S2,
                                                                 const double* __restrict__ loads,
                                                                 FactorOut A, FactorOut B, int64_t total) {
  pdl_wait();
  const int64_t e = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kFactorLanes;
  const int sub = threadIdx.x & (kFactorLanes - 1);
  if (e >= total) return;  // whole warps leave together
  int a = 0;
  while (a + 1 < g.d && e >= (int64_t)R * g.off[a + 1]) ++a;
  const int n = g.n[a];
  const int64_t local = e - (int64_t)R * g.off[a];
  const int r = (int)(local / n), j = (int)(local - (int64_t)r * n);
  const double* S = a == 0 ? S0 : (a == 1 ? S1 : S2);
  const double* row = S + (int64_t)j * n;
  const double* L = loads + (int64_t)R * g.off[a] + (int64_t)r * n;
  double acc = 0.0;
#pragma unroll 8
  for (int k = sub; k < n; k += kFactorLanes) acc = fma(row[k], L[k], acc);
#pragma unroll
  for (int o = kFactorLanes / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
  if (sub == 0) {
    // terms r < A.R belong to the first list, the others to the second
    const bool second = r >= A.R;
    const FactorOut& F = second ? B : A;
    const int64_t o = (int64_t)F.R * g.off[a] + (int64_t)(second ? r - A.R : r) * n + j;
    const double v = F.muInv ? acc * F.muInv[g.off[a] + j] : acc;
    F.fac[o] = v;
    if (F.fac32) F.fac32[o] = (float)v;
  }
}

__global__ void divide_axis_mu_kernel(Geom g, int R, const double* __restrict__ muM, double* __restrict__ x,
                                      float* __restrict__ x32) {
  const int a = blockIdx.z;
  const int r = blockIdx.y;
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= g.d || r >= R || j >= g.n[a]) return;
  const int64_t idx = (int64_t)R * g.off[a] + (int64_t)r * g.n[a] + j;
  const double v = x[idx] / muM[g.off[a] + j];
  x[idx] = v;
  if (x32) x32[idx] = (float)v;
}

// out[J] = sum_r w_r prod_a fac[R*off[a] + r*n_a + j_a]
struct TermWeights {
  double w[PE_MAX_TERMS];
};
__global__ void outer_sum_kernel(Geom g, int R, const double* __restrict__ fac, TermWeights W,
                                 double* __restrict__ out, int accumulate) {
  pdl_wait();
  const int64_t J = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (J >= g.ndof) return;
  int j[PE_MAX_D];
  unflatten(g, J, j);
  double acc = 0.0;
  for (int r = 0; r < R; ++r) {
    double P = fac[(int64_t)R * g.off[0] + (int64_t)r * g.n[0] + j[0]];
#pragma unroll
    for (int a = 1; a < PE_MAX_D; ++a) if (a < g.d) P *= fac[(int64_t)R * g.off[a] + (int64_t)r * g.n[a] + j[a]];
    acc += W.w[r] * P;
  }
  out[J] = accumulate ? out[J] + acc : acc;
}

__global__ void scale_mu_kernel(Geom g, const double* __restrict__ muM, double* __restrict__ x, int inverse) {
  const int64_t J = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (J >= g.ndof) return;
  int j[PE_MAX_D];
  unflatten(g, J, j);
  double mu = muM[g.off[0] + j[0]];
#pragma unroll
  for (int a = 1; a < PE_MAX_D; ++a) if (a < g.d) mu *= muM[g.off[a] + j[a]];
  x[J] = inverse ? x[J] / mu : x[J] * mu;
}

}  // namespace

// Rows d of the inverse: the coefficient of x^d of the polynomial through values at the Chebyshev nodes
// x_i = cos(pi (2 i + 1) / (2 n)), from the discrete Chebyshev transform and T_k's own coefficients.
static RespInv response_inverse(int n) {
  double T[8][8] = {};  // T_k in monomials
  T[0][0] = 1.0;
  if (n > 1) T[1][1] = 1.0;
  for (int k = 2; k < n; ++k)
    for (int d = 0; d < n; ++d) T[k][d] = (d ? 2.0 * T[k - 1][d - 1] : 0.0) - T[k - 2][d];
  RespInv I{};
  for (int d = 0; d < n; ++d)
    for (int i = 0; i < n; ++i) {
      double s = 0.0;
      for (int k = 0; k < n; ++k)
        s += (k ? 2.0 : 1.0) / n * cos(M_PI * k * (2.0 * i + 1.0) / (2.0 * n)) * T[k][d];
      I.m[d][i] = s;
    }
  return I;
}

pe_status setup_response_nodes(pe_ctx* c) {
  // the range of lam over the whole grid, zero aside
  double lo = 0.0, hi = 0.0, least = INFINITY;
  bool zero = true;
  for (int a = 0; a < c->gn.d; ++a) {
    const int n = c->gn.n[a];
    auto ratio = [&](double th) {
      const double sh = sin(0.5 * th);
      return ((4.0 / c->h[a]) * sh * sh) / ((c->h[a] / 3.0) * (2.0 + cos(th)));
    };
    if (c->gn.per[a]) {
      if (n > 1) least = std::min(least, ratio(2.0 * M_PI / n));
      hi += ratio(2.0 * M_PI * (n / 2) / n);
    } else {
      zero = false;
      lo += ratio(M_PI / (n + 1));
      hi += ratio(M_PI * n / (n + 1));
    }
  }
  if (zero) lo = least;
  lo *= c->D * (1.0 - 1e-9);
  hi *= c->D * (1.0 + 1e-9);
  // no table for spectra beyond the normal range of a double
  if (!(lo > 1e-300 && hi < 1e300)) return PE_OK;
  const bool f32 = c->precision == PE_MIXED;
  const int bits = f32 ? Resp<float>::bits : Resp<double>::bits, nodes = f32 ? Resp<float>::nodes : Resp<double>::nodes;
  const int comp = f32 ? Resp<float>::comp : Resp<double>::comp;
  auto lead = [bits](double v) {
    int64_t u;
    memcpy(&u, &v, sizeof(u));
    return (int)(u >> (52 - bits));
  };
  const int base = lead(lo), T = lead(hi) - base + 1;
  // a node costs about what eight modes save (200 x 117 modes in float64, 4200 nodes: 9 us slower with the table)
  // (the whole grid decides, for a shard too: its weights are the unsharded solve's, bit for bit)
  if ((int64_t)(T + 1) * nodes * 8 > c->gn.ndof) return PE_OK;
  if (cudaMalloc((void**)&c->resp_nodes, sizeof(double) * (size_t)(T + 1) * nodes * (1 + c->q)) != cudaSuccess ||
      cudaMalloc(&c->resp, (f32 ? sizeof(float) : sizeof(double)) * (size_t)PE_MAX_TERMS * (T + 1) * 2 * comp) !=
          cudaSuccess) {
    cudaGetLastError();
    return pe_fail(PE_ENOMEM, "pe_setup: response-table allocation failed");
  }
  c->resp_base = base;
  c->resp_T = T;
  c->resp_lo = lo;
  c->resp_hi = hi;
  Lag LF{};
  for (int i = 0; i < PE_MAX_S; ++i)
    for (int m = 0; m < PE_MAX_S; ++m) LF.a[i][m] = c->lagF[i][m];
  response_nodes_kernel<<<((T + 1) * nodes + 63) / 64, 64, 0, c->stream>>>(base, T, bits, nodes, c->dt, c->q, LF,
                                                                          c->resp_nodes);
  c->launches += 1;
  PE_CUDA_TRY(cudaGetLastError());
  return PE_OK;
}

// Whether the tabulated weights of a term are as exact as the form rounds, relative to the weight itself on every
// mode.  A term that persists, or grows and is counted from the slice's end, has weights of the size of int e^{-lam s} ds, in
// which the table's error is bounded.  For e^{-alpha t} the weight is int_0^dT e^{-lam s} e^{-alpha (dT - s)} ds:
// its n-th derivative in lam is the weight times a mean of s^n, at most dT^n and, where lam > alpha, n! / (lam - alpha)^n.  With
// n! >= (n/e)^n the interpolation error on an interval of width w lam, 2 (w lam / 4)^n max |H^(n)| / n!, is at most
//   2 ((w lam / 4) min(e dT / n, 1 / (lam - alpha)))^n H,
// largest where the two meet, lam = alpha + n / (e dT), or at the end of the spectrum next to it.  One source, lam_min about 20,
// relative L2 by the table and directly: dT = 1.5, alpha = 30, 7.2e-5 and 9.1e-9 (mixed, 160^2 modes), 4.4e-11 and 4.3e-16
// (float64, 208^2); dT = 3, alpha = 40, 3.4e-3 and 3.0e-8, 1.2e-8 and 2.2e-15; just inside the rule by the table: 1.0e-7 and
// 4.0e-16.
static bool response_exact(const pe_ctx* c, const pe_term& t) {
  if (t.tkind == PE_T_SIN || !(t.tp[0] < 0.0)) return true;
  const bool f32 = c->precision == PE_MIXED;
  const double n = f32 ? Resp<float>::nodes : Resp<double>::nodes, w = ldexp(1.0, -(f32 ? Resp<float>::bits : Resp<double>::bits));
  const double alpha = -t.tp[0], reach = n / (M_E * c->dT);
  const double lam = std::min(std::max(alpha + reach, c->resp_lo), c->resp_hi);
  const double f = 0.25 * w * lam / std::max(reach, lam - alpha);
  return 2.0 * pow(f, n) <= (f32 ? 0x1p-24 : 0x1p-53);
}

// The current problem's weights come from the table (not with the learned correction, whose bands the
// direct kernel adds).  All of them or none: one term beyond the table's reach takes the problem to the direct kernel.
static bool uses_response(const pe_ctx* c) { return c->resp && c->resp_on && !c->mlp; }

// The current problem's response table, after its time tables.
static pe_status launch_response(pe_ctx* c) {
  if (!uses_response(c)) return PE_OK;
  const dim3 grid((unsigned)(c->resp_T + 1));
  if (c->precision == PE_MIXED) {
    static const RespInv I = response_inverse(Resp<float>::nodes);
    PE_CUDA_TRY(launch_pdl(response_kernel<float>, grid, dim3(160), 0, c->stream, c->cols, c->tab, c->R, c->M, c->q,
                           c->resp_T, I, (const double*)c->resp_nodes, (float*)c->resp));
  } else {
    static const RespInv I = response_inverse(Resp<double>::nodes);
    PE_CUDA_TRY(launch_pdl(response_kernel<double>, grid, dim3(160), 0, c->stream, c->cols, c->tab, c->R, c->M, c->q,
                           c->resp_T, I, (const double*)c->resp_nodes, (double*)c->resp));
  }
  c->launches += 1;
  return PE_OK;
}

pe_status launch_time_tables(pe_ctx* c) {
  const int R = c->R;
  if (R == 0) return PE_OK;
  TermsDev T = pack_terms(c->terms, R);
  Nodes nF{}, nG{};
  for (int i = 0; i < PE_MAX_S; ++i) {
    nF.c[i] = c->cF[i];
    nG.c[i] = c->cG[i];
  }
  // columns: one per exponential term, two per sinusoid
  StageCols C{};
  for (int r = 0; r < R; ++r) {
    C.first[r] = (signed char)C.K;
    C.term[C.K] = (signed char)r;
    C.kind[C.K++] = 0;
    if (c->terms[r].tkind == PE_T_SIN) {
      C.term[C.K] = (signed char)r;
      C.kind[C.K++] = 1;
    }
  }
  c->cols = C;
  c->K = C.K;
  c->resp_on = c->resp && std::all_of(c->terms, c->terms + R, [c](const pe_term& t) { return response_exact(c, t); });
  const int total = c->N * C.K + (c->q + c->p) * C.K + R * (chain_steps(c->M) + 1);
  const int threads = 128;
  PE_CUDA_TRY(launch_pdl(time_tables_kernel, dim3((unsigned)((total + threads - 1) / threads)), dim3(threads), 0,
                         c->stream, T, C, c->tab, c->N, c->M, c->q, c->p, c->t0, c->dT, c->dt, nF, nG));
  c->launches += 1;
  PE_CUDA_TRY(cudaGetLastError());
  return launch_response(c);
}

// Room for the weights of K columns in one table.
template <typename T>
static pe_status grow_weights(pe_ctx* c, T** W, int* cap) {
  const int K = c->K;
  if (K <= *cap) return PE_OK;
  PE_CUDA_TRY(cudaStreamSynchronize(c->stream));
  if (*W) {
    drop_loop_graph(c);  // it was captured with the address given back here
    cudaFree(*W);
  }
  *W = nullptr;
  *cap = 0;
  if (cudaMalloc((void**)W, (size_t)K * (size_t)c->g.ndof * sizeof(T)) != cudaSuccess) {
    cudaGetLastError();
    return pe_fail(PE_ENOMEM, "pe_set_problem: column-weight table allocation failed");
  }
  *cap = K;
  return PE_OK;
}

// Terms per thread of the weights kernel: one while the modes alone leave the GPU short of warps
// (each term's chain is a serial run of its own), then a few, so that the tables of the mode are
// read less often; all of them with the learned correction, whose band position costs a logarithm.
static int weights_tpt(const pe_ctx* c, bool learned) {
  if (learned) return c->R;
  return c->g.ndof < ((int64_t)1 << 19) ? 1 : std::min(c->R, 4);
}

template <typename T>
static pe_status column_weights(pe_ctx* c, T* V, T* G, const LearnedTerms& L) {
  const int threads = 256, tpt = weights_tpt(c, L.Ktab != nullptr);
  const dim3 grid((unsigned)((c->g.ndof + threads - 1) / threads), (unsigned)((c->R + tpt - 1) / tpt));
  const T *axisF, *coef, *coefG;
  if constexpr (sizeof(T) == 8) {
    axisF = c->axisF;
    coef = c->coefF;
    coefG = c->coefG + c->g.ndof;
  } else {
    axisF = c->axisF32;
    coef = c->coefF32;
    coefG = c->coefG32;
  }
  // the table serves the form it was made in (a mixed context's float64 weights are evaluated directly)
  if (uses_response(c) && V && (sizeof(T) == 8) == (c->precision != PE_MIXED)) {
    PE_CUDA_TRY(launch_pdl(response_weights_kernel<T>, grid, dim3(threads), 0, c->stream, c->g, c->cols, c->tab, c->R,
                           c->p, tpt, c->resp_base, c->resp_T, (const T*)c->resp, axisF, coefG, V, G,
                           (const double*)c->lam));
    c->launches += 1;
    return PE_OK;
  }
  PE_CUDA_TRY(launch_pdl(column_weights_kernel<T>, grid, dim3(threads), 0, c->stream, c->g, c->cols, c->tab, c->R, c->M,
                         c->q, c->p, tpt, axisF, coef, coefG, V, G, L, (const double*)c->axisF,
                         (const double*)c->lam));
  c->launches += 1;
  PE_CUDA_TRY(cudaGetLastError());
  return PE_OK;
}

pe_status launch_column_weights(pe_ctx* c) {
  LearnedTerms L{};
  if (c->mlp) PE_TRY(launch_learned_tables(c, &L));
  c->V64_valid = false;
  if (c->precision == PE_MIXED) {
    // the float32 sweeps need only float32 weights; pe_refine makes its float64 ones.  The general
    // path's coarse forcing is float64 in either form.
    PE_TRY(grow_weights(c, &c->V32, &c->capV32));
    if (c->forcing_path == PE_FORCING_GENERAL) {
      PE_TRY(grow_weights(c, &c->G64, &c->capG64));
      PE_TRY(column_weights<double>(c, nullptr, c->G64, L));
      return column_weights<float>(c, c->V32, nullptr, L);
    }
    PE_TRY(grow_weights(c, &c->G32, &c->capG32));
    return column_weights<float>(c, c->V32, c->G32, L);
  }
  PE_TRY(grow_weights(c, &c->V64, &c->capV64));
  PE_TRY(grow_weights(c, &c->G64, &c->capG64));
  PE_TRY(column_weights<double>(c, c->V64, c->G64, L));
  c->V64_valid = true;
  return PE_OK;
}

pe_status launch_column_weights_f64(pe_ctx* c) {
  if (c->V64_valid) return PE_OK;
  PE_TRY(grow_weights(c, &c->V64, &c->capV64));
  PE_TRY(column_weights<double>(c, c->V64, nullptr, LearnedTerms{}));
  c->V64_valid = true;
  return PE_OK;
}

// Rows of the whole-axis per-axis tables (layout of gf) that a sharded context owns, in its
// own layout (gl): out[R off_l[a] + r n_l[a] + j] = in[R off_f[a] + r n_f[a] + j + base_a],
// base_0 = the first owned axis-0 mode, base_a = 0 for the other axes.
__global__ void compact_axis_kernel(Geom gf, Geom gl, int base0, int R, const double* __restrict__ in,
                                    double* __restrict__ out, float* __restrict__ out32) {
  const int a = blockIdx.z;
  const int r = blockIdx.y;
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= gl.d || r >= R || j >= gl.n[a]) return;
  const int jf = j + (a == 0 ? base0 : 0);
  const double v = in[(int64_t)R * gf.off[a] + (int64_t)r * gf.n[a] + jf];
  const int64_t o = (int64_t)R * gl.off[a] + (int64_t)r * gl.n[a] + j;
  out[o] = v;
  if (out32) out32[o] = (float)v;
}

static pe_status separable_factors_whole(pe_ctx* c, const pe_term* terms, int nterms, double* axis_out, int mode,
                                         const signed char (*lk)[PE_MAX_D]);

pe_status compact_axis_tables(pe_ctx* c, int R, const double* in, double* out, float* out32) {
  int nmax = 1;
  for (int a = 0; a < c->g.d; ++a) nmax = c->g.n[a] > nmax ? c->g.n[a] : nmax;
  dim3 grid((nmax + 127) / 128, R, c->g.d);
  compact_axis_kernel<<<grid, 128, 0, c->stream>>>(c->gn, c->g, c->base0, R, in, out, out32);
  c->launches += 1;
  PE_CUDA_TRY(cudaGetLastError());
  return PE_OK;
}

// mode 0: 1D loads only (axis_out gets loads); mode 1: modal factors (S_a F)/mu^M;
// mode 2: S_a F only (the modal coefficients V^T y of a separable nodal vector y).
// lk (may be NULL): per-term, per-axis load kinds of the Dirichlet lifting (TermsDev).
// A sharded context computes the factors of the whole axes and keeps the rows of its modes.
pe_status launch_separable_factors(pe_ctx* c, const pe_term* terms, int nterms, double* axis_out, int mode,
                                   const signed char (*lk)[PE_MAX_D]) {
  if (!c->sharded) return separable_factors_whole(c, terms, nterms, axis_out, mode, lk);
  if (nterms == 0) return PE_OK;
  if (mode != 1) return pe_fail(PE_EINVAL, "a context that owns a block of modes takes separable modal factors only");
  const Geom gl = c->g;
  double* mu_l = c->muM_axis;
  c->g = c->gn;
  c->muM_axis = c->muM_full;
  const pe_status st = separable_factors_whole(c, terms, nterms, c->fac_full, 1, lk);
  c->g = gl;
  c->muM_axis = mu_l;
  PE_TRY(st);
  const bool f32 = (axis_out == c->axisF) && c->precision == PE_MIXED;
  return compact_axis_tables(c, nterms, c->fac_full, axis_out, f32 ? c->axisF32 : nullptr);
}

static bool matrix_factors(const pe_ctx* c, int nterms) {
  // the matrix form over every SM while its float64 work stays small (R sum_a n_a^2 <= 8M FMAs)
  int64_t work = 0;
  for (int a = 0; a < c->g.d; ++a) work += (int64_t)nterms * c->g.n[a] * c->g.n[a];
  return c->muM_inv && work <= ((int64_t)8 << 20);
}

// 1D loads of the terms, then their factors in matrix form into A (and B)
static pe_status loads_of(pe_ctx* c, const TermsDev& T, double* loads) {
  const Gauss G = make_gauss(c->quad_pts);
  int nmax = 1;
  for (int a = 0; a < c->g.d; ++a) nmax = c->g.n[a] > nmax ? c->g.n[a] : nmax;
  dim3 lgrid((nmax + 31) / 32, T.n, c->g.d);  // 32 nodes of eight lanes per CTA
  PE_CUDA_TRY(launch_pdl(loads_1d_kernel, lgrid, dim3(32 * kLoadLanes), 0, c->stream, T, c->g, c->lo[0], c->lo[1],
                         c->lo[2], c->h[0], c->h[1], c->h[2], G, loads));
  c->launches += 1;
  return PE_OK;
}

static pe_status factors_of(pe_ctx* c, const FactorOut& A, const FactorOut& B) {
  const int nterms = A.R + B.R;
  const int64_t total = (int64_t)nterms * (c->g.off[c->g.d - 1] + c->g.n[c->g.d - 1]);
  const unsigned blocks = (unsigned)((total * kFactorLanes + 255) / 256);
  PE_CUDA_TRY(launch_pdl(axis_factor_matrix_kernel, dim3(blocks), dim3(256), 0, c->stream, c->g, nterms,
                         (const double*)c->S[0], (const double*)(c->g.d > 1 ? c->S[1] : c->S[0]),
                         (const double*)(c->g.d > 2 ? c->S[2] : c->S[0]), (const double*)c->loads, A, B, total));
  c->launches += 1;
  return PE_OK;
}

static FactorOut factor_out(const pe_ctx* c, int R, double* out, int mode) {
  return FactorOut{R, out, mode == 1 && out == c->axisF && c->precision == PE_MIXED ? c->axisF32 : nullptr,
                   mode == 1 ? c->muM_inv : nullptr};
}

pe_status launch_separable_factors_two(pe_ctx* c, const pe_term* ta, int na, double* axis_a,
                                       const signed char (*lka)[PE_MAX_D], const pe_term* tb, int nb, double* axis_b,
                                       int mode_b, const signed char (*lkb)[PE_MAX_D]) {
  if (na == 0 || nb == 0 || na + nb > PE_MAX_TERMS || c->sharded || mode_b == 0 || !matrix_factors(c, na + nb)) {
    PE_TRY(launch_separable_factors(c, ta, na, axis_a, 1, lka));
    return launch_separable_factors(c, tb, nb, axis_b, mode_b, lkb);
  }
  TermsDev T = pack_terms(ta, na, lka);
  const TermsDev U = pack_terms(tb, nb, lkb);
  for (int i = 0; i < nb; ++i) {
    T.t[na + i] = U.t[i];
    for (int a = 0; a < PE_MAX_D; ++a) T.lk[na + i][a] = U.lk[i][a];
  }
  T.n = na + nb;
  PE_TRY(loads_of(c, T, c->loads));
  return factors_of(c, factor_out(c, na, axis_a, 1), factor_out(c, nb, axis_b, mode_b));
}

static pe_status separable_factors_whole(pe_ctx* c, const pe_term* terms, int nterms, double* axis_out, int mode,
                                         const signed char (*lk)[PE_MAX_D]) {
  if (nterms == 0) return PE_OK;
  int nmax = 1;
  for (int a = 0; a < c->g.d; ++a) nmax = c->g.n[a] > nmax ? c->g.n[a] : nmax;
  dim3 grid((nmax + 127) / 128, nterms, c->g.d);
  double* loads = mode == 0 ? axis_out : c->loads;
  PE_TRY(loads_of(c, pack_terms(terms, nterms, lk), loads));
  if (mode == 0) return PE_OK;
  const bool f32 = (axis_out == c->axisF) && c->precision == PE_MIXED;
  if (matrix_factors(c, nterms)) return factors_of(c, factor_out(c, nterms, axis_out, mode), FactorOut{});
  if (mode == 1) {
    bool done = false;
    PE_TRY(axis_factors_fused(c, nterms, loads, axis_out, f32 ? c->axisF32 : nullptr, &done));
    if (done) return PE_OK;
  }
  for (int a = 0; a < c->g.d; ++a) {
    const int64_t base = (int64_t)nterms * c->g.off[a];
    PE_TRY(dst_axis_f64(c->S[a], loads + base, axis_out + base, nterms, c->g.n[a], 1, c->stream, c->g.per[a]));
    c->launches += 1;
  }
  if (mode == 2) return PE_OK;  // V^T of nodal values: no division by mu^M
  divide_axis_mu_kernel<<<grid, 128, 0, c->stream>>>(c->g, nterms, c->muM_axis, axis_out,
                                                     f32 ? c->axisF32 : nullptr);
  c->launches += 1;
  PE_CUDA_TRY(cudaGetLastError());
  return PE_OK;
}

static pe_status outer_sum(pe_ctx* c, const double* fac, int R, const TermWeights& W, double* out, int accumulate) {
  const int threads = 256;
  PE_CUDA_TRY(launch_pdl(outer_sum_kernel, dim3((unsigned)((c->g.ndof + threads - 1) / threads)), dim3(threads), 0,
                         c->stream, c->g, R, fac, W, out, accumulate));
  c->launches += 1;
  return PE_OK;
}

// out[J] = sum_r amp_r prod_a fac_{r,a}[j_a] (nodal_loads: fac are 1D loads, out a nodal load vector)
pe_status launch_outer_sum(pe_ctx* c, const double* axis_fac, const pe_term* terms, int nterms, double* out,
                           int accumulate) {
  if (nterms == 0) return PE_OK;
  TermWeights W{};
  for (int r = 0; r < nterms; ++r) W.w[r] = terms[r].amp;
  return outer_sum(c, axis_fac, nterms, W, out, accumulate);
}

pe_status launch_forcing_modal(pe_ctx* c, double t, double* out) {
  TermWeights W{};
  for (int r = 0; r < c->R; ++r) {
    const pe_term& T = c->terms[r];
    W.w[r] = T.amp * (T.tkind == PE_T_SIN ? sin(T.tp[0] * t + T.tp[1]) : exp(T.tp[0] * t));
  }
  return outer_sum(c, c->axisF, c->R, W, out, 0);
}

pe_status launch_scale_by_muM(pe_ctx* c, double* x, int inverse) {
  const int threads = 256;
  scale_mu_kernel<<<(unsigned)((c->g.ndof + threads - 1) / threads), threads, 0, c->stream>>>(c->g, c->muM_axis, x,
                                                                                              inverse);
  c->launches += 1;
  PE_CUDA_TRY(cudaGetLastError());
  return PE_OK;
}
