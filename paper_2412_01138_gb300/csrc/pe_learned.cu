// Learned coarse-propagator correction: a 3-layer MLP (2 -> 64 -> 64 -> 2, tanh)
// with hand-written training (forward, backward, weight gradients, Adam) and
// inference kernels.
//
// Why it can help: G and F share the homogeneous propagator e^{-lam dT}, so
// F^M(v) - G(v) does not depend on v (Algorithm 1 then converges after one
// iteration, and a residual stop confirms at k = 2).  Per mode J and sine source
// term r = amp_r sin(w_r t + phi_r) prod_a g_{r,a}, the difference over slice n is
//   delta_{n,J} = sum_r P_{r,J} amp_r Im( e^{i(w_r T_n + phi_r)} K(lam_J, w_r) ),
//   K(lam, w) = [F^M(0) - G(0)] for the unit source e^{i w t} on [0, dT],
// a smooth function of (lam dT, w dT) alone.  The network learns K from pairs the
// method itself generates (the fine and coarse steps of Eq. (1-7) run on unit
// sources); adding its prediction to the coarse step gives G'(v) = G(v) + delta^.
// F - G' is still iterate-independent and the fixed point of Algorithm 1 is still
// the fine solution, so the network can only change how soon the residual falls
// below tol, never the answer.  If the prediction error is below tol the solve
// stops after one fine sweep instead of two.
//
// Normalisation: features x = (log(lam dT)/6, w dT - 1); target
// K~ = 4 K / (s (w dT)^2) with s = dT/(1 + lam dT) (K~ = O(1) over the spectrum).
#include <cuda_fp16.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "pe_batch.h"
#include "pe_learned.h"
#include "pe_phi.cuh"

namespace {

constexpr int H = PE_MLP_WIDTH;
// parameter layout (floats): W1[H][2], b1[H], W2[H][H], b2[H], W3[2][H], b3[2]
constexpr int OW1 = 0, OB1 = OW1 + 2 * H, OW2 = OB1 + H, OB2 = OW2 + H * H, OW3 = OB2 + H, OB3 = OW3 + 2 * H;
constexpr int NPARAM = OB3 + 2;

struct Cd {
  double re, im;
};

__device__ inline Cd cexpi(double x) {
  double s, c;
  sincos(x, &s, &c);
  return Cd{c, s};
}

// ---------------------------------------------------------------------------
// labels: K(lam, w) = F^M(0) - G(0) for the unit source e^{i w t}, normalised
// ---------------------------------------------------------------------------
__global__ void samples_kernel(int n, const double* __restrict__ lam, const double* __restrict__ om, double dT,
                               int M, int q, int p, Lag LF, Lag LG, Nodes8 cF, Nodes8 cG, float* __restrict__ x,
                               float* __restrict__ y, double* __restrict__ Kraw) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  const double l = lam[s], w = om[s];
  const double dt = dT / (double)M;
  double bF[PE_MAX_S], bG[PE_MAX_S];
  const double E = exp(-l * dt);
  b_weights(-l * dt, q, LF, bF);
  b_weights(-l * dT, p, LG, bG);
  Cd acc{0.0, 0.0};
  for (int m = 0; m < M; ++m) {
    Cd st{0.0, 0.0};
    for (int i = 0; i < q; ++i) {
      const Cd e = cexpi(w * ((double)m + cF.c[i]) * dt);
      st.re = fma(bF[i], e.re, st.re);
      st.im = fma(bF[i], e.im, st.im);
    }
    acc.re = fma(E, acc.re, dt * st.re);
    acc.im = fma(E, acc.im, dt * st.im);
  }
  Cd g{0.0, 0.0};
  for (int i = 0; i < p; ++i) {
    const Cd e = cexpi(w * cG.c[i] * dT);
    g.re = fma(bG[i], e.re, g.re);
    g.im = fma(bG[i], e.im, g.im);
  }
  const double Kre = acc.re - dT * g.re, Kim = acc.im - dT * g.im;
  if (Kraw) {
    Kraw[2 * s] = Kre;
    Kraw[2 * s + 1] = Kim;
  }
  const double wd = w * dT;
  const double scale = 4.0 * (1.0 + l * dT) / (dT * wd * wd);
  x[2 * s] = (float)(log(l * dT) / 6.0);
  x[2 * s + 1] = (float)(wd - 1.0);
  y[2 * s] = (float)(Kre * scale);
  y[2 * s + 1] = (float)(Kim * scale);
}

// ---------------------------------------------------------------------------
// training: one persistent cooperative launch runs every Adam step.  Per step
//   1. every CTA loads the float32 parameters into shared memory and runs the forward and
//      backward pass of its share of the batch in rounds of TR_ROUND samples: the 2 -> 64 and
//      64 -> 2 layers on the CUDA cores, the 64 x 64 layer's three contractions -- forward
//      Z2 = H1 W2^T, backward dH1 = dZ2 W2 and the weight gradient dW2 = dZ2^T H1 -- as warp-level
//      tensor-core MMAs (m16n8k8, TF32 operands split in two, float32 accumulation);
//   2. the other parameters' gradients are summed per thread over the round's samples; each CTA
//      writes its partial gradient as row c of partial[c][k];
//   3. grid barrier; each CTA owns a contiguous range of parameters (a lane per parameter) and
//      adds their G partials in a fixed order (deterministic), then applies Adam (or, for a
//      gradient evaluation, writes the gradient);
//   4. grid barrier (the next step reads the updated parameters).
// A step is a chain of trips to L2, not work (4096 samples are one round of 27 per CTA): so a thread issues all
// its parameter loads, and all its partial-gradient loads, before it uses the first, the barriers arrive
// with a release and poll with an acquire instead of two full fences, and the Adam scalars are made
// while the parameters travel: 13.3 to 11.8 us a step of 4096 samples on 152 SMs.
// Barriers are bounded waits: on expiry the CTA records an error and returns (every other
// CTA then expires at its next wait); the host reports PE_ETIMEOUT.
// ---------------------------------------------------------------------------
constexpr int TR_THREADS = 512;
constexpr int TR_WARPS = TR_THREADS / 32;
constexpr int TR_ROUND = 32;            // samples per CTA per round: the M of the MMA tiles
constexpr int AP = H + 4;               // padded row stride of W2 and the activations in shared memory
constexpr int NPARAM_L = NPARAM + 1;    // the gradient slots plus one slot for the loss
constexpr int NSIMT = NPARAM_L - H * H;  // slots summed on the CUDA cores: all but W2
constexpr int NOTHER = NPARAM - H * H;  // the parameters but W2
static_assert(2 * 4 * TR_THREADS == H * H && OW2 % 4 == 0, "two float4 of W2 per thread");
static_assert(NSIMT <= TR_THREADS, "one CUDA-core gradient slot per thread");
static_assert(TR_WARPS == 16 && TR_ROUND == 32 && H == 64, "MMA tile assignment below");
constexpr long long kGridWaitCycles = 2000000000LL;  // about a second

struct TrainArgs {
  float* params;
  float* adam_m;
  float* adam_v;
  float* partial;        // [G][NPARAM_L]: CTA c's partial gradient in row c
  const float* x;        // [n][2]
  const float* t;        // [n][2]
  int n, batch, steps_per_epoch, total, it0, nsteps;
  float lr, b1, b2, eps;
  long long adam_step0;  // Adam steps taken before this launch
  float inv_n;           // > 0: fixed loss weight (gradient evaluation); 0: 1 / (batch size)
  float* grad_out;       // gradient evaluation: the reduced gradient and loss [NPARAM_L]; else null
  unsigned* bar_count;
  int* err;
  int own_cap;           // parameters a CTA owns at most (its Adam state stays in shared memory)
};

struct TrainSmem {
  float W2[H * AP];  // W2[i][j] at i * AP + j
  float W1[2 * H], b1[H], b2[H], W3[2 * H], b3[2];
  float H1[TR_ROUND * AP], H2[TR_ROUND * AP], DZ1[TR_ROUND * AP], DZ2[TR_ROUND * AP];  // [q][unit]
  float X[TR_ROUND][2], TG[TR_ROUND][2], DY[TR_ROUND][2], L[TR_ROUND];
};

// Grid-wide barrier of a cooperative launch: the arrival counter only grows (the host zeroes it
// before the launch), so barrier b of the launch is passed once it reads G (b + 1); every CTA
// waits on the counter itself (no last-arriver broadcast).  False if the wait expired.
__device__ bool grid_barrier(const TrainArgs& a, unsigned target, int* s_ok) {
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    unsigned* count = (unsigned*)__cvta_generic_to_global(a.bar_count);
    // release: what this CTA's threads wrote before the __syncthreads above; acquire: what the others wrote
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
    const long long t0 = clock64();
    for (;;) {
      unsigned seen;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(count) : "memory");
      if (seen >= target) break;
      if (clock64() - t0 > kGridWaitCycles || *(volatile int*)a.err) {
        atomicExch(a.err, 1);
        ok = 0;
        break;
      }
    }
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

// --- warp-level TF32 MMA (m16n8k8, row-major A, column-major B, float32 accumulators) ---------
__device__ __forceinline__ uint32_t tf32_bits(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return r;
}

// x = hi + lo, both TF32 (10 explicit mantissa bits each): hi + lo carries about 21 bits
__device__ __forceinline__ void tf32_split(float x, uint32_t& hi, uint32_t& lo) {
  hi = tf32_bits(x);
  lo = tf32_bits(x - __uint_as_float(hi));
}

__device__ __forceinline__ void mma_tf32(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// d += A[m0:m0+16, k0:k0+8] B[k0:k0+8, n0:n0+8] with A(m, k) = A_at(m, k), B(k, n) = B_at(k, n).
// Three products of the split operands (lo hi, hi lo, hi hi; the lo lo term is below float32
// rounding).  Fragment layout of m16n8k8: lane = 4 g + t holds A rows g, g + 8 at columns t,
// t + 4, B rows t, t + 4 at column g, and D rows g, g + 8 at columns 2t, 2t + 1.
template <class FA, class FB>
__device__ __forceinline__ void mma3_tf32(float (&d)[4], FA A_at, FB B_at, int m0, int n0, int k0, int lane) {
  const int g = lane >> 2, t = lane & 3;
  const float av[4] = {A_at(m0 + g, k0 + t), A_at(m0 + g + 8, k0 + t), A_at(m0 + g, k0 + t + 4),
                       A_at(m0 + g + 8, k0 + t + 4)};
  const float bv[2] = {B_at(k0 + t, n0 + g), B_at(k0 + t + 4, n0 + g)};
  uint32_t ah[4], al[4], bh[2], bl[2];
#pragma unroll
  for (int i = 0; i < 4; ++i) tf32_split(av[i], ah[i], al[i]);
#pragma unroll
  for (int i = 0; i < 2; ++i) tf32_split(bv[i], bh[i], bl[i]);
  mma_tf32(d, al, bh);
  mma_tf32(d, ah, bl);
  mma_tf32(d, ah, bh);
}

// D fragment element r of a tile at (m0, n0): row and column
__device__ __forceinline__ int frag_row(int m0, int lane, int r) { return m0 + (lane >> 2) + (r >= 2 ? 8 : 0); }
__device__ __forceinline__ int frag_col(int n0, int lane, int r) { return n0 + 2 * (lane & 3) + (r & 1); }

__global__ void __launch_bounds__(TR_THREADS) train_kernel(TrainArgs a) {
  extern __shared__ __align__(16) unsigned char tr_smem[];
  TrainSmem& S = *reinterpret_cast<TrainSmem*>(tr_smem);
  __shared__ int s_ok;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = gridDim.x, c = blockIdx.x;
  // parameters this CTA reduces and updates
  const int k0 = (int)((int64_t)c * NPARAM_L / G), k1 = (int)((int64_t)(c + 1) * NPARAM_L / G);
  // their parameter values and Adam moments, read once per launch and written back at its end
  float* own_p = reinterpret_cast<float*>(tr_smem + sizeof(TrainSmem));
  float* own_m = own_p + a.own_cap;
  float* own_v = own_m + a.own_cap;
  const bool adam = a.grad_out == nullptr;
  if (adam) {
    for (int k = k0 + tid; k < k1 && k < NPARAM; k += TR_THREADS) {
      own_p[k - k0] = a.params[k];
      own_m[k - k0] = a.adam_m[k];
      own_v[k - k0] = a.adam_v[k];
    }
  }
  // this thread's CUDA-core gradient slot: W1 and b1, then b2, W3, b3 and the loss
  const int ks = tid < OW2 ? tid : tid + H * H;
  // MMA tiles: forward / backward (32 x 64 outputs, 16 tiles of 16 x 8): one per warp;
  // weight gradient (64 x 64, 32 tiles): two per warp
  const int fm = (warp >> 3) * 16, fn = (warp & 7) * 8;
  const int gm = (warp >> 2) * 16, gn = (warp & 3) * 16;
  auto load_round = [&](int r0, int cnt) {
    if (tid < TR_ROUND) {
      const bool live = tid < cnt;
      const int smp = r0 + tid;
      const float x0 = live ? a.x[2 * smp] : 0.f, x1 = live ? a.x[2 * smp + 1] : 0.f;
      const float t0 = live ? a.t[2 * smp] : 0.f, t1 = live ? a.t[2 * smp + 1] : 0.f;
      S.X[tid][0] = x0;
      S.X[tid][1] = x1;
      S.TG[tid][0] = t0;
      S.TG[tid][1] = t1;
    }
  };
  for (int s = 0; s < a.nsteps; ++s) {
    const int it = a.it0 + s;
    const int sidx = it % a.steps_per_epoch;
    const int off = sidx * a.batch;
    const int nb = min(a.batch, a.n - off);
    const float inv_n = a.inv_n > 0.f ? a.inv_n : 1.0f / (float)nb;
    // this CTA's samples of the batch
    const int s0 = off + (int)((int64_t)c * nb / G), s1 = off + (int)((int64_t)(c + 1) * nb / G);
    // 1. the first round's samples and the parameters into shared memory (parameters from L2:
    //    other CTAs updated them in the last step), every load of a thread before its first store
    {
      const float4* w2 = reinterpret_cast<const float4*>(a.params + OW2);
      const float4 wa = __ldcg(w2 + tid), wb = __ldcg(w2 + TR_THREADS + tid);
      float other = 0.f;
      if (tid < NOTHER) other = __ldcg(a.params + (tid < OW2 ? tid : tid + H * H));
      load_round(s0, min(TR_ROUND, s1 - s0));
      const int i0 = 4 * tid, i1 = 4 * (TR_THREADS + tid);
      *reinterpret_cast<float4*>(S.W2 + (i0 >> 6) * AP + (i0 & (H - 1))) = wa;
      *reinterpret_cast<float4*>(S.W2 + (i1 >> 6) * AP + (i1 & (H - 1))) = wb;
      if (tid < NOTHER) {
        const int k = tid < OW2 ? tid : tid + H * H;
        if (k < OB1) S.W1[k - OW1] = other;
        else if (k < OW2) S.b1[k - OB1] = other;
        else if (k < OW3) S.b2[k - OB2] = other;
        else if (k < OB3) S.W3[k - OW3] = other;
        else S.b3[k - OB3] = other;
      }
    }
    // the step's Adam scalars, ready before the first barrier
    const long long step = a.adam_step0 + s + 1;
    const float bc1 = 1.f - powf(a.b1, (float)step), bc2 = 1.f - powf(a.b2, (float)step);
    const float cosv = 0.5f * (1.f + cospif((float)it / (float)a.total));
    const float lr_t = a.lr * (0.01f + 0.99f * cosv);
    __syncthreads();
    float gw[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};  // dW2 tiles of this warp
    float gs = 0.f;                                                 // CUDA-core slot ks
    for (int r0 = s0; r0 < s1; r0 += TR_ROUND) {
      const int cnt = min(TR_ROUND, s1 - r0);
      // layer 1 (rows past cnt hold x = 0; their output gradients are zero below)
      for (int e = tid; e < TR_ROUND * H; e += TR_THREADS) {
        const int q = e >> 6, j = e & (H - 1);
        S.H1[q * AP + j] = tanhf(fmaf(S.W1[2 * j], S.X[q][0], fmaf(S.W1[2 * j + 1], S.X[q][1], S.b1[j])));
      }
      __syncthreads();
      // layer 2: Z2 = H1 W2^T (K = 64), H2 = tanh(Z2 + b2)
      {
        float d[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int kk = 0; kk < H; kk += 8)
          mma3_tf32(
              d, [&](int m, int k) { return S.H1[m * AP + k]; }, [&](int k, int n) { return S.W2[n * AP + k]; },
              fm, fn, kk, lane);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int q = frag_row(fm, lane, r), i = frag_col(fn, lane, r);
          S.H2[q * AP + i] = tanhf(d[r] + S.b2[i]);
        }
      }
      __syncthreads();
      // layer 3, loss and the output gradients (a warp per sample)
      for (int q = warp; q < TR_ROUND; q += TR_WARPS) {
        const float h2a = S.H2[q * AP + lane], h2b = S.H2[q * AP + lane + 32];
        float y0 = fmaf(S.W3[lane], h2a, S.W3[lane + 32] * h2b);
        float y1 = fmaf(S.W3[H + lane], h2a, S.W3[H + lane + 32] * h2b);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          y0 += __shfl_xor_sync(0xffffffffu, y0, o);
          y1 += __shfl_xor_sync(0xffffffffu, y1, o);
        }
        y0 += S.b3[0];
        y1 += S.b3[1];
        const bool live = q < cnt;
        const float e0 = y0 - S.TG[q][0], e1 = y1 - S.TG[q][1];
        const float d0 = live ? e0 * inv_n : 0.f, d1 = live ? e1 * inv_n : 0.f;
        S.DZ2[q * AP + lane] = fmaf(S.W3[lane], d0, S.W3[H + lane] * d1) * (1.f - h2a * h2a);
        S.DZ2[q * AP + lane + 32] = fmaf(S.W3[lane + 32], d0, S.W3[H + lane + 32] * d1) * (1.f - h2b * h2b);
        if (lane == 0) {
          S.DY[q][0] = d0;
          S.DY[q][1] = d1;
          S.L[q] = live ? 0.5f * (e0 * e0 + e1 * e1) * inv_n : 0.f;
        }
      }
      __syncthreads();
      // backward through layer 2: dH1 = dZ2 W2 (K = 64), dZ1 = dH1 (1 - H1^2)
      {
        float d[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int kk = 0; kk < H; kk += 8)
          mma3_tf32(
              d, [&](int m, int k) { return S.DZ2[m * AP + k]; }, [&](int k, int n) { return S.W2[k * AP + n]; },
              fm, fn, kk, lane);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int q = frag_row(fm, lane, r), j = frag_col(fn, lane, r);
          const float h = S.H1[q * AP + j];
          S.DZ1[q * AP + j] = d[r] * (1.f - h * h);
        }
      }
      // weight gradient dW2 += dZ2^T H1 (K = the round's 32 samples)
#pragma unroll
      for (int tt = 0; tt < 2; ++tt) {
#pragma unroll
        for (int kk = 0; kk < TR_ROUND; kk += 8)
          mma3_tf32(
              gw[tt], [&](int m, int k) { return S.DZ2[k * AP + m]; },
              [&](int k, int n) { return S.H1[k * AP + n]; }, gm, gn + 8 * tt, kk, lane);
      }
      __syncthreads();
      // 2. the CUDA-core gradient slots over this round's samples
      if (tid < NSIMT) {
        const int k = ks;
        float v = 0.f;
        if (k < OB1) {
          const int j = (k - OW1) >> 1, cc = (k - OW1) & 1;
          for (int q = 0; q < cnt; ++q) v = fmaf(S.DZ1[q * AP + j], S.X[q][cc], v);
        } else if (k < OW2) {
          for (int q = 0; q < cnt; ++q) v += S.DZ1[q * AP + (k - OB1)];
        } else if (k < OW3) {
          for (int q = 0; q < cnt; ++q) v += S.DZ2[q * AP + (k - OB2)];
        } else if (k < OB3) {
          const int o = (k - OW3) / H, i = (k - OW3) % H;
          for (int q = 0; q < cnt; ++q) v = fmaf(S.DY[q][o], S.H2[q * AP + i], v);
        } else if (k < NPARAM) {
          for (int q = 0; q < cnt; ++q) v += S.DY[q][k - OB3];
        } else {
          for (int q = 0; q < cnt; ++q) v += S.L[q];
        }
        gs += v;
      }
      __syncthreads();
      if (r0 + TR_ROUND < s1) {
        load_round(r0 + TR_ROUND, min(TR_ROUND, s1 - r0 - TR_ROUND));
        __syncthreads();
      }
    }
    float* prow = a.partial + (int64_t)c * NPARAM_L;
    if (tid < NSIMT) prow[ks] = gs;
#pragma unroll
    for (int tt = 0; tt < 2; ++tt)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int i = frag_row(gm, lane, r), j = frag_col(gn + 8 * tt, lane, r);
        prow[OW2 + i * H + j] = gw[tt][r];
      }
    if (!grid_barrier(a, (unsigned)G * (unsigned)(2 * s + 1), &s_ok)) return;
    // 3. this CTA's parameters: lane l of warp w adds the partials of parameter kb + l of the
    //    CTAs w, w + 16, ...; warp 0 adds the 16 warp sums in warp order, then Adam (or the
    //    gradient out)
    auto apply = [&](int k, float g) {
      if (!adam) {
        a.grad_out[k] = g;
      } else if (k < NPARAM) {
        const int i = k - k0;
        const float mk = a.b1 * own_m[i] + (1.f - a.b1) * g;
        const float vk = a.b2 * own_v[i] + (1.f - a.b2) * g * g;
        own_m[i] = mk;
        own_v[i] = vk;
        const float pk = own_p[i] - lr_t * (mk / bc1) / (sqrtf(vk / bc2) + a.eps);
        own_p[i] = pk;
        a.params[k] = pk;
      }
    };
    float* wsum = S.H2;  // [TR_WARPS][32] (the activations are dead until the next step)
    for (int kb = k0; kb < k1; kb += 32) {
      const int k = kb + lane;
      float g = 0.f;
      if (k < k1) {
        // (ten rows at a time, all of them in flight: one trip to L2 for 152 CTAs)
        for (int c0 = warp; c0 < G; c0 += 10 * TR_WARPS) {
          float v[10];
#pragma unroll
          for (int u = 0; u < 10; ++u) {
            const int cc = c0 + u * TR_WARPS;
            v[u] = cc < G ? __ldcg(a.partial + (int64_t)cc * NPARAM_L + k) : 0.f;
          }
#pragma unroll
          for (int u = 0; u < 10; ++u)
            if (c0 + u * TR_WARPS < G) g += v[u];
        }
      }
      wsum[warp * 32 + lane] = g;
      __syncthreads();
      if (warp == 0 && k < k1) {
        float tot = 0.f;
#pragma unroll
        for (int w = 0; w < TR_WARPS; ++w) tot += wsum[w * 32 + lane];
        apply(k, tot);
      }
      __syncthreads();
    }
    if (!grid_barrier(a, (unsigned)G * (unsigned)(2 * s + 2), &s_ok)) return;
  }
  if (adam) {
    for (int k = k0 + tid; k < k1 && k < NPARAM; k += TR_THREADS) {
      a.adam_m[k] = own_m[k - k0];
      a.adam_v[k] = own_v[k - k0];
    }
  }
}

__global__ void to_half_kernel(const float* __restrict__ p, __half* __restrict__ h) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < NPARAM) h[k] = __float2half_rn(p[k]);
}

// ---------------------------------------------------------------------------
// inference (float16 weights, float32 accumulation)
// ---------------------------------------------------------------------------
__device__ inline void mlp_eval_half(const __half* __restrict__ P, float x0, float x1, float* y0, float* y1) {
  float h1[H];
#pragma unroll
  for (int j = 0; j < H; ++j)
    h1[j] = tanhf(fmaf(__half2float(P[OW1 + 2 * j]), x0, fmaf(__half2float(P[OW1 + 2 * j + 1]), x1,
                                                                 __half2float(P[OB1 + j]))));
  float a0 = __half2float(P[OB3]), a1 = __half2float(P[OB3 + 1]);
  for (int i = 0; i < H; ++i) {
    float z = __half2float(P[OB2 + i]);
#pragma unroll
    for (int j = 0; j < H; ++j) z = fmaf(__half2float(P[OW2 + H * i + j]), h1[j], z);
    const float h2 = tanhf(z);
    a0 = fmaf(__half2float(P[OW3 + i]), h2, a0);
    a1 = fmaf(__half2float(P[OW3 + H + i]), h2, a1);
  }
  *y0 = a0;
  *y1 = a1;
}

__global__ void forward_kernel(const __half* __restrict__ params16, const float* __restrict__ x, int n,
                               float* __restrict__ y) {
  __shared__ __half P[NPARAM];
  for (int i = threadIdx.x; i < NPARAM; i += blockDim.x) P[i] = params16[i];
  __syncthreads();
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  float y0, y1;
  mlp_eval_half(P, x[2 * s], x[2 * s + 1], &y0, &y1);
  y[2 * s] = y0;
  y[2 * s + 1] = y1;
}

// K^[r][b] for every sine source term r and lam band b (log-spaced band centres).
__global__ void band_table_kernel(const __half* __restrict__ params16, TermsW T, int NB, double loglo,
                                  double logstep, double dT, double* __restrict__ Ktab) {
  __shared__ __half P[NPARAM];
  for (int i = threadIdx.x; i < NPARAM; i += blockDim.x) P[i] = params16[i];
  __syncthreads();
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= T.R * NB) return;
  const int r = idx / NB, b = idx % NB;
  double Kre = 0.0, Kim = 0.0;
  if (T.is_sin[r]) {
    const double w = T.omega[r];
    const double ll = loglo + logstep * (double)b;  // log(lam dT)
    const double ldt = exp(ll);
    const double wd = w * dT;
    float y0, y1;
    mlp_eval_half(P, (float)(ll / 6.0), (float)(wd - 1.0), &y0, &y1);
    const double unscale = (dT * wd * wd) / (4.0 * (1.0 + ldt));
    Kre = (double)y0 * unscale;
    Kim = (double)y1 * unscale;
  }
  Ktab[2 * idx] = Kre;
  Ktab[2 * idx + 1] = Kim;
}

// ---------------------------------------------------------------------------
// batched form: band tables of every problem of a batch, jobs flattened through
// per-problem prefix tables (the owner of job e is the problem with the largest prefix <= e)
// ---------------------------------------------------------------------------
__device__ inline int job_owner(const int64_t* __restrict__ prefix, int P, int64_t e) {
  int lo = 0, hi = P - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (prefix[mid] <= e) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

__global__ void b_band_table_kernel(const __half* __restrict__ params16, const BProb* __restrict__ probs,
                                    const pe_term* __restrict__ terms, const int64_t* __restrict__ prefix, int P,
                                    int64_t total, int NB, double* __restrict__ Kt) {
  __shared__ __half Ps[NPARAM];
  for (int i = threadIdx.x; i < NPARAM; i += blockDim.x) Ps[i] = params16[i];
  __syncthreads();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= total) return;
  const int p = job_owner(prefix, P, e);
  const BProb& B = probs[p];
  const int64_t le = e - prefix[p];
  const int r = (int)(le / NB), band = (int)(le % NB);
  const pe_term& t = terms[B.tf + r];
  double Kre = 0.0, Kim = 0.0;
  if (t.tkind == PE_T_SIN) {
    const double w = t.tp[0];
    const double ll = B.lloglo + B.lstep * (double)band;  // log(lam dT)
    const double wd = w * B.dT;
    float y0, y1;
    mlp_eval_half(Ps, (float)(ll / 6.0), (float)(wd - 1.0), &y0, &y1);
    const double unscale = (B.dT * wd * wd) / (4.0 * (1.0 + exp(ll)));
    Kre = (double)y0 * unscale;
    Kim = (double)y1 * unscale;
  }
  Kt[B.oKt + 2 * le] = Kre;
  Kt[B.oKt + 2 * le + 1] = Kim;
}

}  // namespace

pe_status batch_learned_tables(pe_batch* b, cudaStream_t st) {
  if (!b->mlp) return PE_OK;
  if (b->kt_jobs > 0)
    b_band_table_kernel<<<(unsigned)((b->kt_jobs + 127) / 128), 128, 0, st>>>(
        (const __half*)b->mlp->params16, b->d_probs, b->d_terms, b->d_kt_prefix, b->P, b->kt_jobs,
        kBatchLearnedBands, b->Kt);
  b->launches += 1;
  PE_CUDA_TRY(cudaGetLastError());
  return PE_OK;
}

// ---------------------------------------------------------------------------
// host API
// ---------------------------------------------------------------------------
extern "C" pe_status pe_mlp_create(pe_mlp** out, uint64_t seed) {
  if (!out) return pe_fail(PE_EINVAL, "pe_mlp_create: out is NULL");
  *out = nullptr;
  pe_mlp* m = new (std::nothrow) pe_mlp();
  if (!m) return pe_fail(PE_ENOMEM, "pe_mlp_create: host allocation failed");
  // Xavier-uniform initial weights from SplitMix64, zero biases
  std::vector<float> p(NPARAM, 0.f);
  uint64_t st = seed;
  auto uni = [&st]() {
    st += 0x9E3779B97F4A7C15ull;
    uint64_t z = st;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return (double)(z >> 11) * (1.0 / 9007199254740992.0);
  };
  auto fill = [&](int off, int fan_in, int fan_out, int count) {
    const double a = sqrt(6.0 / (double)(fan_in + fan_out));
    for (int i = 0; i < count; ++i) p[off + i] = (float)((2.0 * uni() - 1.0) * a);
  };
  fill(OW1, 2, H, 2 * H);
  fill(OW2, H, H, H * H);
  fill(OW3, H, 2, 2 * H);
  pe_status s = PE_OK;
  auto al = [&s](void** ptr, size_t bytes) {
    if (s != PE_OK) return;
    if (cudaMalloc(ptr, bytes) != cudaSuccess) {
      cudaGetLastError();
      s = pe_fail(PE_ENOMEM, "pe_mlp_create: cudaMalloc failed");
    }
  };
  al((void**)&m->params, sizeof(float) * NPARAM);
  al((void**)&m->params16, sizeof(__half) * NPARAM);
  al((void**)&m->grad, sizeof(float) * NPARAM_L);
  al((void**)&m->sync, sizeof(unsigned) * 4);
  al((void**)&m->adam_m, sizeof(float) * NPARAM);
  al((void**)&m->adam_v, sizeof(float) * NPARAM);
  al((void**)&m->loss_dev, sizeof(float));
  if (s == PE_OK) {
    cudaMemcpy(m->params, p.data(), sizeof(float) * NPARAM, cudaMemcpyHostToDevice);
    cudaMemset(m->adam_m, 0, sizeof(float) * NPARAM);
    cudaMemset(m->adam_v, 0, sizeof(float) * NPARAM);
    to_half_kernel<<<(NPARAM + 255) / 256, 256>>>(m->params, (__half*)m->params16);
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) s = pe_cuda_fail(e, "pe_mlp_create");
  }
  if (s != PE_OK) {
    pe_mlp_destroy(m);
    return s;
  }
  *out = m;
  return PE_OK;
}

extern "C" void pe_mlp_destroy(pe_mlp* m) {
  if (!m) return;
  void* ptrs[] = {m->params, m->params16, m->grad, m->adam_m, m->adam_v, m->loss_dev, m->partial, m->sync};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  delete m;
}

extern "C" int32_t pe_mlp_num_params(void) { return NPARAM; }

// One launch of the persistent training kernel: nsteps steps from step index it0 of a schedule
// of `total` steps over epochs of steps_per_epoch batches (grad_out != null: one gradient
// evaluation of the whole range, no update).
static pe_status run_train(pe_mlp* m, const float* x, const float* t, int n, int batch, int steps_per_epoch,
                           int total, int it0, int nsteps, float lr, float inv_n, float* grad_out,
                           cudaStream_t st) {
  int dev = 0, sms = 0, coop = 0;
  PE_CUDA_TRY(cudaGetDevice(&dev));
  PE_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  PE_CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
  if (!coop) return pe_fail(PE_ECUDA, "pe_mlp: the device does not support cooperative launches");
  const int own_cap = (NPARAM_L + sms - 1) / sms + 1;
  const size_t smem = sizeof(TrainSmem) + 3 * sizeof(float) * (size_t)own_cap;
  if (smem > 200 * 1024) return pe_fail(PE_ECUDA, "pe_mlp: too few SMs for the training kernel");
  PE_TRY(allow_smem((const void*)train_kernel, smem));
  int per_sm = 0;
  PE_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, train_kernel, TR_THREADS, smem));
  if (per_sm < 1) return pe_fail(PE_ECUDA, "pe_mlp: the training kernel does not fit an SM");
  const int G = sms;  // one CTA per SM: all co-resident, as the grid barriers need
  if (m->partial_cap < G) {
    if (m->partial) cudaFree(m->partial);
    m->partial = nullptr;
    m->partial_cap = 0;
    if (cudaMalloc((void**)&m->partial, sizeof(float) * (size_t)NPARAM_L * G) != cudaSuccess) {
      cudaGetLastError();
      return pe_fail(PE_ENOMEM, "pe_mlp: partial-gradient allocation failed");
    }
    m->partial_cap = G;
  }
  PE_CUDA_TRY(cudaMemsetAsync(m->sync, 0, 3 * sizeof(unsigned), st));  // barrier count, (unused), error
  TrainArgs a{};
  a.params = m->params;
  a.adam_m = m->adam_m;
  a.adam_v = m->adam_v;
  a.partial = m->partial;
  a.x = x;
  a.t = t;
  a.n = n;
  a.batch = batch;
  a.steps_per_epoch = steps_per_epoch;
  a.total = total;
  a.it0 = it0;
  a.nsteps = nsteps;
  a.lr = lr;
  a.b1 = 0.9f;
  a.b2 = 0.999f;
  a.eps = 1e-8f;
  a.adam_step0 = m->step;
  a.inv_n = inv_n;
  a.grad_out = grad_out;
  a.bar_count = m->sync;
  a.err = (int*)(m->sync + 2);
  a.own_cap = own_cap;
  void* args[] = {&a};
  PE_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)train_kernel, dim3(G), dim3(TR_THREADS), args, smem, st));
  PE_CUDA_TRY(cudaGetLastError());
  unsigned herr = 0;
  PE_CUDA_TRY(cudaMemcpyAsync(&herr, m->sync + 2, sizeof(unsigned), cudaMemcpyDeviceToHost, st));
  PE_CUDA_TRY(cudaStreamSynchronize(st));
  if (herr) return pe_fail(PE_ETIMEOUT, "pe_mlp: a grid barrier of the training kernel expired");
  if (!grad_out) m->step += nsteps;
  return PE_OK;
}

extern "C" pe_status pe_mlp_gradient(pe_mlp* m, const float* x, const float* t, int32_t n, float* grad_out,
                                     float* loss_out) {
  if (!m || !x || !t || n < 1) return pe_fail(PE_EINVAL, "pe_mlp_gradient: bad arguments");
  PE_TRY(run_train(m, x, t, n, n, 1, 1, 0, 1, 0.f, 1.0f / (float)n, m->grad, nullptr));
  if (grad_out) PE_CUDA_TRY(cudaMemcpy(grad_out, m->grad, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost));
  if (loss_out) PE_CUDA_TRY(cudaMemcpy(loss_out, m->grad + NPARAM, sizeof(float), cudaMemcpyDeviceToHost));
  return PE_OK;
}

// steps per launch of the persistent kernel (about 0.1 s each)
constexpr int kTrainStepsPerLaunch = 16384;

extern "C" pe_status pe_mlp_train(pe_mlp* m, const float* x, const float* t, int32_t n, int32_t epochs,
                                  int32_t batch, float lr, float* final_loss) {
  if (!m || !x || !t || n < 1 || epochs < 1 || batch < 1) return pe_fail(PE_EINVAL, "pe_mlp_train: bad arguments");
  const int steps_per_epoch = (n + batch - 1) / batch;
  const int64_t total64 = (int64_t)epochs * steps_per_epoch;
  if (total64 > (int64_t)1 << 30) return pe_fail(PE_EINVAL, "pe_mlp_train: too many steps");
  const int total = (int)total64;
  for (int it = 0; it < total; it += kTrainStepsPerLaunch)
    PE_TRY(run_train(m, x, t, n, batch, steps_per_epoch, total, it, std::min(kTrainStepsPerLaunch, total - it), lr,
                     0.f, nullptr, nullptr));
  // mean loss of the final parameters over every sample
  PE_TRY(run_train(m, x, t, n, n, 1, 1, 0, 1, 0.f, 1.0f / (float)n, m->grad, nullptr));
  float last = 0.f;
  PE_CUDA_TRY(cudaMemcpy(&last, m->grad + NPARAM, sizeof(float), cudaMemcpyDeviceToHost));
  to_half_kernel<<<(NPARAM + 255) / 256, 256>>>(m->params, (__half*)m->params16);
  PE_CUDA_TRY(cudaDeviceSynchronize());
  if (final_loss) *final_loss = last;
  return PE_OK;
}

extern "C" pe_status pe_mlp_forward(pe_mlp* m, const float* x, int32_t n, float* y) {
  if (!m || !x || !y || n < 1) return pe_fail(PE_EINVAL, "pe_mlp_forward: bad arguments");
  forward_kernel<<<(n + 127) / 128, 128>>>((const __half*)m->params16, x, n, y);
  PE_CUDA_TRY(cudaGetLastError());
  PE_CUDA_TRY(cudaDeviceSynchronize());
  return PE_OK;
}

extern "C" pe_status pe_mlp_get_params(pe_mlp* m, float* out) {
  if (!m || !out) return pe_fail(PE_EINVAL, "pe_mlp_get_params: NULL argument");
  PE_CUDA_TRY(cudaMemcpy(out, m->params, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost));
  return PE_OK;
}

extern "C" pe_status pe_mlp_set_params(pe_mlp* m, const float* in) {
  if (!m || !in) return pe_fail(PE_EINVAL, "pe_mlp_set_params: NULL argument");
  PE_CUDA_TRY(cudaMemcpy(m->params, in, sizeof(float) * NPARAM, cudaMemcpyHostToDevice));
  to_half_kernel<<<(NPARAM + 255) / 256, 256>>>(m->params, (__half*)m->params16);
  PE_CUDA_TRY(cudaDeviceSynchronize());
  return PE_OK;
}

extern "C" pe_status pe_learned_samples(pe_ctx* c, int32_t n, const double* lam, const double* omega, float* x,
                                        float* y, double* K) {
  if (!c || n < 1 || !lam || !omega || !x || !y) return pe_fail(PE_EINVAL, "pe_learned_samples: bad arguments");
  Lag LF{}, LG{};
  Nodes8 cF{}, cG{};
  for (int i = 0; i < PE_MAX_S; ++i) {
    cF.c[i] = c->cF[i];
    cG.c[i] = c->cG[i];
    for (int k = 0; k < PE_MAX_S; ++k) {
      LF.a[i][k] = c->lagF[i][k];
      LG.a[i][k] = c->lagG[i][k];
    }
  }
  samples_kernel<<<(n + 127) / 128, 128, 0, c->stream>>>(n, lam, omega, c->dT, c->M, c->q, c->p, LF, LG, cF, cG, x,
                                                          y, K);
  PE_CUDA_TRY(cudaGetLastError());
  PE_CUDA_TRY(cudaStreamSynchronize(c->stream));
  return PE_OK;
}

extern "C" pe_status pe_set_learned(pe_ctx* c, const pe_mlp* m) {
  if (!c) return pe_fail(PE_EINVAL, "pe_set_learned: ctx is NULL");
  drop_solve_graphs(c);
  c->mlp = m;
  return PE_OK;
}

// Called by pe_set_problem before the column weights, which take the table in.
pe_status launch_learned_tables(pe_ctx* c, LearnedTerms* L) {
  if (!c->mlp) return pe_fail(PE_ESTATE, "learned G: no network attached");
  if (!c->Ktab) {
    if (cudaMalloc((void**)&c->Ktab, sizeof(double) * 2 * PE_MAX_TERMS * PE_LEARNED_BANDS) != cudaSuccess) {
      cudaGetLastError();
      return pe_fail(PE_ENOMEM, "learned G: band table allocation failed");
    }
  }
  TermsW T{};
  T.R = c->R;
  for (int r = 0; r < c->R; ++r) {
    T.is_sin[r] = c->terms[r].tkind == PE_T_SIN ? 1 : 0;
    T.omega[r] = c->terms[r].tp[0];
    T.phase[r] = c->terms[r].tp[1];
    T.amp[r] = c->terms[r].amp;
  }
  // band range: the closed-form extremes of lam on this grid (slowest and fastest mode)
  double lmin = 0.0, lmax = 0.0;
  for (int a = 0; a < c->gn.d; ++a) {
    const int n = c->gn.n[a];
    auto ratio = [&](int j) {
      const double th = M_PI * (double)j / (double)(n + 1);
      const double sh = sin(0.5 * th);
      return ((4.0 / c->h[a]) * sh * sh) / ((c->h[a] / 3.0) * (2.0 + cos(th)));
    };
    lmin += ratio(1);
    lmax += ratio(n);
  }
  lmin *= c->D;
  lmax *= c->D;
  const int NB = PE_LEARNED_BANDS;
  const double loglo = log(lmin * c->dT) - 1e-6, loghi = log(lmax * c->dT) + 1e-6;
  const double step = (loghi - loglo) / (double)(NB - 1);
  band_table_kernel<<<(c->R * NB + 127) / 128, 128, 0, c->stream>>>((const __half*)c->mlp->params16, T, NB, loglo,
                                                                     step, c->dT, c->Ktab);
  c->launches += 1;
  PE_CUDA_TRY(cudaGetLastError());
  L->NB = NB;
  L->loglo = loglo;
  L->logstep = step;
  L->dT = c->dT;
  L->Ktab = c->Ktab;
  return PE_OK;
}
