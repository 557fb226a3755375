// Tensor-core engine of the mixed-precision fine sweep (pe_options.fine_engine = PE_FINE_TC).
//
// The forced part of the fine propagator over one slice n (the EIFE stage recurrence of
// Sec. 3 with its stage columns contracted) is, per mode J,
//   w_{m+1} = E_F w_m + a_m,   a_m = sum_k W[k][J] Y_n[m][k],   m = 0..M-1,   w_0 = 0,
// and F^M(U^n)_J = exp(-lam_J M dt) U^n_J + w_M.  For a tile of 128 modes and a group of G
// slices the inputs a_m of all G*M substeps form one dense contraction
//   D[J][s*M + m] = sum_k W[k][J] Y_{gG+s}[m][k]        (128 x NR, NR = G*M <= 256, K <= 64),
// which runs on the 5th-generation tensor cores: both operands are split into three
// bfloat16 terms x = x0 + x1 + x2 (about 24 bits together) and the six products whose
// weight is at least 2^-24 (x0y0, x0y1, x1y0, x0y2, x1y1, x2y0) are accumulated in float32
// in tensor memory, the five small ones first.  The recurrence (hi/lo E_F, float32) and
// the float64 homogeneous term then run per mode on the CUDA cores from tcgen05.ld rows.
//
// Kernel roles (one persistent CTA per SM, 288 threads, items = (slice group, mode tile)
// pairs, group-major, a contiguous range per CTA):
//   * warps 0-7 (two warpgroups): the epilogue of each item: wait for its accumulator,
//     read rows with tcgen05.ld, 32 substeps of two slices per read (warp w reads TMEM lanes
//     32 (w % 4) ..; warpgroup h takes the slices h, h + 2, ... of the group), run the
//     recurrence four substeps per step, write F; the next item's epilogue inputs are
//     loaded meanwhile;
//   * warp 8, one thread: bulk copies of the split operands, both prepared once per problem
//     in global memory in the exact shared-memory layout (the time factors of the current
//     slice group; the stage weights of each item's mode tile, a ring of three), and the
//     tcgen05.mma issue into one of two accumulators (2 x NR TMEM columns), released by
//     tcgen05.commit.
// Every mbarrier wait is bounded; on expiry the CTA records an error code, writes a NaN
// into the first output value (so that the Parareal residual reports it), frees its
// tensor memory and exits.
#include <cuda_bf16.h>

#include <algorithm>
#include <mutex>

#include "pe_batch.h"
#include "pe_internal.h"
#include "pe_tc_common.cuh"

namespace {

constexpr int FT_ROWS = 128;                 // modes of a tile (TMEM lanes)
constexpr int FT_WORKERS = 256;              // warps 0-7: two warpgroups
constexpr int FT_THREADS = FT_WORKERS + 32;  // + warp 8 (copies and MMA issue)
constexpr int FT_CHUNK = 16 * 1024;          // bytes per bulk copy instruction
constexpr int FT_MIN_SMEM = 120 * 1024;      // at most one CTA per SM (its TMEM allocation)
constexpr int FT_ABUF = 3;                   // ring of A-operand tiles

// rows of the B operand (G*M) a K padding allows, and the shared-memory budget
__host__ __device__ constexpr int ft_rows_max(int KP) { return KP <= 32 ? 256 : 128; }
__host__ __device__ constexpr int ft_a_bytes(int KP) { return 3 * FT_ROWS * KP * 2; }
__host__ __device__ constexpr int ft_smem_bytes(int KP) {
  return std::max(1024 + 3 * ft_rows_max(KP) * KP * 2 + FT_ABUF * ft_a_bytes(KP), FT_MIN_SMEM);
}

// Operand images use the swizzled K-major layout whose swizzle width equals a row of KP
// bfloat16 (32, 64 or 128 bytes): row r of a term at r * KP * 2 bytes, its 16-byte chunk c
// stored at chunk c ^ ((byte offset >> 7) & (KP / 8 - 1)) (address bits 4.. XOR bits 7..),
// so that the tensor core reads whole rows without bank conflicts.  Terms start on
// 1024-byte boundaries, as the pattern requires.
__host__ __device__ constexpr int ft_kpad(int K) { return K <= 16 ? 16 : (K <= 32 ? 32 : 64); }
__device__ __forceinline__ int64_t ft_swz(int64_t off, int KP) {
  return off ^ (((off >> 7) & (KP / 8 - 1)) << 4);
}
// shared-memory descriptor of a swizzled K-major operand: start address, stride between
// 8-row groups (8 rows of KP * 2 bytes), version 1, layout type 6 / 4 / 2 (32 / 64 / 128-byte
// swizzle); the leading offset is not used by these layouts
__device__ __forceinline__ uint64_t smem_desc_swz(uint32_t saddr, int KP) {
  const uint32_t sbo = 8u * (uint32_t)KP * 2u;
  const uint64_t layout = KP == 16 ? 6 : (KP == 32 ? 4 : 2);
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)((sbo & 0x3FFFFu) >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= layout << 61;
  return d;
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
      "%14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
#pragma unroll
  for (int e = 0; e < 16; ++e) v[e] = __uint_as_float(r[e]);
}
// hi + lo pair squared in float32 arithmetic (a double-float product: the low word collects
// the exact rounding error of hi * hi from an FMA and the cross term 2 hi lo; about 2^-44
// relative)
__device__ __forceinline__ void df_square(float h, float l, float& oh, float& ol) {
  const float p = h * h;
  float e = fmaf(h, h, -p);
  e = fmaf(2.f * h, l, e);
  oh = p + e;
  ol = e - (oh - p);
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
#pragma unroll
  for (int e = 0; e < 32; ++e) v[e] = __uint_as_float(r[e]);
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Three bfloat16 terms of eight consecutive values (x = t0 + t1 + t2 up to about 2^-24
// relative), each packed as one 16-byte core-matrix row.
__device__ __forceinline__ void split8(const float (&x)[8], uint4 (&o)[3]) {
  uint32_t pk[3][4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    float r0 = x[2 * e], r1 = x[2 * e + 1];
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(r0, r1);  // .x = r0 (low half)
      pk[t][e] = *reinterpret_cast<const uint32_t*>(&h);
      r0 -= __low2float(h);
      r1 -= __high2float(h);
    }
  }
#pragma unroll
  for (int t = 0; t < 3; ++t) o[t] = make_uint4(pk[t][0], pk[t][1], pk[t][2], pk[t][3]);
}


// ---------------------------------------------------------------------------
// Batched form: the same engine over the work items (problem p, slice group g, mode tile t)
// of many problems at once, one persistent launch per column padding KP.  Each item reads
// its problem's record (sizes, slice-group shape NR = TG * M, arena offsets); the B operand
// (the group's split time factors) is reloaded when (p, g) changes, the A operand (the tile's
// split stage weights) every item through the same ring; the MMA instruction takes the item's
// N = NR.  Items of converged problems run too (the batched correction leaves those problems
// unchanged), which keeps both pipeline sides' item sequences fixed inside the captured graph.
// ---------------------------------------------------------------------------
struct BtcArgs {
  const BProb* probs;
  const BTcItem* items;
  int64_t n_items;
  const float* coefF32;  // arena: E_hi, E_lo at oCF
  const double* coefF;   // arena: exp(-lam M dt) at oCF + (q + 1) ndof
  const double* U;       // arena at oU
  double* Fbar;          // arena at oS
  const unsigned char* A;
  const unsigned char* B;
  int* err;
};

template <int KP>
__global__ void __launch_bounds__(FT_THREADS, 1) b_fine_tc_kernel(BtcArgs a) {
  constexpr int A_TERM = FT_ROWS * KP * 2;
  constexpr int A_BYTES = 3 * A_TERM;
  constexpr int NRMAX = ft_rows_max(KP);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t fullA[FT_ABUF], emptyA[FT_ABUF], fullD[2], emptyD[2], fullB, freeB, drain;
  __shared__ uint32_t tmem_slot;
  __shared__ int s_fail;
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  unsigned char* sB = smem;
  unsigned char* sA = smem + 3 * NRMAX * KP * 2;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int64_t i0 = (int64_t)blockIdx.x * a.n_items / gridDim.x;
  const int64_t i1 = (int64_t)(blockIdx.x + 1) * a.n_items / gridDim.x;
  constexpr uint32_t ncols = 2 * NRMAX;  // 512 or 256: a power of two
  volatile int* fail = &s_fail;
  auto set_fail = [&](int code) {
    atomicExch(a.err, code);
    *fail = 1;
    a.Fbar[0] = __longlong_as_double(0x7ff8000000000000LL);
  };
  if (tid == 0) {
    for (int b = 0; b < FT_ABUF; ++b) {
      mbar_init(&fullA[b], 1);
      mbar_init(&emptyA[b], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&fullD[b], 1);
      mbar_init(&emptyD[b], FT_WORKERS / 32);
    }
    mbar_init(&fullB, 1);
    mbar_init(&freeB, 1);
    mbar_init(&drain, 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == FT_WORKERS / 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;

  if (warp < FT_WORKERS / 32) {
    const int r = tid & (FT_ROWS - 1), h = tid >> 7, lane = tid & 31;
    struct Pre {
      float eh, el;
      double em;
    };
    Pre P0, P1;
    auto load_epi = [&](Pre& P, int64_t i) {
      const BTcItem it = a.items[i];
      const BProb& B = a.probs[it.p];
      const int64_t nd = B.g.ndof, J = it.t * FT_ROWS + r;
      const bool ok = J < nd;
      P.eh = ok ? a.coefF32[B.oCF + J] : 0.f;
      P.el = ok ? a.coefF32[B.oCF + nd + J] : 0.f;
      P.em = ok ? a.coefF[B.oCF + (int64_t)(B.q + 1) * nd + J] : 0.0;
    };
    auto step = [&](int64_t i, const Pre& cur, Pre& nxt) -> bool {
      const int j = (int)(i - i0);
      if (i + 1 < i1) load_epi(nxt, i + 1);
      const BTcItem it = a.items[i];
      const BProb& B = a.probs[it.p];
      const int M = B.M, TG = B.TG, N = B.N;
      const int64_t nd = B.g.ndof;
      const int64_t J = it.t * FT_ROWS + r;
      const bool ok = J < nd;
      // U^n loaded ahead, as in the single-problem kernel: the first pair's before the wait
      auto load_u = [&](int s) -> double {
        const int64_t n = (int64_t)it.g * TG + s;
        return (ok && s < TG && n < N) ? a.U[B.oU + n * nd + J] : 0.0;
      };
      double u0 = load_u(h), u1 = load_u(h + 2);
      if (!mbar_wait(&fullD[j & 1], (uint32_t)((j >> 1) & 1))) {
        set_fail(5);
        return false;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      float e2h, e2l, e4h, e4l;
      df_square(cur.eh, cur.el, e2h, e2l);
      df_square(e2h, e2l, e4h, e4l);
      const float eh = cur.eh, e2 = e2h, e3 = e2h * eh;
      const uint32_t row = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((j & 1) * NRMAX);
      auto chain4 = [&](float& w, float x0, float x1, float x2, float x3) {
        const float bsum = fmaf(e3, x0, fmaf(e2, x1, fmaf(eh, x2, x3)));
        w = fmaf(e4h, w, fmaf(e4l, w, bsum));
      };
      auto finish = [&](double u, int s, float w) {
        const int64_t n = (int64_t)it.g * TG + s;
        if (ok && n < N) a.Fbar[B.oS + n * nd + J] = fma(cur.em, u, (double)w);
      };
#pragma unroll 1
      for (int pq = 0; pq < 8; ++pq) {
        const int s0 = h + 4 * pq, s1 = s0 + 2;
        if (s0 >= TG) break;
        const bool two = s1 < TG;
        const double n0 = load_u(s0 + 4), n1 = load_u(s1 + 4);
        float w0 = 0.f, w1 = 0.f;
        int m0 = 0;
        for (; m0 + 32 <= M; m0 += 32) {
          float v0[32], v1[32];
          tmem_ld32(row + (uint32_t)(s0 * M + m0), v0);
          if (two) tmem_ld32(row + (uint32_t)(s1 * M + m0), v1);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 32; e += 4) {
            chain4(w0, v0[e], v0[e + 1], v0[e + 2], v0[e + 3]);
            if (two) chain4(w1, v1[e], v1[e + 1], v1[e + 2], v1[e + 3]);
          }
        }
        if (m0 < M) {
          float v0[16], v1[16];
          tmem_ld16(row + (uint32_t)(s0 * M + m0), v0);
          if (two) tmem_ld16(row + (uint32_t)(s1 * M + m0), v1);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 16; e += 4) {
            chain4(w0, v0[e], v0[e + 1], v0[e + 2], v0[e + 3]);
            if (two) chain4(w1, v1[e], v1[e + 1], v1[e + 2], v1[e + 3]);
          }
        }
        finish(u0, s0, w0);
        if (two) finish(u1, s1, w1);
        u0 = n0;
        u1 = n1;
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&emptyD[j & 1]);
      return true;
    };
    if (i0 < i1) load_epi(P0, i0);
    for (int64_t i = i0; i < i1; i += 2) {
      if (*fail || !step(i, P0, P1)) break;
      if (i + 1 < i1 && (*fail || !step(i + 1, P1, P0))) break;
    }
  } else if (tid == FT_WORKERS) {
    const int ta[6] = {2, 1, 0, 1, 0, 0}, tb[6] = {0, 1, 2, 0, 1, 0};
    const int n = (int)(i1 - i0);
    auto load_A = [&](int jj) {
      const int b = jj % FT_ABUF;
      const BTcItem it = a.items[i0 + jj];
      const unsigned char* src = a.A + a.probs[it.p].oTA + it.t * (int64_t)A_BYTES;
      mbar_expect_tx(&fullA[b], (uint32_t)A_BYTES);
      for (int off = 0; off < A_BYTES; off += FT_CHUNK)
        bulk_g2s(sA + b * A_BYTES + off, src + off, (uint32_t)(A_BYTES - off < FT_CHUNK ? A_BYTES - off : FT_CHUNK),
                 &fullA[b]);
    };
    int nl = 0;
    for (; nl < FT_ABUF && nl < n; ++nl) load_A(nl);
    int j = 0;
    int cur_p = -1, cur_g = -1, nB = 0;
    bool issued = false;
    for (; j < n; ++j) {
      const BTcItem it = a.items[i0 + j];
      const BProb& B = a.probs[it.p];
      const int NR = B.NR;
      if (it.p != cur_p || it.g != cur_g) {
        if (cur_p >= 0) {
          mma_commit(&freeB);
          if (!mbar_wait(&freeB, (uint32_t)((nB - 1) & 1))) {
            set_fail(6);
            break;
          }
        }
        const int B_BYTES = 3 * NR * KP * 2;
        mbar_expect_tx(&fullB, (uint32_t)B_BYTES);
        const unsigned char* src = a.B + B.oTB + (int64_t)it.g * B_BYTES;
        for (int off = 0; off < B_BYTES; off += FT_CHUNK)
          bulk_g2s(sB + off, src + off, (uint32_t)(B_BYTES - off < FT_CHUNK ? B_BYTES - off : FT_CHUNK), &fullB);
        if (!mbar_wait(&fullB, (uint32_t)(nB & 1))) {
          set_fail(7);
          break;
        }
        ++nB;
        cur_p = it.p;
        cur_g = it.g;
      }
      const int b = j % FT_ABUF;
      if (!mbar_wait(&fullA[b], (uint32_t)((j / FT_ABUF) & 1))) {
        set_fail(8);
        break;
      }
      if (j >= 2 && !mbar_wait(&emptyD[j & 1], (uint32_t)(((j >> 1) - 1) & 1))) {
        set_fail(9);
        break;
      }
      if (*fail) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t idesc = instr_desc_bf16(FT_ROWS, NR);
      const uint32_t a0 = smem_u32(sA + b * A_BYTES), b0 = smem_u32(sB);
      const uint32_t d = tmem + (uint32_t)((j & 1) * NRMAX);
      bool first = true;
#pragma unroll
      for (int q = 0; q < 6; ++q) {
#pragma unroll
        for (int ks = 0; ks < KP / 16; ++ks) {
          const uint64_t da = smem_desc_swz(a0 + ta[q] * A_TERM + 32 * ks, KP);
          const uint64_t db = smem_desc_swz(b0 + tb[q] * (NR * KP * 2) + 32 * ks, KP);
          mma_bf16(d, da, db, idesc, first ? 0u : 1u);
          first = false;
        }
      }
      mma_commit(&fullD[j & 1]);
      mma_commit(&emptyA[b]);
      issued = true;
      if (j >= 1 && j + FT_ABUF - 1 < n) {
        if (!mbar_wait(&emptyA[(j - 1) % FT_ABUF], (uint32_t)(((j - 1) / FT_ABUF) & 1))) {
          set_fail(11);
          break;
        }
        load_A(j + FT_ABUF - 1);
        ++nl;
      }
    }
    if (*fail)
      for (int jj = j; jj < nl; ++jj) mbar_wait(&fullA[jj % FT_ABUF], (uint32_t)((jj / FT_ABUF) & 1));
    if (issued) {
      mma_commit(&drain);
      if (!mbar_wait(&drain, 0)) set_fail(10);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == FT_WORKERS / 32) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
  }
}

// Split images of every problem of a batch.  Job index e of a prefix table: the problem whose
// first job is the largest prefix <= e (binary search), then that problem's local job.
__device__ inline int prefix_owner(const int64_t* __restrict__ prefix, int P, int64_t e) {
  int lo = 0, hi = P - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (prefix[mid] <= e) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

__global__ void b_split_time_kernel(const BProb* __restrict__ probs, const int64_t* __restrict__ prefix, int P,
                                    int64_t total, const float* __restrict__ AF32, unsigned char* __restrict__ Bimg) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= total) return;
  const int p = prefix_owner(prefix, P, e);
  const BProb& B = probs[p];
  const int KP = B.KP, chunks = KP / 8, NR = B.NR, M = B.M, K = B.K, KC = (K + 3) / 4 * 4;
  const int64_t le = e - prefix[p];
  const int c = (int)(le % chunks);
  const int64_t gr = le / chunks;
  const int rr = (int)(gr % NR);
  const int g = (int)(gr / NR);
  const int sl = rr / M, m = rr - sl * M, n = g * B.TG + sl;
  float x[8];
#pragma unroll
  for (int jj = 0; jj < 8; ++jj) {
    const int k = 8 * c + jj;
    x[jj] = (n < B.N && k < K) ? AF32[B.oAF32 + ((int64_t)n * M + m) * KC + k] : 0.f;
  }
  uint4 o[3];
  split8(x, o);
  const int64_t term = (int64_t)NR * KP * 2;
  uint4* dst = reinterpret_cast<uint4*>(Bimg + B.oTB);
#pragma unroll
  for (int t = 0; t < 3; ++t) dst[(((int64_t)g * 3 + t) * term + ft_swz((int64_t)rr * KP * 2 + c * 16, KP)) / 16] = o[t];
}

__global__ void b_split_w_kernel(const BProb* __restrict__ probs, const int64_t* __restrict__ prefix, int P,
                                 int64_t total, const float* __restrict__ W32, unsigned char* __restrict__ Aimg) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= total) return;
  const int p = prefix_owner(prefix, P, e);
  const BProb& B = probs[p];
  const int KP = B.KP, chunks = KP / 8, K = B.K;
  const int64_t nd = B.g.ndof;
  const int64_t le = e - prefix[p];
  const int rr = (int)(le % FT_ROWS);
  const int64_t rest = le / FT_ROWS;
  const int c = (int)(rest % chunks);
  const int64_t tile = rest / chunks;
  const int64_t J = tile * FT_ROWS + rr;
  float x[8];
#pragma unroll
  for (int jj = 0; jj < 8; ++jj) {
    const int k = 8 * c + jj;
    x[jj] = (J < nd && k < K) ? W32[B.oW + (int64_t)k * nd + J] : 0.f;
  }
  uint4 o[3];
  split8(x, o);
  const int64_t term = (int64_t)FT_ROWS * KP * 2;
  uint4* dst = reinterpret_cast<uint4*>(Aimg + B.oTA);
#pragma unroll
  for (int t = 0; t < 3; ++t) dst[((tile * 3 + t) * term + ft_swz((int64_t)rr * KP * 2 + c * 16, KP)) / 16] = o[t];
}

template <int KP>
pe_status btc_launch(const BtcArgs& args, int grid, cudaStream_t st) {
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  std::call_once(once, [] {
    attr = cudaFuncSetAttribute(b_fine_tc_kernel<KP>, cudaFuncAttributeMaxDynamicSharedMemorySize, ft_smem_bytes(KP));
  });
  if (attr != cudaSuccess) return pe_cuda_fail(attr, "batched fine sweep (tensor cores): shared-memory attribute");
  b_fine_tc_kernel<KP><<<grid, FT_THREADS, ft_smem_bytes(KP), st>>>(args);
  PE_CUDA_TRY(cudaGetLastError());
  return PE_OK;
}

}  // namespace

static bool fine_tc_supported(int M) { return M >= 16 && M <= 128 && M % 16 == 0; }

// slice-group shape of a column padding KP at M substeps: G slices, NR = G * M rows
static void ft_shape(int KP, int M, int N, int* G, int* NR, int* ngroups) {
  *G = std::max(1, ft_rows_max(KP) / M);
  *NR = *G * M;
  *ngroups = (N + *G - 1) / *G;
}

// ---------------------------------------------------------------------------
// batched form (pe_batch with fine_engine = PE_FINE_TC)
// ---------------------------------------------------------------------------
bool batch_tc_shape(int K, int M, int* KP, int* TG, int* NR) {
  if (!fine_tc_supported(M) || K < 1 || K > 64) return false;
  *KP = ft_kpad(K);
  int ng = 0;
  ft_shape(*KP, M, 1, TG, NR, &ng);
  return true;
}

pe_status batch_tc_prepare(pe_batch* b, cudaStream_t st) {
  const unsigned threads = 256;
  if (b->tc.y_jobs > 0)
    b_split_time_kernel<<<(unsigned)((b->tc.y_jobs + threads - 1) / threads), threads, 0, st>>>(
        b->d_probs, b->tc.d_y_prefix, b->P, b->tc.y_jobs, b->AF32, b->tc.B);
  if (b->tc.w_jobs > 0)
    b_split_w_kernel<<<(unsigned)((b->tc.w_jobs + threads - 1) / threads), threads, 0, st>>>(
        b->d_probs, b->tc.d_w_prefix, b->P, b->tc.w_jobs, b->W32, b->tc.A);
  b->launches += 2;
  PE_CUDA_TRY(cudaGetLastError());
  return PE_OK;
}

pe_status batch_tc_fine(pe_batch* b, cudaStream_t st) {
  for (int cls = 0; cls < 3; ++cls) {
    const int n = b->tc.begin[cls + 1] - b->tc.begin[cls];
    if (n == 0) continue;
    BtcArgs args{};
    args.probs = b->d_probs;
    args.items = b->tc.d_items + b->tc.begin[cls];
    args.n_items = n;
    args.coefF32 = b->coefF32;
    args.coefF = b->coefF;
    args.U = b->U;
    args.Fbar = b->Fbar;
    args.A = b->tc.A;
    args.B = b->tc.B;
    args.err = b->tc.err;
    const int grid = std::min(n, b->sm_count);
    if (cls == 0) PE_TRY(btc_launch<16>(args, grid, st));
    else if (cls == 1) PE_TRY(btc_launch<32>(args, grid, st));
    else PE_TRY(btc_launch<64>(args, grid, st));
  }
  return PE_OK;
}

pe_status batch_tc_status(pe_batch* b) {
  if (!b->tc.err) return PE_OK;
  int herr = 0;
  PE_CUDA_TRY(cudaMemcpy(&herr, b->tc.err, sizeof(int), cudaMemcpyDeviceToHost));
  if (herr != 0) {
    cudaMemset(b->tc.err, 0, sizeof(int));
    return pe_fail(PE_ETIMEOUT, "batched fine sweep (tensor cores): a pipeline wait expired (code " +
                                    std::to_string(herr) + ")");
  }
  return PE_OK;
}
