// Host side of the batched solver (pe_setup_batch / pe_batch_*): validation,
// arena layout, work-item lists, the captured Parareal iteration graph and
// the launch-shape autotuner.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <fstream>
#include <new>
#include <sstream>
#include <string>
#include <vector>

#include "pe_batch.h"
#include "pe_contract.cuh"

namespace {

template <typename T>
pe_status balloc(T** p, size_t count) {
  cudaError_t e = cudaMalloc((void**)p, sizeof(T) * (count ? count : 1));
  if (e != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    return pe_fail(PE_ENOMEM, "batch: cudaMalloc of " + std::to_string(sizeof(T) * count) + " bytes failed");
  }
  return PE_OK;
}

template <typename T>
pe_status upload(T** d, const std::vector<T>& h, cudaStream_t st) {
  PE_TRY(balloc(d, h.size()));
  if (!h.empty()) PE_CUDA_TRY(cudaMemcpyAsync(*d, h.data(), sizeof(T) * h.size(), cudaMemcpyHostToDevice, st));
  return PE_OK;
}

void free_batch(pe_batch* b) {
  if (!b) return;
  for (cudaGraphExec_t g : b->graph_exec)
    if (g) cudaGraphExecDestroy(g);
  void* ptrs[] = {b->d_probs, b->d_terms, b->d_mode_items, b->walk128.d_items, b->walk256.d_items,
                  b->d_factor_jobs, b->d_mu_prefix, b->d_tt_prefix, b->muM, b->ratio, b->rows, b->scratch, b->coefF, b->coefG,
                  b->coefF32, b->coefG32, b->U, b->axisF, b->axisU0, b->axisF32, b->partials, b->active,
                  b->kcount, b->resid, b->counter, b->dflags, b->Y, b->Z, b->chain, b->xs, b->Y32, b->Z32,
                  b->chain32, b->xs32, b->V, b->G, b->V32, b->G32, b->d_cols, b->d_first, b->Kt, b->d_kt_prefix};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  if (b->h_flags) cudaFreeHost(b->h_flags);
  for (cudaEvent_t e : b->ev)
    if (e) cudaEventDestroy(e);
  if (b->ev_order) cudaEventDestroy(b->ev_order);
  if (b->stream) cudaStreamDestroy(b->stream);
  delete b;
}

uint64_t fnv1a(uint64_t h, const void* data, size_t n) {
  const unsigned char* p = (const unsigned char*)data;
  for (size_t i = 0; i < n; ++i) {
    h ^= p[i];
    h *= 0x100000001B3ull;
  }
  return h;
}

// Walk items (problem, `threads` modes; the item runs every slice of its problem), longest (most
// slices) first; the residual slots of a problem are consecutive from oItems.
pe_status build_walk_items(pe_batch* b, int threads, WalkItems* out) {
  std::vector<WalkItem> items;
  std::vector<int> order((size_t)b->P);
  for (int p = 0; p < b->P; ++p) order[(size_t)p] = p;
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return b->probs[x].N > b->probs[y].N; });
  for (int p : order) {
    const BProb& B = b->probs[p];
    int slot = (int)B.oItems;
    for (int64_t J0 = 0; J0 < B.g.ndof; J0 += threads) items.push_back(WalkItem{p, slot++, J0});
  }
  if (items.size() > (size_t)INT32_MAX) return pe_fail(PE_EINVAL, "batch: too many work items");
  out->n = (int)items.size();
  return upload(&out->d_items, items, b->stream);
}

}  // namespace

extern "C" pe_status pe_setup_batch(pe_batch** out, int32_t n_problems, const pe_problem* problems,
                                    const pe_options* opt) {
  if (!out) return pe_fail(PE_EINVAL, "pe_setup_batch: out is NULL");
  *out = nullptr;
  if (n_problems < 1 || !problems) return pe_fail(PE_EINVAL, "pe_setup_batch: need at least one problem");
  pe_options o{};
  if (opt) o = *opt;
  if (o.precision != PE_FP64 && o.precision != PE_MIXED) return pe_fail(PE_EINVAL, "pe_setup_batch: bad precision");
  if (o.quad_pts == 0) o.quad_pts = 3;
  if (o.quad_pts < 1 || o.quad_pts > 8) return pe_fail(PE_EINVAL, "pe_setup_batch: quad_pts must be in 1..8");
  if (o.fine_engine != PE_FINE_SIMT && o.fine_engine != PE_FINE_TC)
    return pe_fail(PE_EINVAL, "pe_setup_batch: bad fine_engine");
  if (o.fine_engine == PE_FINE_TC && o.precision != PE_MIXED)
    return pe_fail(PE_EINVAL, "pe_setup_batch: PE_FINE_TC needs PE_MIXED");

  pe_batch* b = new (std::nothrow) pe_batch();
  if (!b) return pe_fail(PE_ENOMEM, "pe_setup_batch: host allocation failed");
  b->P = n_problems;
  b->precision = o.precision;
  b->fine_engine = o.fine_engine;
  b->quad_pts = o.quad_pts;
  b->user_stream = (cudaStream_t)o.cuda_stream;
  b->gauss = make_gauss(o.quad_pts);
  pe_status st = PE_OK;
  {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&b->sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
      st = pe_cuda_fail(cudaGetLastError(), "pe_setup_batch: device query");
    }
  }
  if (st == PE_OK && cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) != cudaSuccess)
    st = pe_cuda_fail(cudaGetLastError(), "pe_setup_batch: stream");
  if (st != PE_OK) {
    free_batch(b);
    return st;
  }

  // ---- validate and lay out every problem --------------------------------
  int64_t oU = 0, oCF = 0, oCG = 0, oAx = 0, oAxU = 0, oY = 0, oY32 = 0, oMu = 0, oItems = 0;
  int64_t oV = 0, oZ = 0, oCh = 0, oXs = 0;
  std::vector<int64_t> mu_prefix, tt_prefix;
  std::vector<short> cols, first;
  int64_t tt = 0;
  uint64_t sig = 0xcbf29ce484222325ull;
  b->probs.resize(n_problems);
  for (int p = 0; p < n_problems && st == PE_OK; ++p) {
    const pe_problem& q = problems[p];
    BProb& B = b->probs[p];
    memset(&B, 0, sizeof(B));
    const std::string tag = "problem " + std::to_string(p) + ": ";
    if (q.d < 1 || q.d > PE_MAX_D) { st = pe_fail(PE_EINVAL, tag + "d must be 1..3"); break; }
    if (!(q.D > 0.0) || !(q.T > 0.0) || !isfinite(q.D) || !isfinite(q.T) || !isfinite(q.t0)) {
      st = pe_fail(PE_EINVAL, tag + "D and T must be positive");
      break;
    }
    if (q.n_slices < 1 || q.n_substeps < 1) { st = pe_fail(PE_EINVAL, tag + "slices/substeps must be >= 1"); break; }
    int64_t ndof = 1;
    int nsum = 0;
    for (int a = 0; a < PE_MAX_D; ++a) {
      if (a < q.d) {
        if (q.n[a] < 1 || q.n[a] > 4096) { st = pe_fail(PE_EINVAL, tag + "n_a must be in 1..4096"); break; }
        if (!(q.box[2 * a + 1] > q.box[2 * a])) { st = pe_fail(PE_EINVAL, tag + "box needs lo < hi"); break; }
        B.g.n[a] = q.n[a];
        B.g.off[a] = nsum;
        B.lo[a] = q.box[2 * a];
        B.h[a] = (q.box[2 * a + 1] - q.box[2 * a]) / (double)(q.n[a] + 1);
        ndof *= q.n[a];
        nsum += q.n[a];
        b->nmax = std::max(b->nmax, q.n[a]);
      } else {
        B.g.n[a] = 1;
        B.g.off[a] = nsum;
        B.lo[a] = 0.0;
        B.h[a] = 1.0;
      }
    }
    if (st != PE_OK) break;
    B.g.d = q.d;
    B.g.ndof = ndof;
    B.N = q.n_slices;
    B.M = q.n_substeps;
    B.D = q.D;
    B.t0 = q.t0;
    B.dT = q.T / (double)q.n_slices;
    B.dt = B.dT / (double)q.n_substeps;
    if ((st = pe_resolve_nodes(&q.fine, "fine", &B.q, B.cF)) != PE_OK) break;
    if ((st = pe_resolve_nodes(&q.coarse, "coarse", &B.p, B.cG)) != PE_OK) break;
    pe_lagrange_coeffs(B.q, B.cF, B.lagF);
    pe_lagrange_coeffs(B.p, B.cG, B.lagG);
    if (q.u0.kind != PE_FIELD_TERMS_SEPARABLE) {
      st = pe_fail(PE_EINVAL, tag + "a batch takes separable initial data (PE_FIELD_TERMS_SEPARABLE)");
      break;
    }
    const int nf = q.forcing.n_terms;
    if (nf > PE_BATCH_MAX_TERMS) { st = pe_fail(PE_EINVAL, tag + "at most 20 forcing terms in a batch"); break; }
    if ((st = pe_validate_terms(nf, q.forcing.terms, q.d, "forcing")) != PE_OK) break;
    if ((st = pe_validate_terms(q.u0.n_terms, q.u0.terms, q.d, "u0")) != PE_OK) break;
    B.tf = (int)b->terms.size();
    if (nf == 0) {
      pe_term z;
      memset(&z, 0, sizeof(z));
      b->terms.push_back(z);
      B.R = 1;
    } else {
      for (int i = 0; i < nf; ++i) b->terms.push_back(q.forcing.terms[i]);
      B.R = nf;
    }
    B.tu = (int)b->terms.size();
    if (q.u0.n_terms == 0) {
      pe_term z;
      memset(&z, 0, sizeof(z));
      b->terms.push_back(z);
      B.Ru = 1;
    } else {
      for (int i = 0; i < q.u0.n_terms; ++i) b->terms.push_back(q.u0.terms[i]);
      B.Ru = q.u0.n_terms;
    }
    if (B.Ru > PE_MAX_TERMS) { st = pe_fail(PE_EINVAL, tag + "too many u0 terms"); break; }
    // source columns: one per exponential term, two per sinusoid
    B.oCol = (int64_t)cols.size();
    B.oFirst = (int64_t)first.size();
    for (int r = 0; r < B.R; ++r) {
      first.push_back((short)((int64_t)cols.size() - B.oCol));
      cols.push_back((short)(r << 1));
      if (b->terms[B.tf + r].tkind == PE_T_SIN) cols.push_back((short)((r << 1) | 1));
    }
    B.K = (int)((int64_t)cols.size() - B.oCol);
    b->Kmax = std::max(b->Kmax, B.K);
    b->ndof_max = std::max(b->ndof_max, ndof);
    B.oU = oU; oU += (int64_t)(B.N + 1) * ndof;
    B.oCF = oCF; oCF += (int64_t)(B.q + 2) * ndof;
    B.oCG = oCG; oCG += (int64_t)(B.p + 1) * ndof;
    B.oAx = oAx; oAx += (int64_t)B.R * nsum;
    B.oAxU = oAxU; oAxU += (int64_t)B.Ru * nsum;
    const int KC = (B.K + 3) / 4 * 4;
    const int64_t steps = chain_steps(B.M);
    B.oY = oY; oY += (int64_t)B.N * B.K;
    B.oY32 = oY32; oY32 += (int64_t)B.N * 2 * KC;
    B.oV = oV; oV += (int64_t)B.K * ndof;
    B.oZ = oZ; oZ += (int64_t)(B.q + B.p) * B.K;
    B.oCh = oCh; oCh += steps * B.R * 4;
    B.oXs = oXs; oXs += B.R;
    B.oMu = oMu;
    mu_prefix.push_back(oMu);
    oMu += nsum;
    tt_prefix.push_back(tt);
    tt += (int64_t)(B.N + B.q + B.p) * B.K + (int64_t)B.R * (steps + 1);  // b_time_tables_kernel's threads
    B.oItems = oItems;
    oItems += (ndof + 127) / 128;  // residual slots for the smaller item
    if (b->fine_engine == PE_FINE_TC && (B.M < 16 || B.M > 128 || B.M % 16 != 0)) {
      st = pe_fail(PE_EINVAL, tag + "PE_FINE_TC needs M a multiple of 16 in 16..128");
      break;
    }
    sig = fnv1a(sig, &B.g, sizeof(B.g));
    sig = fnv1a(sig, &B.N, sizeof(int) * 6);
  }
  if (st != PE_OK) {
    free_batch(b);
    return st;
  }
  b->signature = fnv1a(fnv1a(sig, &b->precision, sizeof(int)), &b->fine_engine, sizeof(int));
  b->mu_total = oMu;
  b->tt_total = tt;

  // ---- arenas --------------------------------------------------------------
  const bool mixed = b->precision == PE_MIXED;
  b->u_total = (size_t)oU;
  if (st == PE_OK) st = balloc(&b->muM, oMu);
  if (st == PE_OK) st = balloc(&b->ratio, oMu);
  if (st == PE_OK) st = balloc(&b->rows, oMu);
  if (st == PE_OK) st = balloc(&b->scratch, 2 * (size_t)b->ndof_max);
  if (st == PE_OK) st = balloc(&b->coefF, oCF);
  if (st == PE_OK && mixed) st = balloc(&b->coefF32, oCF);
  if (st == PE_OK) st = balloc(&b->coefG, oCG);
  if (st == PE_OK && mixed) st = balloc(&b->coefG32, oCG);
  if (st == PE_OK) st = balloc(&b->U, oU);
  if (st == PE_OK) st = balloc(&b->axisF, oAx);
  if (st == PE_OK && mixed) st = balloc(&b->axisF32, oAx);
  if (st == PE_OK) st = balloc(&b->axisU0, oAxU);
  // time tables and column weights in the form's own arithmetic
  if (st == PE_OK) st = mixed ? balloc(&b->Y32, oY32) : balloc(&b->Y, oY);
  if (st == PE_OK) st = mixed ? balloc(&b->Z32, oZ) : balloc(&b->Z, oZ);
  if (st == PE_OK) st = mixed ? balloc(&b->chain32, 2 * oCh) : balloc(&b->chain, oCh);
  if (st == PE_OK) st = mixed ? balloc(&b->xs32, 2 * oXs) : balloc(&b->xs, oXs);
  if (st == PE_OK) st = mixed ? balloc(&b->V32, oV) : balloc(&b->V, oV);
  if (st == PE_OK) st = mixed ? balloc(&b->G32, oV) : balloc(&b->G, oV);
  if (st == PE_OK) st = balloc(&b->partials, 2 * (size_t)oItems);
  if (st == PE_OK) st = balloc(&b->active, (size_t)b->P);
  if (st == PE_OK) st = balloc(&b->kcount, (size_t)b->P);
  if (st == PE_OK) st = balloc(&b->resid, (size_t)b->P);
  if (st == PE_OK) st = balloc(&b->counter, 1);
  if (st == PE_OK) st = balloc(&b->dflags, 2);
  for (cudaEvent_t& e : b->ev)
    if (st == PE_OK && cudaEventCreate(&e) != cudaSuccess) st = pe_cuda_fail(cudaGetLastError(), "pe_setup_batch: event");
  if (st == PE_OK && cudaEventCreateWithFlags(&b->ev_order, cudaEventDisableTiming) != cudaSuccess)
    st = pe_cuda_fail(cudaGetLastError(), "pe_setup_batch: event");
  if (st == PE_OK && cudaMallocHost((void**)&b->h_flags, 2 * sizeof(int)) != cudaSuccess) {
    cudaGetLastError();
    st = pe_fail(PE_ENOMEM, "pe_setup_batch: pinned allocation failed");
  }
  if (st != PE_OK) {
    free_batch(b);
    return st;
  }
  b->n_active = b->dflags;
  b->nonfinite = b->dflags + 1;

  // ---- work items ----------------------------------------------------------
  {
    std::vector<ModeItem> mitems;
    for (int p = 0; p < b->P; ++p)
      for (int64_t J0 = 0; J0 < b->probs[p].g.ndof; J0 += 256) mitems.push_back(ModeItem{p, 0, J0});
    b->n_mode_items = (int)mitems.size();
    std::vector<FactorJob> jobs;
    for (int p = 0; p < b->P; ++p) {
      const BProb& B = b->probs[p];
      for (int a = 0; a < B.g.d; ++a) {
        for (int r = 0; r < B.R; ++r) jobs.push_back(FactorJob{p, a, r, 0});
        for (int r = 0; r < B.Ru; ++r) jobs.push_back(FactorJob{p, a, r, 1});
      }
    }
    std::stable_sort(jobs.begin(), jobs.end(), [&](const FactorJob& x, const FactorJob& y) {
      return b->probs[x.p].g.n[x.axis] > b->probs[y.p].g.n[y.axis];
    });
    b->n_factor_jobs = (int)jobs.size();
    st = upload(&b->d_probs, b->probs, b->stream);
    if (st == PE_OK) st = upload(&b->d_terms, b->terms, b->stream);
    if (st == PE_OK) st = upload(&b->d_mode_items, mitems, b->stream);
    if (st == PE_OK) st = upload(&b->d_factor_jobs, jobs, b->stream);
    if (st == PE_OK) st = upload(&b->d_mu_prefix, mu_prefix, b->stream);
    if (st == PE_OK) st = upload(&b->d_tt_prefix, tt_prefix, b->stream);
    if (st == PE_OK) st = upload(&b->d_cols, cols, b->stream);
    if (st == PE_OK) st = upload(&b->d_first, first, b->stream);
    if (st == PE_OK) st = build_walk_items(b, 128, &b->walk128);
    if (st == PE_OK) st = build_walk_items(b, 256, &b->walk256);
  }
  if (st == PE_OK) st = batch_set_attributes(b);
  if (st == PE_OK) st = batch_launch_axis_tables(b);
  if (st == PE_OK) st = batch_launch_coef_tables(b);
  if (st == PE_OK) {
    cudaError_t e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) st = pe_cuda_fail(e, "pe_setup_batch");
  }
  if (st != PE_OK) {
    free_batch(b);
    return st;
  }
  *out = b;
  return PE_OK;
}

extern "C" void pe_batch_destroy(pe_batch* b) {
  if (!b) return;
  cudaStreamSynchronize(b->stream);
  free_batch(b);
}

namespace {

pe_status reset_iteration_state(pe_batch* b) {
  PE_CUDA_TRY(cudaMemsetAsync(b->active, 1, sizeof(int) * b->P, b->stream));  // any nonzero value: active
  PE_CUDA_TRY(cudaMemsetAsync(b->kcount, 0, sizeof(int) * b->P, b->stream));
  PE_CUDA_TRY(cudaMemsetAsync(b->resid, 0, sizeof(double) * b->P, b->stream));
  PE_CUDA_TRY(cudaMemsetAsync(b->dflags, 0, 2 * sizeof(int), b->stream));
  return PE_OK;
}

// The graphs of the first iteration (which = 1) and of the others (0).
pe_status ensure_graphs(pe_batch* b, double tol) {
  if (b->graph_exec[0] && b->graph_exec[1] && b->graph_tol == tol && b->graph_threads == b->tune_threads &&
      b->graph_ctas == b->tune_ctas)
    return PE_OK;
  for (int which = 0; which < 2; ++which) {
    cudaGraphExec_t& ex = b->graph_exec[which];
    if (ex) {
      cudaGraphExecDestroy(ex);
      ex = nullptr;
    }
    PE_CUDA_TRY(cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal));
    pe_status st = batch_enqueue_iteration(b, b->stream, tol, which == 1);
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamEndCapture(b->stream, &g);
    if (st == PE_OK && e != cudaSuccess) st = pe_cuda_fail(e, "batch: graph capture");
    if (st == PE_OK) {
      e = cudaGraphInstantiate(&ex, g, 0);
      if (e != cudaSuccess) {
        ex = nullptr;
        st = pe_cuda_fail(e, "batch: graph instantiation");
      }
    }
    if (g) cudaGraphDestroy(g);
    PE_TRY(st);
  }
  b->graph_tol = tol;
  b->graph_threads = b->tune_threads;
  b->graph_ctas = b->tune_ctas;
  return PE_OK;
}

float ms_between(cudaEvent_t a, cudaEvent_t b) {
  float ms = 0.f;
  cudaEventElapsedTime(&ms, a, b);
  return ms;
}

}  // namespace

// What the caller's stream (the legacy default stream where the batch was given none) still has to do with a network it
// attached comes before the work on the batch's own stream, which waits for no other by itself.
static pe_status after_caller(pe_batch* b) {
  PE_CUDA_TRY(cudaEventRecord(b->ev_order, b->user_stream));
  PE_CUDA_TRY(cudaStreamWaitEvent(b->stream, b->ev_order, 0));
  return PE_OK;
}

namespace {

// The fastest launch shape of the walk on a prepared state; the timed walks write iterates.
pe_status time_shapes(pe_batch* b, int* threads, int* ctas) {
  PE_TRY(reset_iteration_state(b));
  PE_TRY(batch_launch_prepare(b));
  const int cand_threads[2] = {128, 256};
  float best = 1e30f;
  for (int ti = 0; ti < 2; ++ti) {
    for (int ct = 1; ct <= 4; ++ct) {
      float ms = 0.f, tot = 0.f;
      PE_TRY(batch_time_walk(b, cand_threads[ti], ct, &ms));  // warm
      for (int rep = 0; rep < 2; ++rep) {
        PE_TRY(batch_time_walk(b, cand_threads[ti], ct, &ms));
        tot += ms;
      }
      if (tot < best) {
        best = tot;
        *threads = cand_threads[ti];
        *ctas = ct;
      }
    }
  }
  return PE_OK;
}

// What a finished solve can still be asked for (iterates, k, residuals), kept in `buf` or put back from it.
size_t result_bytes(const pe_batch* b) { return sizeof(double) * (b->u_total + b->P) + sizeof(int) * b->P; }
pe_status copy_result(pe_batch* b, double* buf, bool back) {
  const auto part = [&](void* own, void* kept, size_t bytes) {
    return cudaMemcpyAsync(back ? own : kept, back ? kept : own, bytes, cudaMemcpyDeviceToDevice, b->stream);
  };
  PE_CUDA_TRY(part(b->U, buf, sizeof(double) * b->u_total));
  PE_CUDA_TRY(part(b->resid, buf + b->u_total, sizeof(double) * b->P));
  PE_CUDA_TRY(part(b->kcount, buf + b->u_total + b->P, sizeof(int) * b->P));
  return PE_OK;
}

}  // namespace

extern "C" pe_status pe_batch_autotune(pe_batch* b, const char* cache_path) {
  if (!b) return pe_fail(PE_EINVAL, "pe_batch_autotune: NULL batch");
  cudaDeviceProp prop;
  int dev = 0;
  PE_CUDA_TRY(cudaGetDevice(&dev));
  PE_CUDA_TRY(cudaGetDeviceProperties(&prop, dev));
  char key[320];
  // (the kernel whose shape was timed is part of the key: a file of another one's choices is left alone)
  snprintf(key, sizeof(key), "%s|walk|%016llx", prop.name, (unsigned long long)b->signature);
  for (char* c = key; *c; ++c)
    if (*c == ' ') *c = '_';
  if (cache_path) {
    std::ifstream in(cache_path);
    std::string line;
    while (std::getline(in, line)) {
      std::istringstream ss(line);
      std::string k;
      int th = 0, ct = 0;
      if (ss >> k >> th >> ct && k == key && (th == 128 || th == 256) && ct >= 1 && ct <= 8) {
        b->tune_threads = th;
        b->tune_ctas = ct;
        return PE_OK;
      }
    }
  }
  PE_TRY(after_caller(b));
  // a finished solve stays as it is; without room to keep it the launch shape stays as it is
  double* kept = nullptr;
  if (b->have_problem) {
    if (cudaMalloc((void**)&kept, result_bytes(b)) != cudaSuccess) {
      cudaGetLastError();
      return PE_OK;
    }
    const pe_status st = copy_result(b, kept, false);
    if (st != PE_OK) {
      cudaFree(kept);
      return st;
    }
  }
  int best_t = 128, best_c = 4;
  pe_status st = time_shapes(b, &best_t, &best_c);
  if (kept) {
    const pe_status back = copy_result(b, kept, true);
    cudaStreamSynchronize(b->stream);
    cudaFree(kept);
    if (st == PE_OK) st = back;
  }
  PE_TRY(st);
  b->tune_threads = best_t;
  b->tune_ctas = best_c;
  if (cache_path) {
    std::ofstream outf(cache_path, std::ios::app);
    if (outf) outf << key << " " << best_t << " " << best_c << "\n";
  }
  return PE_OK;
}

extern "C" pe_status pe_batch_solve(pe_batch* b, double tol, pe_batch_result* res) {
  if (!b) return pe_fail(PE_EINVAL, "pe_batch_solve: NULL batch");
  if (!(tol >= 0.0)) return pe_fail(PE_EINVAL, "pe_batch_solve: tol must be >= 0");
  cudaEvent_t* ev = b->ev;
  PE_TRY(after_caller(b));
  b->launches = 0;
  PE_TRY(reset_iteration_state(b));
  PE_TRY(ensure_graphs(b, tol));
  PE_CUDA_TRY(cudaEventRecord(ev[0], b->stream));
  PE_TRY(batch_launch_prepare(b));
  PE_CUDA_TRY(cudaEventRecord(ev[1], b->stream));
  int replays = 0;
  int maxN = 0;
  for (const BProb& B : b->probs) maxN = std::max(maxN, B.N);
  for (;;) {
    PE_CUDA_TRY(cudaGraphLaunch(b->graph_exec[replays == 0 ? 1 : 0], b->stream));
    PE_CUDA_TRY(cudaStreamSynchronize(b->stream));
    ++replays;
    b->launches += 2;  // graph: walk, reduction
    if (b->h_flags[1]) {
      b->have_problem = false;
      return pe_fail(PE_ENONFINITE, "batch: a problem's Parareal residual is not finite");
    }
    if (b->h_flags[0] == 0 || replays >= maxN) break;
  }
  PE_CUDA_TRY(cudaEventRecord(ev[2], b->stream));
  PE_CUDA_TRY(cudaEventSynchronize(ev[2]));
  b->have_problem = true;
  if (b->user_stream) {
    PE_CUDA_TRY(cudaEventRecord(b->ev_order, b->stream));
    PE_CUDA_TRY(cudaStreamWaitEvent(b->user_stream, b->ev_order, 0));
  }
  if (res) {
    std::vector<int> k((size_t)b->P);
    std::vector<double> r((size_t)b->P);
    PE_CUDA_TRY(cudaMemcpy(k.data(), b->kcount, sizeof(int) * b->P, cudaMemcpyDeviceToHost));
    PE_CUDA_TRY(cudaMemcpy(r.data(), b->resid, sizeof(double) * b->P, cudaMemcpyDeviceToHost));
    res->graph_replays = replays;
    res->max_k = 0;
    res->max_residual = 0.0;
    res->fine_dof_substeps = 0;
    for (int p = 0; p < b->P; ++p) {
      const BProb& B = b->probs[p];
      res->max_k = std::max(res->max_k, k[p]);
      res->max_residual = std::max(res->max_residual, r[p]);
      res->fine_dof_substeps += B.g.ndof * (int64_t)B.N * B.M * k[p];
    }
    res->ms_prepare = ms_between(ev[0], ev[1]);
    res->ms_iterations = ms_between(ev[1], ev[2]);
    res->kernel_launches = b->launches;
    res->threads = b->tune_threads;
    res->ctas_per_sm = b->tune_ctas;
  }
  return PE_OK;
}

extern "C" pe_status pe_batch_get_modal(pe_batch* b, int32_t problem, int32_t slice, double* out) {
  if (!b || !out) return pe_fail(PE_EINVAL, "pe_batch_get_modal: NULL argument");
  if (problem < 0 || problem >= b->P) return pe_fail(PE_EINVAL, "pe_batch_get_modal: problem out of range");
  const BProb& B = b->probs[problem];
  if (slice < 0 || slice > B.N) return pe_fail(PE_EINVAL, "pe_batch_get_modal: slice out of range");
  if (!b->have_problem) return pe_fail(PE_ESTATE, "pe_batch_get_modal: no solve has completed");
  const bool dev = pe_is_device_ptr(out);
  // fetches run on the caller's stream (the batch's own has nothing left to do after a solve): after whatever that
  // still does with the buffer, without an event in between (1 us a fetch)
  const cudaStream_t st = b->user_stream;
  PE_CUDA_TRY(cudaMemcpyAsync(out, b->U + B.oU + (int64_t)slice * B.g.ndof, sizeof(double) * B.g.ndof,
                              dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, st));
  PE_CUDA_TRY(cudaStreamSynchronize(st));
  return PE_OK;
}

extern "C" pe_status pe_batch_get_solution(pe_batch* b, int32_t problem, double* nodal_out) {
  if (!b || !nodal_out) return pe_fail(PE_EINVAL, "pe_batch_get_solution: NULL argument");
  if (problem < 0 || problem >= b->P) return pe_fail(PE_EINVAL, "pe_batch_get_solution: problem out of range");
  if (!b->have_problem) return pe_fail(PE_ESTATE, "pe_batch_get_solution: no solve has completed");
  const BProb& B = b->probs[problem];
  int n[PE_MAX_D] = {B.g.n[0], B.g.n[1], B.g.n[2]};
  const double* last = b->U + B.oU + (int64_t)B.N * B.g.ndof;
  double* rows[PE_MAX_D] = {nullptr, nullptr, nullptr};
  for (int a = 0; a < B.g.d; ++a) rows[a] = b->rows + B.oMu + B.g.off[a];
  const bool dev = pe_is_device_ptr(nodal_out);
  double* out = dev ? nodal_out : b->scratch + b->ndof_max;
  const cudaStream_t stream = b->user_stream;  // (as in pe_batch_get_modal)
  std::lock_guard<std::mutex> lock(b->fetch);
  pe_status st = dst_rows_f64(B.g.d, n, rows, last, out, b->scratch, stream);
  if (st == PE_OK && !dev) {
    cudaError_t e = cudaMemcpyAsync(nodal_out, out, sizeof(double) * B.g.ndof, cudaMemcpyDeviceToHost, stream);
    if (e != cudaSuccess) st = pe_cuda_fail(e, "pe_batch_get_solution");
  }
  cudaError_t e = cudaStreamSynchronize(stream);
  if (st == PE_OK && e != cudaSuccess) st = pe_cuda_fail(e, "pe_batch_get_solution");
  return st;
}

// Learned correction for every problem: the band range of each problem (its slowest and fastest
// closed-form lam, times dT), table offsets and job prefixes; the tables themselves are made by
// the next pe_batch_solve (batch_learned_tables).
extern "C" pe_status pe_batch_set_learned(pe_batch* b, const pe_mlp* m) {
  if (!b) return pe_fail(PE_EINVAL, "pe_batch_set_learned: NULL batch");
  if (!m) {
    b->mlp = nullptr;
    return PE_OK;
  }
  PE_CUDA_TRY(cudaStreamSynchronize(b->stream));
  const int NB = kBatchLearnedBands;
  std::vector<int64_t> kp;
  int64_t okt = 0;
  for (int p = 0; p < b->P; ++p) {
    BProb& B = b->probs[p];
    double lmin = 0.0, lmax = 0.0;
    for (int a = 0; a < B.g.d; ++a) {
      const int n = B.g.n[a];
      auto ratio = [&](int j) {
        const double th = M_PI * (double)j / (double)(n + 1);
        const double sh = sin(0.5 * th);
        return ((4.0 / B.h[a]) * sh * sh) / ((B.h[a] / 3.0) * (2.0 + cos(th)));
      };
      lmin += ratio(1);
      lmax += ratio(n);
    }
    const double loglo = log(B.D * lmin * B.dT) - 1e-6, loghi = log(B.D * lmax * B.dT) + 1e-6;
    B.lloglo = loglo;
    B.lstep = (loghi - loglo) / (double)(NB - 1);
    B.oKt = okt;
    kp.push_back(okt / 2);
    okt += 2 * (int64_t)B.R * NB;
  }
  if (b->Kt) cudaFree(b->Kt);
  if (b->d_kt_prefix) cudaFree(b->d_kt_prefix);
  b->Kt = nullptr;
  b->d_kt_prefix = nullptr;
  PE_TRY(balloc(&b->Kt, (size_t)okt));
  PE_TRY(upload(&b->d_kt_prefix, kp, b->stream));
  PE_CUDA_TRY(cudaMemcpyAsync(b->d_probs, b->probs.data(), sizeof(BProb) * b->P, cudaMemcpyHostToDevice, b->stream));
  PE_CUDA_TRY(cudaStreamSynchronize(b->stream));
  b->kt_jobs = okt / 2;
  b->mlp = m;
  return PE_OK;
}

extern "C" pe_status pe_batch_status(pe_batch* b, double* residuals, int32_t* iterations) {
  if (!b) return pe_fail(PE_EINVAL, "pe_batch_status: NULL batch");
  if (residuals)
    PE_CUDA_TRY(cudaMemcpy(residuals, b->resid, sizeof(double) * b->P, cudaMemcpyDeviceToHost));
  if (iterations)
    PE_CUDA_TRY(cudaMemcpy(iterations, b->kcount, sizeof(int) * b->P, cudaMemcpyDeviceToHost));
  return PE_OK;
}
