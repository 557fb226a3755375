"""Benchmark: Parareal EIFE-linear on the 2D 255^2 workload, float64 vs mixed precision.

One step = one pe_solve of the workload: phi/b tables, P_h f tables, the
projection of u0 (forward tensor DST-I), the coarse sweep, Parareal
iterations (fine sweep from every slice + correction + float64 residual)
until the relative residual reaches 1e-6, and the inverse DST of the final
slice.  The metric is fine DoF*substeps per second:
    Ndof * N * M * (fine sweeps executed) / step time.

Workload: d = 2, 255 x 255 interior Q1 nodes on (0,1)^2, D = 0.1, t in [0,1],
u0 = nodal values of sin(pi x) sin(pi y), f = manufactured term + 8 seeded
Gaussian bumps modulated by sin(w t + phi), 32 slices x 64 substeps, RK4 fine
(c = 0, 1/4, 1/2, 3/4), 2-stage coarse with seeded random nodes.  The main
line is the float64 path; "chosen" reports the mixed-precision form on the
same workload with the loop on the device and its phases replayed as graphs ("mixed_simt": the
same kernels under the host-driven loop).  --impl reference times the CPU oracle instead.

Usage: python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]
       (N > 1: launch with torch.distributed.run; ranks solve independent
       replicas of the workload, no collective on the data path)
"""
from __future__ import annotations

import argparse
import json
import math
import os
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from paper_2412_01138_gb300 import inputs as I  # noqa: E402

METRIC = "time to rel-L2 1e-6 & fine DoF·substeps/s: chosen form vs plain FP64, 1 GB300"
UNIT = "fine DoF*substeps/s"
TOL = 1e-6
L2_BYTES = 129 * 1024 * 1024


_FLUSH = None


def timed_solves(s, steps, warmup, barrier, **kw):
    """Mean device time (ms) of `steps` solves of one Solver and their reports: each solve is
    enqueued with pe_solve_async between CUDA events on the current stream (the solver's), L2
    flushed before each (a 258 MB write), the report read after the closing event."""
    import torch

    global _FLUSH
    if _FLUSH is None:
        _FLUSH = torch.empty(2 * L2_BYTES // 4, dtype=torch.float32, device="cuda")
    stream = torch.cuda.current_stream()
    for _ in range(warmup):
        s.solve(**kw)
    barrier()
    total, infos = 0.0, []
    for _ in range(steps):
        _FLUSH.fill_(1.0)
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        s.solve_async(**kw)
        e1.record(stream)
        infos.append(s.wait())
        e1.synchronize()
        total += e0.elapsed_time(e1)
    barrier()
    return total / steps, infos


def cur_stream():
    import torch

    return torch.cuda.current_stream()


def chosen_kw(pe, prec):
    """Solver options of a separable-path solve: the mixed form (the chosen form) runs its Parareal
    loop on the device, with the set-up and output phases of a repeated solve replayed as graphs;
    float64 is the plain form (host-driven loop of Algorithm 1).  Both fine engines run the same kernels."""
    if prec == pe.PE_MIXED:
        return {"fine_engine": pe.PE_FINE_SIMT, "device_loop": 2}
    return {"fine_engine": pe.PE_FINE_SIMT}


def workload():
    return I.config2()


def nodal_u0(prob):
    """Synthetic initial data: sin(pi x) sin(pi y) at the interior nodes."""
    xs = []
    for a in range(prob.d):
        lo, hi = prob.box[a]
        h = (hi - lo) / (prob.n[a] + 1)
        xs.append(lo + h * np.arange(1, prob.n[a] + 1))
    out = np.ones(())
    for x in xs:
        out = np.multiply.outer(out, np.sin(np.pi * x))
    return np.ascontiguousarray(out.reshape(-1))


def stage_columns(prob) -> int:
    """K: stage-contracted columns of the fine step (one per exponential, two per sinusoid)."""
    return sum(2 if t.tkind == I.T_SIN else 1 for t in prob.forcing) if prob.forcing else 1


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as fh:
            return json.load(fh)
    return None


def fp64_peak_tflops(sm_mhz: float):
    """FP64 FMA peak: 152 SMs x 2 FP64 FMA lanes per clock x 2 FLOPs x clock."""
    return 152 * 2 * 2 * sm_mhz * 1e6 / 1e12


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled every 200 ms while running."""

    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device_index: int):
        self.dev = device_index
        self.proc = None
        # raw samples: PE_BENCH_CLOCKS_DIR if set, else the system's temporary directory (the
        # JSON line carries their summary)
        import tempfile

        out_dir = os.environ.get("PE_BENCH_CLOCKS_DIR") or tempfile.gettempdir()
        self.path = os.path.join(out_dir, f"clocks_bench_rank{device_index}.csv")

    def __enter__(self):
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.fh = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.dev}", f"--query-gpu={self.QUERY}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=self.fh, stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None
        return self

    def __exit__(self, *a):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
            self.fh.close()

    def summary(self):
        if self.proc is None or not os.path.exists(self.path):
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        sm, smax, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        with open(self.path) as fh:
            for line in fh:
                parts = [p.strip() for p in line.split(",")]
                if len(parts) < 9:
                    continue
                try:
                    sm.append(float(parts[1]))
                    smax = float(parts[2])
                except ValueError:
                    continue
                for name, v in zip(names, parts[5:9]):
                    if v.lower().startswith("active"):
                        reasons.add(name)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": smax, "reasons": ["no samples"]}
        return {"sm_mhz": float(np.median(sm)), "sm_max_mhz": smax, "reasons": sorted(reasons),
                "samples": len(sm)}


def oracle_chunk(payload):
    """Worker of the all-cores oracle run: Parareal on one contiguous block of modes."""
    from oracle import fem
    from oracle import solver as osolver

    prob, idx, u0_nodal = payload
    t0 = time.perf_counter()
    sys_ = osolver.ModalSystem(prob, modes=idx)
    basis = fem.ClosedFormBasis(prob.n, prob.box, prob.D)
    sys_.c0 = basis.to_modal_from_nodal(u0_nodal.reshape(prob.n)).reshape(-1)[idx]
    res = osolver.parareal(sys_, tol=TOL, keep_history=False)
    return len(idx) * prob.N * prob.M * res.k, time.perf_counter() - t0


def oracle_all_cores(prob, u0_nodal):
    """The oracle as it stands over every host core: modes split into one contiguous block per
    process (spawned, so no CUDA state is inherited); the pool is started before the timed region."""
    import multiprocessing as mp

    cores = os.cpu_count() or 1
    blocks = np.array_split(np.arange(prob.ndof), cores)
    with mp.get_context("spawn").Pool(cores) as pool:
        pool.map(abs, range(cores))  # workers up
        t0 = time.perf_counter()
        out = pool.map(oracle_chunk, [(prob, b, u0_nodal) for b in blocks])
        wall = time.perf_counter() - t0
    units = sum(u for u, _ in out)
    return {"value": units / wall, "unit": UNIT, "cores": cores, "kind": "oracle",
            "sample": f"the whole workload split into {cores} blocks of modes, one process each, {wall:.1f} s"}


def oracle_sample(prob, n_modes: int, seed: int = 0, u0_nodal=None):
    """Run the oracle's Parareal (to the same residual tolerance) on a random sample of modes.

    Modes are independent after the diagonalisation, so the sample is an exact
    restriction of the full solve.  u0_nodal: nodal initial data (as the bench
    feeds the library), else P_h of the descriptor.  Returns the rate in fine
    DoF*substeps/s and the pieces needed for a parity check.
    """
    from oracle import fem
    from oracle import solver as osolver

    rng = np.random.default_rng(seed)
    idx = np.sort(rng.choice(prob.ndof, size=min(n_modes, prob.ndof), replace=False))
    t0 = time.perf_counter()
    sys_ = osolver.ModalSystem(prob, modes=idx)
    if u0_nodal is not None:
        basis = fem.ClosedFormBasis(prob.n, prob.box, prob.D)
        sys_.c0 = basis.to_modal_from_nodal(u0_nodal.reshape(prob.n)).reshape(-1)[idx]
    res = osolver.parareal(sys_, tol=TOL, keep_history=False)
    dt = time.perf_counter() - t0
    units = len(idx) * prob.N * prob.M * res.k
    return units / dt, dt, len(idx), res.k, sys_, res, idx


def run_batch_learned(pe, args, barrier, probs):
    """The batched workload in the mixed, batched, learned-G form: a network trained on pairs the
    method generates over the batch family's ranges of lam dT and w dT (problems of the held-apart
    seed 7: their slice lengths, source frequencies and spectra), attached to every problem."""
    import torch

    dev = torch.device("cuda")
    rng = np.random.default_rng(77)
    ref = I.config4_problem(0)
    dT0 = ref.T / ref.N
    LT, WT = [], []
    for i in range(400):  # held-apart problems of the family (base seed 7)
        pr = I.config4_problem(i, base_seed=7)
        dT = pr.T / pr.N
        lmin = pr.D * sum(np.pi ** 2 / (hi - lo) ** 2 for lo, hi in pr.box)
        lmax = pr.D * sum(12.0 * (n + 1) ** 2 / (hi - lo) ** 2 for n, (lo, hi) in zip(pr.n, pr.box))
        ws = [t.tp[0] for t in pr.forcing if t.tkind == I.T_SIN]
        ls = np.exp(rng.uniform(np.log(lmin * dT), np.log(lmax * dT), 256))
        LT.append(np.repeat(ls, len(ws)))
        WT.append(np.tile(np.array(ws) * dT, 256))
    LT, WT = np.concatenate(LT), np.concatenate(WT)
    perm = rng.permutation(LT.size)
    out = {"training_pairs": int(LT.size), "seeds": "batch family, base seed 7, problems 0..399"}
    with pe.Solver(ref, precision=pe.PE_MIXED) as s:  # the unit response is a function of (lam dT, w dT)
        lam_d = torch.tensor(LT[perm] / dT0, device=dev)
        om_d = torch.tensor(WT[perm] / dT0, device=dev)
        x = torch.empty((LT.size, 2), device=dev, dtype=torch.float32)
        t = torch.empty((LT.size, 2), device=dev, dtype=torch.float32)
        s.learned_samples(lam_d, om_d, x, t)
    net = pe.MLP(seed=5)
    t1 = time.perf_counter()
    out["final_loss"] = net.train(x, t, epochs=max(1, 60000 // ((LT.size + 4095) // 4096)), batch=4096, lr=3e-3)
    torch.cuda.synchronize()
    out["seconds_training"] = time.perf_counter() - t1
    with pe.BatchSolver(probs, precision=pe.PE_MIXED, fine_engine=pe.PE_FINE_TC) as b:
        b.set_learned(net)
        for _ in range(max(1, args.warmup)):
            b.solve(tol=TOL)
        barrier()
        t0 = time.perf_counter()
        infos = [b.solve(tol=TOL) for _ in range(args.steps)]
        barrier()
        dt = (time.perf_counter() - t0) / args.steps
        r, k = b.status()
    out.update({"form": "batched, learned coarse correction", "time_to_tol_ms": 1e3 * dt,
                "value": infos[-1]["fine_dof_substeps"] / dt, "unit": UNIT,
                "iterations_histogram": {int(v): int((k == v).sum()) for v in np.unique(k)},
                "max_residual": float(r.max()), "graph_replays": infos[-1]["graph_replays"],
                "ms_prepare": infos[-1]["ms_prepare"], "ms_iterations": infos[-1]["ms_iterations"]})
    net.close()
    return out


def run_batch(pe, args, barrier):
    """512 uneven 2D problems: batched persistent mixed form vs a per-problem float64 loop."""
    probs = I.config4(count=args.batch_count)
    out = {"workload": f"{len(probs)} uneven 2D problems (n 31..511, 16-64 slices x 32 substeps, RK4/RK2)"}
    for name, eng, form in (("chosen", pe.PE_FINE_TC, "batched launches over (problem, mode block) items, CUDA graph per "
                                                      "iteration, float32 column sums, float64 recurrence and residual"),
                            ("simt", pe.PE_FINE_SIMT, "the same kernels through fine_engine = PE_FINE_SIMT")):
        with pe.BatchSolver(probs, precision=pe.PE_MIXED, fine_engine=eng) as b:
            b.autotune(None)
            for _ in range(max(1, args.warmup)):
                b.solve(tol=TOL)
            barrier()
            t0 = time.perf_counter()
            infos = [b.solve(tol=TOL) for _ in range(args.steps)]
            barrier()
            dt = (time.perf_counter() - t0) / args.steps
            r, k = b.status()
        units = infos[-1]["fine_dof_substeps"]
        out[name] = {"form": form, "time_to_tol_ms": 1e3 * dt, "value": units / dt, "unit": UNIT,
                     "max_iterations": int(k.max()), "max_residual": float(r.max()),
                     "graph_replays": infos[-1]["graph_replays"], "launch_shape": [infos[-1]["threads"],
                                                                                  infos[-1]["ctas_per_sm"]],
                     "ms_prepare": infos[-1]["ms_prepare"], "ms_iterations": infos[-1]["ms_iterations"],
                     "gpu_launches": infos[-1]["kernel_launches"]}
    if not args.no_learned:
        out["learned"] = run_batch_learned(pe, args, barrier, probs)
    dt = out["chosen"]["time_to_tol_ms"] / 1e3
    # plain: one problem after another, float64, host-driven iteration loop (solvers set up
    # before the timed region, as the batch is)
    solvers = [pe.Solver(prob, precision=pe.PE_FP64) for prob in probs]
    try:
        barrier()
        t0 = time.perf_counter()
        units_p = 0
        for prob, s in zip(probs, solvers):
            info = s.solve(tol=TOL)
            units_p += prob.ndof * prob.N * prob.M * info["fine_sweeps"]
        barrier()
        dtp = time.perf_counter() - t0
    finally:
        for s in solvers:
            s.close()
    out["plain"] = {"form": "float64, one problem per launch sequence", "time_to_tol_ms": 1e3 * dtp,
                    "value": units_p / dtp, "unit": UNIT}
    out["speedup_time_to_tol"] = dtp / dt
    return out


def run_config1(pe, args, barrier):
    """The 1D workload (63 interior nodes, 8 x 16, RK2/RK2, manufactured e^{-t} sin(pi x)): float64 to
    its own residual tolerance 1e-12 and to 1e-6, and the chosen mixed form
    to 1e-6; every mode checked against the oracle (a launch- and latency-bound size)."""
    from oracle import solver as osolver

    prob = I.config1()
    sys_ = osolver.ModalSystem(prob)
    out = {"workload": prob.label}
    for name, prec, tol in (("fp64_tol1e-12", pe.PE_FP64, 1e-12), ("fp64", pe.PE_FP64, TOL),
                            ("chosen", pe.PE_MIXED, TOL)):
        with pe.Solver(prob, precision=prec, stream=cur_stream(), **chosen_kw(pe, prec)) as s:
            ms, infos = timed_solves(s, max(10, args.steps), max(3, args.warmup), barrier, tol=tol)
            dt = ms / 1e3
            modal = s.modal(prob.N)
        ref = osolver.parareal(sys_, tol=tol)
        out[name] = {"time_to_tol_ms": 1e3 * dt, "iterations": infos[-1]["k"], "tol": tol,
                     "value": prob.ndof * prob.N * prob.M * infos[-1]["fine_sweeps"] / dt, "unit": UNIT,
                     "rel_l2_vs_oracle": osolver.rel_l2(modal, ref.U[-1], sys_.norm_w),
                     "gpu_launches": infos[-1]["kernel_launches"],
                     "phases_ms": {k: infos[-1][k] for k in ("ms_tables", "ms_prepare", "ms_iterations",
                                                             "ms_output")},
                     "options": {k: v for k, v in chosen_kw(pe, prec).items()}}
    out["speedup_time_to_tol"] = out["fp64"]["time_to_tol_ms"] / out["chosen"]["time_to_tol_ms"]
    return out


def run_learned(pe, args, barrier):
    """511^2 workload, 128 x 32: plain coarse step vs the learned coarse correction (mixed form).

    The network is trained on pairs the method generates from the source frequencies of the
    held-apart seeds 100000..101999 (lam log-uniform over the grid's spectrum); the solve is on seed 1.
    """
    import torch

    prob = I.config5(seed=1)
    dev = torch.device("cuda")
    out = {"workload": prob.label}
    with pe.Solver(prob, precision=pe.PE_MIXED, stream=cur_stream(), **chosen_kw(pe, pe.PE_MIXED)) as s:
        lam = s.lam()
        lo, hi = np.log(lam.min()), np.log(lam.max())
        rng = np.random.default_rng(2024)
        L, W = [], []
        for seed in range(100000, 102000):
            ws = [t.tp[0] for t in I.config5(seed=seed, n=prob.n[0]).forcing]
            ls = np.exp(rng.uniform(lo, hi, 64))
            L.append(np.repeat(ls, len(ws)))
            W.append(np.tile(ws, 64))
        L, W = np.concatenate(L), np.concatenate(W)
        perm = rng.permutation(L.size)
        lam_d = torch.tensor(L[perm], device=dev)
        om_d = torch.tensor(W[perm], device=dev)
        x = torch.empty((L.size, 2), device=dev, dtype=torch.float32)
        t = torch.empty((L.size, 2), device=dev, dtype=torch.float32)
        t0 = time.perf_counter()
        s.learned_samples(lam_d, om_d, x, t)
        torch.cuda.synchronize()
        t_samples = time.perf_counter() - t0
        net = pe.MLP(seed=3)
        epochs = max(1, 60000 // ((L.size + 4095) // 4096))
        t1 = time.perf_counter()
        loss = net.train(x, t, epochs=epochs, batch=4096, lr=3e-3)
        torch.cuda.synchronize()
        t_train = time.perf_counter() - t1
        steps = epochs * ((L.size + 4095) // 4096)
        # 6 FLOP per weight and sample (2 forward, 4 backward: input and weight gradients)
        weights = 2 * 64 + 64 * 64 + 64 * 2
        flops = 6.0 * weights * float(L.size) * epochs
        out["training"] = {"pairs": int(L.size), "seeds": "100000..101999", "final_loss": loss,
                           "adam_steps": steps, "batch": 4096, "seconds_samples": t_samples,
                           "seconds_training": t_train, "training_tflops": flops / t_train / 1e12,
                           "flops_note": "6 FLOP per weight (4352 weights) per sample and step"}
        res = {}
        for name, mlp in (("plain_G", None), ("learned_G", net)):
            s.set_learned(mlp)
            ms, infos = timed_solves(s, args.steps, max(1, args.warmup), barrier, tol=TOL)
            dt = ms / 1e3
            modal = s.modal(prob.N)
            res[name] = {"time_to_tol_ms": 1e3 * dt, "iterations": infos[-1]["k"],
                         "value": prob.ndof * prob.N * prob.M * infos[-1]["fine_sweeps"] / dt, "unit": UNIT,
                         "residual": infos[-1]["residual"], "modal": modal}
        s.set_learned(None)
    # the plain float64 form on the same workload (plain G)
    with pe.Solver(prob, precision=pe.PE_FP64, stream=cur_stream()) as s:
        ms, infos = timed_solves(s, max(1, min(args.steps, 3)), max(1, args.warmup), barrier, tol=TOL)
        dt = ms / 1e3
        res["fp64_plain_G"] = {"time_to_tol_ms": 1e3 * dt, "iterations": infos[-1]["k"],
                               "value": prob.ndof * prob.N * prob.M * infos[-1]["fine_sweeps"] / dt, "unit": UNIT,
                               "residual": infos[-1]["residual"], "modal": s.modal(prob.N)}
    rate, dtc, nm, k_or, sys_, ref, idx = oracle_sample(prob, 1024, seed=11)
    w = sys_.norm_w
    for name in res:
        m = res[name].pop("modal")
        res[name]["rel_l2_vs_oracle"] = float(np.sqrt(np.sum(w * (m[idx] - ref.U[-1]) ** 2)) /
                                              np.sqrt(np.sum(w * ref.U[-1] ** 2)))
    out.update(res)
    out["speedup_time_to_tol"] = res["plain_G"]["time_to_tol_ms"] / res["learned_G"]["time_to_tol_ms"]
    out["speedup_vs_fp64"] = res["fp64_plain_G"]["time_to_tol_ms"] / res["learned_G"]["time_to_tol_ms"]
    # the mixed, batched, learned-G form: four problems of the family (seeds 1..4) in one batch
    probs = [I.config5(seed=sd) for sd in (1, 2, 3, 4)]
    bat = {"workload": "4 problems of the family (seeds 1..4), one batch"}
    with pe.BatchSolver(probs, precision=pe.PE_MIXED, fine_engine=pe.PE_FINE_TC) as b:
        for name, mlp in (("batched_plain_G", None), ("batched_learned_G", net)):
            b.set_learned(mlp)
            for _ in range(max(1, args.warmup)):
                b.solve(tol=TOL)
            barrier()
            t1 = time.perf_counter()
            steps = max(1, min(args.steps, 5))
            infos = [b.solve(tol=TOL) for _ in range(steps)]
            barrier()
            dt = (time.perf_counter() - t1) / steps
            r, k = b.status()
            bat[name] = {"time_to_tol_ms": 1e3 * dt, "iterations": [int(v) for v in k],
                         "max_residual": float(r.max()), "value": infos[-1]["fine_dof_substeps"] / dt, "unit": UNIT,
                         "ms_prepare": infos[-1]["ms_prepare"], "ms_iterations": infos[-1]["ms_iterations"]}
            if mlp is not None:
                m1 = b.modal(0, prob.N)
        b.set_learned(None)
    bat["rel_l2_vs_oracle_problem0"] = float(np.sqrt(np.sum(w * (m1[idx] - ref.U[-1]) ** 2)) /
                                             np.sqrt(np.sum(w * ref.U[-1] ** 2)))
    # the plain form on the same four problems: float64, one problem after another
    solvers = [pe.Solver(pr, precision=pe.PE_FP64) for pr in probs]
    try:
        for sv in solvers:
            sv.solve(tol=TOL)
        barrier()
        t1 = time.perf_counter()
        for sv in solvers:
            sv.solve(tol=TOL)
        barrier()
        bat["fp64_per_problem_loop_ms"] = 1e3 * (time.perf_counter() - t1)
    finally:
        for sv in solvers:
            sv.close()
    bat["speedup_vs_fp64"] = bat["fp64_per_problem_loop_ms"] / bat["batched_learned_G"]["time_to_tol_ms"]
    out["batched"] = bat
    net.close()
    return out


def run_precision(pe, args, barrier):
    """The 3D 127^3 workload (64 slices x 32 substeps, 16 bumps): plain float64 against the mixed
    form, its error against the oracle before and after one float64 refinement iteration."""
    prob = I.config3()
    out = {"workload": prob.label}
    steps = max(1, min(args.steps, 2))
    rate, dtc, nm, k_or, sys_, ref, idx = oracle_sample(prob, 512, seed=13)
    w = sys_.norm_w

    def rel(m):
        return float(np.sqrt(np.sum(w * (m[idx] - ref.U[-1]) ** 2)) / np.sqrt(np.sum(w * ref.U[-1] ** 2)))

    for name, prec in (("fp64", pe.PE_FP64), ("mixed", pe.PE_MIXED)):
        with pe.Solver(prob, precision=prec, stream=cur_stream(), **chosen_kw(pe, prec)) as s:
            ms, infos = timed_solves(s, steps, 1, barrier, tol=TOL)
            dt = ms / 1e3
            rec = {"time_to_tol_ms": 1e3 * dt, "iterations": infos[-1]["k"],
                   "value": prob.ndof * prob.N * prob.M * infos[-1]["fine_sweeps"] / dt, "unit": UNIT,
                   "rel_l2_vs_oracle": rel(s.modal(prob.N))}
            if prec == pe.PE_MIXED:
                barrier()
                t0 = time.perf_counter()
                s.refine()
                barrier()
                rec["refine_ms"] = 1e3 * (time.perf_counter() - t0)
                rec["rel_l2_after_refine"] = rel(s.modal(prob.N))
            out[name] = rec
    out["speedup_time_to_tol"] = out["fp64"]["time_to_tol_ms"] / out["mixed"]["time_to_tol_ms"]
    out["oracle_sample"] = f"{nm} random modes of {prob.ndof}"
    return out


def run_cached(pe, args, barrier, u0_dev, u0_host):
    """The main workload with the forced part F^M(0) of every slice kept after the first sweep
    (exact, the fine propagator being affine); later iterations run no fine sweep.  Reported as
    time to tolerance only: the reused forced parts are not counted as fine substeps."""
    prob = workload()
    out = {"workload": prob.label + " with cached F^M(0)"}
    rate, dtc, nm, k_or, sys_, ref, idx = oracle_sample(prob, 1024, seed=17, u0_nodal=u0_host)
    w = sys_.norm_w
    for name, prec in (("fp64", pe.PE_FP64), ("mixed", pe.PE_MIXED)):
        with pe.Solver(prob, precision=prec, cache_forced=True, stream=cur_stream(), **chosen_kw(pe, prec)) as s:
            ms, infos = timed_solves(s, args.steps, max(1, args.warmup), barrier, tol=TOL,
                                     u0_kind=pe.PE_FIELD_NODAL, nodal=u0_dev)
            dt = ms / 1e3
            m = s.modal(prob.N)
        out[name] = {"time_to_tol_ms": 1e3 * dt, "iterations": infos[-1]["k"],
                     "fine_sweeps_executed": infos[-1]["fine_sweeps"],
                     "rel_l2_vs_oracle": float(np.sqrt(np.sum(w * (m[idx] - ref.U[-1]) ** 2)) /
                                               np.sqrt(np.sum(w * ref.U[-1] ** 2)))}
    return out


def dirichlet_problem():
    """The main workload with non-homogeneous Dirichlet data: two separable data terms (an
    exponentially decaying bilinear ramp and an oscillating sine product) on the closed box."""
    prob = workload()
    poly = lambda c0, c1: I.Factor(I.S_POLY, (c0, c1, 0.0, 0.0))  # noqa: E731
    g = (I.Term(0.8, (poly(1.0, 0.5), poly(0.5, -1.0)), I.T_EXP, (-0.5, 0.0)),
         I.Term(0.3, (I.Factor(I.S_SIN, (2.0, 0.4)), I.Factor(I.S_SIN, (1.5, 0.2))), I.T_SIN, (6.0, 0.3)))
    return I.Problem(prob.d, prob.n, prob.box, prob.D, prob.t0, prob.T, prob.N, prob.M, prob.fine_nodes,
                     prob.coarse_nodes, prob.u0, prob.forcing, prob.quad_pts, prob.tol, None,
                     prob.label + "_dirichlet2", g)


def run_dirichlet(pe, args, barrier):
    """Time to tolerance of the main workload with Dirichlet data (each data term adds 1 + d
    forcing terms), both forms.  Parity of this path is checked against the oracle in the GPU
    tests on smaller grids (the oracle's full-grid lifting route is too slow at 255^2)."""
    prob = dirichlet_problem()
    out = {"workload": prob.label}
    for name, prec in (("fp64", pe.PE_FP64), ("mixed", pe.PE_MIXED)):
        with pe.Solver(prob, precision=prec, stream=cur_stream(), **chosen_kw(pe, prec)) as s:
            ms, infos = timed_solves(s, args.steps, max(1, args.warmup), barrier, tol=TOL)
            dt = ms / 1e3
        out[name] = {"time_to_tol_ms": 1e3 * dt, "iterations": infos[-1]["k"],
                     "value": prob.ndof * prob.N * prob.M * infos[-1]["fine_sweeps"] / dt, "unit": UNIT}
    return out


def periodic_problem():
    """The main workload's forcing and slices on a grid periodic along x (256 nodes) and
    Dirichlet along y (255 interior nodes)."""
    prob = workload()
    return I.Problem(prob.d, (256, 255), prob.box, prob.D, prob.t0, prob.T, prob.N, prob.M, prob.fine_nodes,
                     prob.coarse_nodes, prob.u0, prob.forcing, prob.quad_pts, prob.tol, None,
                     "d2_n256p_x_255_N32_M64_bumps8", (), (True, False))


def run_periodic(pe, args, barrier):
    """Time to tolerance with a periodic axis (DHT basis along x), both forms, and the error
    against the oracle on sampled modes."""
    prob = periodic_problem()
    out = {"workload": prob.label}
    rate, dtc, nm, k_or, sys_, ref, idx = oracle_sample(prob, 1024, seed=19)
    w = sys_.norm_w
    for name, prec in (("fp64", pe.PE_FP64), ("mixed", pe.PE_MIXED)):
        with pe.Solver(prob, precision=prec, stream=cur_stream(), **chosen_kw(pe, prec)) as s:
            ms, infos = timed_solves(s, args.steps, max(1, args.warmup), barrier, tol=TOL)
            dt = ms / 1e3
            m = s.modal(prob.N)
        out[name] = {"time_to_tol_ms": 1e3 * dt, "iterations": infos[-1]["k"],
                     "value": prob.ndof * prob.N * prob.M * infos[-1]["fine_sweeps"] / dt, "unit": UNIT,
                     "rel_l2_vs_oracle": float(np.sqrt(np.sum(w * (m[idx] - ref.U[-1]) ** 2)) /
                                               np.sqrt(np.sum(w * ref.U[-1] ** 2)))}
    return out


DST_SHAPE = (511, 511, 255)


def run_dst(pe, args, barrier):
    """Tensor DST-I of a (511, 511, 255) grid (every axis, n + 1 a power of two: the FFT kernels)
    in float64 and float32, and the tcgen05 split-bf16 form (float32 in/out).  Algorithmic bytes per
    call: one read and one write of the grid per axis pass.  L2 flushed before every call."""
    import torch

    dev = torch.device("cuda")
    n = DST_SHAPE
    size = int(np.prod(n))
    flush = torch.empty(2 * L2_BYTES // 4, dtype=torch.float32, device=dev)
    peaks = measured_peaks() or {}
    hbm = float(peaks.get("hbm_gbs", 6800.0))
    stream = torch.cuda.current_stream(dev)
    out = {"shape": list(n), "hbm_peak_gbs": hbm}
    forms = (("f64", torch.float64, lambda x, y: pe.dst(3, n, x, y)),
             ("f32", torch.float32, lambda x, y: pe.dst(3, n, x, y, f32=True)),
             ("tc_bf16x3", torch.float32, lambda x, y: pe.dst_tc(3, n, x, y, nsplit=3)))
    gen = torch.Generator(device=dev).manual_seed(5)
    for name, dt, fn in forms:
        x = torch.randn(size, dtype=dt, device=dev, generator=gen)
        y = torch.empty_like(x)
        for _ in range(max(1, args.warmup)):
            fn(x, y)
        barrier()
        times = []
        for _ in range(max(1, args.steps)):
            flush.fill_(1.0)
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            fn(x, y)
            e1.record(stream)
            e1.synchronize()
            times.append(e0.elapsed_time(e1))
        ms = float(np.median(times))
        nbytes = 3 * 2 * size * x.element_size()
        out[name] = {"ms": ms, "algorithmic_bytes": nbytes, "gbs": nbytes / (ms / 1e3) / 1e9,
                     "frac_hbm": nbytes / (ms / 1e3) / 1e9 / hbm}
        del x, y
    return out


def run_general(pe, args, barrier, u0_dev, u0_host):
    """The 255^2 workload through the general forcing path: the source at every one of the
    32 x 64 x 4 fine stage times, per sweep (products of transformed axis factors).  Parity against the oracle on
    1024 sampled modes (the source is separable: the oracle's element quadrature of it equals
    its per-axis route, which runs on a mode subset)."""
    prob = workload()
    out = {"workload": prob.label + " general forcing path (source at every stage time)"}
    rate, dtc, nm, k_or, sys_, ref, idx = oracle_sample(prob, 1024, seed=23, u0_nodal=u0_host)
    w = sys_.norm_w
    for name, prec in (("fp64", pe.PE_FP64), ("mixed", pe.PE_MIXED)):
        with pe.Solver(prob, precision=prec, forcing_path=pe.PE_FORCING_GENERAL, stream=cur_stream()) as s:
            ms, infos = timed_solves(s, max(1, args.steps // 2), max(1, args.warmup), barrier, tol=TOL,
                                     u0_kind=pe.PE_FIELD_NODAL, nodal=u0_dev)
            dt = ms / 1e3
            m = s.modal(prob.N)
        sweeps = infos[-1]["fine_sweeps"]
        out[name] = {"time_to_tol_ms": 1e3 * dt, "iterations": infos[-1]["k"],
                     "value": prob.ndof * prob.N * prob.M * sweeps / dt, "unit": UNIT,
                     "source_evaluations_per_step": sweeps * prob.N * prob.M * prob.q + prob.N * prob.p,
                     "rel_l2_vs_oracle": float(np.sqrt(np.sum(w * (m[idx] - ref.U[-1]) ** 2)) /
                                               np.sqrt(np.sum(w * ref.U[-1] ** 2)))}
    return out


EX4_PAIRS = ((0.01, 1.0), (0.01, 10.0), (0.1, 1.0), (0.1, 10.0))


def run_example4(pe, args, barrier):
    """Example 4 of Sec. 5 at the paper's size (N_x = 1024, 4 x 16 slices, three stage and three
    coarse nodes, moving hat source) through the general forcing path: set-up plus k = 4 Parareal
    iterations for every (alpha, f) pair, float64 and mixed.  A launch-bound 1D workload."""

    out = {"workload": "ex4_Nx1024_4x16_q3_p3 general forcing path, k = 4"}
    for alpha, freq in EX4_PAIRS:
        prob = I.example4(1024, alpha, freq, 4, 16, 3, 3)
        rec = {}
        for name, prec in (("fp64", pe.PE_FP64), ("mixed", pe.PE_MIXED)):
            with pe.Solver(prob, precision=prec, forcing_path=pe.PE_FORCING_GENERAL) as s:
                def run():
                    s.set_problem()
                    return [s.iterate() for _ in range(4)]
                for _ in range(max(1, args.warmup)):
                    run()
                barrier()
                t0 = time.perf_counter()
                for _ in range(args.steps):
                    res = run()
                barrier()
                dt = (time.perf_counter() - t0) / args.steps
            rec[name] = {"ms": 1e3 * dt, "residuals": res,
                         "value": prob.ndof * prob.N * prob.M * 4 / dt, "unit": UNIT}
        out[f"a{alpha}_f{freq}"] = rec
    return out


def chosen_rooflines(prob, chosen, plain, fma):
    """Rooflines of the sweeps' kernels: CUDA-event times measured inside the library on the
    launching stream (host-driven loop), algorithmic work of the solve's passes.  The walk takes
    six float64 operations per mode and slice in the first pass (which makes the coarse iterate
    too) and five in each further one; counted as one FMA each."""
    peaks = measured_peaks() or {}
    hbm = float(peaks.get("hbm_gbs", 6788.6))
    nd, N = prob.ndof, prob.N
    out = []
    for name, rec, key, nbytes in (
            ("walk_kernel (chosen)", chosen, "ms_fine_launch", 8 * N * nd + 16 * N * nd * (chosen["k"] - 1)),
            ("walk_kernel (float64)", plain, "ms_corr_launch", 24 * N * nd * plain["k"])):
        ms = rec[key] * rec["k"]
        flops = 2 * N * nd * (6 + 5 * (rec["k"] - 1))
        out.append({"kernel": name, "bound": "alu", "ms": ms, "achieved": flops / (ms / 1e3) / 1e12,
                    "peak": fma["fp64_tflops"], "unit": "TFLOP/s", "frac": flops / (ms / 1e3) / 1e12 / fma["fp64_tflops"],
                    "passes": rec["k"], "hbm_gbs": nbytes / (ms / 1e3) / 1e9, "hbm_frac": nbytes / (ms / 1e3) / 1e9 / hbm,
                    "peak_source": "pe_measure_fma_peak(PE_FP64)",
                    "note": "float64 operations of the recurrences and residual sums; the chosen form's float32 "
                            "column sums run under them"})
    return out


def allmax(x, dist=None, device="cpu"):
    """The maximum of x over all ranks (x itself without a process group): the timed region of
    a replica run ends when the slowest rank ends."""
    if dist is None:
        return x
    import torch

    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def replica_throughput(units_per_rank, max_ms, world):
    """Whole-job throughput of `world` independent replicas: all ranks' units over the slowest
    rank's time (weak scaling: the per-rank workload is fixed)."""
    return units_per_rank * world / (max_ms / 1e3)


def run_reference(args, rank, world):
    """The reference arm: the CPU oracle as it stands, on a bounded sample of the workload."""
    if rank != 0:
        return
    prob = workload()
    n_modes = 16384
    for _ in range(args.warmup):
        oracle_sample(prob, 32, seed=99)
    t_total, units_total = 0.0, 0
    for s in range(args.steps):
        rate, dt, nm, k, *_ = oracle_sample(prob, n_modes, seed=s)
        t_total += dt
        units_total += nm * prob.N * prob.M * k
    value = units_total / t_total
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * t_total / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": prob.label, "ndof": prob.ndof, "slices": prob.N, "substeps": prob.M,
                   "fine_stages": prob.q, "forcing_terms": prob.R},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle",
                         "sample": f"{n_modes} random modes of {prob.ndof} per step, full Parareal to rel "
                                   f"residual {TOL} (k=2 fine sweeps of {prob.N}x{prob.M} substeps)"},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="native", choices=["native", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-batch", action="store_true", help="skip the 512-problem batched workload")
    ap.add_argument("--no-learned", action="store_true", help="skip the learned coarse correction workload")
    ap.add_argument("--no-general", action="store_true", help="skip the general forcing path workload")
    ap.add_argument("--batch-count", type=int, default=512,
                    help="problems in the batched workload (512; fewer only for small profiling captures)")
    ap.add_argument("--no-dst", action="store_true", help="skip the standalone DST-I measurement")
    ap.add_argument("--no-precision", action="store_true", help="skip the 3D 127^3 precision workload")
    ap.add_argument("--no-cached", action="store_true", help="skip the cached-F^M(0) line")
    ap.add_argument("--no-dirichlet", action="store_true", help="skip the Dirichlet-data line")
    ap.add_argument("--no-periodic", action="store_true", help="skip the periodic-axis line")
    ap.add_argument("--no-example4", action="store_true", help="skip the Example 4 paper-size line")
    ap.add_argument("--no-config1", action="store_true", help="skip the 1D 63-node workload line")
    ap.add_argument("--only", choices=["batch", "learned", "general", "dst", "precision", "cached", "dirichlet",
                                       "periodic", "example4", "config1"],
                    help="run one secondary workload alone and print its record (for profiling)")
    args = ap.parse_args()

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))

    if args.impl == "reference":
        run_reference(args, rank, world)
        return

    import torch

    dist = None
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    else:
        torch.cuda.set_device(0)

    from paper_2412_01138_gb300 import pe

    prob = workload()
    dev = torch.device("cuda", local if world > 1 else 0)
    stream = torch.cuda.current_stream(dev)
    u0_host = nodal_u0(prob)
    u0_dev = torch.from_numpy(u0_host).to(dev)
    flush = torch.empty(2 * L2_BYTES // 4, dtype=torch.float32, device=dev)
    out_dev = torch.empty(prob.ndof, dtype=torch.float64, device=dev)

    def barrier():
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize(dev)

    def timed_steps(solver, steps, warmup, nodal):
        for _ in range(warmup):
            solver.solve(tol=TOL, u0_kind=pe.PE_FIELD_NODAL, nodal=nodal)
        barrier()
        total_ms, infos = 0.0, []
        for _ in range(steps):
            flush.fill_(1.0)  # evict the working set from L2 between steps
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            # the whole solve enqueued through the stream-ordered API (with the loop on the device
            # nothing in it waits for the host), the report read after the closing event
            e0.record(stream)
            solver.solve_async(tol=TOL, u0_kind=pe.PE_FIELD_NODAL, nodal=nodal, out=out_dev)
            e1.record(stream)
            info = solver.wait()
            e1.synchronize()
            total_ms += e0.elapsed_time(e1)
            infos.append(info)
        barrier()
        return total_ms, infos

    if args.only:
        run = {"batch": lambda: run_batch(pe, args, barrier), "learned": lambda: run_learned(pe, args, barrier),
               "general": lambda: run_general(pe, args, barrier, u0_dev, u0_host),
               "config1": lambda: run_config1(pe, args, barrier),
               "dst": lambda: run_dst(pe, args, barrier),
               "precision": lambda: run_precision(pe, args, barrier),
               "cached": lambda: run_cached(pe, args, barrier, u0_dev, u0_host),
               "dirichlet": lambda: run_dirichlet(pe, args, barrier),
               "periodic": lambda: run_periodic(pe, args, barrier),
               "example4": lambda: run_example4(pe, args, barrier)}[args.only]
        rec = run()
        if rank == 0:
            print(json.dumps({"section": args.only, **rec}))
        return

    # measured FMA peaks of the CUDA cores (outside every timed region)
    measured_fma = {"fp64_tflops": pe.measure_fma_peak(pe.PE_FP64, stream),
                    "fp32_tflops": pe.measure_fma_peak(pe.PE_MIXED, stream)}
    results = {}
    with ClockSampler(local if world > 1 else 0) as clocks:
        for name, precision, eng, dl in (("fp64", pe.PE_FP64, pe.PE_FINE_SIMT, 0),
                                         ("mixed_simt", pe.PE_MIXED, pe.PE_FINE_SIMT, 0),
                                         ("mixed", pe.PE_MIXED, pe.PE_FINE_TC, 2)):
            with pe.Solver(prob, precision=precision, stream=stream, fine_engine=eng, device_loop=dl) as s:
                total_ms, infos = timed_steps(s, args.steps, args.warmup, u0_dev)
                modal = s.modal(prob.N)
                # end to end through the C-ABI with host buffers: H2D of u0, D2H of the solution
                out_host = np.empty(prob.ndof)
                s.solve(tol=TOL, u0_kind=pe.PE_FIELD_NODAL, nodal=u0_host, out=out_host)
                barrier()
                t0 = time.perf_counter()
                for _ in range(args.steps):
                    s.solve(tol=TOL, u0_kind=pe.PE_FIELD_NODAL, nodal=u0_host, out=out_host)
                e2e_s = time.perf_counter() - t0
            results[name] = dict(total_ms=total_ms, infos=infos, modal=modal, e2e_s=e2e_s)
        # per-kernel device times of the chosen form's kernels (its device-resident loop does not
        # time kernels one by one): the same solve with the host-driven loop
        with pe.Solver(prob, precision=pe.PE_MIXED, stream=stream, fine_engine=pe.PE_FINE_TC) as s:
            _, kinfos = timed_steps(s, args.steps, args.warmup, u0_dev)
        results["mixed"]["kernel_infos"] = kinfos
        batch = None if args.no_batch else run_batch(pe, args, barrier)
        learned = None if args.no_learned else run_learned(pe, args, barrier)
        general = None if args.no_general else run_general(pe, args, barrier, u0_dev, u0_host)
        config1 = None if args.no_config1 else run_config1(pe, args, barrier)
        dst = None if args.no_dst else run_dst(pe, args, barrier)
        precision = None if args.no_precision else run_precision(pe, args, barrier)
        cached = None if args.no_cached else run_cached(pe, args, barrier, u0_dev, u0_host)
        dirichlet = None if args.no_dirichlet else run_dirichlet(pe, args, barrier)
        periodic = None if args.no_periodic else run_periodic(pe, args, barrier)
        example4 = None if args.no_example4 else run_example4(pe, args, barrier)
    clock = clocks.summary()

    # max over ranks
    for r in results.values():
        r["total_ms"] = allmax(r["total_ms"], dist, dev)
        r["e2e_s"] = allmax(r["e2e_s"], dist, dev)

    if rank != 0:
        if dist is not None:
            dist.destroy_process_group()
        return

    def summarize(r):
        k = r["infos"][-1]["k"]
        kin = r.get("kernel_infos", r["infos"])
        units = prob.ndof * prob.N * prob.M * sum(i["fine_sweeps"] for i in r["infos"])
        value = replica_throughput(units, r["total_ms"], world)
        e2e_units = prob.ndof * prob.N * prob.M * k * args.steps * world
        ms_fine = np.mean([i["ms_fine_kernel"] / max(i["fine_sweeps"], 1) for i in kin])
        phases = {key: float(np.mean([i[key] for i in r["infos"]]))
                  for key in ("ms_tables", "ms_prepare", "ms_iterations", "ms_output", "ms_coarse_kernel")}
        for key in ("ms_fine_kernel", "ms_correction_kernel"):
            phases[key] = float(np.mean([i[key] for i in kin]))
        ms_corr = np.mean([i["ms_correction_kernel"] / max(i["k"], 1) for i in kin])
        return dict(value=value, k=k, ms_per_step=r["total_ms"] / args.steps, e2e=e2e_units / r["e2e_s"],
                    ms_fine_launch=ms_fine, ms_corr_launch=float(ms_corr),
                    ms_coarse=phases["ms_coarse_kernel"], launches=r["infos"][-1]["kernel_launches"],
                    residual=r["infos"][-1]["residual"], phases=phases)

    plain = summarize(results["fp64"])
    chosen = summarize(results["mixed"])
    simt = summarize(results["mixed_simt"])

    # parity of both forms on sampled modes against the oracle (outside the timed region);
    # the same run is the CPU baseline (the oracle as it stands, one core)
    # every mode of the workload: the parity check covers the whole field; the oracle is
    # repeated (up to 3 passes, about 10 s of one core) for the CPU rate
    rate, dt, nm, k_or, sys_, ref, idx = oracle_sample(prob, prob.ndof, seed=7, u0_nodal=u0_host)
    w = sys_.norm_w
    cpu_passes, cpu_s, cpu_units = 1, dt, nm * prob.N * prob.M * k_or
    while not args.no_cpu_baseline and cpu_s < 10.0 and cpu_passes < 3:
        r2 = oracle_sample(prob, prob.ndof, seed=7, u0_nodal=u0_host)
        cpu_passes, cpu_s, cpu_units = cpu_passes + 1, cpu_s + r2[1], cpu_units + r2[2] * prob.N * prob.M * r2[3]

    all_cores = None
    if not args.no_cpu_baseline and rank == 0:
        all_cores = oracle_all_cores(prob, u0_host)

    def rel(a):
        return float(np.sqrt(np.sum(w * (a[idx] - ref.U[-1]) ** 2)) / np.sqrt(np.sum(w * ref.U[-1] ** 2)))

    err_plain, err_chosen = rel(results["fp64"]["modal"]), rel(results["mixed"]["modal"])
    err_simt = rel(results["mixed_simt"]["modal"])
    cpu = None
    if not args.no_cpu_baseline:
        cpu = {"value": cpu_units / cpu_s, "unit": UNIT, "cores": 1, "kind": "oracle",
               "sample": f"the whole workload ({nm} of {prob.ndof} modes), Parareal to rel residual {TOL} "
                         f"(k={k_or} sweeps of {prob.N}x{prob.M} substeps), {cpu_passes} pass(es), {cpu_s:.1f} s",
               "all_cores": all_cores}

    # the float64 form's forced parts: both propagators' in the first pass, the fine one's after it
    flops_solve = 2 * stage_columns(prob) * prob.ndof * prob.N * (plain["k"] + 1)
    ms_forced = plain["ms_fine_launch"] * plain["k"]
    achieved = flops_solve / (ms_forced / 1e3) / 1e12
    sm_mhz = clock.get("sm_max_mhz") or 2070.0
    peak = fp64_peak_tflops(sm_mhz)
    fma = measured_fma
    kernel_rooflines = chosen_rooflines(prob, chosen, plain, fma)

    line = {
        "metric": METRIC,
        "value": plain["value"],
        "unit": UNIT,
        "n_gpus": world,
        "steps": args.steps,
        "warmup": args.warmup,
        "ms_per_step": plain["ms_per_step"],
        "higher_is_better": True,
        "scaling": "weak",
        "vs_baseline": None,
        "dtype": "f64",
        "data": "synthetic",
        "config": {"workload": prob.label, "d": prob.d, "n": list(prob.n), "slices": prob.N,
                   "substeps": prob.M, "fine_stages": prob.q, "coarse_stages": prob.p, "forcing_terms": prob.R,
                   "tol": TOL, "l2": "flushed between steps (256 MiB write)",
                   "parallelism": f"replicas x{world}"},
        "time_to_tol_ms": plain["ms_per_step"],
        "iterations": plain["k"],
        "rel_l2_vs_oracle": err_plain,
        "substeps": "fine DoF*substeps are the method's (Ndof x slices x substeps x fine sweeps run): a sweep "
                    "evaluates F^M on every mode and slice, its M substeps of q stages contracted exactly to one "
                    "sum over the source's time columns",
        "chosen": {"form": "mixed: float32 column sums under float64 recurrences, correction and residual, one kernel "
                           "per iteration (the coarse sweep in the first); Parareal loop on the device (one CUDA graph "
                           "with a conditional while node), set-up and output phases replayed as CUDA graphs, "
                           "the solve enqueued with pe_solve_async and its nodal output written by the solve; "
                           "kernel times from the same solve with the host-driven loop",
                   "value": chosen["value"], "unit": UNIT, "time_to_tol_ms": chosen["ms_per_step"],
                   "iterations": chosen["k"], "rel_l2_vs_oracle": err_chosen, "dtype": "f32",
                   "speedup_time_to_tol": plain["ms_per_step"] / chosen["ms_per_step"],
                   "iteration_kernel_ms": chosen["ms_fine_launch"],
                   "e2e": chosen["e2e"], "phases_ms": chosen["phases"]},
        "mixed_simt": {"form": "the same kernels through fine_engine = PE_FINE_SIMT",
                       "value": simt["value"], "unit": UNIT, "time_to_tol_ms": simt["ms_per_step"],
                       "iterations": simt["k"], "rel_l2_vs_oracle": err_simt,
                       "iteration_kernel_ms": simt["ms_fine_launch"],
                       "e2e": simt["e2e"]},
        "phases_ms": plain["phases"],
        "roofline": {"kernel": "forced_f64_kernel", "bound": "alu", "achieved": achieved, "peak": peak,
                     "unit": "TFLOP/s", "frac": achieved / peak, "traffic": None,
                     "peak_source": "derived: 152 SMs x 2 FP64 FMA/clk x 2 FLOP x max SM clock",
                     "peak_measured": fma["fp64_tflops"], "frac_of_measured": achieved / fma["fp64_tflops"],
                     "peak_measured_source": "pe_measure_fma_peak(PE_FP64): independent FMA chains, best of 5",
                     "flops_per_solve": flops_solve, "ms_per_solve": ms_forced,
                     "unit_of_work": "2 K FLOP per mode, slice and propagator (K = 17 time columns: one per "
                                     "exponential, two per sinusoid); k + 1 of them per solve, the coarse forcing "
                                     "in the first pass and the fine one in each"},
        "kernel_rooflines": kernel_rooflines,
        "measured_fma_peaks": fma,
        "e2e": {"value": plain["e2e"], "unit": UNIT, "h2d_bytes_per_step": prob.ndof * 8,
                "d2h_bytes_per_step": prob.ndof * 8 + 16 * plain["k"]},
        "gpu_launches": int(plain["launches"] + 0) * args.steps,
        "clocks": clock,
        "cpu_baseline": cpu,
        "config1": config1,
        "batched": batch,
        "learned": learned,
        "general": general,
        "dst": dst,
        "precision": precision,
        "affine_cached": cached,
        "dirichlet": dirichlet,
        "periodic": periodic,
        "example4": example4,
    }
    print(json.dumps(line))
    if dist is not None:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
