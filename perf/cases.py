"""The workloads by which this framework's speed is followed.

Each case is one call, or one short sequence of calls, that a program using the binding
(``paper_2412_01138_gb300.pe``) makes in earnest: a solve to tolerance on a line, a plane or a
box, a batch of uneven problems, a solve with a moving source, a standalone sine transform, the
training of the learned coarse correction.  Grids and time partitions are those of the
workloads in ``paper_2412_01138_gb300/inputs.py`` and of the tests; ``draw`` spreads over the
same ranges.

What a program keeps between calls (the solver of one grid and time partition, the buffers, the
problem's descriptors) is made by ``prepare``; ``run`` is the call.  Initial data and sources
follow the seed.  The mixed-precision form states a relative error of 1e-6, the accuracy of
float32, so a program hands its field on as float32 and that is what is returned here; float64
solves return float64.
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_2412_01138_gb300 import inputs as I

_PRECISIONS = ("float64", "mixed")


def _device() -> torch.device:
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _solve(name, n, N, M, q, p, bumps, D, precision, **more):
    """A Parareal solve on n interior nodes per axis, N slices of M substeps, q fine and p coarse
    stages, `bumps` oscillating Gaussian sources beside the manufactured exponential one."""
    case = {"name": name, "kind": "solve", "d": len(n), "n0": n[0], "n1": n[1] if len(n) > 1 else 1,
            "n2": n[2] if len(n) > 2 else 1, "N": N, "M": M, "q": q, "p": p, "bumps": bumps, "D": D, "T": 1.0,
            "omega": 20.0, "precision": precision, "tensor_cores": False, "loop": 0, "u0": "nodal",
            "random_coarse": False, "boundary": 0, "periodic": False, "host": False, "tol": 1e-6}
    case.update(more)
    return case


def listed():
    return [
        # The smallest problem: a 63-node line, descriptors in, host array out, default options.
        # What counts is the number of launches and waits.
        _solve("line_63_float64", (63,), 8, 16, 2, 2, 0, 1.0, "float64", u0="terms", host=True, tol=1e-12),
        # The plain method at its usual size: 255 x 255 nodes in float64, host-driven loop.
        _solve("plane_255_float64", (255, 255), 32, 64, 4, 2, 8, 0.1, "float64", random_coarse=True),
        # The same workload in the form chosen for speed: mixed precision, the stream-ordered call,
        # a problem solved again and again (device-side loop, replayed set-up).
        _solve("plane_255_mixed", (255, 255), 32, 64, 4, 2, 8, 0.1, "mixed", tensor_cores=True, loop=2,
               random_coarse=True),
        # Grid sizes without an FFT form, non-homogeneous Dirichlet data, three stages, float64.
        _solve("plane_200x117_dirichlet", (200, 117), 20, 24, 3, 2, 5, 0.15, "float64", loop=1, boundary=2,
               tol=1e-10),
        # The long time interval of the learned workload: 511 x 511 nodes, 128 slices, fast sources.
        _solve("plane_511_mixed", (511, 511), 128, 32, 4, 2, 12, 0.02, "mixed", tensor_cores=True, loop=1, T=2.0,
               omega=50.0),
        # Three dimensions at full size, the largest state (an array of 64 slices of 2.05M values).
        _solve("space_127_mixed", (127, 127, 127), 64, 32, 4, 2, 16, 0.05, "mixed", tensor_cores=True, loop=1,
               u0="terms"),
        # A periodic axis (Hartley transform) with the default engine and loop of the mixed form.
        _solve("plane_256_periodic_mixed", (256, 255), 32, 64, 4, 2, 8, 0.1, "mixed", periodic=True),
        # Many uneven problems advanced together, then every solution fetched.
        {"name": "batch_64_mixed", "kind": "batch", "count": 64, "family": 4, "precision": "mixed",
         "tensor_cores": True, "tol": 1e-6},
        # A source that moves: the load is assembled and transformed at every stage time.
        {"name": "hat_255x127_float64", "kind": "hat", "d": 2, "n0": 255, "n1": 127, "N": 8, "M": 32, "q": 4, "p": 2,
         "bumps": 3, "precision": "float64", "tol": 1e-6},
        # The sine transform alone, as a spectral program calls it: a large box in float32 ...
        {"name": "transform_511x511x255_float32", "kind": "transform", "d": 3, "n0": 511, "n1": 511, "n2": 255,
         "float32": True},
        # ... and one plane in float64.
        {"name": "transform_255x255_float64", "kind": "transform", "d": 2, "n0": 255, "n1": 255, "n2": 1,
         "float32": False},
        # A new network for the learned correction: training steps, then inference.
        {"name": "train_64_steps", "kind": "train", "samples": 65536, "batch": 4096, "epochs": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("line", "plane", "plane", "plane", "space", "batch", "hat", "transform", "transform", "train"))
    if kind == "train":
        batch = _log(rng, 256, 8192)
        steps = _log(rng, 4, 24)
        return {"kind": "train", "samples": batch * steps - rng.randrange(batch // 2), "batch": batch,
                "epochs": rng.randint(1, 4)}
    if kind == "transform":
        single = rng.random() < 0.5
        d = rng.randint(1, 3)
        while True:
            n = [_log(rng, 7, (4000, 1023, 511)[d - 1]) for _ in range(d)]
            fft = [2 ** round(math.log2(v + 1)) - 1 if rng.random() < 0.5 else v for v in n]
            ragged, n = fft != [2 ** round(math.log2(v + 1)) - 1 for v in n], fft + [1] * (3 - d)
            # axes without an FFT form cost n operations a value, most of all in float64
            if n[0] * n[1] * n[2] <= 511 * 511 * 255 // ((4 if single else 16) if ragged else 1):
                break
        return {"kind": "transform", "d": d, "n0": n[0], "n1": n[1], "n2": n[2], "float32": single}
    if kind == "hat":
        n0, n1, N, q = _log(rng, 31, 255), _log(rng, 31, 127), rng.randint(4, 8), rng.randint(2, 4)
        M = min(rng.randint(4, 32), max(4, 12000000 // (n0 * n1 * N * q)))
        return {"kind": "hat", "d": 2, "n0": n0, "n1": n1, "N": N, "M": M, "q": q, "p": 2, "bumps": rng.randint(0, 3),
                "precision": rng.choice(_PRECISIONS), "tol": 1e-6}
    if kind == "batch":
        precision = rng.choice(_PRECISIONS)
        return {"kind": "batch", "count": _log(rng, 4, 64 if precision == "mixed" else 8),
                "family": rng.randint(5, 1 << 20), "precision": precision,
                "tensor_cores": precision == "mixed" and rng.random() < 0.5, "tol": 1e-6}
    precision = rng.choice(_PRECISIONS)
    N, M = _log(rng, 4, 128), _log(rng, 4, 96)
    cores = precision == "mixed" and rng.random() < 0.5
    if cores:
        M = 16 * rng.randint(1, 6)
    lim = 3e9 if precision == "mixed" else 1e8
    while True:
        if kind == "line":
            n = (_log(rng, 31, 8191),)
        elif kind == "plane":
            n = (_log(rng, 31, 511), _log(rng, 31, 511))
        else:
            n = (_log(rng, 9, 127), _log(rng, 9, 127), _log(rng, 9, 127))
        if rng.random() < 0.4:
            n = tuple(2 ** round(math.log2(v + 1)) - 1 for v in n)
        if math.prod(n) * N * M <= lim:
            break
        N = max(4, N // 2)
    boundary = rng.choice((0, 0, 0, 1, 2)) if len(n) < 3 else 0
    return _solve("", n, N, M, rng.randint(2, 4), 2, rng.randint(0, 16 - 4 * boundary),
                  math.exp(rng.uniform(math.log(0.01), 0.0)), precision, tensor_cores=cores, loop=rng.randint(0, 2),
                  u0=rng.choice(("nodal", "nodal", "terms")), random_coarse=rng.random() < 0.3, boundary=boundary,
                  periodic=not boundary and rng.random() < 0.2) | {"name": "solve"}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _boundary_terms(rng, d, count):
    out = []
    for i in range(count):
        facs = tuple(I.Factor(I.S_POLY, (1.0 + 0.3 * a, rng.uniform_range(-0.5, 0.5), 0.2, 0.0)) for a in range(d))
        out.append(I.Term(rng.uniform_range(0.3, 0.8), facs, I.T_EXP, (-rng.uniform(), 0.0)) if i % 2 == 0 else
                   I.Term(rng.uniform_range(0.3, 0.8), facs, I.T_SIN, (rng.uniform_range(1.0, 5.0), rng.uniform())))
    return tuple(out)


def _problem(case, seed) -> I.Problem:
    rng = I.SplitMix64(1000003 * seed + 17)
    d = case["d"]
    n = (case["n0"], case["n1"], case.get("n2", 1))[:d]
    box = ((0.0, 1.0),) * d
    if case["kind"] == "hat":
        u0, f, _ = I.sin_mode(d, box, 0.05)
        hat = I.Term(rng.uniform_range(2.0, 4.0),
                     (I.Factor(I.S_MOVING_HAT, (0.5, 0.35, rng.uniform_range(1.0, 2.0), 0.1)),
                      I.Factor(I.S_GAUSS, (rng.uniform_range(0.4, 0.6), 0.15))))
        return I.Problem(d, n, box, 0.05, 0.0, 1.0, case["N"], case["M"], I.uniform_nodes(case["q"]),
                         I.uniform_nodes(case["p"]), u0, f + (hat,) + I.gaussian_bumps(rng, d, case["bumps"]), 3,
                         case["tol"])
    D = case["D"]
    u0, f, _ = I.sin_mode(d, box, D)
    u0 = tuple(dataclasses.replace(t, amp=rng.uniform_range(0.5, 1.5)) for t in u0)
    coarse = I.draw_random_nodes(case["p"], 2) if case["random_coarse"] else I.uniform_nodes(case["p"])
    bumps = I.gaussian_bumps(rng, d, case["bumps"], omega=(1.0, case["omega"]))
    periodic = (True,) + (False,) * (d - 1) if case["periodic"] else ()
    return I.Problem(d, n, box, D, 0.0, case["T"], case["N"], case["M"], I.uniform_nodes(case["q"]), coarse, u0,
                     f + bumps, 3, case["tol"], None, "", _boundary_terms(rng, d, case["boundary"]), periodic)


def _nodal_u0(case, seed) -> torch.Tensor:
    """Smooth nodal data: four separable products of low sine modes (cosines along a periodic axis)."""
    rng = I.SplitMix64(7919 * seed + 3)
    d = case["d"]
    dev = _device()
    out = None
    for _ in range(4):
        term = torch.full((), rng.normal(), dtype=torch.float64, device=dev)
        for a in range(d):
            n = case["n%d" % a]
            j = rng.randint(1, 4)
            if a == 0 and case["periodic"]:
                x = torch.cos(torch.arange(n, dtype=torch.float64, device=dev) * (2.0 * math.pi * j / n))
            else:
                x = torch.sin(torch.arange(1, n + 1, dtype=torch.float64, device=dev) * (math.pi * j / (n + 1)))
            term = term.unsqueeze(-1) * x
        out = term if out is None else out + term
    return out.reshape(-1).contiguous()


def _batch_problems(case, seed):
    out = []
    for i in range(case["count"]):
        p = I.config4_problem(i, case["family"])
        rng = I.SplitMix64(((seed + 1) << 20) + i)
        bumps = I.gaussian_bumps(rng, 2, p.R - 1)
        out.append(dataclasses.replace(p, forcing=p.forcing[:1] + bumps))
    return out


def _values(case, seed):
    g = torch.Generator(device=_device()).manual_seed(seed)
    n = case["n0"] * case["n1"] * case["n2"]
    return torch.randn(n, generator=g, device=_device(), dtype=torch.float32 if case["float32"] else torch.float64)


def _training_set(case, seed):
    """Features over the network's range and a smooth target of the size of the normalised one."""
    g = torch.Generator(device=_device()).manual_seed(seed)
    x = torch.rand((case["samples"], 2), generator=g, device=_device()) * 2.0 - 1.0
    t = torch.stack([torch.sin(2.0 * x[:, 0] + x[:, 1]), torch.cos(1.5 * x[:, 0]) * x[:, 1]], dim=1) * 0.5
    w = np.random.RandomState(seed % (1 << 31)).standard_normal(4482).astype(np.float32)
    w *= np.concatenate([np.full(128, 0.5), np.full(64, 0.1), np.full(4096, 0.15), np.full(64, 0.1),
                         np.full(130, 0.15)]).astype(np.float32)
    return x.contiguous(), t.contiguous(), w


def prepare(case, seed):
    from paper_2412_01138_gb300 import pe

    kind = case["kind"]
    state = {"kind": kind, "case": case}
    if kind == "train":
        state["x"], state["t"], state["w"] = _training_set(case, seed)
        state["y"] = torch.empty_like(state["x"])
        return state
    if kind == "transform":
        state["in"] = _values(case, seed)
        state["out"] = torch.empty_like(state["in"])
        return state
    mixed = case["precision"] == "mixed"
    precision = pe.PE_MIXED if mixed else pe.PE_FP64
    if kind == "batch":
        probs = _batch_problems(case, seed)
        engine = pe.PE_FINE_TC if case["tensor_cores"] else pe.PE_FINE_SIMT
        state["solver"] = pe.BatchSolver(probs, precision=precision, fine_engine=engine)
        buf = torch.empty(sum(p.ndof for p in probs), dtype=torch.float64, device=_device())
        state["all"] = buf
        state["parts"] = list(torch.split(buf, [p.ndof for p in probs]))
        return state
    prob = _problem(case, seed)
    state["out"] = torch.empty(prob.ndof, dtype=torch.float64, device=_device())
    if kind == "hat":
        state["solver"] = pe.Solver(prob, precision=precision, forcing_path=pe.PE_FORCING_GENERAL)
        state["nodal"] = None
        return state
    if case["host"]:
        state["out"] = np.empty(prob.ndof)
    state["nodal"] = _nodal_u0(case, seed) if case["u0"] == "nodal" else None
    state["solver"] = pe.Solver(prob, precision=precision, device_loop=case["loop"],
                                fine_engine=pe.PE_FINE_TC if case["tensor_cores"] else pe.PE_FINE_SIMT)
    return state


def run(state):
    from paper_2412_01138_gb300 import pe

    kind, case = state["kind"], state["case"]
    if kind == "train":
        net = pe.MLP(seed=1)
        net.set_params(state["w"])
        loss = net.train(state["x"], state["t"], epochs=case["epochs"], batch=case["batch"], lr=2e-3)
        net.forward(state["x"], state["y"])
        w = net.params()
        net.close()
        return {"weights": w, "loss": loss, "y": state["y"]}
    if kind == "transform":
        n = (case["n0"], case["n1"], case["n2"])[:case["d"]]
        pe.dst(case["d"], n, state["in"], state["out"], f32=case["float32"])
        return state["out"]
    s = state["solver"]
    if kind == "batch":
        s.solve(case["tol"])
        for i, part in enumerate(state["parts"]):
            s.solution(i, out=part)
        u = state["all"]
        return {"u": u.float() if case["precision"] == "mixed" else u, "k": s.status()[1]}
    out, nodal = state["out"], state["nodal"]
    u0_kind = pe.PE_FIELD_TERMS_SEPARABLE if nodal is None else pe.PE_FIELD_NODAL
    if kind == "solve" and case["loop"]:
        s.solve_async(u0_kind=u0_kind, nodal=nodal, out=out)
        info = s.wait()
    else:
        info = s.solve(u0_kind=u0_kind, nodal=nodal, out=out)
    return {"u": out.float() if case["precision"] == "mixed" else out, "k": info["k"]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """Bytes: inputs read once, outputs written once.  Operations: for a solve, two iterations
    (one reaches the fine solution, the second confirms it), each of which has to know the value
    of every column of the source (one per exponential, two per sinusoid) on every mode and
    slice, besides the step itself: 2 (columns + 1) per mode, slice and iteration.  A moving source has
    its load made and transformed at every stage time.  A transform: 5 log2 per value and axis
    for its FFT, two real pencils per complex one."""
    kind = case["kind"]
    if kind == "train":
        steps = case["epochs"] * -(-case["samples"] // case["batch"])
        return {"bytes": 16.0 * case["samples"] * case["epochs"] + 16.0 * case["samples"] + 8.0 * 4482,
                "flops": 6.0 * 4352 * case["samples"] * case["epochs"] + 4.0 * 4352 * case["samples"] + 20.0 * 4482 * steps}
    if kind == "transform":
        count = float(case["n0"] * case["n1"] * case["n2"])
        logs = sum(math.log2(case[a] + 1) for a in ("n0", "n1", "n2") if case[a] > 1)
        return {"bytes": count * (8.0 if case["float32"] else 16.0), "flops": 2.5 * count * logs}
    if kind == "batch":
        probs = [I.config4_problem(i, case["family"]) for i in range(case["count"])]
        out = 12.0 if case["precision"] == "mixed" else 8.0
        return {"bytes": sum(out * p.ndof for p in probs),
                "flops": sum(4.0 * p.ndof * p.N * (2.0 * p.R) for p in probs)}
    count = float(case["n0"] * case["n1"] * case.get("n2", 1))
    out = 4.0 if case["precision"] == "mixed" else 8.0
    if kind == "hat":
        logs = math.log2(case["n0"] + 1) + math.log2(case["n1"] + 1)
        stages = 2.0 * case["N"] * case["M"] * case["q"]
        return {"bytes": out * count, "flops": stages * count * (2.0 * (2 + case["bumps"]) + 2.5 * logs + 2.0)}
    columns = 1 + 2 * case["bumps"] + 2 * case["boundary"]
    return {"bytes": count * (out + (8.0 if case["u0"] == "nodal" else 0.0)),
            "flops": 4.0 * count * case["N"] * (columns + 1)}


# ---------------------------------------------------------------------------
# the same results in plain float64 torch: the method stage by stage, nothing regrouped
# ---------------------------------------------------------------------------

def _phi(z, s):
    """phi_1 .. phi_s at z <= 0: Taylor series for |z| < 2, the recurrence beyond."""
    small = z.abs() < 2.0
    zs = torch.where(small, z, torch.zeros_like(z))
    zl = torch.where(small, torch.full_like(z, -3.0), z)
    low, high = [], [torch.expm1(zl) / zl]
    for j in range(1, s):
        high.append((high[-1] - 1.0 / math.factorial(j)) / zl)
    for j in range(1, s + 1):
        acc = torch.full_like(zs, 1.0 / math.factorial(j + 30))
        for k in range(29, -1, -1):
            acc = acc * zs + 1.0 / math.factorial(j + k)
        low.append(acc)
    return [torch.where(small, a, b) for a, b in zip(low, high)]


def _stage_weights(z, nodes):
    """b_i(z) = int_0^1 e^{z (1 - s)} l_i(s) ds for the Lagrange basis of the nodes."""
    ph = _phi(z, len(nodes))
    out = []
    for i, ci in enumerate(nodes):
        poly = np.polynomial.Polynomial([1.0])
        for j, cj in enumerate(nodes):
            if j != i:
                poly = poly * np.polynomial.Polynomial([-cj, 1.0]) / (ci - cj)
        out.append(sum(c * math.factorial(m) * ph[m] for m, c in enumerate(poly.coef)))
    return torch.stack(out)


def _factor_at(f, x, t=None):
    p = f.params4()
    if f.kind == I.S_SIN:
        return torch.sin(p[0] * x + p[1])
    if f.kind == I.S_GAUSS:
        return torch.exp(-(x - p[0]) ** 2 / (2.0 * p[1] ** 2))
    if f.kind == I.S_POLY:
        return p[0] + x * (p[1] + x * (p[2] + x * p[3]))
    if f.kind == I.S_MOVING_HAT:
        c = p[0] + p[1] * torch.sin(2.0 * math.pi * p[2] * t)
        return torch.clamp(1.0 - (x - c.reshape(-1, *([1] * x.dim()))).abs() / p[3], min=0.0)
    return torch.ones_like(x)


def _time_at(term, t, derivative=False):
    a, b = term.tp
    if term.tkind == I.T_SIN:
        return a * np.cos(a * t + b) if derivative else np.sin(a * t + b)
    return (a if derivative else 1.0) * np.exp(a * t)


class _Axis:
    def __init__(self, prob, a, dev):
        lo, hi = prob.box[a]
        self.n = n = prob.n[a]
        self.periodic = bool(prob.periodic and prob.periodic[a])
        self.h = (hi - lo) / (n if self.periodic else n + 1)
        self.lo = lo
        f64 = dict(dtype=torch.float64, device=dev)
        j = torch.arange(n, dtype=torch.int64, device=dev) + (0 if self.periodic else 1)
        if self.periodic:
            ang = (torch.outer(j, j) % n).to(torch.float64) * (2.0 * math.pi / n)
            self.S = (torch.cos(ang) + torch.sin(ang)) / math.sqrt(n)
            th = j.to(torch.float64) * (2.0 * math.pi / n)
        else:
            ang = (torch.outer(j, j) % (2 * (n + 1))).to(torch.float64) * (math.pi / (n + 1))
            self.S = math.sqrt(2.0 / (n + 1)) * torch.sin(ang)
            th = j.to(torch.float64) * (math.pi / (n + 1))
        self.mass = self.h / 3.0 * (2.0 + torch.cos(th))
        self.ratio = 4.0 / self.h * torch.sin(0.5 * th) ** 2 / self.mass
        s, w = np.polynomial.legendre.leggauss(prob.quad_pts)
        self.s = torch.tensor(0.5 * (s + 1.0), **f64)
        self.w = torch.tensor(0.5 * w, **f64)
        self.elements = torch.arange(n if self.periodic else n + 1, **f64)
        self.nodes = lo + self.h * torch.arange(0, n + 2, **f64)

    def load(self, f, t=None):
        """int f phi_k (one row per time for a factor that moves)."""
        x = self.lo + (self.elements[:, None] + self.s[None, :]) * self.h
        v = _factor_at(f, x, t) * self.w
        right, left = (v * self.s).sum(-1) * self.h, (v * (1.0 - self.s)).sum(-1) * self.h
        if self.periodic:
            return torch.roll(right, 1, -1) + left
        return right[..., :-1] + left[..., 1:]

    def rows(self, f, kind):
        """Interior rows of the mass or stiffness matrix of all nodes, or the interior values."""
        g = _factor_at(f, self.nodes)
        if kind == "mass":
            return self.h / 6.0 * (g[:-2] + 4.0 * g[1:-1] + g[2:])
        if kind == "stiffness":
            return (2.0 * g[1:-1] - g[:-2] - g[2:]) / self.h
        return g[1:-1]

    def modal(self, load):
        return load @ self.S / self.mass


def _outer(vectors):
    out = vectors[0]
    for v in vectors[1:]:
        out = out.unsqueeze(-1) * v
    return out.reshape(-1)


def _transform(axes, x):
    for a, ax in enumerate(axes):
        x = torch.tensordot(ax.S, x.reshape([b.n for b in axes]), dims=([1], [a])).movedim(0, a)
    return x.reshape(-1).contiguous()


def _fine_solution(prob, nodal, dev):
    """The sequential fine solution at the end of the interval, nodal values."""
    axes = [_Axis(prob, a, dev) for a in range(prob.d)]
    lam = axes[0].ratio
    for ax in axes[1:]:
        lam = lam.unsqueeze(-1) + ax.ratio
    lam = prob.D * lam.reshape(-1)
    terms = []  # (function of time, modal values of the spatial product)
    moving = []
    for t in prob.forcing:
        if any(f.kind == I.S_MOVING_HAT for f in t.factors):
            moving.append(t)
        else:
            terms.append((lambda s, t=t: t.amp * _time_at(t, s),
                          _outer([ax.modal(ax.load(f)) for ax, f in zip(axes, t.factors)])))
    for g in prob.boundary:
        rows = [{k: ax.modal(ax.rows(f, k)) for k in ("mass", "stiffness")} for ax, f in zip(axes, g.factors)]
        terms.append((lambda s, g=g: -g.amp * _time_at(g, s, True), _outer([r["mass"] for r in rows])))
        for a in range(prob.d):
            terms.append((lambda s, g=g: -g.amp * prob.D * _time_at(g, s),
                          _outer([r["stiffness" if b == a else "mass"] for b, r in enumerate(rows)])))
    if nodal is not None:
        c = _transform(axes, nodal)
        for g in prob.boundary:
            c = c - g.amp * _time_at(g, prob.t0) * _transform(
                axes, _outer([ax.rows(f, "value") for ax, f in zip(axes, g.factors)]))
    else:
        c = sum(t.amp * _outer([ax.modal(ax.load(f)) for ax, f in zip(axes, t.factors)]) for t in prob.u0)
        for g in prob.boundary:
            c = c - g.amp * _time_at(g, prob.t0) * _outer(
                [ax.modal(ax.rows(f, "mass")) for ax, f in zip(axes, g.factors)])
    dT = prob.T / prob.N
    dt = dT / prob.M
    times = np.array([[prob.t0 + n * dT + (m + ci) * dt for ci in prob.fine_nodes]
                      for n in range(prob.N) for m in range(prob.M)])
    E = torch.exp(-lam * dt)
    B = dt * _stage_weights(-lam * dt, prob.fine_nodes)
    A = torch.tensor(np.stack([np.broadcast_to(f(times), times.shape) for f, _ in terms], -1), device=dev)
    P = torch.stack([v for _, v in terms])
    tt = torch.tensor(times, device=dev)
    tracks = []
    for t in moving:
        amp = torch.tensor(t.amp * np.broadcast_to(_time_at(t, times), times.shape), device=dev)
        facs = []
        for ax, f in zip(axes, t.factors):
            v = ax.modal(ax.load(f, tt.reshape(-1))) if f.kind == I.S_MOVING_HAT else ax.modal(ax.load(f))
            facs.append(v.reshape(*times.shape, -1) if v.dim() == 2 else v)
        tracks.append((amp, facs))
    for s in range(times.shape[0]):
        g = A[s] @ P
        for amp, facs in tracks:
            for i in range(prob.q):
                g[i] += amp[s, i] * _outer([v[s, i] if v.dim() == 3 else v for v in facs])
        c = E * c + (B * g).sum(0)
    u = _transform(axes, c)
    for g in prob.boundary:
        u = u + g.amp * _time_at(g, prob.t0 + prob.T) * _outer(
            [ax.rows(f, "value") for ax, f in zip(axes, g.factors)])
    return u


def _trained(case, seed):
    x, t, w = _training_set(case, seed)
    x, t = x.double(), t.double()
    w = torch.tensor(w.astype(np.float64), device=x.device)
    shapes = ((64, 2), (64,), (64, 64), (64,), (2, 64), (2,))

    def loss_of(w, x, t):
        W1, b1, W2, b2, W3, b3 = (v.reshape(s) for v, s in
                                  zip(torch.split(w, [math.prod(s) for s in shapes]), shapes))
        y = torch.tanh(torch.tanh(x @ W1.T + b1) @ W2.T + b2) @ W3.T + b3
        return 0.5 * ((y - t) ** 2).sum() / x.shape[0]

    m, v = torch.zeros_like(w), torch.zeros_like(w)
    per = -(-case["samples"] // case["batch"])
    total = per * case["epochs"]
    for it in range(total):
        lo = (it % per) * case["batch"]
        w.requires_grad_(True)
        g, = torch.autograd.grad(loss_of(w, x[lo:lo + case["batch"]], t[lo:lo + case["batch"]]), w)
        w = w.detach()
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        lr = 2e-3 * (0.01 + 0.99 * 0.5 * (1.0 + math.cos(math.pi * it / total)))
        w = w - lr * (m / (1.0 - 0.9 ** (it + 1))) / (torch.sqrt(v / (1.0 - 0.999 ** (it + 1))) + 1e-8)
    return {"weights": w, "loss": float(loss_of(w, x, t)), "y": None}


def exact(case, seed):
    dev = _device()
    kind = case["kind"]
    if kind == "train":
        return _trained(case, seed)
    if kind == "transform":
        n = (case["n0"], case["n1"], case["n2"])[:case["d"]]
        x = _values(case, seed).double()
        for a, v in enumerate(n):
            j = torch.arange(1, v + 1, dtype=torch.int64, device=dev)
            S = math.sqrt(2.0 / (v + 1)) * torch.sin((torch.outer(j, j) % (2 * (v + 1))).double() * (math.pi / (v + 1)))
            x = torch.tensordot(S, x.reshape(n), dims=([1], [a])).movedim(0, a)
        return x.reshape(-1).contiguous()
    if kind == "batch":
        return {"u": torch.cat([_fine_solution(p, None, dev) for p in _batch_problems(case, seed)]), "k": None}
    nodal = _nodal_u0(case, seed) if case.get("u0") == "nodal" else None
    return {"u": _fine_solution(_problem(case, seed), nodal, dev), "k": None}
