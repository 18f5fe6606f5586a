"""Performance cases: what users of this library have it do, through its Python entry points.

Every grid side is a power of two (the library takes no other), so the arrays are the odd
sizes N + 1 = 65 ... 8193, and every level below is odd too. The kinds:

  solve   mg_solve on device arrays from u = 0
  host    mg_solve_host on pinned host arrays (copies included)
  cycle   one mg_cycle on a given iterate (a user's own outer iteration)
  steps   smoothing, residual, restriction and interpolation of the finest level, each by
          its own entry point (a user's own cycle driver)
  batch   mg_batch_solve of many uneven problems

A case carries every option that it does not take from the library's defaults.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2008_03885_gb300 as mg

SOLVE = dict(kind="solve", order=4, coarsening="redblack", op="galerkin", boundary="dirichlet", mixed=False, fma=0,
             nu1=2, nu2=1, gamma=1, omega=1.0, n_min=2, transfer=2, rtol=1e-10, rhs="normal")


def listed():
    return [
        # The smallest calls: a user's own cycle driver on a 65 x 65 grid, launch bound.
        dict(SOLVE, name="steps_fp64_o2_64", kind="steps", n=64, order=2, nu1=1),
        # The same driver on an ordinary fourth-order grid.
        dict(SOLVE, name="steps_fp64_o4_2048", kind="steps", n=2048),
        # A small FP64 solve: every level is latency bound.
        dict(SOLVE, name="solve_fp64_o4_128", n=128),
        # An ordinary second-order V(1,1) solve called on host arrays, as a CPU program does.
        dict(SOLVE, name="host_fp64_o2_1024", kind="host", n=1024, order=2, nu1=1),
        # Periodic boundaries, the paper's own setting.
        dict(SOLVE, name="solve_fp64_periodic_o4_512", n=512, boundary="periodic"),
        # Standard coarsening, the comparison method, with its optimal omega.
        dict(SOLVE, name="solve_fp64_standard_o4_2048", n=2048, coarsening="standard", omega=1.1),
        # The library's headline: FP64, fourth order, red-black Galerkin, smooth data, 4097^2.
        dict(SOLVE, name="solve_fp64_o4_4096", n=4096, rhs="sine"),
        # The served requests: mixed precision to 1e-8, dense coarsest solve; small, Galerkin ...
        dict(SOLVE, name="solve_mixed_o4_256", n=256, mixed=True, fma=1, n_min=16, rtol=1e-8),
        # ... and larger, with the 5-point coarse operators.
        dict(SOLVE, name="solve_mixed_nongalerkin_o4_2048", n=2048, op="nongalerkin", mixed=True, fma=1, n_min=16,
             rtol=1e-8),
        # The headline problem in mixed precision.
        dict(SOLVE, name="solve_mixed_o4_4096", n=4096, rhs="sine", mixed=True, fma=1),
        # The largest: second order, 8193^2, mixed precision.
        dict(SOLVE, name="solve_mixed_o2_8192", n=8192, order=2, nu1=1, mixed=True, fma=1),
        # Many uneven problems at once: sides 129 ... 2049, orders 2 and 4, mixed precision.
        dict(SOLVE, name="batch_mixed_48", kind="batch", n=2048, count=48, mixed=True, fma=1, n_min=16, rtol=1e-8),
    ]


def draw(rng: random.Random):
    kind = rng.choices(["fp64", "mixed", "steps", "host", "cycle", "batch"], [35, 30, 12, 8, 7, 8])[0]
    order = rng.choices([2, 4, 6], [45, 45, 10])[0]
    c = dict(SOLVE, order=order, nu1=rng.choice([1, 2, 2, 3]) if order > 2 else rng.choice([1, 1, 2]),
             nu2=rng.choice([1, 1, 1, 2]), omega=rng.choice([1.0, 1.0, round(rng.uniform(0.95, 1.1), 3)]),
             op=rng.choices(["galerkin", "nongalerkin", "g1", "gn"], [60, 25, 7, 8])[0],
             coarsening=rng.choices(["redblack", "standard", "variable"], [75, 15, 10])[0],
             rtol=10.0 ** round(rng.uniform(-9.5, -6), 2), rhs=rng.choice(["normal", "sine"]))
    if order == 6:
        c["op"] = "galerkin"
    elif c["coarsening"] != "redblack":
        c["op"] = rng.choice(["galerkin", "nongalerkin"])
    if c["coarsening"] == "standard" and rng.random() < 0.25:
        c["transfer"] = 4
    if kind == "batch":
        c.update(kind="batch", n=2 ** rng.randint(9, 11), count=rng.randint(8, 48), mixed=rng.random() < 0.8, fma=1,
                 n_min=16, coarsening="redblack", op="galerkin", transfer=2, order=4, nu1=2, nu2=1, omega=1.0)
        if not c["mixed"]:
            c.update(n=512, fma=0)
        return c
    if kind == "mixed":
        c.update(mixed=True, fma=rng.choice([0, 1, 1]), n=2 ** rng.randint(6, 12), n_min=rng.choice([2, 8, 16]))
        if rng.random() < 0.1 and c["coarsening"] == "redblack":
            c.update(boundary="periodic", n_min=2)
        return c
    if kind == "steps":
        c.update(kind="steps", n=2 ** rng.randint(5, 12), transfer=2)
        return c
    c.update(fma=rng.choice([0, 0, 0, 1]), n=2 ** rng.randint(6, 11), n_min=rng.choice([2, 2, 8, 16]))
    if kind == "host":
        c.update(kind="host", mixed=rng.random() < 0.5)
    elif kind == "cycle":
        c.update(kind="cycle", gamma=rng.choice([1, 1, 3]))
    elif rng.random() < 0.15 and c["coarsening"] == "redblack":
        c.update(boundary="periodic", n_min=2)
    return c


# ---- inputs -------------------------------------------------------------------------
def _rhs(n: int, kind: str, boundary: str, gen) -> torch.Tensor:
    """White noise or 16 smooth sine modes on the unknowns (zero mean if periodic)."""
    f = torch.zeros((n + 1, n + 1), dtype=torch.float64, device="cuda")
    if kind == "sine" and boundary != "periodic":
        kmax = max(1, min(64, n // 4))
        k = torch.randint(max(1, kmax // 16), kmax + 1, (2, 16), generator=gen, device="cuda").to(torch.float64)
        a = torch.randn(16, dtype=torch.float64, generator=gen, device="cuda")
        x = torch.arange(n + 1, dtype=torch.float64, device="cuda") * (math.pi / n)
        s, t = torch.sin(k[0][:, None] * x), torch.sin(k[1][:, None] * x)
        f[1:-1, 1:-1] = ((s * a[:, None]).T @ t)[1:-1, 1:-1]
    elif boundary == "periodic":
        g = torch.randn((n, n), dtype=torch.float64, generator=gen, device="cuda")
        f[:n, :n] = g - g.mean()
    else:
        f[1:-1, 1:-1] = torch.randn((n - 1, n - 1), dtype=torch.float64, generator=gen, device="cuda")
    return f


def _gen(seed: int):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _problems(case):
    """(n, order) of every problem of a batch: sides 128 ... n, both orders, seeded by the case alone."""
    r = random.Random(case["count"])
    top = int(math.log2(case["n"]))
    return [(2 ** r.randint(7, top), r.choice([2, 4])) for _ in range(case["count"])]


def _handle(case, n=None, order=None):
    o = dict(nu1=case["nu1"], nu2=case["nu2"], gamma=case["gamma"], omega=case["omega"], n_min=case["n_min"],
             boundary=case["boundary"], transfer_order=case["transfer"], fma_contract=case["fma"],
             precision=mg.MG_PREC_MIXED_FP32 if case["mixed"] else mg.MG_PREC_FP64)
    return mg.mg_setup(n or case["n"], order or case["order"], case["coarsening"], case["op"], **o)


def _start_iterate(n: int, gen) -> torch.Tensor:
    u = torch.zeros((n + 1, n + 1), dtype=torch.float64, device="cuda")
    u[1:-1, 1:-1] = torch.randn((n - 1, n - 1), dtype=torch.float64, generator=gen, device="cuda") / n
    return u


def prepare(case, seed):
    gen = _gen(seed)
    n, kind = case["n"], case["kind"]
    if kind == "batch":
        ps = _problems(case)
        hs = [_handle(case, m, order) for m, order in ps]
        fs = [_rhs(m, case["rhs"], case["boundary"], gen) for m, _ in ps]
        return dict(case=case, handles=hs, f=fs, u=[torch.zeros_like(x) for x in fs], batch=mg.mg_batch_create(hs))
    f = _rhs(n, case["rhs"], case["boundary"], gen)
    s = dict(case=case, handle=_handle(case))
    if kind == "host":
        s.update(f=f.cpu().pin_memory(), u=torch.zeros((n + 1, n + 1), dtype=torch.float64).pin_memory())
        return s
    s.update(f=f, u=torch.zeros_like(f))
    if kind in ("cycle", "steps"):
        s["u0"] = _start_iterate(n, gen)
    if kind == "steps":
        s.update(d=torch.zeros_like(f), fc=mg.level_array(s["handle"], 1), w=torch.zeros_like(f))
    return s


def run(state):
    case = state["case"]
    u, f = state["u"], state["f"]
    if case["kind"] == "batch":
        for x in u:
            x.zero_()
        cycles, _ = mg.mg_batch_solve(state["batch"], u, f, rtol=case["rtol"], max_cycles=60)
        return {"u": u, "cycles": torch.tensor(cycles)}
    h = state["handle"]
    if case["kind"] == "steps":
        d, fc, w = state["d"], state["fc"], state["w"]
        u.copy_(state["u0"])
        mg.mg_level_smooth(h, 0, u, f, case["nu1"])
        mg.mg_level_residual(h, 0, u, f, d)
        mg.mg_level_restrict(h, 0, d, fc)
        w.copy_(state["u0"])
        mg.mg_level_prolong_add(h, 0, w, fc)
        return {"u": u, "d": d, "fc": fc, "w": w}
    if case["kind"] == "cycle":
        u.copy_(state["u0"])
        return {"u": u, "rel": mg.mg_cycle(h, u, f)}
    u.zero_()
    solve = mg.mg_solve_host if case["kind"] == "host" else mg.mg_solve
    cycles, history = solve(h, u, f, rtol=case["rtol"], max_cycles=60)
    return {"u": u, "cycles": cycles, "history": np.array(history)}


# ---- the least work of one pass -------------------------------------------------------
TERMS = {2: 5, 4: 9, 6: 13}


def _cycles(case) -> float:
    """Cycles to the tolerance at about 0.02 a cycle (0.1 for standard and non-Galerkin coarsening)."""
    rate = 0.02 if case["coarsening"] == "redblack" and case["op"] == "galerkin" else 0.1
    return max(1.0, math.ceil(math.log(case["rtol"]) / math.log(rate)))


def _solve_work(case, n, order):
    """A cycle reads u and f and writes u once before and once after the coarse correction, on
    every level (the levels add a factor 2, or 4/3 for standard coarsening); flops: 2 s + 3 a
    node and sweep, 2 s a node for the residual, 8 for each transfer. A refinement step does
    that in FP32 and reads u, f (FP64 residual), reads and writes u (update) in FP64."""
    pts = float((n + 1) ** 2)
    s = TERMS[order]
    levels = 4 / 3 if case["coarsening"] == "standard" else 2.0
    word = 4 if case["mixed"] else 8
    sweeps = case["nu1"] + case["nu2"]
    flops = levels * (sweeps * (2 * s + 3) + 2 * s + 16)
    nbytes = levels * 6 * word + (16 + 16 + 8 if case["mixed"] else 0)
    k = 1.0 if case["kind"] == "cycle" else _cycles(case)
    return pts * k * nbytes, pts * k * (flops + (2 * s if case["mixed"] else 0))


def work(case):
    if case["kind"] == "batch":
        w = [_solve_work(case, m, order) for m, order in _problems(case)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    n, s = case["n"], TERMS[case["order"]]
    pts = float((n + 1) ** 2)
    if case["kind"] == "steps":
        # smooth (u, f -> u), residual (-> d), restriction (-> fc), interpolation (u0, fc -> w)
        ratio = 0.25 if case["coarsening"] == "standard" else 0.5
        return {"bytes": pts * 8 * (2 + 1 + 1 + ratio + 1),
                "flops": pts * (case["nu1"] * (2 * s + 3) + 2 * s + 16)}
    nbytes, flops = _solve_work(case, n, case["order"])
    return {"bytes": nbytes, "flops": flops}


# ---- the same results in 64 bits, without the library ----------------------------------
def _dst(a: torch.Tensor, axis: int) -> torch.Tensor:
    """DST-I of the interior along one axis, by an FFT of the odd extension."""
    m = a.shape[axis]
    shape = list(a.shape)
    shape[axis] = 1
    zero = torch.zeros(shape, dtype=a.dtype, device=a.device)
    x = torch.cat([zero, a, zero, -a.flip(axis)], dim=axis)
    return -torch.fft.rfft(x, dim=axis).imag.narrow(axis, 1, m) / 2


def _symbol(n: int, order: int, device) -> torch.Tensor:
    """Eigenvalues of the 1D operator on sin(k pi x), k = 1 ... n - 1 (odd reflection at the ends)."""
    t = torch.arange(1, n, dtype=torch.float64, device=device) * (math.pi / n)
    h2 = 1.0 / (float(n) * n)
    if order == 2:
        return (2 - 2 * torch.cos(t)) / h2
    if order == 4:
        return (30 - 32 * torch.cos(t) + 2 * torch.cos(2 * t)) / (12 * h2)
    return (490 - 540 * torch.cos(t) + 54 * torch.cos(2 * t) - 4 * torch.cos(3 * t)) / (180 * h2)


def _solution(f: torch.Tensor, order: int) -> torch.Tensor:
    n = f.shape[0] - 1
    g = _dst(_dst(f[1:-1, 1:-1], 0), 1)
    lam = _symbol(n, order, f.device)
    g /= lam[:, None] + lam[None, :]
    u = torch.zeros_like(f)
    u[1:-1, 1:-1] = _dst(_dst(g, 0), 1) * (2.0 / n) ** 2
    return u


def _operator(u: torch.Tensor, order: int):
    """(L u, diagonal of L) on the interior, ghosts by odd reflection."""
    n = u.shape[0] - 1
    w = {2: [2.0, -1.0], 4: [30.0, -16.0, 1.0], 6: [490.0, -270.0, 27.0, -2.0]}[order]
    scale = float(n) * n / {2: 1, 4: 12, 6: 180}[order]
    r = len(w) - 1

    def line(axis):
        m = u.movedim(axis, 0)
        e = torch.cat([-m[1:r].flip(0), m, -m[n + 1 - r:n].flip(0)], 0) if r > 1 else m
        s = sum(w[abs(k)] * e[r + k:r + k + n - 1] for k in range(-r, r + 1))
        return s.movedim(0, axis)

    d = torch.full((n - 1,), w[0], dtype=torch.float64, device=u.device)
    for k in range(2, r + 1):  # reflected terms that land on the node itself
        if k % 2 == 0:
            d[k // 2 - 1] -= w[k]
            d[n - 1 - k // 2] -= w[k]
    return scale * (line(0)[:, 1:-1] + line(1)[1:-1, :]), scale * (d[:, None] + d[None, :])


def _steps(case, seed):
    gen = _gen(seed)
    n, order = case["n"], case["order"]
    f = _rhs(n, case["rhs"], case["boundary"], gen)
    u0 = _start_iterate(n, gen)
    u = u0.clone()
    i = torch.arange(1, n, device="cuda")
    red = ((i[:, None] + i[None, :]) % 2 == 1).to(torch.float64)
    for _ in range(case["nu1"]):
        for colour in (red, 1 - red):
            a, diag = _operator(u, order)
            u[1:-1, 1:-1] += colour * (case["omega"] * (f[1:-1, 1:-1] - a) / diag)
    d = torch.zeros_like(f)
    d[1:-1, 1:-1] = f[1:-1, 1:-1] - _operator(u, order)[0]
    return {"u": u, "d": d, "fc": None, "w": None}


def exact(case, seed):
    if case["kind"] == "cycle" or case["boundary"] == "periodic":
        return None
    if case["kind"] == "steps":
        return _steps(case, seed)
    gen = _gen(seed)
    if case["kind"] == "batch":
        return {"u": [_solution(_rhs(m, case["rhs"], case["boundary"], gen), order) for m, order in _problems(case)],
                "cycles": None}
    u = _solution(_rhs(case["n"], case["rhs"], case["boundary"], gen), case["order"])
    return {"u": u.cpu() if case["kind"] == "host" else u, "cycles": None, "history": None}
