"""The scale of the fixed-point refinement residual (csrc/fixed.cuh): it comes only from entries
of u that the 5-point rows read. The four corners of the grid are read by no row, so what a
caller's array holds there (with Dirichlet data the boundary entries are the caller's) must
not change a bit of a solve, alone or in a batch. And the scale costs no node precision: rows
whose values lose bits in it are evaluated in FP64, so every residual stays within what an
FP64 row can be off at that node, however large the values elsewhere in the tile."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2008_03885_gb300 as mg  # noqa: E402

MIXED = dict(precision=mg.MG_PREC_MIXED_FP32, dirichlet_data=1, fma_contract=1)


def boundary_start(n, corner):
    """Zero iterate with O(1) Dirichlet data and `corner` in the four corners."""
    g = synth.uniform_pm1(4, (n + 1) ** 2).reshape(n + 1, n + 1)
    g[1:-1, 1:-1] = 0.0
    g[0, 0] = g[0, -1] = g[-1, 0] = g[-1, -1] = corner
    return torch.tensor(g, device="cuda")


@pytest.mark.parametrize("corner", [1e10, -1e30, 1e300])
@pytest.mark.parametrize("n", [8, 64, 256])
def test_corner_entries_do_not_change_a_solve(n, corner):
    f = torch.tensor(synth.rhs_normal(n, 9), device="cuda")
    h = mg.mg_setup(n, 2, **MIXED)
    try:
        out = []
        for c in (0.0, corner):
            u = boundary_start(n, c)
            _, hist = mg.mg_solve(h, u, f, rtol=0.0, max_cycles=6, raise_not_converged=False)
            rel = mg.mg_cycle(h, u, f)
            out.append((u[1:-1, 1:-1].clone(), hist, rel))
        assert out[0][1] == out[1][1] and out[0][2] == out[1][2]
        assert torch.equal(out[0][0], out[1][0])
        assert out[0][1][-1] < 1e-3 * out[0][1][0]  # and the solve converges (0.3 a cycle would do)
    finally:
        h.close()


def test_corner_entries_do_not_change_a_batch():
    ns = [8, 64, 128]
    hs = [mg.mg_setup(n, 2, **MIXED) for n in ns]
    fs = [torch.tensor(synth.rhs_normal(n, 9 + n), device="cuda") for n in ns]
    b = mg.mg_batch_create(hs, solo_min_n=32768)  # level-synchronous
    try:
        out = []
        for c in (0.0, 1e30):
            us = [boundary_start(n, c) for n in ns]
            cyc, rel = mg.mg_batch_solve(b, us, fs, rtol=1e-8, max_cycles=40)
            out.append((cyc, rel, [u[1:-1, 1:-1].clone() for u in us]))
        assert out[0][:2] == out[1][:2]
        assert all(torch.equal(x, y) for x, y in zip(out[0][2], out[1][2]))
    finally:
        b.close()
        for h in hs:
            h.close()


# ---- precision by place ---------------------------------------------------------------
LD = np.longdouble


def rows(u, n):
    """(4; -1) sums of the interior in extended precision (times s = n^2: L u)."""
    U = u.astype(LD)
    return 4 * U[1:-1, 1:-1] - (U[:-2, 1:-1] + U[1:-1, :-2] + U[1:-1, 2:] + U[2:, 1:-1])


def local_max(u):
    a = np.abs(u)
    return np.max([a[1:-1, 1:-1], a[:-2, 1:-1], a[1:-1, :-2], a[1:-1, 2:], a[2:, 1:-1]], axis=0)


def start_norm(u, f, n):
    """||f - L u|| as a mixed solve finds it."""
    h = mg.mg_setup(n, 2, precision=mg.MG_PREC_MIXED_FP32)
    try:
        _, hist = mg.mg_solve(h, torch.tensor(u, device="cuda"), torch.tensor(f, device="cuda"), rtol=0.0, max_cycles=0,
                              raise_not_converged=False)
    finally:
        h.close()
    F = f.astype(LD)
    return LD(hist[0]) * np.sqrt((F * F).sum())


def check_rounding_level(u, n, exact_nodes=None):
    """f = L u rounded, so that the residual is at rounding level: its norm is within what an FP64
    row can be off at each node: 13 roundings of at most s 8 max |its five values| (0 at
    exact_nodes, whose rows hold exact sums), and m + 14 roundings of the two norms."""
    s = LD(n) * n
    t = rows(u, n)
    f = np.zeros_like(u)
    f[1:-1, 1:-1] = (s * t).astype(np.float64)
    r = f[1:-1, 1:-1].astype(LD) - s * t
    off = s * 8 * 13 * LD(2.0) ** -53 * local_max(u)
    if exact_nodes is not None:
        assert not np.any(r[exact_nodes])
        off[exact_nodes] = 0
    want = np.sqrt((r * r).sum())
    got = start_norm(u, f, n)
    assert abs(got - want) <= np.sqrt((off * off).sum()) + (n * n + 14) * LD(2.0) ** -52 * (want + got)


@pytest.mark.parametrize("n", [8, 64, 256])
def test_integers_give_a_zero_residual(n):
    """Values and sums of at most 53 bits: every row is exact, whatever the tile's scale."""
    rng = np.random.default_rng(n)
    u = np.zeros((n + 1, n + 1))
    u[1:-1, 1:-1] = rng.integers(-2 ** 50, 2 ** 50, (n - 1, n - 1)) // 2 ** rng.integers(0, 48, (n - 1, n - 1))
    f = np.zeros_like(u)
    f[1:-1, 1:-1] = n * n * rows(u, n)
    assert start_norm(u, f, n) == 0


@pytest.mark.parametrize("small", [1e-3, 1e-10, 1e-200])
@pytest.mark.parametrize("n", [64, 256])
def test_small_values_beside_a_large_one(n, small):
    """A one in every 16 x 16 nodes, zeros around it, small values elsewhere: a residual at the
    small values' rounding level, far below the last bit of 1."""
    rng = np.random.default_rng(n)
    u = np.zeros((n + 1, n + 1))
    u[1:-1, 1:-1] = small * rng.uniform(-1, 1, (n - 1, n - 1))
    exact = np.zeros((n + 1, n + 1), bool)
    for j in range(8, n, 16):
        for i in range(8, n, 16):
            u[j - 2:j + 3, i - 2:i + 3] = 0.0
            u[j, i] = 1.0
            exact[j - 1:j + 2, i - 1:i + 2] = True
    check_rounding_level(u, n, exact[1:-1, 1:-1])


@pytest.mark.parametrize("kind", ["corner", "smooth", "rough", "tiles"])
@pytest.mark.parametrize("n", [8, 64, 256])
def test_rounding_level(n, kind):
    x = np.arange(n + 1) / n
    rng = np.random.default_rng(n)
    if kind == "corner":  # falls to 0 like (x y)^2 in a corner of the grid
        u = np.outer((x * (1 - x)) ** 2, (x * (1 - x)) ** 2)
    elif kind == "smooth":
        u = np.outer(np.sin(np.pi * x), np.sin(3 * np.pi * x))
    else:
        u = rng.uniform(-1, 1, (n + 1, n + 1))
        if kind == "tiles":  # another magnitude in every 32 x 16 nodes
            k = np.add.outer(np.arange(n + 1) // 16, np.arange(n + 1) // 32)
            u *= 2.0 ** (-20.0 * (k % 3))
    u[0, :] = u[-1, :] = u[:, 0] = u[:, -1] = 0.0
    check_rounding_level(u, n)
