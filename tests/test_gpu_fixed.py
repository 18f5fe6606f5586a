"""The refinement residual of a mixed solve, through its history with no cycle: the norm
against extended precision on the host. Second order goes in fixed point (csrc/fixed.cuh):
a value of the tile's largest exponent keeps 6 bits below its last one, so the stencil sum is
off by at most W / 2 units of 2^-6 ulp(max |u|), W = 8 the sum of the |weights|; r takes one
more rounding, and the norm's sum of squares m + 10 roundings at most. Fourth order, and
tiles of tiny values, go through FP64 rows: every product and partial sum (13 at most, each
at most s W max |u|) rounded. Inputs: smooth with heavy cancellation, rough, zero, tiny and
huge, values over 200 decades, infinities; grids from one ragged tile up, Dirichlet data."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2008_03885_gb300 as mg  # noqa: E402

LD = np.longdouble


def inputs(kind, n):
    x = np.arange(n + 1) / n
    smooth = np.outer(np.sin(np.pi * x), np.sin(2 * np.pi * x))
    noise = synth.uniform_pm1(3, (n + 1) ** 2).reshape(n + 1, n + 1)
    u = {"smooth": 3.0 * smooth, "rough": noise, "zero": 0.0 * noise, "tiny": 1e-300 * noise, "huge": 1e140 * noise,
         "decades": noise * 10.0 ** (100 * noise[::-1])}[kind].copy()
    u[0, :] = u[-1, :] = u[:, 0] = u[:, -1] = 0.0
    return u


def exact_norm(u, f, order, n, data):
    """(norm of f - L u, norm of f, s) over the interior in extended precision."""
    s = n * n / 12.0 if order == 4 else float(n * n)
    U = u.astype(LD)
    e = np.zeros((n + 3, n + 3), LD)
    e[1:-1, 1:-1] = U
    if not data:  # odd reflection
        e[0, 1:-1], e[-1, 1:-1], e[1:-1, 0], e[1:-1, -1] = -U[1], -U[-2], -U[:, 1], -U[:, -2]
    c = e[2:-2, 2:-2]

    def at(dy, dx):
        return e[2 + dy:n + 1 + dy, 2 + dx:n + 1 + dx]

    near = at(-1, 0) + at(0, -1) + at(0, 1) + at(1, 0)
    far = at(-2, 0) + at(0, -2) + at(0, 2) + at(2, 0)
    t = far - 16 * near + 60 * c if order == 4 else 4 * c - near
    F = f[1:-1, 1:-1].astype(LD)
    r = F - LD(s) * t
    return np.sqrt((r * r).sum()), np.sqrt((F * F).sum()), s


@pytest.mark.parametrize("kind", ["smooth", "rough", "zero", "tiny", "huge", "decades"])
@pytest.mark.parametrize("n,order", [(8, 2), (64, 2), (64, 4), (256, 2)])
@pytest.mark.parametrize("fma", [0, 1])
def test_residual_norm_within_the_bound_of_the_format(n, order, kind, fma):
    u = inputs(kind, n)
    f = synth.rhs_normal(n, 9)
    check(u, f, n, order, dict(fma_contract=fma))


@pytest.mark.parametrize("n", [8, 64])
def test_dirichlet_data(n):
    u = synth.uniform_pm1(4, (n + 1) ** 2).reshape(n + 1, n + 1)
    check(u, synth.rhs_normal(n, 9), n, 2, dict(dirichlet_data=1))


def check(u, f, n, order, opts):
    h = mg.mg_setup(n, order, precision=mg.MG_PREC_MIXED_FP32, **opts)
    try:
        _, hist = mg.mg_solve(h, torch.tensor(u, device="cuda"), torch.tensor(f, device="cuda"), rtol=0.0, max_cycles=0,
                              raise_not_converged=False)
    finally:
        h.close()
    rn, fn, s = exact_norm(u, f, order, n, "dirichlet_data" in opts)
    m = (n - 1) ** 2
    big = np.abs(u).max()
    node = s * 8 / 2 * 2.0 ** -6 * 2.0 ** -52 * big
    if order == 4 or big < 1e-250:  # rows in FP64
        node = s * (128 if order == 4 else 8) * 13 * 2.0 ** -53 * big
    bound = np.sqrt(m) * node + (m + 14) * 2.0 ** -53 * float(rn)
    assert abs(hist[0] * float(fn) - float(rn)) <= bound + (m + 14) * 2.0 ** -53 * float(rn)


def test_infinity_is_reported():
    n = 64
    u = inputs("rough", n)
    u[20, 30] = np.inf
    h = mg.mg_setup(n, 2, precision=mg.MG_PREC_MIXED_FP32)
    try:
        with pytest.raises(mg.MGError) as e:
            mg.mg_solve(h, torch.tensor(u, device="cuda"), torch.tensor(synth.rhs_normal(n, 9), device="cuda"),
                        max_cycles=0)
        assert e.value.status == mg.MG_ERR_NONFINITE
    finally:
        h.close()
