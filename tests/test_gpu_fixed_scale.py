"""The scale of the fixed-point refinement residual (csrc/fixed.cuh): it comes only from entries
of u that the 5-point rows read. The four corners of the grid are read by no row, so what a
caller's array holds there (with Dirichlet data the boundary entries are the caller's) must
not change a bit of a solve, alone or in a batch."""
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
