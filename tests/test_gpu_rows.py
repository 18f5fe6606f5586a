"""Operator rows evaluated by octets of lanes (csrc/rows.cuh): the nodes off a level's fast
rectangle, and every node of a small level. Bit for bit against the oracle on levels on
both sides of the small-level threshold, axis and rotated, with the longest rows
(sixth order, true high-order Galerkin, 45 points), and on grids so small that every node
is a class of its own; Dirichlet data, whose class rows drop the boundary columns; and the
fused-multiply-add order against the exact one within its rounding bound."""
import numpy as np
import pytest

import synth
from oracle.mg import GALERKIN, NONGALERKIN, REDBLACK, STANDARD, TRUE_HIGH, VARIABLE, Oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2008_03885_gb300 as mg  # noqa: E402


def to_dev(h, level, vec):
    i, j, row, col = mg.level_nodes(h, level)
    a = mg.level_array(h, level)
    a[torch.as_tensor(row), torch.as_tensor(col)] = torch.as_tensor(vec, dtype=torch.float64).cuda()
    return a


def from_dev(h, level, a):
    i, j, row, col = mg.level_nodes(h, level)
    return a.cpu().numpy()[row, col]


@pytest.mark.parametrize("n,order,co,op", [(256, 4, REDBLACK, GALERKIN), (256, 6, STANDARD, NONGALERKIN),
                                           (256, 2, VARIABLE, GALERKIN), (32, 6, REDBLACK, TRUE_HIGH),
                                           (4, 4, REDBLACK, GALERKIN), (8, 6, STANDARD, GALERKIN)])
def test_smooth_and_residual_bitwise(n, order, co, op):
    o = Oracle(n, order, co, op)
    h = mg.mg_setup(n, order, co, op)
    try:
        for l, lev in enumerate(o.levels):
            u = synth.uniform_pm1(10 + l, lev.size) * 3.0
            f = synth.uniform_pm1(20 + l, lev.size) * 1e3
            du, df, out = to_dev(h, l, u), to_dev(h, l, f), mg.level_array(h, l)
            mg.mg_level_residual(h, l, du, df, out)
            assert np.array_equal(from_dev(h, l, out), o.residual(l, u, f)), ("residual", l)
            mg.mg_level_smooth(h, l, du, df, 2)
            assert np.array_equal(from_dev(h, l, du), o.smooth(l, o.smooth(l, u, f), f)), ("smooth", l)
    finally:
        h.close()


@pytest.mark.parametrize("n", [4, 8, 64])
def test_dirichlet_data_bitwise(n):
    o = Oracle(n, 2, REDBLACK, GALERKIN)
    g = synth.uniform_pm1(5, (n + 1) ** 2).reshape(n + 1, n + 1)
    f = synth.uniform_pm1(6, o.levels[0].size) * 10.0
    h = mg.mg_setup(n, 2, REDBLACK, GALERKIN, dirichlet_data=1)
    o.set_boundary(g)
    try:
        u = torch.tensor(g, device="cuda")
        out = mg.level_array(h, 0)
        mg.mg_level_residual(h, 0, u, to_dev(h, 0, f), out)
        ref = o.residual(0, o.to_vec(g), f)
        assert np.array_equal(from_dev(h, 0, out), ref)
    finally:
        h.close()


@pytest.mark.parametrize("n,order,co", [(64, 4, REDBLACK), (256, 2, STANDARD)])
def test_fma_order_stays_within_its_rounding_bound(n, order, co):
    """|fma - exact| <= 2 (t + 2) eps (|f| + sum |a_pq| |u_q|) for a row of t terms."""
    o = Oracle(n, order, co, GALERKIN)
    h = mg.mg_setup(n, order, co, GALERKIN, fma_contract=1)
    try:
        for l, lev in enumerate(o.levels):
            u = synth.uniform_pm1(30 + l, lev.size)
            f = synth.uniform_pm1(40 + l, lev.size)
            out = mg.level_array(h, l)
            mg.mg_level_residual(h, l, to_dev(h, l, u), to_dev(h, l, f), out)
            t = np.diff(lev.A.indptr).max()
            bound = 2 * (t + 2) * 2.0 ** -53 * (np.abs(f) + abs(lev.A) @ np.abs(u))
            assert np.all(np.abs(from_dev(h, l, out) - o.residual(l, u, f)) <= bound), l
    finally:
        h.close()


def test_steps_in_a_caller_captured_graph_with_a_joined_stream():
    """Small-level kernels start early (programmatic dependent launch): in a caller's graph
    whose first step joins a second stream, and replayed on new data, they still see the
    other stream's writes and give the bits of eager calls."""
    n = 64
    h = mg.mg_setup(n, 4, REDBLACK, GALERKIN)
    try:
        f = torch.tensor(synth.rhs_normal(n, 3), device="cuda")
        src = torch.zeros_like(f)
        u, d, u2, d2 = (torch.zeros_like(f) for _ in range(4))
        fc, fc2 = mg.level_array(h, 1), mg.level_array(h, 1)
        side, main = torch.cuda.Stream(), torch.cuda.Stream()
        g = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=main):
            side.wait_stream(main)
            with torch.cuda.stream(side):
                u.copy_(src)
            main.wait_stream(side)
            mg.mg_level_smooth(h, 0, u, f, 2, stream=main)
            mg.mg_level_residual(h, 0, u, f, d, stream=main)
            mg.mg_level_restrict(h, 0, d, fc, stream=main)
            mg.mg_level_prolong_add(h, 0, u, fc, stream=main)
        for seed in range(3):
            src.copy_(torch.tensor(synth.rhs_normal(n, 7 + seed), device="cuda"))
            g.replay()
            u2.copy_(src)
            mg.mg_level_smooth(h, 0, u2, f, 2)
            mg.mg_level_residual(h, 0, u2, f, d2)
            mg.mg_level_restrict(h, 0, d2, fc2)
            mg.mg_level_prolong_add(h, 0, u2, fc2)
            torch.cuda.synchronize()
            assert torch.equal(u, u2) and torch.equal(d, d2) and torch.equal(fc, fc2), seed
    finally:
        h.close()
