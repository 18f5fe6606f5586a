"""The shared-memory tail (csrc/kernels.cu, k_tail_smem): the small levels of a cycle in one
kernel. Every branch of it gives the bits of the same cycle as separate launches
(tail_unknowns = -1), and in FP64 with the exact order those of the oracle: both precisions,
exact and FMA rows, red-black with and without pre-smoothing, Jacobi, periodic levels, the
dense coarsest solve, standard coarsening, and rows without group records."""
import numpy as np
import pytest

import synth
from oracle.mg import GALERKIN, PERIODIC, REDBLACK, STANDARD, TRUE_HIGH, Options, Oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2008_03885_gb300 as mg  # noqa: E402

SMOOTH = {"rb0": dict(nu1=0, nu2=2), "rb1": dict(nu1=1, nu2=1), "rb2": dict(nu1=2, nu2=1),
          "jacobi": dict(nu1=2, nu2=1, smoother=mg.MG_SMOOTH_JACOBI, omega=0.8)}
SETTING = {  # n, order, coarsening, coarse operator, options
    "dirichlet": (32, 4, REDBLACK, GALERKIN, {}), "dense8": (64, 4, REDBLACK, GALERKIN, dict(n_min=8)),
    "dense16": (64, 2, REDBLACK, GALERKIN, dict(n_min=16)), "standard": (64, 4, STANDARD, GALERKIN, {}),
    "no_records": (16, 4, REDBLACK, TRUE_HIGH, {}), "periodic": (16, 4, REDBLACK, GALERKIN, dict(boundary="periodic"))}
CYCLES = 2


def rhs(setting):
    n, per = SETTING[setting][0], "boundary" in SETTING[setting][4]
    return synth.rhs_periodic_normal(n, seed=5) if per else synth.rhs_normal(n, seed=5)


def solve(setting, smooth, **opts):
    """(u, history, launches of one more cycle)."""
    n, order, co, op, extra = SETTING[setting]
    f = torch.tensor(rhs(setting), dtype=torch.float64, device="cuda")
    u = torch.zeros_like(f)
    h = mg.mg_setup(n, order, co, op, **{**extra, **SMOOTH[smooth], **opts})
    try:
        _, hist = mg.mg_solve(h, u, f, rtol=0.0, max_cycles=CYCLES, raise_not_converged=False)
        out = u.cpu().numpy()
        mg.mg_reset_counters(h)
        mg.mg_cycle(h, u, f)
        return out, hist, mg.mg_get_counters(h)[0]
    finally:
        h.close()


@pytest.mark.parametrize("precision", [mg.MG_PREC_FP64, mg.MG_PREC_MIXED_FP32])
@pytest.mark.parametrize("fma", [0, 1])
@pytest.mark.parametrize("smooth", SMOOTH)
@pytest.mark.parametrize("setting", SETTING)
def test_w_cycles_have_the_bits_of_separate_launches(setting, smooth, fma, precision):
    o = dict(gamma=2, precision=precision, fma_contract=fma)
    u, hist, launches = solve(setting, smooth, **o)
    u2, hist2, launches2 = solve(setting, smooth, tail_unknowns=-1, **o)
    assert np.array_equal(u, u2) and hist == hist2
    if setting != "dense16":  # there the levels above the dense one may be past the budget
        assert launches < launches2


@pytest.mark.parametrize("smooth", SMOOTH)
@pytest.mark.parametrize("setting", SETTING)
def test_fp64_w_cycles_match_the_oracle(setting, smooth):
    n, order, co, op, extra = SETTING[setting]
    s = SMOOTH[smooth]
    keys = {k: v for k, v in {**s, **extra}.items() if k in ("nu1", "nu2", "omega", "n_min")}
    if "smoother" in s:
        keys["smoother"] = "jacobi"
    o = Oracle(n, order, co, op, Options(gamma=2, **keys), **(dict(boundary=PERIODIC) if "boundary" in extra else {}))
    uo, ho = o.solve(o.to_vec(rhs(setting)), max_cycles=CYCLES, fixed_cycles=True)
    u, hist, _ = solve(setting, smooth, gamma=2)
    assert np.array_equal(u[o.levels[0].pj, o.levels[0].pi], uo)
    assert np.max(np.abs(np.array(hist) - np.array(ho)) / np.array(ho)) <= 1e-12


@pytest.mark.parametrize("tail", [dict(gamma=2), dict(gamma=2, tail_unknowns=300), dict(tail_unknowns=300)])
@pytest.mark.parametrize("levels", [1, 3, 4])
def test_levels_of_the_bfloat16_trial_are_not_in_a_tail(levels, tail):
    """Every value stored on the finest k levels is rounded, whatever kernel runs the level."""
    o = dict(precision=mg.MG_PREC_MIXED_FP32, bf16_levels=levels)
    u, hist, _ = solve("dirichlet", "rb2", **o, **tail)
    u2, hist2, _ = solve("dirichlet", "rb2", **o, **{**tail, "tail_unknowns": -1})
    assert np.array_equal(u, u2) and hist == hist2


@pytest.mark.parametrize("precision", [mg.MG_PREC_FP64, mg.MG_PREC_MIXED_FP32])
@pytest.mark.parametrize("fma", [0, 1])
@pytest.mark.parametrize("gamma", [1, 3])
@pytest.mark.parametrize("setting", ["dirichlet", "dense8", "standard", "periodic"])
def test_v_cycles_with_jacobi_have_a_tail(setting, gamma, fma, precision):
    """Jacobi levels are launches of one thread per class node; the small ones stay in the tail."""
    o = dict(gamma=gamma, precision=precision, fma_contract=fma)
    u, hist, launches = solve(setting, "jacobi", **o)
    u2, hist2, launches2 = solve(setting, "jacobi", tail_unknowns=-1, **o)
    assert np.array_equal(u, u2) and hist == hist2
    assert launches < launches2


@pytest.mark.parametrize("precision", [mg.MG_PREC_FP64, mg.MG_PREC_MIXED_FP32])
@pytest.mark.parametrize("fma", [0, 1])
@pytest.mark.parametrize("setting", ["dirichlet", "dense8", "standard"])
def test_v_cycles_with_one_kernel_sweeps_have_a_tail(setting, fma, precision):
    o = dict(precision=precision, fma_contract=fma, sweep_kernel=2)
    u, hist, launches = solve(setting, "rb2", **o)
    u2, hist2, launches2 = solve(setting, "rb2", tail_unknowns=-1, **o)
    assert np.array_equal(u, u2) and hist == hist2
    assert launches < launches2


@pytest.mark.parametrize("boundary", ["dirichlet", "periodic"])
@pytest.mark.parametrize("n", [16, 64])
def test_fma_rows_of_cubic_transfers_by_octets_and_by_threads(n, boundary):
    """Rows of up to 121 terms in groups of one to eight: an octet of lanes hands the FMA sum from
    lane to lane (separate launches), a thread walks it term by term (tail); the same bits."""
    f = synth.rhs_periodic_normal(n, seed=7) if boundary == "periodic" else synth.rhs_normal(n, seed=7)
    out = []
    for tail in (0, -1):
        u = torch.zeros((n + 1, n + 1), dtype=torch.float64, device="cuda")
        h = mg.mg_setup(n, 4, STANDARD, GALERKIN, nu1=2, gamma=2, fma_contract=1, transfer_order=4, boundary=boundary,
                        tail_unknowns=tail)
        try:
            _, hist = mg.mg_solve(h, u, torch.tensor(f, device="cuda"), rtol=0.0, max_cycles=CYCLES,
                                  raise_not_converged=False)
        finally:
            h.close()
        out.append((u.cpu().numpy(), hist))
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]
