"""hx_variant = 2 in a batch: FP32 products by pair removal on every problem that
it serves, variant 3 for the others and for FP64."""
import numpy as np
import pytest

import pd_inputs

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_2001_01978_gb300")

pytestmark = pytest.mark.gpu


def solve(sizes, tol, **opt):
    ps = [(om, n, *pd_inputs.separable_noise(om, seed=11 + i)) for i, (om, n) in enumerate(sizes)]
    before = pd.pairdiag_kernel_launches()
    r = pd.pairdiag_batch_ground_state(ps, tol, pd.pairdiag_default_options(**opt))
    return r, pd.pairdiag_kernel_launches() - before


def test_removal_where_the_automatic_rule_takes_it():
    """The same kernels as variant 0 on problems of at least 15000 states: the
    same bits (sums have a fixed order) and the same launches."""
    sizes = [(17, 8), (18, 9), (22, 5)]
    a, la = solve(sizes, 1e-5, precision=pd.PD_PREC_MIXED, hx_variant=2)
    b, lb = solve(sizes, 1e-5, precision=pd.PD_PREC_MIXED, hx_variant=0)
    assert np.array_equal(a["e0"], b["e0"]) and np.array_equal(a["iterations"], b["iterations"])
    assert la == lb


def test_removal_of_small_problems():
    """Below that line too: two launches per product instead of one; (12, 6) has
    no high orbits and (16, 16) one state, so both go row by row beside them."""
    tol = 1e-5
    r, l2 = solve([(13, 12), (14, 7), (16, 3), (16, 15)], tol, precision=pd.PD_PREC_MIXED, hx_variant=2)
    _, l3 = solve([(13, 12), (14, 7), (16, 3), (16, 15)], tol, precision=pd.PD_PREC_MIXED, hx_variant=3)
    ref, _ = solve([(13, 12), (14, 7), (16, 3), (16, 15)], 1e-9, precision=pd.PD_PREC_FP64)
    assert l2 != l3
    assert np.all(np.abs(np.array(r["e0"]) - np.array(ref["e0"])) <= 2 * tol * np.abs(ref["e0"]))
    r, _ = solve([(12, 6), (14, 7), (16, 16)], tol, precision=pd.PD_PREC_MIXED, hx_variant=2)
    ref, _ = solve([(12, 6), (14, 7), (16, 16)], 1e-9, precision=pd.PD_PREC_FP64)
    assert np.all(np.abs(np.array(r["e0"]) - np.array(ref["e0"])) <= 2 * tol * np.abs(ref["e0"]))


def test_fp64_as_variant_3():
    sizes = [(14, 7), (17, 8), (20, 6)]
    a, la = solve(sizes, 1e-11, precision=pd.PD_PREC_FP64, hx_variant=2)
    b, lb = solve(sizes, 1e-11, precision=pd.PD_PREC_FP64, hx_variant=3)
    assert np.array_equal(a["e0"], b["e0"]) and la == lb
