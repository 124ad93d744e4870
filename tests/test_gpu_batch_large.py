"""The batched solver's larger problems: vectors cut into more than 32 chunks,
and FP32 products by pair removal with all of a class's problems in one launch
(tiles of two widths, problems that finish at different times)."""
import math

import numpy as np
import pytest

import pd_inputs

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_2001_01978_gb300")

pytestmark = pytest.mark.gpu


def problems(sizes, seed):
    return [(om, n, *pd_inputs.separable_noise(om, seed=seed + 7 * i)) for i, (om, n) in enumerate(sizes)]


# 131072 = 32 chunks of 4096 elements; 256 chunks at most
@pytest.mark.parametrize("sizes", [[(20, 9), (21, 10)], [(19, 9), (22, 11), (9, 4)], [(24, 10)]])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_energies_of_single_solves(sizes, prec):
    tol = 1e-8
    p = pd.PD_PREC_FP64 if prec == "fp64" else pd.PD_PREC_MIXED
    ps = problems(sizes, 3)
    r = pd.pairdiag_batch_ground_state(ps, tol, pd.pairdiag_default_options(precision=p))
    for (om, n, e, G), e0 in zip(ps, r["e0"]):
        with pd.Solver(om, n, e, G) as s:
            ref = pd.pairdiag_ground_state_dev(s.h, tol)["e0"]
        assert abs(e0 - ref) <= 2 * tol * abs(ref)      # the residual bounds the distance of each


# Ω up to 24 and up to 32: two tile widths; (14, 7) goes row by row beside them
@pytest.mark.parametrize("sizes", [[(17, 8), (18, 9), (19, 8), (20, 12), (22, 11)], [(23, 6), (26, 6), (25, 5), (14, 7), (18, 6)]])
def test_removal_needs_no_more_steps_than_rows(sizes):
    """With the FP32 cycles alone (tolerance at the hand-over): the same energies
    as with row-by-row products, within the residuals, and as many steps give or
    take a cycle."""
    tol = 1e-5
    ps = problems(sizes, 5)
    got = pd.pairdiag_batch_ground_state(ps, tol, pd.pairdiag_default_options(precision=pd.PD_PREC_MIXED))
    ref = pd.pairdiag_batch_ground_state(ps, tol, pd.pairdiag_default_options(precision=pd.PD_PREC_MIXED, hx_variant=3))
    for a, b, ia, ib in zip(got["e0"], ref["e0"], got["iterations"], ref["iterations"]):
        assert abs(a - b) <= 2 * tol * abs(b)
        assert abs(ia - ib) <= 20                        # one cycle
