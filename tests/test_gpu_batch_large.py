"""The batched solver's larger problems: vectors cut into more than 32 chunks."""
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
