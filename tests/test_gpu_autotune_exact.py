"""The autotuner takes pair removal (variant 2) only where its rows are no less
exact than row by row: not in small spaces above two thirds filling."""
import pytest

import pd_inputs

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_2001_01978_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("omega,n,candidate", [(22, 19, False), (18, 13, False), (18, 12, True), (24, 19, True), (14, 7, True)])
def test_candidates(omega, n, candidate):
    e, G = pd_inputs.separable_noise(omega, seed=1)
    try:
        best, every = pd.pairdiag_autotune(omega, n, e, G, pd.PD_PREC_MIXED, 1)
    finally:
        pd.pairdiag_tune_set(omega, n, pd.PD_PREC_MIXED, 0, 0)
    assert any(t["hx_variant"] == 2 for t in every) == candidate
    assert best["hx_variant"] != 2 or candidate
