"""The FP32 product by pair removal (variant 2) where most high words leave few
low words (far from half filling over many orbits): several blocks per tile in
the removal, one thread per row in the addition.  Rows element by element
against the oracle with blocks of 1, 12 and 66 words from both ends of the
filling, elements that cannot be split, and the dot product of the addition."""
import math

import numpy as np
import pytest

import oracle
import pd_inputs
from helpers import abs_row_scale
from test_gpu_removal import product32, removal_eps

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_2001_01978_gb300")

pytestmark = pytest.mark.gpu


# 26 to 32 and 33 to 40 orbits are two widths of a tile; (25, 20) has the blocks
# of 66, 12 and 1 words at the other end, and a class without rows of its own
@pytest.mark.parametrize("omega,n", [(25, 20), (26, 6), (30, 5), (32, 5), (33, 5), (34, 5), (40, 4)])
def test_rows_vs_oracle(omega, n):
    e, G = pd_inputs.separable_noise(omega, seed=omega + n)
    b = oracle.basis(omega, n)
    x32 = pd_inputs.random_vector(len(b), omega + n).astype(np.float32)
    x32[::5] *= np.float32(1e-10)
    x = x32.astype(np.float64)
    with pd.Solver(omega, n, e, G, precision=pd.PD_PREC_MIXED, hx_variant=2) as s:
        got = product32(s, x32)
        again = product32(s, x32)
    assert np.array_equal(got, again)
    bound = removal_eps(omega, n) * abs_row_scale(omega, n, e, G, x, basis=b)
    err = np.abs(got - oracle.hx(omega, n, e, G, x, b))
    assert np.all(err <= bound), np.max(err / np.maximum(bound, 1e-300))


@pytest.mark.parametrize("value", [np.inf, np.nan, np.finfo(np.float32).max])
def test_elements_that_cannot_be_split(value):
    omega, n = 30, 5
    e, G = pd_inputs.separable_noise(omega, seed=4)
    x32 = pd_inputs.random_vector(math.comb(omega, n), 3).astype(np.float32)
    bad = x32.copy()
    bad[::20011] = value
    with pd.Solver(omega, n, e, G, precision=pd.PD_PREC_MIXED, hx_variant=2) as s, \
            pd.Solver(omega, n, e, G, precision=pd.PD_PREC_MIXED, hx_variant=3) as r:
        got, ref = product32(s, bad), product32(r, bad)
        clean = product32(s, x32)
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    assert np.array_equal(np.isinf(got), np.isinf(ref))
    assert np.all(np.isfinite(clean))


def test_fused_dot():
    """Lanczos on the mixed handle takes x^T H x from the addition kernels: the
    lowest energy is that of the FP64 handle."""
    omega, n = 30, 5
    e, G = pd_inputs.separable_noise(omega, seed=6)
    with pd.Solver(omega, n, e, G, precision=pd.PD_PREC_MIXED, hx_variant=2) as s, pd.Solver(omega, n, e, G) as r:
        a = pd.pairdiag_ground_state_dev(s.h, 1e-7)["e0"]
        b = pd.pairdiag_ground_state_dev(r.h, 1e-10)["e0"]
    assert abs(a - b) <= 1e-6 * max(1.0, abs(b))   # the tolerance asked for, with a factor of ten
