"""A wait of the FP32 product by pair removal that runs out (a limit of no polls:
the wait gives up at once, the kernel then waits for its product and returns).
The rows are NaN instead of half-made sums, a solve reports PD_ETIMEOUT and says
which wait it was, and the handle goes on working.  Sizes: one set of blocks, rows
class by class after small blocks, tiles of 16, 24, 32 and 40 columns."""
import math

import pytest

import pd_inputs

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_2001_01978_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("omega,n", [(12, 6), (14, 3), (18, 9), (24, 12), (30, 5), (40, 4)])
def test_rows_of_an_expired_product_are_nan(omega, n):
    e, G = pd_inputs.separable_noise(omega, seed=omega)
    with pd.Solver(omega, n, e, G, precision=pd.PD_PREC_MIXED, hx_variant=2) as s:
        gen = torch.Generator(device="cuda").manual_seed(1)
        x = torch.randn(s.dim, dtype=torch.float32, device="cuda", generator=gen)
        good, y = torch.empty_like(x), torch.zeros_like(x)
        pd.pairdiag_hx_dev(s.h, pd.PD_PREC_MIXED, x, good)
        pd.pairdiag_set_wait_limit(s.h, 0)
        pd.pairdiag_hx_dev(s.h, pd.PD_PREC_MIXED, x, y)
        torch.cuda.synchronize()
        assert bool(torch.isnan(y).all())
        pd.pairdiag_set_wait_limit(s.h, 1 << 14)
        pd.pairdiag_hx_dev(s.h, pd.PD_PREC_MIXED, x, y)
        torch.cuda.synchronize()
        assert torch.equal(y, good)


def test_a_solve_reports_its_own_waits_only():
    omega, n = 18, 9
    e, G = pd_inputs.separable_noise(omega, seed=2)
    with pd.Solver(omega, n, e, G, precision=pd.PD_PREC_MIXED, hx_variant=2) as s:
        x = torch.ones(math.comb(omega, n), dtype=torch.float32, device="cuda")
        pd.pairdiag_set_wait_limit(s.h, 0)
        pd.pairdiag_hx_dev(s.h, pd.PD_PREC_MIXED, x, torch.empty_like(x))
        pd.pairdiag_set_wait_limit(s.h, 1 << 14)
        first = pd.pairdiag_ground_state_dev(s.h, 1e-6)       # not failed by the product before it
        pd.pairdiag_set_wait_limit(s.h, 0)
        with pytest.raises(pd.PairDiagError, match="pair removal") as err:
            pd.pairdiag_ground_state_dev(s.h, 1e-6)
        assert err.value.code == pd.PD_ETIMEOUT
        pd.pairdiag_set_wait_limit(s.h, 1 << 14)
        assert pd.pairdiag_ground_state_dev(s.h, 1e-6)["e0"] == first["e0"]


def test_limits_out_of_range_are_refused():
    e, G = pd_inputs.separable_noise(6, seed=1)
    with pd.Solver(6, 3, e, G) as s:
        for polls in (-1, (1 << 20) + 1):
            with pytest.raises(pd.PairDiagError):
                pd.pairdiag_set_wait_limit(s.h, polls)
