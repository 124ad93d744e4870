"""One element of x that is not finite touches its own rows only: the others keep
the bits of the product by pair removal, and the product takes no longer than
forming those rows costs."""
import math

import numpy as np
import pytest

import oracle
import pd_inputs

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_2001_01978_gb300")

pytestmark = pytest.mark.gpu


def neighbours(omega, n, index):
    b = oracle.basis(omega, n)
    w = b ^ b[index]
    return np.array([bin(int(v)).count("1") <= 2 for v in w])


# one set of blocks, without and with rows of no low pairs; the kernels of small blocks
@pytest.mark.parametrize("omega,n", [(18, 9), (22, 5), (30, 4)])
@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_rows_it_does_not_reach(omega, n, value):
    e, G = pd_inputs.separable_noise(omega, seed=1)
    x = torch.from_numpy(pd_inputs.random_vector(math.comb(omega, n), 2).astype(np.float32)).cuda()
    bad = x.clone()
    bad[4321] = value
    with pd.Solver(omega, n, e, G, precision=pd.PD_PREC_MIXED, hx_variant=2) as s:
        good, y, zero = torch.empty_like(x), torch.empty_like(x), torch.empty_like(x)
        pd.pairdiag_hx_dev(s.h, pd.PD_PREC_MIXED, x, good)
        pd.pairdiag_hx_dev(s.h, pd.PD_PREC_MIXED, bad, y)
        torch.cuda.synchronize()
    reached = torch.from_numpy(neighbours(omega, n, 4321)).cuda()
    assert torch.equal(y[~reached], good[~reached])
    assert not bool(torch.isfinite(y[reached]).any())


def test_time():
    """C(24, 12) has 2.7e6 rows, of which one element reaches 145 and a vector
    full of NaN makes every row NaN at once."""
    omega, n = 24, 12
    e, G = pd_inputs.separable_noise(omega, seed=1)
    with pd.Solver(omega, n, e, G, precision=pd.PD_PREC_MIXED, hx_variant=2) as s:
        pd.pairdiag_set_stream(s.h, torch.cuda.current_stream())
        x = torch.randn(s.dim, dtype=torch.float32, device="cuda")
        one, every = x.clone(), torch.full_like(x, float("nan"))
        one[12345] = float("inf")
        y = torch.empty_like(x)

        def ms(v):
            t = []
            for _ in range(7):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                pd.pairdiag_hx_dev(s.h, pd.PD_PREC_MIXED, v, y)
                b.record()
                torch.cuda.synchronize()
                t.append(a.elapsed_time(b))
            return sorted(t)[3]

        usual = ms(x)
        assert ms(one) < 6 * usual and ms(every) < 6 * usual, (usual, ms(one), ms(every))
