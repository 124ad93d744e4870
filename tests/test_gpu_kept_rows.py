"""The truncated product by lists of kept rows (variants 2 to 5) against the one
that looks every state up in the map (variant 1), at the sizes where it can go
wrong: one kept state, blocks of at most 32 kept rows and of several per thread,
all but a few states kept, few and many high orbits."""
import math

import numpy as np
import pytest

import pd_inputs

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_2001_01978_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("omega,n,limit,low", [(9, 4, 1, 0), (12, 6, 923, 0), (13, 6, 40, 12), (16, 8, 12000, 13),
                                               (17, 3, 300, 5), (20, 10, 150000, 12), (22, 18, 2000, 0),
                                               (21, 7, 50000, 9)])
@pytest.mark.parametrize("precision", [0, 1])
def test_kept_rows_vs_map(omega, n, limit, low, precision):
    e, G = pd_inputs.separable_noise(omega, seed=omega + n)
    dt = torch.float64 if precision == pd.PD_PREC_FP64 else torch.float32
    eps = 2.0 ** -52 if precision == pd.PD_PREC_FP64 else 2.0 ** -23
    out = []
    for variant in (1, 3):
        with pd.Solver(omega, n, e, G, low_bits=low, hx_variant=variant) as s:
            kept = pd.pairdiag_truncate(s.h, limit)
            assert limit <= kept < math.comb(omega, n)
            gen = torch.Generator(device="cuda").manual_seed(3)
            for _ in range(2):                   # a second vector: nothing is left of the first
                x = torch.randn(kept, dtype=dt, device="cuda", generator=gen)
                y = torch.full_like(x, float("nan"))
                pd.pairdiag_hx_dev(s.h, precision, x, y)
            out.append(y.double().cpu().numpy())
            xs = float(x.abs().max())
    # both are sums of the same terms: 4 terms eps times a bound on |H| |x|
    terms = n * (omega - n) + 2
    row = float(np.abs(G).max()) * terms + float(np.sum(np.abs(2 * e + np.diag(G))))
    assert np.all(np.abs(out[0] - out[1]) <= 8.0 * terms * eps * row * xs)
