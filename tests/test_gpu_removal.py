"""The FP32 product by pair removal on the tensor cores (variant 2): rows
element by element against the oracle at the edges of its tiles (128 words of
one pair less per tile, 12 low orbits, columns padded to 16, 24, 32 and 40),
elements that cannot be split, and the class-by-class form of a large space."""
import math

import numpy as np
import pytest

import oracle
import pd_inputs
from helpers import abs_row_scale

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_2001_01978_gb300")

pytestmark = pytest.mark.gpu


def removal_eps(omega, n):
    """Error of a row of sum_i [sum_j G_ij V_j] relative to its sum of absolute
    terms: each inner sum adds three split products per (padded) orbit in FP32
    (2^-23 per addition, which covers an accumulator that truncates), the outer
    one n + 2 terms; the splits and the FP32 rounding of G drop below 8 x 2^-23."""
    return (3 * (omega + 8) + n + 2 + 8) * 2.0 ** -23


def product32(s, x32):
    xt = torch.from_numpy(x32).cuda()
    yt = torch.full_like(xt, float("nan"))
    pd.pairdiag_hx_dev(s.h, pd.PD_PREC_MIXED, xt, yt)
    return yt.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("omega,n", [(2, 1), (5, 2), (11, 5), (12, 1), (12, 6), (12, 11), (13, 12), (16, 8), (17, 1), (17, 9),
                                     (21, 10), (24, 5), (24, 12), (25, 6), (25, 23), (32, 4), (33, 3), (40, 3)])
def test_rows_vs_oracle(omega, n):
    e, G = pd_inputs.separable_noise(omega, seed=3 * omega + n)
    G[0, 1] = G[1, 0] = 0.0                      # a hop of zero strength
    b = oracle.basis(omega, n)
    x32 = pd_inputs.random_vector(len(b), omega + 2 * n).astype(np.float32)
    x32[::7] *= np.float32(1e-12)                # elements of very different size side by side
    x = x32.astype(np.float64)
    with pd.Solver(omega, n, e, G, precision=pd.PD_PREC_MIXED, hx_variant=2) as s:
        got = product32(s, x32)
        again = product32(s, x32)
    assert np.array_equal(got, again)            # sums in a fixed order
    bound = removal_eps(omega, n) * abs_row_scale(omega, n, e, G, x, basis=b)
    err = np.abs(got - oracle.hx(omega, n, e, G, x, b))
    assert np.all(err <= bound), np.max(err / np.maximum(bound, 1e-300))


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, np.finfo(np.float32).max])
def test_elements_that_cannot_be_split(value):
    """Infinities, NaN and a value that overflows when rounded to TF32: the same
    rows are non-finite, in the same way, as in the row-by-row kernel, the others
    agree, and the next product is clean."""
    omega, n = 18, 8
    e, G = pd_inputs.separable_noise(omega, seed=4)
    x32 = pd_inputs.random_vector(math.comb(omega, n), 3).astype(np.float32)
    bad = x32.copy()
    bad[12345] = value
    with pd.Solver(omega, n, e, G, precision=pd.PD_PREC_MIXED, hx_variant=2) as s, \
            pd.Solver(omega, n, e, G, precision=pd.PD_PREC_MIXED, hx_variant=3) as r:
        got, ref = product32(s, bad), product32(r, bad)
        clean, ref_clean = product32(s, x32), product32(r, x32)
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    assert np.array_equal(np.isinf(got), np.isinf(ref))
    inf = np.isinf(ref)
    assert np.array_equal(got[inf], ref[inf])
    fin = np.isfinite(ref)
    scale = abs_row_scale(omega, n, e, G, np.where(np.isfinite(bad), bad, 0.0).astype(np.float64))
    tol = (removal_eps(omega, n) + 4.0 * (n * (omega - n) + 2) * 2.0 ** -23) * scale
    assert np.all(np.abs(got - ref)[fin] <= tol[fin])
    assert np.all(np.isfinite(clean)) and np.all(np.abs(clean - ref_clean) <= tol)


def test_class_by_class_vs_float_float():
    """C(30,15): more scratch than is taken at once, so the rows go class by
    class; every row against the float-float product of the same vector."""
    omega, n = 30, 15
    e, G = pd_inputs.separable_noise(omega, seed=2)
    d = 2.0 * e + np.diag(G)
    with pd.Solver(omega, n, e, G, precision=pd.PD_PREC_MIXED) as s, \
            pd.Solver(omega, n, (np.abs(d) - np.abs(np.diag(G))) / 2.0, np.abs(G)) as a:
        gen = torch.Generator(device="cuda").manual_seed(5)
        x = torch.randn(s.dim, dtype=torch.float32, device="cuda", generator=gen)
        y = torch.empty_like(x)
        ref = torch.empty(s.dim, dtype=torch.float64, device="cuda")
        scale = torch.empty_like(ref)
        pd.pairdiag_hx_dev(s.h, pd.PD_PREC_MIXED, x, y)
        pd.pairdiag_hx_dev(s.h, pd.PD_HX_FLOATFLOAT, x, ref)
        pd.pairdiag_hx_dev(a.h, pd.PD_HX_FLOATFLOAT, x.abs(), scale)
        torch.cuda.synchronize()
        assert bool(((y.double() - ref).abs() <= removal_eps(omega, n) * scale).all())


@pytest.mark.parametrize("omega,n,i,j", [(12, 6, 1, 2), (14, 7, 12, 3), (18, 9, 16, 15), (24, 12, 1, 2), (30, 4, 29, 0)])
def test_rows_with_one_dominant_hop(omega, n, i, j):
    """Every other coefficient 1e-12 times smaller: the row is one term, of which
    the split may drop 4 x 2^-23 and the FP32 rounding of G 2^-24; each of the K / 8
    steps after the term is in the accumulator, the alignment in its own step and the
    two additions that follow (rows, high orbits) may cut one unit in the last place,
    2^-23, of which at most 40 / 8 + 1 + 2 are."""
    e, G = pd_inputs.separable_noise(omega, seed=omega)
    e, G = e * 1e-12, G * 1e-12
    G[i, j] = G[j, i] = 0.3331111
    b = oracle.basis(omega, n)
    x32 = pd_inputs.random_vector(len(b), omega + n).astype(np.float32)
    x = x32.astype(np.float64)
    rows = ((b >> np.uint64(i)) ^ (b >> np.uint64(j))) & np.uint64(1) == 1
    with pd.Solver(omega, n, e, G, precision=pd.PD_PREC_MIXED, hx_variant=2) as s:
        got = product32(s, x32)
    err = np.abs(got - oracle.hx(omega, n, e, G, x, b))[rows]
    scale = abs_row_scale(omega, n, e, G, x, basis=b)[rows]
    assert np.all(err <= (4.5 + 40 / 8 + 1 + 2) * 2.0 ** -23 * scale), np.max(err / scale) * 2 ** 23


def test_class_by_class_40_columns():
    """C(38, 10), 4.7e8 states: tiles of 40 columns, one set of partial results,
    classes with small blocks in launches of their own; every row against the
    float-float product."""
    omega, n = 38, 10
    e, G = pd_inputs.separable_noise(omega, seed=4)
    d = 2.0 * e + np.diag(G)
    with pd.Solver(omega, n, e, G, precision=pd.PD_PREC_MIXED) as s, \
            pd.Solver(omega, n, (np.abs(d) - np.abs(np.diag(G))) / 2.0, np.abs(G)) as a:
        gen = torch.Generator(device="cuda").manual_seed(7)
        x = torch.randn(s.dim, dtype=torch.float32, device="cuda", generator=gen)
        y = torch.full_like(x, float("nan"))
        pd.pairdiag_hx_dev(s.h, pd.PD_PREC_MIXED, x, y)
        err = torch.empty(s.dim, dtype=torch.float64, device="cuda")
        pd.pairdiag_hx_dev(s.h, pd.PD_HX_FLOATFLOAT, x, err)
        torch.cuda.synchronize()
        err.sub_(y).abs_()
        del y
        scale = torch.empty_like(err)
        pd.pairdiag_hx_dev(a.h, pd.PD_HX_FLOATFLOAT, x.abs_(), scale)
        torch.cuda.synchronize()
        assert bool((err <= scale.mul_(removal_eps(omega, n))).all())
