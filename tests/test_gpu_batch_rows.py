"""Rows of the batched FP32 product by pair removal, problem by problem against the
oracle: tiles of two widths in one call, a problem beside them that goes row by
row, one that is skipped, one with an element that is not finite, repeated
products (the tickets of every problem are back at zero)."""
import ctypes
import math

import numpy as np
import pytest

import oracle
import pd_inputs
from helpers import abs_row_scale
from test_gpu_removal import removal_eps

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_2001_01978_gb300")

pytestmark = pytest.mark.gpu


def products(sizes, xs, skip, reps, **opt):
    fn = pd.lib().pairdiag_batch_product_for_tests
    fn.restype = ctypes.c_int
    ptr = ctypes.c_void_p
    fn.argtypes = [ctypes.c_int, ptr, ptr, ptr, ptr, ptr, ctypes.c_int, ptr, ptr, ptr, ptr]
    ham = [pd_inputs.separable_noise(om, seed=3 * om + n) for om, n in sizes]
    om = np.array([s[0] for s in sizes], dtype=np.int32)
    nn = np.array([s[1] for s in sizes], dtype=np.int32)
    e = np.ascontiguousarray(np.concatenate([h[0] for h in ham]))
    G = np.ascontiguousarray(np.concatenate([h[1].ravel() for h in ham]))
    off = np.cumsum([0] + [(len(x) + 3) // 4 * 4 for x in xs])
    x = np.zeros(off[-1], dtype=np.float32)
    for o, v in zip(off, xs):
        x[o:o + len(v)] = v
    y = np.empty_like(x)
    sk = np.array(skip, dtype=np.int32)
    taken = ctypes.c_int()
    o = pd.pairdiag_default_options(precision=pd.PD_PREC_MIXED, **opt)
    torch.cuda.init()
    st = fn(len(sizes), om.ctypes.data, nn.ctypes.data, e.ctypes.data, G.ctypes.data, ctypes.addressof(o), reps,
            x.ctypes.data, y.ctypes.data, sk.ctypes.data, ctypes.addressof(taken))
    assert st == pd.PD_OK
    return ham, [y[a:a + len(v)].astype(np.float64) for a, v in zip(off, xs)], taken.value


def vectors(sizes):
    return [pd_inputs.random_vector(math.comb(om, n), om + n).astype(np.float32) for om, n in sizes]


# (9, 4) and (12, 6) have no removal (12 orbits or fewer), (14, 7) too few states
@pytest.mark.parametrize("sizes,removal", [([(17, 8), (9, 4), (26, 5), (18, 9), (14, 7), (25, 6), (12, 6)], 4),
                                           ([(22, 11)], 1), ([(16, 8), (13, 6)], 0)])
def test_rows_vs_oracle(sizes, removal):
    xs = vectors(sizes)
    for reps in (1, 3):
        ham, ys, taken = products(sizes, xs, [0] * len(sizes), reps)
        assert taken == removal
        for (om, n), (e, G), x, y in zip(sizes, ham, xs, ys):
            b = oracle.basis(om, n)
            x64 = x.astype(np.float64)
            rows = (4 * n * (om - n) + 8) * 2.0 ** -23               # row by row: a chain of hops
            bound = max(removal_eps(om, n), rows) * abs_row_scale(om, n, e, G, x64, basis=b)
            assert np.all(np.abs(y - oracle.hx(om, n, e, G, x64, b)) <= bound), (om, n)


def test_the_bits_of_a_single_handle():
    """Where the handle runs the same kernels: fewer than 2000 small blocks (with
    more, another kernel adds the high orbits' diagonal in another order)."""
    sizes = [(17, 8), (25, 4), (18, 9), (26, 4), (22, 6)]
    xs = vectors(sizes)
    ham, ys, taken = products(sizes, xs, [0] * 5, 2, hx_variant=2)
    assert taken == 5
    for (om, n), (e, G), x, y in zip(sizes, ham, xs, ys):
        with pd.Solver(om, n, e, G, precision=pd.PD_PREC_MIXED, hx_variant=2) as s:
            xt = torch.from_numpy(x).cuda()
            yt = torch.empty_like(xt)
            pd.pairdiag_hx_dev(s.h, pd.PD_PREC_MIXED, xt, yt)
            assert np.array_equal(yt.cpu().numpy().astype(np.float64), y)


def test_skipped_and_not_finite():
    sizes = [(17, 8), (18, 9), (17, 6), (22, 5), (26, 5)]
    xs = vectors(sizes)
    clean = products(sizes, xs, [0] * 5, 1)[1]
    bad = [x.copy() for x in xs]
    bad[3][777] = np.inf
    got = products(sizes, bad, [0, 1, 0, 0, 0], 2)[1]
    assert np.all(np.isnan(got[1]))                                   # nothing was written
    for p in (0, 2, 4):
        assert np.array_equal(got[p], clean[p])
    om, n = sizes[3]
    b = oracle.basis(om, n)
    reached = np.array([bin(int(w)).count("1") <= 2 for w in b ^ b[777]])
    assert not np.any(np.isfinite(got[3][reached]))
    assert np.array_equal(got[3][~reached], clean[3][~reached])
