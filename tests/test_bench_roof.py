"""The benchmark's roofline of a product: a fraction of its floor, not of bytes that
the kernel does not move."""
import pytest


def test_roofline_is_a_fraction_of_the_floor():
    bench = pytest.importorskip("bench")
    # C(24, 12): 3.9e8 multiply-adds against 22 MB moved
    nnz, dim = 2704156 * 144, 2704156
    r = bench.hx_roof(nnz, dim, 4, 96e-6, 74.0, 6700.0)
    assert r["bound"] == "fma" and r["unit"] == "TFLOP/s"
    assert r["frac"] == pytest.approx(2 * nnz / 74e12 / 96e-6) and r["frac"] < 1
    assert r["achieved"] / r["peak"] == pytest.approx(r["frac"])
    # one pair in two orbits: two elements moved per hop
    r = bench.hx_roof(2 * 10 ** 6, 10 ** 6, 4, 1e-5, 74.0, 6700.0)
    assert r["bound"] == "hbm" and r["achieved"] / r["peak"] == pytest.approx(r["frac"])
