"""Memory that only makes products faster (the scratch of the pair removal, the
full-space vectors of a truncated handle) makes way for the solver's own vectors:
allocations that fail once on the host side, as they would on a full device."""
import math

import pytest

import pd_inputs

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_2001_01978_gb300")

pytestmark = pytest.mark.gpu

OMEGA, N, LOW = 20, 10, 10                       # removal by the automatic rule; its row kernel has 10 low orbits
DIM = math.comb(OMEGA, N)
E, G = pd_inputs.separable_noise(OMEGA, seed=3)


@pytest.fixture(autouse=True)
def no_failures_left():
    yield
    pd.pairdiag_fail_alloc(0, 0)


def solver(**kw):
    return pd.Solver(OMEGA, N, E, G, **kw)


def product(s, precision=None, seed=1):
    precision = pd.PD_PREC_MIXED if precision is None else precision
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(pd.pairdiag_dim(s.h), dtype=torch.float32 if precision else torch.float64, device="cuda", generator=gen)
    y = torch.full_like(x, float("nan"))
    pd.pairdiag_hx_dev(s.h, precision, x, y)
    torch.cuda.synchronize()
    return y


# the FP32 window, the FP64 pair of the refinement, the FP64 window of its cycles
@pytest.mark.parametrize("nbytes,count", [(4 * 20 * DIM, 1), (8 * DIM, 1), (8 * 20 * DIM, 1)])
def test_solve_goes_on_without_the_scratch(nbytes, count):
    with solver(precision=pd.PD_PREC_MIXED) as s, solver(precision=pd.PD_PREC_MIXED, hx_variant=3, low_bits=LOW) as rows:
        ref = pd.pairdiag_ground_state_dev(rows.h, 1e-8)["e0"]
        assert not torch.equal(product(s), product(rows))
        pd.pairdiag_fail_alloc(nbytes, count)
        got = pd.pairdiag_ground_state_dev(s.h, 1e-8)["e0"]
        assert abs(got - ref) <= 2e-8 * abs(ref)
        assert torch.equal(product(s), product(rows))        # row by row from then on


def test_without_anything_to_give_the_call_fails_and_the_handle_goes_on():
    with solver(precision=pd.PD_PREC_MIXED) as s:
        for nbytes, count in ((4 * 20 * DIM, 2), (4 * DIM, 100)):      # the retry fails too; then the work vector
            pd.pairdiag_fail_alloc(nbytes, count)
            with pytest.raises(pd.PairDiagError) as err:
                pd.pairdiag_ground_state_dev(s.h, 1e-6)
            assert err.value.code == pd.PD_ENOMEM
            pd.pairdiag_fail_alloc(0, 0)
        assert pd.pairdiag_ground_state_dev(s.h, 1e-6)["converged"]


def test_a_work_vector_that_fails_after_its_window():
    """The window fits and the work vector does not: the next call allocates it."""
    with solver(precision=pd.PD_PREC_FP64) as s:
        pd.pairdiag_fail_alloc(0, 0)
        pd.pairdiag_release_cache()
        pd.pairdiag_hx(s.h, [0.0] * DIM)                     # (v64 and w64 exist)
        pd.pairdiag_fail_alloc(8 * DIM, 100)
        with pytest.raises(pd.PairDiagError):
            pd.pairdiag_ground_state_dev(s.h, 1e-6)
        pd.pairdiag_fail_alloc(0, 0)
        assert pd.pairdiag_ground_state_dev(s.h, 1e-6)["converged"]


@pytest.mark.parametrize("precision", [0, 1])
def test_truncated_solve_goes_on_through_the_map(precision):
    form = pd.PD_PREC_MIXED if precision else pd.PD_PREC_FP64
    with solver(precision=form) as s, solver(precision=form, hx_variant=1, low_bits=LOW) as by_map:
        kept = pd.pairdiag_truncate(s.h, 20000)
        assert pd.pairdiag_truncate(by_map.h, 20000) == kept
        ref = pd.pairdiag_ground_state_dev(by_map.h, 1e-8)["e0"]
        pd.pairdiag_fail_alloc((4 if precision else 8) * 20 * kept, 1)
        got = pd.pairdiag_ground_state_dev(s.h, 1e-8)["e0"]
        assert abs(got - ref) <= 2e-8 * abs(ref)
        assert torch.equal(product(s, precision), product(by_map, precision))


def test_a_captured_product_keeps_its_memory():
    with solver(precision=pd.PD_PREC_MIXED) as s:
        gen = torch.Generator(device="cuda").manual_seed(1)
        x = torch.randn(DIM, dtype=torch.float32, device="cuda", generator=gen)
        want, y = product(s), torch.empty_like(x)
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            pd.pairdiag_set_stream(s.h, torch.cuda.current_stream())
            pd.pairdiag_hx_dev(s.h, pd.PD_PREC_MIXED, x, y)
        pd.pairdiag_set_stream(s.h, torch.cuda.current_stream())
        pd.pairdiag_fail_alloc(4 * 20 * DIM, 1)
        with pytest.raises(pd.PairDiagError):
            pd.pairdiag_ground_state_dev(s.h, 1e-6)
        pd.pairdiag_truncate(s.h, 20000)
        pd.pairdiag_truncate(s.h, 0)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, want)


def test_a_truncated_handle_holds_no_scratch():
    """And a handle back in the full space takes it again."""
    with solver(precision=pd.PD_PREC_MIXED) as s:
        full = product(s)
        pd.pairdiag_release_cache()
        pd.pairdiag_truncate(s.h, 20000)
        # rows of 0..10 low pairs (12 low orbits, 8 high ones), FP32
        scratch = 4 * sum(math.comb(8, p) * p * math.comb(12, N - p) for p in range(9))
        assert pd.pairdiag_release_cache() >= scratch
        truncated = product(s)
        pd.pairdiag_truncate(s.h, 0)
        assert torch.equal(product(s), full)
        pd.pairdiag_truncate(s.h, 20000)
        assert torch.equal(product(s), truncated)


def test_fp32_product_of_a_truncated_fp64_handle():
    """Its full-space FP32 vector is made at the first product; without room, and
    under capture, the product goes through the map."""
    with solver(precision=pd.PD_PREC_MIXED) as m, solver(precision=pd.PD_PREC_FP64) as s, \
            solver(precision=pd.PD_PREC_FP64) as t, solver(precision=pd.PD_PREC_FP64, hx_variant=1, low_bits=LOW) as by_map:
        for h in (m, s, t, by_map):
            pd.pairdiag_truncate(h.h, 20000)
        assert torch.equal(product(s), product(m))
        pd.pairdiag_fail_alloc(4 * DIM, 1)
        assert torch.equal(product(t), product(by_map))
        assert torch.equal(product(t), product(by_map))


def batch(sizes, tol, **kw):
    ps = [(o, n, *pd_inputs.separable_noise(o, seed=5 + o)) for o, n in sizes]
    before = pd.pairdiag_kernel_launches()
    r = pd.pairdiag_batch_ground_state(ps, tol, pd.pairdiag_default_options(precision=pd.PD_PREC_MIXED, **kw))
    return list(r["e0"]), pd.pairdiag_kernel_launches() - before


def scratch_bytes(sizes):
    return 4 * sum(math.comb(o - 12, p) * p * math.comb(12, n - p) for o, n in sizes for p in range(o - 11) if p <= n)


def vector_elements(sizes):
    return sum((math.comb(o, n) + 3) // 4 * 4 for o, n in sizes)


def test_batch_takes_its_vectors_before_the_scratch():
    """The first allocation of the scratch's size or more is the FP32 window: its
    failure is the call's.  The failure of the FP64 window makes the scratch go,
    and the call ends as without it."""
    sizes = [(17, 8), (18, 9), (19, 8)]
    assert scratch_bytes(sizes) < 4 * 20 * vector_elements(sizes)
    ref = batch(sizes, 1e-9)
    assert ref[1] != batch(sizes, 1e-9, hx_variant=3)[1]      # two launches per FP32 product
    pd.pairdiag_fail_alloc(scratch_bytes(sizes), 1)
    with pytest.raises(pd.PairDiagError) as err:
        batch(sizes, 1e-9)
    assert err.value.code == pd.PD_ENOMEM
    pd.pairdiag_fail_alloc(8 * 20 * vector_elements(sizes), 1)
    assert batch(sizes, 1e-9) == ref


def test_batch_without_the_scratch_goes_row_by_row():
    """A window of four vectors is smaller than the scratch of C(22, 11)."""
    sizes = [(22, 11)]
    assert scratch_bytes(sizes) > 4 * 4 * vector_elements(sizes)
    rows = batch(sizes, 1e-5, window=4, hx_variant=3)
    assert batch(sizes, 1e-5, window=4)[1] != rows[1]
    pd.pairdiag_fail_alloc(scratch_bytes(sizes), 1)
    assert batch(sizes, 1e-5, window=4) == rows
