"""Creating a handle: its tables are built on the host, block by block."""
import time

import pytest

import pd_inputs

torch = pytest.importorskip("torch")
pd = pytest.importorskip("paper_2001_01978_gb300")

pytestmark = pytest.mark.gpu


def test_time_of_many_blocks():
    """C(30, 15) has 262,000 basis blocks: 2 ms; a rank and a sort step for each
    block take 64 ms."""
    e, G = pd_inputs.separable_noise(30, seed=1)
    t = []
    for _ in range(5):
        t0 = time.perf_counter()
        s = pd.Solver(30, 15, e, G)
        t.append(time.perf_counter() - t0)
        s.close()
    assert sorted(t)[2] < 0.02, t
