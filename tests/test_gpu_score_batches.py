"""Batches of schedules at the edges of the counting kernels, against the oracle bit for bit: rows of whole 16-byte vectors
(asynchronous copies) and others, one vector more than a CTA's tile, pad bits, an odd schedule at the end, short step chunks,
one wave of CTAs (totals by the last CTA) and more (totals in a second launch), a CTA per schedule with many steps."""
import numpy as np
import pytest

from paper_2508_13231_b200 import workloads as wl
from gpu_util import both_problems, to_dev, u64

pytestmark = pytest.mark.gpu
GB = 10 ** 9


@pytest.fixture(scope="module")
def kvp():
    from paper_2508_13231_b200 import kvp
    return kvp


@pytest.mark.parametrize("U,S,n", [(8192, 512, 40), (8316, 512, 41), (8290, 512, 41), (65659, 130, 25), (65700, 131, 24),
                                   (16384, 257, 64), (262144, 3, 64), (20000, 300, 7), (65664, 20, 8),
                                   # a CTA per schedule, many steps: whole and single words, chunks of 1024 steps and what is left
                                   (1000, 1030, 2), (2040, 513, 3), (420, 1500, 2), (4090, 2049, 1), (250, 1024, 150), (1020, 160, 600)])
def test_batches(kvp, oracle, U, S, n):
    A = wl.random_access(U, S, 0.2, seed=U)
    g, o = both_problems(kvp, oracle, U, 8192, S, A, U // 8, (4900 * GB, 900 * GB, 500 * GB))
    rng = np.random.default_rng(n)
    scheds = rng.integers(0, 2 ** 32, (n, S, A.shape[1]), dtype=np.uint64).astype(np.uint32)
    scheds[::2] &= rng.integers(0, 2 ** 32, (1, S, A.shape[1]), dtype=np.uint64).astype(np.uint32)   # pad bits are ignored
    dev = to_dev(scheds)
    out, counts = g.eval(dev), g.eval_counts(dev)
    for i in sorted({0, min(1, n - 1), n // 2, max(0, n - 2), n - 1}):
        ref = o.eval(scheds[i])
        assert int(u64(out["total_ticks"])[i]) == ref["total_ticks"]
        assert np.array_equal(u64(out["step_ticks"])[i], ref["step_ticks"])
        assert int(out["bad_step"][i]) == ref["bad_step"]
    again = g.eval(dev[-1:].contiguous())
    assert int(u64(again["total_ticks"])[0]) == int(u64(out["total_ticks"])[n - 1])
    one = g.eval_counts(dev[-1:].contiguous())
    assert np.array_equal(one[0].cpu().numpy(), counts[n - 1].cpu().numpy())
