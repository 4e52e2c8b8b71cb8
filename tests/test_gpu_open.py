"""From trace to problem at the edges of the kernels' tiles, against the oracle bit for bit: selections that the largest keys
of the lanes bound and those they cannot, problems whose bitmap is one row or column tile, one more, or a part of one."""
import numpy as np
import pytest

from paper_2508_13231_b200 import workloads as wl
from gpu_util import both_problems, to_dev, to_np, trace_on_gpu

pytestmark = pytest.mark.gpu
GB, Q16 = 10 ** 9, 65536


@pytest.fixture(scope="module")
def kvp():
    from paper_2508_13231_b200 import kvp
    return kvp


@pytest.mark.parametrize("G,n,k", [(2, 4096, 192), (2, 4096, 193), (1, 4097, 24), (2, 8192, 768), (3, 512, 96), (3, 512, 97),
                                   (2, 1000, 1), (1, 2081, 2081), (37, 4096, 205)])
@pytest.mark.parametrize("flags", [0, 1])
def test_selection(kvp, oracle, G, n, k, flags):
    rng = np.random.default_rng(n + k)
    hot = rng.integers(-Q16, Q16, size=G * n)
    hot[: n // 2] += 40 * Q16                        # half of a group far above the rest: a bound that keeps many keys
    tp = dict(groups=G, units_per_group=n, steps=3, topk=k, seed=5, rho_q=int(0.9 * Q16), c_q=int(0.4 * Q16), sigma_q=Q16,
              base=hot.astype(np.int32))
    assert np.array_equal(to_np(trace_on_gpu(kvp, tp, flags)), oracle.trace_generate(**tp))
    tp.update(sigma_q=0, c_q=0, base=np.zeros(G * n, np.int32))       # one value: ties only
    assert np.array_equal(to_np(trace_on_gpu(kvp, tp, flags)), oracle.trace_generate(**tp))


@pytest.mark.parametrize("U,S", [(1, 1), (32, 32), (33, 33), (1024, 64), (1025, 65), (511, 128), (513, 129), (257, 256),
                                 (300, 257), (3, 2049), (40000, 40), (140000, 5)])
@pytest.mark.parametrize("grow", [False, True])
def test_problem(kvp, oracle, U, S, grow):
    """The static row (access counts, ties), the initial columns and the winner's way back to rows."""
    A = wl.random_access(U, S, 0.2, seed=U)
    cap, writes = U // 3, dict(hw=[1] * S, ew=list(range(S)))
    if grow:
        birth = np.random.default_rng(S).integers(0, S, size=U).astype(np.uint32)
        u, s = np.arange(U), np.arange(S)[:, None]
        keep = np.zeros((S, A.shape[1] * 32), bool)
        keep[:, :U] = birth[None, u] <= s
        A = A & np.packbits(keep, axis=1, bitorder="little").view(np.uint32)
        args = (cap, 4900 * GB, 900 * GB, 500 * GB)
        g = kvp.Problem(U, 8192, S, to_dev(A), *args, birth=to_dev(birth), **writes)
        o = oracle.Problem(U, 8192, S, A, *args, birth=birth, **writes)
    else:
        g, o = both_problems(kvp, oracle, U, 8192, S, A, cap, (4900 * GB, 900 * GB, 500 * GB), **writes)
    for init in (kvp.INIT_STATIC_FREQ, kvp.INIT_STATIC_FIRST):
        kw = dict(chains=2, moves=200, seed=3, levels=4, p0=0.2, init_mode=init)
        out, ref = g.anneal(g.make_params(**kw)), o.anneal(o.make_params(**kw))
        assert out["best_ticks"] == ref["best_ticks"]
        assert np.array_equal(to_np(out["best_schedule"]), ref["best_schedule"])
