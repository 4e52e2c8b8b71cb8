"""The chain kernels' variants at the sizes where they can go wrong, against the oracle bit for bit: every number of warps
per chain, window edges (steps around multiples of 32), vector columns (two and four words), columns longer than half a
warp, schedules in shared and in global memory, weights for which the cost is not linear in migrations, replica exchange
inside CTAs and in launches."""
import numpy as np
import pytest
import torch

from paper_2508_13231_b200 import workloads as wl
from gpu_util import both_problems, to_np

pytestmark = pytest.mark.gpu
GB = 10 ** 9
NARROW, WIDE = (1, 2, 35, 36), (3, 18, 20)       # kvp_test_hooks.warps_per_chain


@pytest.fixture(scope="module")
def kvp():
    from paper_2508_13231_b200 import kvp
    return kvp


def _warps(hook):
    """Warps per chain that a value of the hook stands for."""
    return 1 if hook == 3 else hook & 15 if hook >= 16 else hook


def _same(g, o, **kw):
    out = g.anneal(g.make_params(**kw), want_per_chain=True)
    ref = o.anneal(o.make_params(**kw))
    assert [r.astuple() for r in out["per_chain"]] == [r.astuple() for r in ref["per_chain"]]
    assert np.array_equal(to_np(out["best_schedule"]), ref["best_schedule"])
    return out["stats"]


SHARED = [(2, 2, 1), (31, 32, 9), (40, 31, 0), (40, 33, 40), (65, 64, 20), (33, 97, 10), (7000, 64, 2000), (5000, 128, 900),
          (3000, 257, 700), (300, 2050, 90)]
# above what two chains of an SM can hold in shared memory: columns of 1, 2, 3, 4, 5, 9 and 65 words
GLOBAL = [(30011, 32, 9000), (15004, 64, 4000), (10001, 90, 900), (8003, 128, 1500), (6001, 129, 2000), (3601, 257, 700), (500, 2050, 90)]


@pytest.mark.parametrize("warps", NARROW + WIDE)
@pytest.mark.parametrize("U,S,cap", SHARED + GLOBAL)
def test_shapes(kvp, oracle, hooks, warps, U, S, cap):
    hooks(warps_per_chain=warps)
    A = wl.random_access(U, S, 0.2, seed=U + S)
    g, o = both_problems(kvp, oracle, U, 8192, S, A, cap, (4900 * GB, 900 * GB, 500 * GB))
    for p0 in (0.8, 1e-4):
        st = _same(g, o, chains=5, moves=1500, seed=U, levels=6, p0=p0, early_stop_permille=1, early_stop_from_level=4)
        assert (st.wide_kernel, st.warps_per_chain) == (warps in WIDE, _warps(warps))
        assert st.shared_schedules == ((U, S, cap) in SHARED) and st.bucket_log2 == 0


@pytest.mark.parametrize("link", [900, 500])
@pytest.mark.parametrize("warps", (3, 18))
@pytest.mark.parametrize("U,S", [(30011, 32), (30004, 30), (15004, 64), (15001, 63), (10001, 90), (10004, 90), (7503, 97), (6001, 129),
                                 (3301, 257)])
def test_buckets_of_eight_columns(kvp, oracle, hooks, warps, U, S, link):
    """Buckets of a slice in global memory taken over as vectors (30004, 15004, 10004 and 7503 units) and word by word (slices
    that do not begin at a vector), the last one shorter than the others; columns of 1, 2, 3, 4, 5 and 9 words; one and two
    warps per chain; a link faster and slower than the DRAM channels."""
    hooks(warps_per_chain=warps, overlay=2)
    A = wl.random_access(U, S, 0.2, seed=U + S)
    g, o = both_problems(kvp, oracle, U, 8192, S, A, U // 3, (8000 * GB, link * GB, 900 * GB))
    for p0 in (0.8, 1e-4):
        st = _same(g, o, chains=5, moves=1500, seed=U, levels=6, p0=p0)
        assert (st.wide_kernel, st.warps_per_chain, st.shared_schedules, st.bucket_log2) == (1, _warps(warps), 0, 3) and U % 8


@pytest.mark.parametrize("bw,flags", [((4900, 500, 900), 3), ((4900, 500, 900), 1), ((3, 1, 1), 0)])
def test_weights(kvp, oracle, hooks, bw, flags):
    """A link slower than the DRAM channels (the cost is not linear in migrations), migrations free on a side or both."""
    A = wl.random_access(90, 70, 0.3, seed=1)
    g, o = both_problems(kvp, oracle, 90, 8192, 70, A, 30, tuple(b * GB for b in bw), mig_flags=flags)
    for warps in (2, 18):
        hooks(warps_per_chain=warps)
        _same(g, o, chains=6, moves=2000, seed=4, levels=4, p0=0.3)


@pytest.mark.parametrize("warps", (0,) + NARROW + (18,))
@pytest.mark.parametrize("U,S,cap", [(31, 32, 9), (40, 33, 40), (65, 64, 20), (33, 97, 10), (7000, 64, 2000), (5000, 128, 900),
                                     (3000, 257, 700), (15004, 64, 4000), (8003, 128, 1500), (3601, 257, 700)])
def test_link_slower_than_dram(kvp, oracle, hooks, warps, U, S, cap):
    """Eq. 4's maximum is over three terms then, each of which leads at some steps: the link in either direction, the DRAM
    channels. Written units on either side shift which one does."""
    hooks(warps_per_chain=warps)
    A = wl.random_access(U, S, 0.2, seed=U + S)
    rng = np.random.default_rng(U)
    hw, ew = rng.integers(0, 3, S), rng.integers(0, 4, S) * (rng.random(S) < 0.5)
    g, o = both_problems(kvp, oracle, U, 8192, S, A, cap, (4900 * GB, 500 * GB, 700 * GB), hw=hw, ew=ew)
    for p0 in (0.8, 1e-4):
        st = _same(g, o, chains=5, moves=1500, seed=U, levels=6, p0=p0, early_stop_permille=1, early_stop_from_level=4)
        assert st.shared_schedules == (U * ((S + 31) // 32) < 25000)      # words of a schedule


@pytest.mark.parametrize("warps", [0, 2, 3])
@pytest.mark.parametrize("chains,rungs", [(24, 3), (40, 20)])
def test_exchange_with_slow_link(kvp, oracle, hooks, warps, chains, rungs):
    hooks(warps_per_chain=warps)
    A = wl.random_access(120, 90, 0.25, seed=2)
    g, o = both_problems(kvp, oracle, 120, 8192, 90, A, 30, (8000 * GB, 400 * GB, 900 * GB))
    kw = dict(chains=chains, moves=701, seed=9, levels=rungs, p0=1e-2, alpha=0.7)
    out = g.anneal_exchange(g.make_params(**kw), rungs, 100)
    ref = o.anneal_exchange(o.make_params(**kw), rungs, 100, want_best=True)
    assert [r.astuple() for r in out["per_chain"]] == [r.astuple() for r in ref["per_chain"]]
    assert out["final_rung"] == ref["final_rung"].tolist()
    assert np.array_equal(to_np(out["best_schedule"]), ref["best_schedule"])


@pytest.mark.parametrize("warps", [0, 2, 3, 18])
@pytest.mark.parametrize("chains,rungs", [(24, 3), (40, 8), (36, 12), (40, 20)])
def test_exchange_rounds(kvp, oracle, hooks, warps, chains, rungs):
    """Ladders that fill a CTA exactly, leave chains of it idle, or do not fit one (a launch per round); both kernels."""
    hooks(warps_per_chain=warps)
    A = wl.random_access(120, 90, 0.25, seed=2)
    g, o = both_problems(kvp, oracle, 120, 8192, 90, A, 30, (8000 * GB, 900 * GB, 900 * GB))
    kw = dict(chains=chains, moves=701, seed=9, levels=rungs, p0=1e-2, alpha=0.7)
    out = g.anneal_exchange(g.make_params(**kw), rungs, 100)
    ref = o.anneal_exchange(o.make_params(**kw), rungs, 100, want_best=True)
    assert [r.astuple() for r in out["per_chain"]] == [r.astuple() for r in ref["per_chain"]]
    assert out["final_rung"] == ref["final_rung"].tolist() and out["n_exchanged"] == ref["n_exchanged"].tolist()
    assert np.array_equal(to_np(out["best_schedule"]), ref["best_schedule"])


@pytest.mark.parametrize("chains", [3, 1184])
def test_horizon_that_fills_shared_memory(kvp, oracle, chains):
    """18,600 steps: the state of one chain takes all of an SM's shared memory with one warp and does not fit with four."""
    U, S = 40, 18600
    A = wl.random_access(U, S, 0.1, seed=3)
    g, o = both_problems(kvp, oracle, U, 8192, S, A, 8, (8000 * GB, 900 * GB, 900 * GB))
    kw = dict(chains=chains, moves=60, seed=9, levels=2, p0=1e-4)
    out = g.anneal(g.make_params(**kw), want_per_chain=True)
    for c in (0, 1, chains - 1):
        want, _, _ = o.anneal_chains(o.make_params(**kw), c, 1)
        assert out["per_chain"][c].astuple() == want[0].astuple()


@pytest.mark.parametrize("busy", [False, True])
@pytest.mark.parametrize("p0,init", [(1e-6, 1), (1e-6, 0), (0.3, 1)])
def test_choice_in_global_memory(kvp, oracle, busy, p0, init):
    """The library's own choice between the kernels: by the start temperature and by which side of Eq. 2 is the larger one in
    the most-accessed placement, whatever placement the chains start from. Both give the oracle's chains."""
    U, S, cap = 16384, 64, 1600
    A = wl.random_access(U, S, 0.05, seed=4)
    if busy:
        rng = np.random.default_rng(3)
        hot = rng.permutation(U) < 1700                       # the same tenth of the units at every step, most of it in HBM
        A = wl.pack_bits(np.broadcast_to(hot, (S, U)) & (rng.random((S, U)) < 0.95))
    g, o = both_problems(kvp, oracle, U, 8192, S, A, cap, (8000 * GB, 900 * GB, 900 * GB))
    ratio = g.weights["kh"] / g.weights["ke"]
    counts = g.eval_counts(g.chain_state(g.make_params(1, 1, temps=[1.0], levels=1), 0, 0)[0])[0].cpu().numpy().astype(np.int64)
    hits, reads = counts[:, 0].sum(), wl.unpack_bits(A, U).sum(dtype=np.int64)
    assert (hits * ratio >= 0.9 * (reads - hits)) == busy
    kw = dict(chains=1184, moves=400, seed=2, levels=4, p0=p0, init_mode=init)
    out = g.anneal(g.make_params(**kw), want_per_chain=True)
    assert out["stats"].wide_kernel == (0 if busy or p0 > 0.1 else 1)
    op = o.make_params(**kw)
    for c in (0, 591, 1183):
        want, _, _ = o.anneal_chains(op, c, 1)
        assert out["per_chain"][c].astuple() == want[0].astuple(), c


@pytest.mark.parametrize("U,S,cap,chains,warps", [
    (63, 63, 20, 200, 1), (64, 63, 20, 200, 3), (63, 64, 20, 200, 2),          # units and steps
    (90, 70, 12, 889, 1), (90, 70, 12, 888, 2),                                # chains per SM: 7 and 6
    (90, 70, 80, 1184, 2)])                                                    # a placement that serves more than half of the reads
def test_choice_of_warps_in_shared_memory(kvp, oracle, U, S, cap, chains, warps):
    """Both sides of the lines below which a near-greedy chain has one warp: units and steps, chains per SM, the share of the
    reads that the static placement serves (a little above cap / U here)."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        warps = None                                                           # (the chains per SM are others)
    A = wl.random_access(U, S, 0.2, seed=U + S)
    g, o = both_problems(kvp, oracle, U, 8192, S, A, cap, (8000 * GB, 900 * GB, 900 * GB))
    kw = dict(chains=chains, moves=1200, seed=3, levels=4, p0=1e-6)
    out = g.anneal(g.make_params(**kw), want_per_chain=True)
    assert not out["stats"].wide_kernel and out["stats"].shared_schedules and warps in (None, out["stats"].warps_per_chain)
    op = o.make_params(**kw)
    for c in (0, 1, chains // 2, chains - 1):
        want, _, _ = o.anneal_chains(op, c, 1)
        assert out["per_chain"][c].astuple() == want[0].astuple(), c


@pytest.mark.parametrize("U,S,link,warps,chains,moves,ahead", [
    (10001, 90, 900, 3, 5, 640, 1), (10001, 90, 900, 3, 5, 512, 0), (10001, 90, 900, 3, 5, 1152, 0),       # rows of a level: 5, 4, 9
    (10001, 90, 900, 18, 5, 384, 1), (10001, 90, 900, 18, 5, 640, 0), (10001, 90, 500, 3, 5, 384, 1), (10001, 90, 500, 3, 5, 640, 0),
    (30011, 32, 900, 3, 5, 40000, 0), (15004, 64, 500, 18, 5, 512, 0),
    (8003, 128, 900, 3, 5, 40000, 1), (8003, 128, 900, 18, 5, 512, 1), (8003, 128, 500, 18, 5, 512, 0),    # vectors of four words
    (15004, 64, 900, 3, 5, 384, 0), (15004, 64, 900, 18, 5, 384, 0),                                       # of two
    (20000, 1400, 900, 18, 1184, 256, 1), (20000, 1400, 900, 18, 740, 256, 0),                             # over and under 196 KB
    (4096, 512, 500, 3, 2368, 256, 1), (65536, 512, 500, 3, 2368, 256, 0)])                                # one wave for two, two for two
def test_choice_of_columns_ahead(kvp, oracle, hooks, U, S, link, warps, chains, moves, ahead):
    """Both sides of the lines between two rows of proposals at a time and one whose columns were loaded a row ahead."""
    hooks(warps_per_chain=warps)
    A = wl.random_access(U, S, 0.1, seed=U + S)
    g, o = both_problems(kvp, oracle, U, 8192, S, A, U // 6, (8000 * GB, link * GB, 900 * GB))
    kw = dict(chains=chains, moves=moves, seed=3, levels=4, p0=1e-3)
    out = g.anneal(g.make_params(**kw), want_per_chain=True)
    st = out["stats"]
    assert (st.wide_kernel, st.warps_per_chain, st.shared_schedules) == (1, _warps(warps), 0)
    if chains < 148 or torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert st.columns_ahead == ahead
    op = o.make_params(**kw)
    for c in sorted({0, 1, chains // 2, chains - 1}):
        want, _, _ = o.anneal_chains(op, c, 1)
        assert out["per_chain"][c].astuple() == want[0].astuple(), c


@pytest.mark.parametrize("link", [900, 500])
@pytest.mark.parametrize("warps", [3, 18])
def test_exchange_with_columns_ahead(kvp, oracle, hooks, warps, link):
    """Replica exchange in global memory on the wide kernel, which loads columns ahead whatever the job."""
    hooks(warps_per_chain=warps)
    U, S = 10001, 90
    A = wl.random_access(U, S, 0.2, seed=2)
    g, o = both_problems(kvp, oracle, U, 8192, S, A, 1000, (8000 * GB, link * GB, 900 * GB))
    kw = dict(chains=20, moves=701, seed=9, levels=5, p0=0.5, alpha=0.7)
    out = g.anneal_exchange(g.make_params(**kw), 5, 100)
    ref = o.anneal_exchange(o.make_params(**kw), 5, 100, want_best=True)
    assert (out["stats"].columns_ahead, out["stats"].warps_per_chain) == (1, _warps(warps))
    assert [r.astuple() for r in out["per_chain"]] == [r.astuple() for r in ref["per_chain"]]
    assert np.array_equal(to_np(out["best_schedule"]), ref["best_schedule"])


@pytest.mark.parametrize("scale", [1, 2 ** 10, 2 ** 20])
def test_accept_table_rows(kvp, oracle, scale):
    """Rows built as geometric sequences against exp() for every entry, at temperatures around powers of two."""
    temps = np.sort(np.concatenate([[0.3, 1.0, 1.0, 44.5, 44.6], scale * np.geomspace(1.0, 1000.0, 300)]))[::-1].copy()
    table, shifts = kvp.accept_table(temps)
    want, wshifts = oracle.accept_table(temps)
    assert np.array_equal(to_np(table), np.asarray(want, dtype=np.uint32)) and np.array_equal(to_np(shifts), np.asarray(wshifts, dtype=np.uint32))
