"""Timed cases of the library's public entry points (`paper_2508_13231_b200.kvp`), over the range of problems that the
repository's configurations, figures and benchmark put through them.

A case is a dict of plain values. `op` says which call, or which short run of calls, one pass makes:
  anneal    kvp_anneal on a problem that is kept: best schedule and bound
  growing   layered trace with births -> problem -> anneal: one search on a growing cache, from nothing
  exchange  kvp_anneal_exchange on a problem that is kept: replica exchange over a temperature ladder
  open      trace -> problem -> two schedules scored: what precedes a search on a new trace
  eval      a batch of schedules scored (kvp_eval; kvp_eval_noalloc with the caller's outputs when noalloc is set)
  wr        the paper's annealer: T(W, R) on the whole grid, the (W, R) walk, the schedule of the best pair
  policies  the comparison strategies (static, reactive, page), each generated and scored
All results are whole numbers, bits, or one fp64 product of a whole number, so outputs are compared exactly.
"""
import math

import numpy as np
import torch

from paper_2508_13231_b200 import kvp, workloads as wl

# B_h, B_k, B_d: the two bandwidth sets of the configurations and the paper's Table I
BW = {"8:0.9": (8 * wl.TB, 9 * wl.TB // 10, 9 * wl.TB // 10),
      "8:0.45": (8 * wl.TB, 45 * wl.TB // 100, 45 * wl.TB // 100),
      "gh200": (49 * wl.TB // 10, 9 * wl.TB // 10, 5 * wl.TB // 10)}
BYTES_PER_UNIT = 8192


def _shape(op, groups, units_per_group, steps, topk, cap, bw="8:0.9", rho=0.95, zipf_lo=0.0, zipf_hi=0.0, burst_p=0.0, **more):
    """One problem: `groups` (layer, head) pairs of `units_per_group` blocks, `topk` of them read per group and step."""
    return dict(op=op, groups=groups, units_per_group=units_per_group, steps=steps, topk=topk, cap=cap, bw=bw, rho=rho,
                zipf_lo=zipf_lo, zipf_hi=zipf_hi, burst_p=burst_p, **more)


def listed():
    return [
        # The smallest search: 16 blocks, 64 chains. Launches, copies and the latency of one chain are all there is.
        dict(_shape("anneal", 1, 16, 32, 4, 6, rho=0.9, chains=64, moves=10_000, p0=1e-6), name="anneal tiny"),
        # One attention head, the schedules in shared memory, near-greedy start: the ordinary search of one head.
        dict(_shape("anneal", 1, 256, 512, 26, 64, zipf_lo=1.1, zipf_hi=1.1, chains=1024, moves=100_000, p0=1e-6),
             name="anneal head"),
        # The same at the paper's (and the API's default) start temperature: a fifth of the proposals change the schedule.
        dict(_shape("anneal", 1, 256, 512, 26, 64, zipf_lo=1.1, zipf_hi=1.1, chains=1024, moves=100_000, p0=0.8),
             name="anneal head hot"),
        # One layer of an 8B-class model, few chains per SM, schedules in global memory.
        dict(_shape("anneal", 8, 2048, 256, 256, 4915, rho=0.98, zipf_lo=0.8, zipf_hi=1.4, chains=1024, moves=200_000, p0=1e-6),
             name="anneal layer"),
        # The benchmark's workload: a 70B-class model at long context, 2.6M blocks, 8192 chains of a million moves.
        dict(_shape("anneal", 640, 4096, 64, 205, 262_144, bw="8:0.45", burst_p=0.01, chains=8192, moves=1_000_000, p0=1e-6),
             name="anneal model"),
        # A growing cache: 32 layers x 8 heads, 480 prompt tokens and 32 decoded ones, (token, layer) steps.
        dict(op="growing", layers=32, heads=8, units_per_group=512, prompt=480, topk=51, cap=26_214, bw="8:0.9", rho=0.97,
             zipf_lo=0.8, zipf_hi=1.4, chains=1024, moves=100_000, p0=1e-6, name="growing model"),
        # Replica exchange on one head: 128 ladders of 8 temperatures, an exchange round every 1000 moves.
        dict(_shape("exchange", 1, 256, 512, 26, 64, zipf_lo=1.1, zipf_hi=1.1, chains=1024, moves=100_000, p0=1e-3, alpha=0.5,
                    rungs=8, every=1000), name="exchange head"),
        # What a new trace costs before its search starts, at the largest size: generate, lay out, score two schedules.
        dict(_shape("open", 640, 4096, 64, 205, 262_144, bw="8:0.45", burst_p=0.01), name="open model"),
        # One schedule of one head scored: the call inside a control loop, all latency.
        dict(_shape("eval", 1, 256, 512, 26, 64, zipf_lo=1.1, zipf_hi=1.1, batch=1, noalloc=False), name="eval one"),
        # A batch of full-size schedules scored: streaming from memory.
        dict(_shape("eval", 640, 4096, 64, 205, 262_144, bw="8:0.45", burst_p=0.01, batch=96, noalloc=False), name="eval batch"),
        # The paper's own search at token granularity (80% sparsity): 64 x 11 policies simulated, scored and walked.
        dict(_shape("wr", 1, 4096, 512, 819, 1024, zipf_lo=1.1, zipf_hi=1.1, w_max=64, n_ratio=11, chains=64, iters=2000),
             name="wr search"),
        # The strategies it is compared with, at the paper's 60% sparsity.
        dict(_shape("policies", 1, 4096, 512, 1638, 1024, zipf_lo=1.1, zipf_hi=1.1, page=16), name="policies"),
    ]


def _log(rng, lo, hi):
    """Whole number, its logarithm uniform over lo..hi."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _problem(rng, op, units_lo, units_hi, steps_hi, bits, **more):
    """A random problem of units_lo..units_hi blocks and 32..steps_hi steps, of at most `bits` block-steps."""
    units = _log(rng, units_lo, units_hi)
    steps = _log(rng, 32, max(32, min(steps_hi, bits // units)))
    groups = _log(rng, max(1, -(-units // 4096)), max(1, -(-units // 4096), min(640, units // 64)))
    n = max(4, units // groups)
    zipf = rng.choice([None, (1.1, 1.1), (0.8, 1.4)]) if groups <= 64 else None    # drawn per group on the host
    lo, hi = zipf or (0.0, 0.0)
    return _shape(op, groups, n, steps, max(1, int(n * rng.uniform(0.05, 0.2))), max(1, int(groups * n * rng.uniform(0.1, 0.35))),
                  bw=rng.choice(sorted(BW) if units < 2_000_000 else ["8:0.9", "8:0.45"]),    # ticks of Table I need 31 bits
                  rho=round(rng.uniform(0.9, 0.98), 3), zipf_lo=lo, zipf_hi=hi,
                  burst_p=rng.choice([0.0, 0.0, 0.01]), **more)


def draw(rng):
    op = rng.choice(["anneal", "anneal", "anneal", "growing", "exchange", "open", "eval", "eval", "wr", "policies"])
    if op == "anneal":
        c = _problem(rng, op, 16, 2_621_440, 512, 167_000_000)
        hot = rng.random() < 0.25
        chains = _log(rng, 32, 4096)
        # near-greedy chains do some 10^10 moves per second, hot ones a tenth of that
        c.update(chains=chains, moves=_log(rng, 5_000, max(5_000, min(1_000_000 if not hot else 60_000,
                                                                   (1_500_000_000 if not hot else 60_000_000) // chains))),
                 p0=0.8 if hot else rng.choice([1e-6, 1e-6, 1e-3]))
        return c
    if op == "growing":
        layers, decoded = _log(rng, 2, 32), _log(rng, 4, 32)
        n = _log(rng, decoded + 8, 512)
        heads = _log(rng, 1, 8)
        return dict(op=op, layers=layers, heads=heads, units_per_group=n, prompt=n - decoded, topk=max(2, n // 10),
                    cap=max(1, int(layers * heads * n * rng.uniform(0.1, 0.3))), bw=rng.choice(sorted(BW)),
                    rho=round(rng.uniform(0.9, 0.98), 3), zipf_lo=0.8, zipf_hi=1.4, chains=_log(rng, 32, 1024),
                    moves=_log(rng, 5_000, 100_000), p0=1e-6)
    if op == "exchange":
        rungs = rng.randint(3, 12)
        return _problem(rng, op, 16, 512, 512, 131_072, chains=rungs * _log(rng, 4, 1024 // rungs), moves=_log(rng, 10_000, 100_000),
                        p0=1e-3, alpha=rng.choice([0.5, 0.7]), rungs=rungs, every=_log(rng, 500, 5_000))
    if op == "open":
        return _problem(rng, op, 256, 2_621_440, 512, 167_000_000)
    if op == "eval":
        c = _problem(rng, op, 64, 2_621_440, 512, 167_000_000)
        row = (c["groups"] * c["units_per_group"] + 31) // 32 * 4
        batch = _log(rng, 1, max(1, min(1024, 2_000_000_000 // (row * c["steps"]))))
        c.update(batch=batch, noalloc=batch * c["steps"] <= 65_536 and rng.random() < 0.5)
        return c
    if op == "wr":
        return _problem(rng, op, 256, 8192, 512, 4096 * 512, w_max=_log(rng, 8, 64), n_ratio=11, chains=_log(rng, 16, 128),
                        iters=_log(rng, 500, 2000))
    c = _problem(rng, op, 256, 16_384, 512, 4096 * 512 * 2)
    c["page"] = rng.choice([4, 8, 16, 32])
    c["groups"], c["units_per_group"] = 1, min(8192, -(-c["groups"] * c["units_per_group"] // 32) * 32)  # pages divide the units
    c["topk"] = max(1, int(c["units_per_group"] * rng.uniform(0.05, 0.4)))
    c["cap"] = max(32, int(c["units_per_group"] * rng.uniform(0.1, 0.35)))
    return c


# ------------------------------------------------------------------------------------------------------------------

def _trace_args(case, seed):
    """Arguments of kvp.trace_generate, the static importance on the GPU."""
    zipf = (case["zipf_lo"], case["zipf_hi"]) if case["zipf_hi"] else None
    if case["op"] == "growing":
        groups, steps = case["layers"] * case["heads"], case["layers"] * (case["units_per_group"] - case["prompt"] + 1)
    else:
        groups, steps = case["groups"], case["steps"]
    tp = wl.custom_trace_params(groups, case["units_per_group"], steps, case["topk"], case["rho"], zipf=zipf, seed=seed)
    if case.get("burst_p"):
        tp.update(burst_jump=4 * wl.Q16, burst_thr=int(case["burst_p"] * 2 ** 32))
    if tp["base"] is not None:
        tp["base"] = torch.from_numpy(tp["base"]).cuda()
    return tp


def _open(case, access, birth=None):
    groups = case["layers"] * case["heads"] if case["op"] == "growing" else case["groups"]
    return kvp.Problem(groups * case["units_per_group"], BYTES_PER_UNIT, access.shape[0], access, case["cap"], *BW[case["bw"]],
                       birth=birth)


def _schedules(case, n, seed):
    """n schedules on the GPU: a static row of about an eighth of the units, a few per cent of them moved at each step."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    w32 = (case["groups"] * case["units_per_group"] + 31) // 32

    def bits(rows, thin):
        r = torch.randint(-2 ** 31, 2 ** 31 - 1, (n, rows, w32), dtype=torch.int32, device="cuda", generator=g)
        for _ in range(thin):
            r &= torch.randint(-2 ** 31, 2 ** 31 - 1, r.shape, dtype=torch.int32, device="cuda", generator=g)
        return r

    return bits(case["steps"], 4).bitwise_xor_(bits(1, 2))


def prepare(case, seed):
    op = case["op"]
    tp = _trace_args(case, seed)
    st = dict(case=case, trace=tp)
    if op == "growing":
        c = dict(layers=case["layers"], heads=case["heads"], units_per_group=case["units_per_group"], prompt=case["prompt"])
        st["birth"] = torch.from_numpy(wl.growing_births(c).astype(np.int32)).cuda()
        st["seed"] = seed
        return st
    if op == "open":
        st["schedules"] = _schedules(case, 2, seed)
        return st
    prob = st["problem"] = _open(case, kvp.trace_generate(**tp))
    if op == "anneal":
        st["params"] = prob.make_params(case["chains"], case["moves"], seed=seed, p0=case["p0"])
    elif op == "exchange":
        st["params"] = prob.make_params(case["chains"], case["moves"], seed=seed, levels=case["rungs"], p0=case["p0"],
                                        alpha=case["alpha"])
    elif op == "eval":
        st["schedules"] = _schedules(case, case["batch"], seed)
        if case["noalloc"]:
            n, S = case["batch"], case["steps"]
            new = lambda shape, t: torch.empty(shape, dtype=t, device="cuda")  # noqa: E731
            st["out"] = [new((n, S), torch.int64), new(n, torch.int64), new((n, S), torch.float64), new(n, torch.float64),
                         new(n, torch.int32)]
    elif op == "wr":
        st["params"] = kvp.wr_params(chains=case["chains"], iters=case["iters"], seed=seed, levels=32)
    return st


def _found(r):
    """What a search is run for: the schedule, the bound and how it was reached."""
    s = r["stats"]
    return dict(schedule=r["best_schedule"], seconds=r["best_seconds"],
                whole=np.array([r["best_ticks"], s.init_ticks, s.best_chain, s.best_move, s.moves_total, s.calib_mean_delta,
                                s.winner_hits, s.winner_accessed], np.uint64).view(np.int64))


def run(st):
    case = st["case"]
    op = case["op"]
    if op == "anneal":
        return _found(st["problem"].anneal(st["params"]))
    if op == "growing":
        access = kvp.trace_generate(**st["trace"], layers=case["layers"], birth=st["birth"])
        prob = _open(case, access, birth=st["birth"])
        r = _found(prob.anneal(prob.make_params(case["chains"], case["moves"], seed=st["seed"], p0=case["p0"])))
        prob.close()
        return dict(r, access=access)
    if op == "exchange":
        r = st["problem"].anneal_exchange(st["params"], case["rungs"], case["every"])
        return dict(_found(r), rungs=np.array(r["final_rung"], np.int64), exchanged=np.array(r["n_exchanged"], np.int64))
    if op == "open":
        access = kvp.trace_generate(**st["trace"])
        prob = _open(case, access)
        r = prob.eval(st["schedules"])
        prob.close()
        return dict(r, access=access)
    if op == "eval":
        if case["noalloc"]:
            st["problem"].eval_noalloc(st["schedules"], *st["out"])
            return st["out"]
        return st["problem"].eval(st["schedules"])
    prob = st["problem"]
    if op == "wr":
        table = prob.wr_grid(case["w_max"], case["n_ratio"])
        chains, best = kvp.wr_anneal(table, st["params"])
        schedule = prob.policy_lookahead([best.best_w], [1000 * best.best_r // (case["n_ratio"] - 1)])
        return dict(table=table, chains=np.array([c.astuple() for c in chains], np.uint64).view(np.int64), schedule=schedule)
    out = {}
    for name, make in (("static", lambda: prob.policy_lookahead([1], [0])), ("reactive", prob.policy_reactive),
                       ("page", lambda: prob.policy_page(case["page"]))):
        schedule = make()
        out[name] = dict(schedule=schedule, ticks=prob.eval(schedule, want_steps=False, want_seconds=False)["total_ticks"],
                         counts=prob.eval_counts(schedule))
    return out


def work(case):
    """Bytes: every input bitmap read once, every result written once. Operations: whole-number operations of the method
    (a proposal is some 130: the ten rounds of its Philox block, its decoding, the two placement windows and the verdict;
    a synthesised score 130: its Philox block and recurrence; a policy or a score of a schedule a few per word)."""
    op = case["op"]
    if op == "growing":
        groups, steps = case["layers"] * case["heads"], case["layers"] * (case["units_per_group"] - case["prompt"] + 1)
    else:
        groups, steps = case["groups"], case["steps"]
    units = groups * case["units_per_group"]
    bitmap = (units + 31) // 32 * 4 * steps
    if op in ("anneal", "exchange"):
        return {"bytes": 2 * bitmap, "flops": 130 * case["chains"] * case["moves"]}
    if op == "growing":
        tokens = steps // case["layers"]
        return {"bytes": 3 * bitmap, "flops": 130 * (case["chains"] * case["moves"] + units * tokens)}
    if op == "open":
        return {"bytes": 4 * bitmap, "flops": 130 * units * steps}
    if op == "eval":
        return {"bytes": bitmap * (1 + case["batch"]) + 16 * case["batch"] * steps, "flops": bitmap / 4 * 6 * case["batch"]}
    if op == "wr":
        # a policy looks at every unit's accesses in every step's window and writes one row
        return {"bytes": 2 * bitmap + 8 * case["w_max"] * case["n_ratio"],
                "flops": 8 * units * steps * case["w_max"] * case["n_ratio"]}
    return {"bytes": bitmap * 4, "flops": 24 * units * steps}


def tolerance(case):
    return "exact"
