"""Performance cases of the execution-plan search: what its users have it do, end to end.

A training job reports a failure set and wants a recovery plan (one at a time, lowest
latency), or a planner works through many failure sets ahead of time (batches, with and
without sharing, both execution orders, both cost modes, with the transition time in the
objective), or it looks at the space itself (enumerate / select / decode, the cost of many
single candidates).  Jobs are the four of the repository's workloads -- 8, 32, 64 and 256
devices -- with layer times and failure sets drawn from the seed.
"""
import math
from dataclasses import dataclass, field

import numpy as np
import torch

from paper_2508_21613_b200 import binding, workloads

# the jobs of workloads.py by device count: grid, layers, layer bytes, links, search window
JOBS = {
    "8dev": dict(L=8, dp=2, pp=4, micro=8, act=8_000_000, p2p=8_000_000, par=50_000_000, cap=80_000_000_000,
                 intra=25, inter=25, window=(1, 7, 1, 8), layers=workloads.LAYERS_FULL, batch=workloads.BATCH_FULL, kappa=1 << 62),
    "32dev": dict(L=32, dp=4, pp=8, micro=32, act=2048 * 4096 * 2, p2p=2048 * 4096 * 2, par=12 * 4096 * 4096 * 2,
                  cap=80_000_000_000, intra=400, inter=25, window=(3, 5, 4, 12), layers=workloads.LAYERS_REMAINDER,
                  batch=workloads.BATCH_REMAINDER, kappa=1 << 16),
    "64dev": dict(L=80, dp=2, pp=32, micro=64, act=34 * 2048 * 8192, p2p=2048 * 8192 * 2, par=12 * 8192 * 8192 * 2,
                  cap=80_000_000_000, intra=400, inter=25, window=(1, 3, 16, 48), layers=workloads.LAYERS_REMAINDER,
                  batch=workloads.BATCH_REMAINDER, kappa=1 << 16),
    "256dev": dict(L=96, dp=8, pp=32, micro=128, act=2048 * 12288 * 2, p2p=2048 * 12288 * 2, par=12 * 12288 * 12288 * 2,
                   cap=120_000_000_000, intra=400, inter=25, window=(7, 9, 30, 34), layers=workloads.LAYERS_REMAINDER,
                   batch=workloads.BATCH_REMAINDER, kappa=1 << 13),
}
MOST_FAILED = {"8dev": 2, "32dev": 4, "64dev": 8, "256dev": 16}
MOST_SETS = {"8dev": 256, "32dev": 3000, "64dev": 200, "256dev": 384}
PLAN_BYTES = 232

# cm_plan as numpy sees it (the C struct of include/chameleon.h)
PLAN = np.dtype([("policy", "<i4"), ("feasible", "<i4"), ("cost", "<f8"), ("cost_ns", "<i8"), ("strategy", "<u4"),
                 ("n_pipes", "<u4"), ("split_rank", "<u8"), ("stages", "<u2", 16), ("micro", "<u2", 16), ("kappa", "<u8", 16)])
# the numbers of cm_transition (its device assignment left out: several matchings of one plan can be optimal,
# and the definition fixes their total, not the assignment)
TRANS = np.dtype([("policy", "<i4"), ("feasible", "<i4"), ("rank", "<i4"), ("n_survivors", "<i4"), ("xfer_bytes", "<i8"),
                  ("t_trans", "<f8"), ("t_trans_ns", "<i8"), ("objective", "<f8"), ("rounds", "<i4"), ("domains", "<i4"),
                  ("t_sync", "<f8"), ("t_sync_ns", "<i8"), ("assign", "<u2", 256)])


def _case(kind, job, sets=1, fail_lo=1, fail_hi=1, micro=0, cost=0, order=0, sharing=False, rounds=0, count=0, indexed=False):
    return dict(kind=kind, job=job, sets=sets, fail_lo=fail_lo, fail_hi=fail_hi, micro=micro or JOBS[job]["micro"],
                cost=cost, order=order, sharing=sharing, rounds=rounds, count=count, indexed=indexed)


def listed():
    return [
        # a failure is being handled now: one set, plan wanted as soon as possible
        dict(_case("one", "8dev"), name="one failure 8 devices"),
        dict(_case("one", "32dev", fail_lo=2, fail_hi=2), name="one failure 32 devices"),
        # deep pipelines, most compositions rejected by memory; integer nanoseconds
        dict(_case("one", "64dev", fail_lo=3, fail_hi=3, cost=1), name="one failure 64 devices int64"),
        # a node of eight lost from the largest job
        dict(_case("one", "256dev", fail_lo=8, fail_hi=8), name="one failure 256 devices"),
        # the step-by-step interface: enumerate the three spaces, select, decode the layer cuts
        dict(_case("select", "32dev", fail_lo=1, fail_hi=1), name="enumerate and select 32 devices"),
        # plans for many potential failure sets, computed ahead of time
        dict(_case("batch", "32dev", sets=2576, fail_lo=1, fail_hi=4), name="batch 2576 32 devices"),
        dict(_case("batch", "64dev", sets=64, fail_lo=1, fail_hi=8, cost=1), name="batch 64 64 devices int64"),
        dict(_case("batch", "256dev", sets=1024, fail_lo=1, fail_hi=16), name="batch 1024 256 devices"),
        # the same with identical searches shared, as the plan cache does
        dict(_case("batch", "256dev", sets=1000, fail_lo=1, fail_hi=16, sharing=True), name="shared batch 1000 256 devices"),
        # the second execution order
        dict(_case("batch", "32dev", sets=515, fail_lo=1, fail_hi=4, order=1), name="batch 515 32 devices all-forward"),
        # transition time in the objective: shortlist, migrations, synchronisation rounds
        dict(_case("objective", "256dev", sets=64, fail_lo=1, fail_hi=8, rounds=1), name="objective 64 256 devices"),
        # cost and feasibility of many single candidates, by index
        dict(_case("evaluate", "256dev", fail_lo=3, fail_hi=3, count=200_000, indexed=True), name="evaluate 200000 256 devices"),
    ]


def _log_uniform(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["one", "one", "select", "batch", "batch", "batch", "objective", "evaluate"])
    job = rng.choice(list(JOBS))
    if kind == "evaluate" and job == "64dev":   # (next to none of its candidates fits in memory: nothing to look at)
        job = "256dev"
    base = JOBS[job]["micro"]
    micro = rng.randint(base - 2, base + 1) if job == "8dev" else rng.randint(int(base * 0.7), int(base * 1.2))
    order = 1 if job != "64dev" and kind in ("one", "batch") and rng.random() < 0.2 else 0   # (a 64-device job stashes too much for it)
    hi = rng.randint(1, MOST_FAILED[job])
    lo = rng.randint(1, hi) if kind in ("batch", "objective") else hi
    cost = 1 if rng.random() < 0.4 else 0
    sets, count, rounds, sharing, indexed = 1, 0, 0, False, False
    if kind == "batch":
        sets = _log_uniform(rng, 2, MOST_SETS[job] // (3 if order else 1))
        sharing = rng.random() < 0.3
    elif kind == "objective":
        sets = _log_uniform(rng, 1, MOST_SETS[job] // 3)
        rounds = rng.randint(0, 1)
    elif kind == "evaluate":
        count = _log_uniform(rng, 1000, 300_000)
        indexed = job == "256dev" or rng.random() < 0.5
    return _case(kind, job, sets, lo, hi, micro, cost, order, sharing, rounds, count, indexed)


def _profile(case, rng):
    j = JOBS[case["job"]]
    L, pp = j["L"], j["pp"]
    if case["job"] == "8dev":
        fwd = rng.uniform(1e6, 3e6, L)
        bwd = 2.0 * fwd * rng.uniform(0.9, 1.1, L)
    else:
        fwd = 10e6 * (1.0 + 0.05 * np.clip(rng.standard_normal(L), -6, 6))
        if case["job"] == "64dev":   # embedding and head weigh twice a layer
            fwd[0] *= 2.0
            fwd[-1] *= 2.0
        bwd = 2.0 * fwd
    per, extra = divmod(L, pp)
    cuts = np.concatenate([[0], np.cumsum([per + (1 if s >= pp - extra else 0) for s in range(pp)])])
    return workloads.make_profile_ns(L, j["dp"], pp, case["micro"], fwd, bwd, j["act"], j["par"], 6 * j["par"], j["p2p"], cuts,
                                     j["cap"], 8, j["intra"], j["inter"])


@dataclass
class Session:
    """A context with a loaded profile, as a planner process keeps it, and one pass's inputs."""
    case: dict
    ctx: object
    opts: object
    failed: list
    packed: object = None
    objective: object = None
    space: object = None
    out: dict = field(default_factory=dict)

    def __del__(self):
        try:
            if self.space is not None:
                binding.cm_space_free(self.space)
            binding.cm_destroy(self.ctx)
        except Exception:   # interpreter shutdown
            pass


def _failure_set(case, rng):
    n = JOBS[case["job"]]["dp"] * JOBS[case["job"]]["pp"]
    k = int(rng.integers(case["fail_lo"], case["fail_hi"] + 1))
    if k == 8 and case["kind"] == "one":   # a whole node
        first = 8 * int(rng.integers(0, n // 8))
        return list(range(first, first + 8))
    return [int(d) for d in np.sort(rng.choice(n, k, replace=False))]


def prepare(case, seed):
    rng = np.random.default_rng([seed & 0x7FFFFFFF, 2508])
    j = JOBS[case["job"]]
    profile = _profile(case, rng)
    opts = workloads.SearchOptions(*j["window"], j["layers"], j["batch"], j["kappa"], case["cost"], case["order"])
    failed = [_failure_set(case, rng) for _ in range(case["sets"])]
    ctx = binding.cm_create(0)
    s = Session(case, ctx, opts, failed)
    binding.cm_load_profile(ctx, profile)
    binding.cm_set_sharing(ctx, case["sharing"])
    if case["kind"] == "one":
        # a program that waits for failures searches some set of the size it expects beforehand
        s.packed = binding.PackedScenarios(failed)
        warm = binding.PackedScenarios([_failure_set(case, rng)])
        for _ in range(3):
            warm.search(ctx, opts, latency=True)
    elif case["kind"] in ("batch", "objective"):
        s.packed = binding.PackedScenarios(failed)
        s.objective = workloads.ObjectiveOptions(sync_rounds=case["rounds"])
    elif case["kind"] == "evaluate":
        s.space, n = binding.cm_enumerate(ctx, binding.CM_DYNPAR, failed[0], opts)
        count = case["count"]
        s.out = {"first": 0, "idx": None}
        if case["indexed"] or count > n:
            s.out["idx"] = torch.from_numpy(np.sort(rng.integers(0, n, count)).astype(np.int64)).cuda()
        else:
            s.out["first"] = int(rng.integers(0, n - count + 1))
        s.out["cost"] = torch.empty(count, dtype=torch.int64 if case["cost"] else torch.float64, device="cuda")
        s.out["feasible"] = torch.empty(count, dtype=torch.uint8, device="cuda")
    return s


def _numbers(array, dtype, skip=()):
    a = np.frombuffer(array, dtype=dtype)
    return {k: a[k] for k in dtype.names if k not in skip}


def _padded(rows, n, width):
    out = np.full((n, width), -1, dtype=np.int64)
    for i, row in enumerate(rows):
        out[i, :len(row)] = row
    return out


def run(state):
    case, ctx, opts = state.case, state.ctx, state.opts
    kind = case["kind"]
    if kind == "one":
        state.packed.search(ctx, opts, latency=True)
        return _numbers(state.packed.best, PLAN), _numbers(state.packed.per_policy, PLAN)
    if kind == "batch":
        state.packed.search(ctx, opts)
        return _numbers(state.packed.best, PLAN), _numbers(state.packed.per_policy, PLAN)
    if kind == "objective":
        best, trans, short, moved, rounds = state.packed.search_objective(ctx, opts, state.objective, shortlist=True)
        return (_numbers(best, PLAN), _numbers(trans, TRANS, skip=("assign",)), _numbers(short, PLAN), moved, rounds)
    if kind == "select":
        spaces = [binding.cm_enumerate(ctx, policy, state.failed[0], opts)
                  for policy in (binding.CM_REROUTE, binding.CM_REDUNDANT, binding.CM_DYNPAR)]
        plan = binding.cm_select(ctx, [h for h, _ in spaces])
        only_dyn = binding.cm_select(ctx, [spaces[2][0]])
        cuts = binding.cm_decode_plan(ctx, spaces[2][0], only_dyn) if only_dyn else []
        for h, _ in spaces:
            binding.cm_space_free(h)
        found = [p for p in (plan, only_dyn) if p]
        return ([n for _, n in spaces], np.array([p.cost for p in found]),
                np.array([(p.policy, p.cost_ns, p.strategy, p.split_rank, p.n_pipes) for p in found]),
                _padded([v for p in found for v in (p.stages, p.micro, p.kappa)], 6, 16),
                _padded(cuts, 16, 65))
    o = state.out
    cost_kw = {"cost_ns_dev": o["cost"]} if case["cost"] else {"cost_dev": o["cost"]}
    binding.cm_evaluate(ctx, state.space, o["first"], case["count"], idx_dev=o["idx"], feasible_dev=o["feasible"], **cost_kw)
    return o["cost"], o["feasible"]


def work(case):
    """What a pass cannot do without: failure sets and profile in, plans out, and -- however the
    candidates are narrowed down -- the recurrence of one plan of every policy per failure set
    (3 operations for each forward and backward of every stage and micro-batch); for single
    candidates their indices and results and the sums of their stages."""
    j = JOBS[case["job"]]
    profile = 8 * 8 * j["L"]
    devices, sets = j["dp"] * j["pp"], case["sets"]
    if case["kind"] == "evaluate":
        n = case["count"]
        return {"bytes": profile + n * (8 + 1 + (8 if case["indexed"] else 0)), "flops": 8.0 * n * j["pp"]}
    plans = sets * 4 + (sets * 9 if case["kind"] == "objective" else 0)
    return {"bytes": profile + sets * 4.0 * (1 + case["fail_hi"]) + plans * PLAN_BYTES, "flops": sets * 3 * 6.0 * devices * case["micro"]}


def tolerance(case):
    """Plans, flags, bytes and integer nanoseconds are whole numbers and stay as they are; fp64
    costs are sums and maxima of doubles along paths of at most a few hundred terms (another
    order of the additions moves them by about 1e-14), stated to the 1e-12 that the oracle's
    comparison asks for."""
    return "exact" if case["cost"] and case["kind"] != "objective" else {"rel": 1e-12}
