"""Batches whose plans and pipelines are taken several to a warp, bounds where the dearer links are the other
ones, and plans that come home in two parts -- against the CPU oracle or the search of one failure at a
time: plan tuples bit-exact, costs equal."""
import numpy as np
import pytest

from paper_2508_21613_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    import torch
    from paper_2508_21613_b200 import binding, build
    build.build()
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device; there is no CPU path")
    return binding


def _job(L, pp, micro, seed=5, per_node=8, intra=300, inter=20, layered=False):
    rng = np.random.default_rng(seed)
    fwd = rng.uniform(2.5e6, 3.5e6, L).round()
    p2p = rng.integers(4_000_000, 12_000_000, L) if layered else 8_000_000
    cuts = [round(i * L / pp) for i in range(pp + 1)]
    return W.make_profile_ns(L, 2, pp, micro, fwd, 2.0 * fwd, 1_000_000, 50_000_000, 300_000_000, p2p, cuts,
                             80_000_000_000, per_node, intra, inter)


# depths on either side of 16 and 40 stages, where the pipelines that share a warp go from eight to three to two; odd and
# even ones side by side; fewer micro-batches than stages as well.  The last number: plans listed at least, in two lists; they
# begin to share warps beyond 7400 to a list
DEPTHS = {"15-16": (36, 16, 24, (2, 2, 15, 16), 0), "17-22": (44, 20, 48, (2, 2, 17, 22), 14801), "39-42": (84, 41, 48, (2, 2, 39, 42), 14801),
          "few-micro-batches": (40, 18, 12, (2, 2, 16, 20), 14801)}


@pytest.mark.parametrize("mode,native", [(0, False), (1, False), (1, True)])
@pytest.mark.parametrize("name", sorted(DEPTHS))
def test_batches_of_pipelines_that_share_warps(gpu, oracle_factory, name, mode, native):
    """5000 failure sets: more listed plans than warps, and more pipelines to complete."""
    L, pp, micro, window, listed = DEPTHS[name]
    profile = _job(L, pp, micro)
    opts = W.SearchOptions(*window, W.LAYERS_REMAINDER, W.BATCH_REMAINDER, 4000, mode)
    sets = [[3], [0, pp + 1], [5, 6, pp]]
    orc = oracle_factory(profile, opts)
    wants = [orc.search(f)[0] for f in sets]
    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, profile)
        gpu.cm_set_int64_arithmetic(ctx, native)
        best = gpu.plans_from_array(gpu.cm_search_batch(ctx, [sets[b % 3] for b in range(5000)], opts)[0])
        st = gpu.cm_last_stats(ctx)
        if listed:
            assert listed <= st["plans_run"] < st["plans_simulated"]
        for b, plan in enumerate(best):
            want = wants[b % 3]
            assert plan.key() == want.key() and plan.cost == want.cost and plan.cost_ns == want.cost_ns, (sets[b % 3], plan, want)
    finally:
        gpu.cm_destroy(ctx)


@pytest.mark.parametrize("mode,native", [(0, False), (1, False), (1, True)])
@pytest.mark.parametrize("n", [3255, 3256, 5000])
def test_tie_break_on_either_side_of_sharing_a_warp(gpu, oracle_factory, n, mode, native):
    """Two shallow pipelines a set: a warp each up to 6511 of them, eight to a warp from 6512 on."""
    profile = _job(36, 16, 24)
    opts = W.SearchOptions(2, 2, 13, 16, W.LAYERS_REMAINDER, W.BATCH_REMAINDER, 1 << 14, mode)
    sets = [[3], [0, 17], [5, 6, 16], [2, 9, 18, 30]]
    orc = oracle_factory(profile, opts)
    wants = [orc.search_policy(f, W.POLICY_DYNPAR) for f in sets]
    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, profile)
        gpu.cm_set_int64_arithmetic(ctx, native)
        _, pol, _ = gpu.cm_search_batch(ctx, [sets[b % 4] for b in range(n)], opts, per_policy=True)
        for b, plan in enumerate(gpu.plans_from_array(pol)[W.POLICY_DYNPAR::3]):
            want = wants[b % 4]
            assert plan.key() == want.key() and plan.cost == want.cost and plan.cost_ns == want.cost_ns, (sets[b % 4], plan, want)
    finally:
        gpu.cm_destroy(ctx)


@pytest.mark.parametrize("layered", [False, True])
@pytest.mark.parametrize("per_node", [3, 8])
def test_bounds_where_links_inside_nodes_are_the_dearer(gpu, oracle_factory, per_node, layered):
    profile = _job(36, 16, 24, per_node=per_node, intra=15, inter=200, layered=layered)
    opts = W.SearchOptions(2, 2, 13, 18, W.LAYERS_REMAINDER, W.BATCH_REMAINDER, 1 << 15)
    sets = [[3], [0, 17]]
    orc = oracle_factory(profile, opts)
    wants = [orc.search(f)[0] for f in sets]
    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, profile)
        best = gpu.plans_from_array(gpu.cm_search_batch(ctx, sets * 60, opts)[0])
        st = gpu.cm_last_stats(ctx)
        assert 0 < st["plans_run"] < st["plans_simulated"]
        for b, plan in enumerate(best):
            assert plan.key() == wants[b % 2].key() and plan.cost == wants[b % 2].cost, (sets[b % 2], plan, wants[b % 2])
    finally:
        gpu.cm_destroy(ctx)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("n", [54, 191, 192, 401])
def test_plans_of_a_batch_come_in_two_parts(gpu, n, mode):
    """From 192 on.  Sets that every policy survives, that rerouting does not (a stage lost in every pipeline), and that nothing
    does (no strategy for the survivors): the same plans as one failure at a time, with and without those per policy."""
    profile = _job(12, 4, 8, per_node=4)
    opts = W.SearchOptions(2, 2, 3, 4, W.LAYERS_REMAINDER, W.BATCH_REMAINDER, 1 << 15, mode)
    sets = ([[1], [1, 5], [0, 4], [0, 4, 1], [], [7]] * 67)[:n]
    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, profile)
        want, want_pol, _ = gpu.cm_search_batch(ctx, sets, opts, per_policy=True, latency=True)
        for per_policy in (True, False):
            best, pol, _ = gpu.cm_search_batch(ctx, sets, opts, per_policy=per_policy)
            assert bytes(best) == bytes(want)
            if per_policy:
                assert bytes(pol) == bytes(want_pol)
        feasible = [p.feasible for p in gpu.plans_from_array(want)]
        assert any(feasible) and not all(feasible)
    finally:
        gpu.cm_destroy(ctx)


def _pairs(n, dp_hi, lo, hi, G):
    """(stages, micro-batches) that occur among the strategies of n survivors: a group of the work layout each."""
    def parts(n, dp, least):
        if dp == 1:
            return [(n,)] if least <= n <= hi else []
        return [(s, *rest) for s in range(least, hi + 1) for rest in parts(n - s, dp - 1, s)]
    found = set()
    for t in (t for dp in range(1, dp_hi + 1) for t in parts(n, dp, lo)):
        m = [G * s // n for s in t]
        found |= {(s, b + k) for s, b in zip(t, m) for k in ((0, 1) if sum(m) < G else (0,))}
    return found


@pytest.mark.parametrize("failures,many", [(2, False), (12, True)])
def test_layouts_of_few_and_of_many_groups(gpu, oracle_factory, failures, many):
    """A block finds its group of segments by a thread per group, or by halving where there are more groups."""
    profile = _job(40, 20, 48, per_node=4)
    opts = W.SearchOptions(1, 2, 14, 26, W.LAYERS_REMAINDER, W.BATCH_REMAINDER, 1 << 15)
    sets = [list(range(0, 3 * k, 3)) for k in range(1, failures + 1)]
    groups = sum(len(_pairs(40 - k, 2, 14, 26, 96)) for k in range(1, failures + 1))
    assert (groups > 128) == many
    orc = oracle_factory(profile, opts)
    wants = [orc.search(f)[0] for f in sets]
    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, profile)
        best = gpu.plans_from_array(gpu.cm_search_batch(ctx, sets * 60, opts)[0])
        st = gpu.cm_last_stats(ctx)
        assert 0 < st["plans_run"] < st["plans_simulated"]
        for b, plan in enumerate(best):
            want = wants[b % failures]
            assert plan.key() == want.key() and plan.cost == want.cost, (sets[b % failures], plan, want)
    finally:
        gpu.cm_destroy(ctx)
