"""cm_evaluate's three ways through a space with deep pipelines (a warp per candidate, binned by depth,
rounds of the binned one), the best split of the full enumeration, and spaces that take over the
buffers of freed ones: at the sizes where they can go wrong, against the CPU oracle."""
import dataclasses

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


def _evaluate(gpu, ctx, space, idx):
    import torch
    dev = torch.tensor(np.asarray(idx, dtype=np.int64), device="cuda")
    cost = torch.zeros(len(idx), dtype=torch.float64, device="cuda")
    cost_ns = torch.zeros(len(idx), dtype=torch.int64, device="cuda")
    feas = torch.zeros(len(idx), dtype=torch.uint8, device="cuda")
    gpu.cm_evaluate(ctx, space, 0, len(idx), dev, cost, cost_ns, feas)
    torch.cuda.synchronize()
    return cost.cpu().numpy(), cost_ns.cpu().numpy(), feas.cpu().numpy()


# 8192 candidates are the most that take a warp each; 40 960 make two rounds of the binned form
@pytest.mark.parametrize("count", [1, 8192, 8193, 40960])
@pytest.mark.parametrize("schedule", [W.SCHED_1F1B, W.SCHED_GPIPE])
@pytest.mark.parametrize("mode,native", [(0, False), (1, False), (1, True)])
def test_evaluate_of_a_deep_space(gpu, oracle_factory, mode, native, schedule, count):
    """Depths 12 .. 61 (registers, a launch per depth, a warp each above 48) in one call, in an order that
    jumps between them, with the first and the last candidate of the space."""
    w = W.deep_pipeline()
    profile = dataclasses.replace(w.profile, mem_capacity_bytes=2_000_000_000)   # some of the plans do not fit
    opts = W.SearchOptions(1, 3, 12, 64, W.LAYERS_REMAINDER, W.BATCH_REMAINDER, 1 << 12, mode, schedule)
    failed = [3]
    orc = oracle_factory(profile, opts)
    n, _, n_seg = orc.count(failed)
    segs = [orc.segment(failed, s) for s in range(n_seg)]
    rng = np.random.default_rng(count)
    idx = np.array([g["first"] + rng.integers(0, max(1, g["K"])) for g in rng.choice(segs, size=count)])
    idx[0], idx[-1] = n - 1, 0
    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, profile)
        gpu.cm_set_int64_arithmetic(ctx, native)
        space, got_n = gpu.cm_enumerate(ctx, W.POLICY_DYNPAR, failed, opts)
        assert got_n == n
        cost, cost_ns, feas = _evaluate(gpu, ctx, space, idx)
        gpu.cm_space_free(space)
    finally:
        gpu.cm_destroy(ctx)
    want, want_ns, want_feas = orc.evaluate(failed, idx=idx)
    assert np.array_equal(feas, want_feas) and (count == 1 or 0 < want_feas.sum() < count)
    ok = want_feas.astype(bool)
    assert (cost_ns[ok] == want_ns[ok]).all() if mode else (cost[ok] == want[ok]).all()


@pytest.mark.parametrize("schedule", [W.SCHED_1F1B, W.SCHED_GPIPE])
@pytest.mark.parametrize("mode,native", [(0, False), (1, False), (1, True)])
def test_evaluate_of_pipelines_without_micro_batches(gpu, oracle_factory, mode, native, schedule):
    """More survivors than micro-batches: some shares are zero, one stage included, and a pipeline that is
    given no work is no plan, however well it fits.  Every candidate of the space, in one call."""
    p = W.random_small(41, L=8, n_dp=3, n_pp=2, n_micro=1).profile
    opts = W.SearchOptions(1, 5, 1, 5, W.LAYERS_FULL, W.BATCH_REMAINDER, 1 << 62, mode, schedule)
    for failed in ([], [0], [1, 4]):
        orc = oracle_factory(p, opts)
        n, _, n_seg = orc.count(failed)
        segs = [orc.segment(failed, s) for s in range(n_seg)]
        idle = np.concatenate([np.arange(g["first"], g["first"] + g["K"] + 1) for g in segs if g["m"] == 0] or [np.zeros(0, int)])
        assert len(idle) and any(g["S"] == 1 and g["m"] == 0 for g in segs)
        want, want_ns, want_feas = orc.evaluate(failed, idx=np.arange(n))
        assert not want_feas[idle].any() and want_feas.any()
        ctx = gpu.cm_create(0)
        try:
            gpu.cm_load_profile(ctx, p)
            gpu.cm_set_int64_arithmetic(ctx, native)
            space, got_n = gpu.cm_enumerate(ctx, W.POLICY_DYNPAR, failed, opts)
            assert got_n == n
            cost, cost_ns, feas = _evaluate(gpu, ctx, space, np.arange(n))
            gpu.cm_space_free(space)
        finally:
            gpu.cm_destroy(ctx)
        assert np.array_equal(feas, want_feas)
        assert np.array_equal(cost_ns, want_ns) if mode else np.array_equal(cost, want)


@pytest.mark.parametrize("n_micro", [1, 2, 7])
@pytest.mark.parametrize("batch_mode", [W.BATCH_FULL, W.BATCH_REMAINDER])
def test_best_split(gpu, oracle_factory, batch_mode, n_micro):
    """One to five pipelines, fewer micro-batches than pipelines included, compositions that do not fit."""
    for seed, tight in ((41, False), (42, True)):
        p = W.random_small(seed, L=8, n_dp=3, n_pp=2, n_micro=n_micro, tight_memory=tight).profile
        for mode in (0, 1):
            opts = W.SearchOptions(1, 5, 1, 5, W.LAYERS_FULL, batch_mode, 1 << 62, mode)
            orc = oracle_factory(p, opts)
            sets = [[], [0], [5], [0, 3], [1, 2], [0, 1, 2], [0, 2, 4, 5]]
            ctx = gpu.cm_create(0)
            try:
                gpu.cm_load_profile(ctx, p)
                best, _, _ = gpu.cm_search_batch(ctx, sets, opts)
                for f, got in zip(sets, gpu.plans_from_array(best)):
                    want = orc.search(f)[0]
                    assert got.feasible == (want is not None and want.feasible)
                    if got.feasible:
                        assert got.key() == want.key() and got.cost == want.cost and got.cost_ns == want.cost_ns
            finally:
                gpu.cm_destroy(ctx)


def _uneven(seed, n_dp, n_pp, n_micro, cap, act):
    """Transfers and stashes that differ between layers: with one more micro-batch memory forces the min-max
    partition elsewhere, at times to cheaper cuts."""
    rng = np.random.default_rng(seed)
    L = 12
    fwd = rng.uniform(1e6, 3e6, L).round()
    p2p = (rng.random(L) < 0.5) * 400_000_000 + 1_000_000
    return W.make_profile_ns(L, n_dp, n_pp, n_micro, fwd, 2 * fwd, (rng.uniform(0.1, 1, L) * act).astype(np.int64),
                             (rng.uniform(0.2, 1, L) * 1e8).astype(np.int64), 300_000_000, p2p,
                             [round(i * L / n_pp) for i in range(n_pp + 1)], int(cap), 4, 30, 20)


@pytest.mark.parametrize("seed,n_dp,n_pp,n_micro,cap,act", [(0, 3, 4, 6, 4e9, 5e8), (5, 3, 4, 6, 7e9, 1e9), (0, 2, 6, 40, 4e9, 5e8),
                                                            (5, 2, 6, 40, 5e9, 1e9), (1, 3, 4, 6, 3e9, 1e9)])
def test_best_split_where_costs_fall(gpu, oracle_factory, seed, n_dp, n_pp, n_micro, cap, act):
    """A pipeline's best cost can fall when it gets one more micro-batch; the least step time over all splits
    and the first split that has it have to be found all the same.  The last case fits nearly nowhere."""
    p = _uneven(seed, n_dp, n_pp, n_micro, cap, act)
    sets = [[0], [1, 7], [2, 3, 8]]
    for mode in (0, 1):
        opts = W.SearchOptions(1, 4, 2, 8, W.LAYERS_MINMAX, W.BATCH_FULL, 1 << 62, mode)
        orc = oracle_factory(p, opts)
        n, _, n_seg = orc.count(sets[0])
        value = orc.evaluate(sets[0], idx=np.arange(n))[mode]
        segs = [orc.segment(sets[0], s) for s in range(n_seg)]
        by = {(g["strategy"], g["pipe"], g["m"]): value[g["first"]] for g in segs}
        assert cap < 4e9 or any(v > by.get((s, q, m + 1), v) for (s, q, m), v in by.items())
        ctx = gpu.cm_create(0)
        try:
            gpu.cm_load_profile(ctx, p)
            best, _, _ = gpu.cm_search_batch(ctx, sets, opts)
            for f, got in zip(sets, gpu.plans_from_array(best)):
                want = orc.search(f)[0]
                assert got.feasible == (want is not None and want.feasible)
                if got.feasible:
                    assert got.key() == want.key() and got.cost == want.cost and got.cost_ns == want.cost_ns
        finally:
            gpu.cm_destroy(ctx)


@pytest.mark.parametrize("layer_mode", [W.LAYERS_REMAINDER, W.LAYERS_MINMAX])
@pytest.mark.parametrize("n_micro", [31, 32, 64])
def test_best_split_of_many_micro_batches(gpu, oracle_factory, n_micro, layer_mode):
    """62, 64 and 128 micro-batches over one to three pipelines."""
    p = W.random_small(43, L=8, n_dp=2, n_pp=4, n_micro=n_micro).profile
    for mode in (0, 1):
        opts = W.SearchOptions(1, 3, 1, 8, layer_mode, W.BATCH_FULL, 1 << 62, mode)
        orc = oracle_factory(p, opts)
        ctx = gpu.cm_create(0)
        try:
            gpu.cm_load_profile(ctx, p)
            sets = [[], [0], [0, 5], [1, 2, 3]]
            best, _, _ = gpu.cm_search_batch(ctx, sets, opts)
            for f, got in zip(sets, gpu.plans_from_array(best)):
                want = orc.search(f)[0]
                assert got.feasible == (want is not None and want.feasible)
                if got.feasible:
                    assert got.key() == want.key() and got.cost == want.cost and got.cost_ns == want.cost_ns
        finally:
            gpu.cm_destroy(ctx)


def test_spaces_that_take_over_buffers(gpu, oracle_factory):
    """Spaces of different sizes made, freed and made again while others live: what a freed one leaves
    behind must not reach the next, and a selection over several sees each of them."""
    w = W.random_small(51, L=9, n_dp=2, n_pp=3)
    opts = dataclasses.replace(w.options, cost_mode=1)
    orc = oracle_factory(w.profile, opts)
    sets = [[0], [0, 1, 2, 3], [5], [1, 4]]
    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, w.profile)
        live = []
        for turn in range(24):
            failed = sets[turn % len(sets)]
            policy = turn % 3
            want = orc.search(failed)[1][policy]
            space, n = gpu.cm_enumerate(ctx, policy, failed, opts)
            live.append((space, want))
            got = gpu.cm_select(ctx, [s for s, _ in live])
            keys = [(p.cost_ns, i) for i, (_, p) in enumerate(live) if p is not None and p.feasible]
            if not keys:
                assert got is None
            else:
                assert got.cost_ns == min(keys)[0]
            one = gpu.cm_select(ctx, [space])
            assert (one is None) == (not want.feasible)
            if one is not None:
                assert one.key() == want.key() and one.cost_ns == want.cost_ns
            if turn % 5 == 4:
                for s, _ in live[:3]:
                    gpu.cm_space_free(s)
                live = live[3:]
        for s, _ in live:
            gpu.cm_space_free(s)
    finally:
        gpu.cm_destroy(ctx)
