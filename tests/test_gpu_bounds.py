"""The bounded search pass (lower bounds decide most plans, the recurrence runs on the few they leave)
and the tie-break pass by bounds, at the sizes where they can go wrong, against the CPU oracle: plan
tuples bit-exact, costs equal."""
import itertools

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


def _small(seed, times=None, tight=False, n_micro=7, p2p=None):
    p = W.random_small(seed, L=13, n_dp=3, n_pp=4, n_micro=n_micro, tight_memory=tight).profile
    fwd = p.fwd_ns if times is None else times(13)
    return W.make_profile_ns(13, 3, 4, n_micro, fwd, 2.0 * np.asarray(fwd), p.act_bytes, p.param_bytes, p.opt_bytes,
                             p.p2p_bytes if p2p is None else p2p, p.base_cuts, p.mem_capacity_bytes, 4, 300, 20)


SETS = [list(c) for k in (1, 2) for c in itertools.combinations(range(12), k)]
CASES = {
    # transfer times that depend on the layer
    "layered-transfers": (_small(31), (1, 3, 2, 6, W.LAYERS_FULL, W.BATCH_REMAINDER), SETS[:20], 160),
    "tight-memory": (_small(33, tight=True), (1, 3, 2, 6, W.LAYERS_FULL, W.BATCH_REMAINDER), SETS[:20], 800),
    # transfer times equal on every boundary; identical layers (most plans tie); fewer micro-batches than stages
    "equal-transfers": (_small(34, p2p=30_000_000), (1, 3, 2, 7, W.LAYERS_FULL, W.BATCH_REMAINDER), SETS[:20], 160),
    "identical-layers": (_small(35, times=lambda n: np.full(n, 3e6), p2p=30_000_000), (1, 3, 2, 6, W.LAYERS_FULL, W.BATCH_REMAINDER), SETS[:20], 160),
    "few-micro-batches": (_small(36, n_micro=2), (1, 3, 2, 8, W.LAYERS_FULL, W.BATCH_REMAINDER), SETS[:20], 640),
}


def _heavy(layer, p2p):
    times = np.linspace(3e6, 3.6e6, 13)
    times[layer] *= 9
    return _small(37, times=lambda n: times, n_micro=20, p2p=p2p)


# a layer that outweighs a pipeline: at either end and inside, transfers equal and by layer
for _layer in (0, 6, 12):
    for _p2p in (None, 30_000_000):
        CASES[f"heavy-layer-{_layer}-{'equal' if _p2p else 'layered'}"] = (
            _heavy(_layer, _p2p), (1, 3, 2, 7, W.LAYERS_FULL, W.BATCH_REMAINDER), SETS[:12], 60)


@pytest.mark.parametrize("schedule", [W.SCHED_1F1B, W.SCHED_GPIPE])
@pytest.mark.parametrize("name", sorted(CASES))
def test_bounded_search_against_the_oracle(gpu, oracle_factory, name, schedule):
    """Each failure set many times over, so that the batch is large enough for bounds; in double,
    integer-valued double and 64-bit integer arithmetic."""
    profile, window, sets, copies = CASES[name]
    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, profile)
        for mode in (0, 1):
            opts = W.SearchOptions(*window, 1 << 62, mode, schedule)
            orc = oracle_factory(profile, opts)
            want = [orc.search(f)[0] for f in sets]
            for native in (False, True)[:1 + mode]:
                gpu.cm_set_int64_arithmetic(ctx, native)
                best, _, _ = gpu.cm_search_batch(ctx, sets * copies, opts)
                st = gpu.cm_last_stats(ctx)
                assert st["plans_run"] < st["plans_simulated"]      # bounds decided the rest
                for b, plan in enumerate(gpu.plans_from_array(best)):
                    w = want[b % len(sets)]
                    assert plan.feasible == (w is not None and w.feasible)
                    if w is not None and w.feasible:
                        assert plan.key() == w.key(), (sets[b % len(sets)], plan, w)
                        assert plan.cost == w.cost and plan.cost_ns == w.cost_ns
    finally:
        gpu.cm_destroy(ctx)


@pytest.mark.parametrize("mode", [0, 1])
def test_search_with_more_ties_than_the_list_holds(gpu, oracle_factory, mode):
    """One layer holds all the time, so every composition of a pipeline ties with a quarter of a million
    others.  (Too little work for bounds: every plan is evaluated at once.  Lists that do overflow:
    test_searches_whose_lists_overflow.)"""
    L = 24
    fwd = np.zeros(L)
    fwd[0] = 5e6
    profile = W.make_profile_ns(L, 2, 8, 4, fwd, 2.0 * fwd, 1_000_000, 50_000_000, 300_000_000, 0,
                                list(range(0, 25, 3)), 80_000_000_000, 4, 300, 20)
    opts = W.SearchOptions(2, 2, 7, 8, W.LAYERS_FULL, W.BATCH_REMAINDER, 1 << 62, mode)
    sets = [[0], [9]]
    orc = oracle_factory(profile, opts)
    want = [orc.search(f)[0] for f in sets]
    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, profile)
        best, _, _ = gpu.cm_search_batch(ctx, sets * 4, opts)
        st = gpu.cm_last_stats(ctx)
        assert st["plans_run"] == st["plans_simulated"] > 1 << 20   # the full search ran in the end
        for b, plan in enumerate(gpu.plans_from_array(best)):
            assert plan.key() == want[b % 2].key() and plan.cost == want[b % 2].cost and plan.cost_ns == want[b % 2].cost_ns
    finally:
        gpu.cm_destroy(ctx)


def test_bounded_shortlist_against_the_oracle(gpu, oracle_factory):
    """The full objective takes the k best step times: every one of them has to be exact, not the first alone."""
    profile, window, sets, copies = CASES["layered-transfers"]
    for mode, topk in ((0, 16), (1, 5)):
        opts = W.SearchOptions(*window, 1 << 62, mode)
        orc = oracle_factory(profile, opts)
        obj = W.ObjectiveOptions(topk=topk)
        want = [orc.search_objective(f, obj) for f in sets[:6]]
        ctx = gpu.cm_create(0)
        try:
            gpu.cm_load_profile(ctx, profile)
            many = sets[:6] * (copies * 2)
            best, trans, short, moved, _ = gpu.cm_search_objective(ctx, many, opts, obj, shortlist=True)
            st = gpu.cm_last_stats(ctx)
            assert st["plans_run"] < st["plans_simulated"]
            short = gpu.plans_from_array(short)
            best = gpu.plans_from_array(best)
            for b in range(len(many)):
                plan, tr = want[b % 6]
                assert best[b].key() == plan.key() and best[b].cost == plan.cost and best[b].cost_ns == plan.cost_ns
                got = [short[b * topk + r] for r in range(topk) if moved[b, r] >= 0]
                assert [p.key() for p in got] == [p.key() for p in tr.shortlist]
                assert [(p.cost, p.cost_ns) for p in got] == [(p.cost, p.cost_ns) for p in tr.shortlist]
        finally:
            gpu.cm_destroy(ctx)


@pytest.mark.parametrize("mode", [0, 1])
def test_bounded_search_of_shared_segments_against_the_oracle(gpu, oracle_factory, mode):
    """Segments that several failure sets have in common are searched once for all of them: each must come
    out exact for the set that needs it most.  Five nodes, sets with equal losses per node among them."""
    rng = np.random.default_rng(61)
    L, n_dp, n_pp = 40, 2, 20
    fwd = rng.uniform(2e6, 6e6, L).round()
    profile = W.make_profile_ns(L, n_dp, n_pp, 48, fwd, 2.0 * fwd, 1_000_000, 50_000_000, 300_000_000, 8_000_000,
                                list(range(0, L + 1, 2)), 80_000_000_000, 8, 300, 20)
    sets = [[3], [5], [12], [20], [27], [38], [0, 1], [2, 7], [0, 9], [8, 30], [39, 15], [17, 31], [1, 6, 33], [4, 35, 2]]
    opts = W.SearchOptions(2, 2, 17, 22, W.LAYERS_REMAINDER, W.BATCH_REMAINDER, 1 << 15, mode)
    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, profile)
        gpu.cm_set_sharing(ctx, True)
        best = gpu.plans_from_array(gpu.cm_search_batch(ctx, sets, opts)[0])
        st = gpu.cm_last_stats(ctx)
        assert st["plans_run"] < st["plans_simulated"], st
        orc = oracle_factory(profile, opts)
        for f, plan in zip(sets, best):
            want = orc.search(f)[0]
            assert plan.key() == want.key() and plan.cost == want.cost and plan.cost_ns == want.cost_ns, (f, plan, want)
    finally:
        gpu.cm_destroy(ctx)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("layer", [0, 13, 39])
def test_bounds_decide_where_one_stage_outweighs_the_others(gpu, oracle_factory, layer, mode):
    """A stage with a layer of twelve times the others is busy from its first forward to its last backward:
    its bound has to say so, or thousands of plans per pipeline are left to the recurrence."""
    rng = np.random.default_rng(71)
    L, n_dp, n_pp = 40, 2, 20
    fwd = rng.uniform(2.8e6, 3.2e6, L).round()
    fwd[layer] *= 12
    profile = W.make_profile_ns(L, n_dp, n_pp, 48, fwd, 2.0 * fwd, 1_000_000, 50_000_000, 300_000_000, 8_000_000,
                                list(range(0, L + 1, 2)), 80_000_000_000, 8, 300, 20)
    sets = [[3], [5], [20], [0, 9], [8, 30]]
    opts = W.SearchOptions(2, 2, 17, 22, W.LAYERS_REMAINDER, W.BATCH_REMAINDER, 1 << 15, mode)
    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, profile)
        best = gpu.plans_from_array(gpu.cm_search_batch(ctx, sets * 12, opts)[0])
        st = gpu.cm_last_stats(ctx)
        assert 0 < st["plans_run"] < st["plans_simulated"] // 100, st
        orc = oracle_factory(profile, opts)
        for f, plan in zip(sets, best):
            want = orc.search(f)[0]
            assert plan.key() == want.key() and plan.cost == want.cost and plan.cost_ns == want.cost_ns, (f, plan, want)
    finally:
        gpu.cm_destroy(ctx)


def _slow_links(deep, p2p, bw):
    """Transfers about as long as the stages, on either link tier: the longest path changes between stages all
    the time and bounds leave a part of the plans open."""
    rng = np.random.default_rng(3 if deep else 1)
    if deep:
        L = 44
        fwd = rng.uniform(5e6, 6e6, L).round()
        profile = W.make_profile_ns(L, 2, 20, 48, fwd, 2.0 * fwd, 1_000_000, 50_000_000, 300_000_000, p2p,
                                    [0] + [round((i + 1) * L / 20) for i in range(20)], 80_000_000_000, 8, bw, bw)
        return profile, W.SearchOptions(2, 2, 17, 22, W.LAYERS_REMAINDER, W.BATCH_REMAINDER, 1 << 16)
    L = 32
    fwd = (10e6 * (1 + 0.05 * rng.standard_normal(L))).round()
    profile = W.make_profile_ns(L, 4, 8, 32, fwd, 2.0 * fwd, 16_777_216, 402_653_184, 2_415_919_104, p2p,
                                list(range(0, 33, 4)), 80_000_000_000, 8, bw, bw)
    return profile, W.SearchOptions(3, 5, 4, 12, W.LAYERS_REMAINDER, W.BATCH_REMAINDER, 1 << 16)


@pytest.mark.parametrize("mode,native", [(0, False), (1, False), (1, True)])
@pytest.mark.parametrize("deep,p2p,bw,copies", [(False, 50_000_000, 1, 0), (False, 16_777_216, 2, 40), (True, 8_000_000, 2, 0),
                                                (True, 8_000_000, 2, 12)])
def test_tie_break_that_bounds_do_not_decide(gpu, oracle_factory, deep, p2p, bw, copies, mode, native):
    """Pipelines that the tie-break leaves open after a few recurrences, a failure on its own (copies 0) and a
    batch, shallow and a launch per depth, and the shortlist's, which go on with a warp each."""
    profile, opts = _slow_links(deep, p2p, bw)
    opts = opts.with_cost_mode(mode)
    sets = [[3], [5, 9], [1, 2, 20]] if not deep else [[3], [0, 9]]
    orc = oracle_factory(profile, opts)
    want = [orc.search(f)[0] for f in sets]
    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, profile)
        gpu.cm_set_int64_arithmetic(ctx, native)
        n_open = 0
        for turn in range(3):   # (from the second on a failure on its own replays a graph)
            for f, w in zip(sets, want) if not copies else [(sets, want)]:
                got = gpu.plans_from_array(gpu.cm_search_batch(ctx, [f] if not copies else f * copies, opts, latency=not copies)[0])
                n_open += gpu.cm_last_stats(ctx)["ties_open"]
                for b, plan in enumerate(got):
                    x = w if not copies else w[b % len(sets)]
                    assert plan.key() == x.key() and plan.cost == x.cost and plan.cost_ns == x.cost_ns, (plan, x)
        assert n_open > 0
        space, _ = gpu.cm_enumerate(ctx, W.POLICY_DYNPAR, sets[0], opts)
        dyn, one = orc.search_policy(sets[0], W.POLICY_DYNPAR), gpu.cm_select(ctx, [space])
        assert one.key() == dyn.key() and (one.cost, one.cost_ns) == (dyn.cost, dyn.cost_ns)
        gpu.cm_space_free(space)
        if not native:
            obj = W.ObjectiveOptions(topk=4)
            best, _, short, moved, _ = gpu.cm_search_objective(ctx, sets[:1], opts, obj, shortlist=True)
            plan, tr = orc.search_objective(sets[0], obj)
            assert gpu.plans_from_array(best)[0].key() == plan.key()
            assert [p.key() for r, p in enumerate(gpu.plans_from_array(short)) if moved[0, r] >= 0] == [p.key() for p in tr.shortlist]
    finally:
        gpu.cm_destroy(ctx)


@pytest.mark.parametrize("mode", [0, 1])
def test_searches_whose_lists_overflow(gpu, oracle_factory, mode):
    """Bounds that leave more plans than the lists hold: the search is repeated without them, searches alike go
    without for a while (twice as long after every refusal), other searches are not held back, and a
    new profile starts afresh.  Plans are the same throughout."""
    profile, opts = _slow_links(True, 8_000_000, 1)
    opts = opts.with_cost_mode(mode)
    sets = [[3], [0, 9]]
    orc = oracle_factory(profile, opts)
    want = [orc.search(f)[0] for f in sets]

    def check(arr):
        for b, plan in enumerate(gpu.plans_from_array(arr)):
            w = want[b % 2]
            assert plan.key() == w.key() and plan.cost == w.cost and plan.cost_ns == w.cost_ns
        return gpu.cm_last_stats(ctx)

    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, profile)
        tried = []
        for call in range(1, 17):
            st = check(gpu.cm_search_batch(ctx, sets * 20, opts)[0])
            assert st["plans_run"] == st["plans_simulated"]
            if st["repeated"]:
                tried.append(call)
        assert tried == [1, 6, 15]
        # another size, then a failure on its own, resident: they find out for themselves
        assert check(gpu.cm_search_batch(ctx, sets * 4, opts)[0])["repeated"] == 1
        tried = [call for call in range(1, 15) if check(gpu.cm_search_batch(ctx, sets[:1], opts, latency=True)[0])["repeated"]]
        assert tried == [1, 5, 13]
        # spaces are made for one selection: the second one knows
        for repeated in (1, 0, 0):
            space, _ = gpu.cm_enumerate(ctx, W.POLICY_DYNPAR, sets[0], opts)
            plan = gpu.cm_select(ctx, [space])
            assert plan.cost == want[0].cost and plan.cost_ns == want[0].cost_ns and plan.kappa == want[0].kappa
            assert gpu.cm_last_stats(ctx)["repeated"] == repeated
            gpu.cm_space_free(space)
        # a prepared batch keeps to what it found out
        packed = gpu.PackedScenarios(sets * 20)
        batch, _ = packed.prepare(ctx, opts)
        for repeated in (1, 0, 0, 0, 0, 0):
            packed.search_prepared(ctx, batch)
            assert check(packed.best)["repeated"] == repeated
        gpu.cm_batch_free(batch)
        gpu.cm_load_profile(ctx, profile)
        assert check(gpu.cm_search_batch(ctx, sets * 20, opts)[0])["repeated"] == 1
    finally:
        gpu.cm_destroy(ctx)


def test_captured_evaluations_outlive_other_calls(gpu, oracle_factory):
    """cm_evaluate in a CUDA graph: spaces that need more of the workspace, and a selection that lays the
    space's own tables out again, must leave what the graph refers to in place."""
    import torch
    profile, opts = _slow_links(True, 8_000_000, 1)
    few = W.SearchOptions(2, 2, 19, 20, opts.layer_mode, opts.batch_mode, opts.kappa_cap)
    stream = torch.cuda.Stream()
    ctx = gpu.cm_create(0, stream.cuda_stream)
    try:
        gpu.cm_load_profile(ctx, profile)
        graphs = []
        for o in (few, opts):
            orc = oracle_factory(profile, o)
            space, n = gpu.cm_enumerate(ctx, W.POLICY_DYNPAR, [3], o)
            idx = np.sort(np.random.default_rng(5).integers(0, n, 20_000)).astype(np.int64)
            want, _, want_feas = orc.evaluate([3], idx=idx)
            dev = torch.from_numpy(idx).cuda()
            cost, feas = torch.zeros(len(idx), dtype=torch.float64, device="cuda"), torch.zeros(len(idx), dtype=torch.uint8, device="cuda")
            torch.cuda.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.stream(stream):
                gpu.cm_evaluate(ctx, space, 0, len(idx), dev, cost, None, feas)
            torch.cuda.synchronize()
            with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
                gpu.cm_evaluate(ctx, space, 0, len(idx), dev, cost, None, feas)
            graphs.append((graph, cost, feas, want, want_feas, space, dev))
        gpu.cm_select(ctx, [graphs[1][5]])
        assert gpu.cm_last_stats(ctx)["repeated"] == 1
        for graph, cost, feas, want, want_feas, _, _ in graphs:
            with torch.cuda.stream(stream):
                cost.zero_()
                feas.zero_()
                graph.replay()
            torch.cuda.synchronize()
            assert np.array_equal(feas.cpu().numpy(), want_feas) and np.array_equal(cost.cpu().numpy(), want)
        del graph, graphs
    finally:
        gpu.cm_destroy(ctx)


def test_feasible_lists_that_find_no_room(gpu):
    """A device whose memory others hold: compositions that cannot be listed are walked in full, with the
    same plans."""
    import torch
    rng = np.random.default_rng(9)
    L = 24
    fwd = rng.uniform(2e6, 4e6, L).round()
    profile = W.make_profile_ns(L, 2, 8, 16, fwd, 2.0 * fwd, 1_000_000_000, 50_000_000, 300_000_000, 8_000_000,
                                list(range(0, 25, 3)), 40_000_000_000, 4, 300, 20)
    opts = W.SearchOptions(2, 2, 7, 8, W.LAYERS_FULL, W.BATCH_FULL, 1 << 62)
    sets = [[0], [9]]
    plans = []
    for hog in (False, True):
        ctx = gpu.cm_create(0)
        held = None
        try:
            gpu.cm_load_profile(ctx, profile)
            gpu.cm_search_batch(ctx, sets, W.SearchOptions(2, 2, 7, 8, W.LAYERS_REMAINDER, W.BATCH_FULL, 1 << 62))
            if hog:   # (the lists take 215 MB)
                torch.cuda.empty_cache()
                held = torch.empty(torch.cuda.mem_get_info()[0] - (120 << 20), dtype=torch.uint8, device="cuda")
            plans.append(gpu.plans_from_array(gpu.cm_search_batch(ctx, sets, opts)[0]))
        finally:
            del held
            torch.cuda.empty_cache()
            gpu.cm_destroy(ctx)
    assert plans[0] == plans[1] and plans[0][0].feasible


@pytest.mark.parametrize("mode,native", [(0, False), (1, False), (1, True)])
@pytest.mark.parametrize("per_node", [1, 2, 3])
def test_bounds_of_pipelines_over_many_nodes(gpu, oracle_factory, per_node, mode, native):
    """Equal transfers, nodes of one to three devices: pipelines of 17 to 22 stages cross five to twenty-one
    node boundaries, on either side of the six that are kept in a list."""
    rng = np.random.default_rng(81)
    L = 40
    fwd = rng.uniform(2.5e6, 3.5e6, L).round()
    profile = W.make_profile_ns(L, 2, 20, 48, fwd, 2.0 * fwd, 1_000_000, 50_000_000, 300_000_000, 8_000_000,
                                list(range(0, L + 1, 2)), 80_000_000_000, per_node, 300, 12)
    sets = [[3], [20], [0, 9]]
    opts = W.SearchOptions(2, 2, 17, 22, W.LAYERS_REMAINDER, W.BATCH_REMAINDER, 1 << 15, mode)
    orc = oracle_factory(profile, opts)
    wants = [orc.search(f)[0] for f in sets]
    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, profile)
        gpu.cm_set_int64_arithmetic(ctx, native)
        best = gpu.plans_from_array(gpu.cm_search_batch(ctx, sets * 20, opts)[0])
        st = gpu.cm_last_stats(ctx)
        assert 0 < st["plans_run"] < st["plans_simulated"]
        for b, plan in enumerate(best):
            want = wants[b % 3]
            assert plan.key() == want.key() and plan.cost == want.cost and plan.cost_ns == want.cost_ns, (sets[b % 3], plan, want)
    finally:
        gpu.cm_destroy(ctx)


@pytest.mark.parametrize("mode,native", [(0, False), (1, False), (1, True)])
@pytest.mark.parametrize("per_node,layered", [(1, False), (1, True), (8, False), (8, True)])
def test_bounds_of_few_segments(gpu, oracle_factory, per_node, layered, mode, native):
    """Four to 33 segments to a block, over two or three dear boundaries and over sixteen and more: up to 32 segments
    over more than six boundaries the lanes take a composition each, else a segment each.  Groups of one, 22 and thousands of
    compositions."""
    rng = np.random.default_rng(83)
    L = 45
    fwd = rng.uniform(2.5e6, 3.5e6, L).round()
    p2p = 8_000_000 if not layered else rng.integers(4_000_000, 12_000_000, L)
    profile = W.make_profile_ns(L, 2, 20, 96, fwd, 2.0 * fwd, 1_000_000, 50_000_000, 300_000_000, p2p,
                                [round(i * L / 20) for i in range(21)], 80_000_000_000, per_node, 300, 20)
    opts = W.SearchOptions(2, 2, 17, 22, W.LAYERS_REMAINDER, W.BATCH_REMAINDER, 16000, mode)
    sets = [[3], [20]]
    orc = oracle_factory(profile, opts)
    wants = [orc.search(f)[0] for f in sets]
    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, profile)
        gpu.cm_set_int64_arithmetic(ctx, native)
        for n in (4, 7, 8, 9, 32, 33):
            best = gpu.plans_from_array(gpu.cm_search_batch(ctx, [sets[b % 2] for b in range(n)], opts)[0])
            st = gpu.cm_last_stats(ctx)
            assert 0 < st["plans_run"] < st["plans_simulated"]
            for b, plan in enumerate(best):
                want = wants[b % 2]
                assert plan.key() == want.key() and plan.cost == want.cost and plan.cost_ns == want.cost_ns, (n, sets[b % 2], plan, want)
    finally:
        gpu.cm_destroy(ctx)
