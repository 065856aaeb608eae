"""The search by bounds where its work lists, its workspaces or the device memory run out -- against the CPU
oracle: plan tuples bit-exact, costs equal."""
import copy
import ctypes as C

import numpy as np
import pytest

from paper_2508_21613_b200 import workloads as W

from test_gpu_bounds import _slow_links, gpu  # noqa: F401

pytestmark = pytest.mark.gpu


def _same(got, want):
    assert got.key() == want.key() and got.cost == want.cost and got.cost_ns == want.cost_ns, (got, want)


def _fast_links(profile):
    """The same job over links that bounds decide: the work layout depends on sizes alone."""
    p = copy.copy(profile)
    p.bw_intra_Bpns, p.bw_inter_Bpns = 400, 25
    return p


@pytest.mark.parametrize("mode,native", [(0, False), (1, False), (1, True)])
def test_lists_that_fill_while_other_blocks_look(gpu, oracle_factory, mode, native):
    """Every block of the compare pass asks whether the lists are full while others fill them: a few sets, whose
    layout is small enough for a block per part, and a batch whose parts are listed (two launches more)."""
    profile, opts = _slow_links(True, 8_000_000, 1)
    opts = W.SearchOptions(2, 2, 19, 20, opts.layer_mode, opts.batch_mode, opts.kappa_cap, mode)
    sets = [[3], [9]]
    orc = oracle_factory(profile, opts)
    want = [orc.search(f)[0] for f in sets]
    ctx = gpu.cm_create(0)
    try:
        launches = []
        for links in (_fast_links(profile), profile):
            gpu.cm_load_profile(ctx, links)
            gpu.cm_set_int64_arithmetic(ctx, native)
            for many in (sets * 4, sets * 200):
                best = gpu.plans_from_array(gpu.cm_search_batch(ctx, many, opts)[0])
                st = gpu.cm_last_stats(ctx)
                if links is not profile:
                    assert st["plans_run"] < st["plans_simulated"] and st["repeated"] == 0
                    launches.append(st["cost_kernel_launches"])
                    continue
                assert st["repeated"] == 1
                for b, plan in enumerate(best):
                    _same(plan, want[b % 2])
        assert launches[1] == launches[0] + 2
    finally:
        gpu.cm_destroy(ctx)


class _Hog:
    """Holds the device's memory but for `leave` bytes (below 1 GB) and what is left in pieces of less than 1 MB."""

    def __init__(self, leave):
        import torch
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.lib = C.CDLL("libcudart.so.12")
        self.lib.cudaMalloc.argtypes, self.lib.cudaFree.argtypes = [C.POINTER(C.c_void_p), C.c_size_t], [C.c_void_p]
        self.blocks = []
        for size in (1 << 30, 64 << 20, 2 << 20, 1 << 20):
            while len(self.blocks) < 4096:   # (183 GB: 183 + 16 + 32 and what is scattered)
                p = C.c_void_p()
                if self.lib.cudaMalloc(C.byref(p), size):
                    self.lib.cudaGetLastError()
                    break
                self.blocks.append(p)
        if leave:   # out of the first block, of 1 GB
            self.lib.cudaFree(self.blocks.pop(0))
            p = C.c_void_p()
            assert self.lib.cudaMalloc(C.byref(p), (1 << 30) - leave) == 0
            self.blocks.append(p)

    def __enter__(self):
        return self

    def __exit__(self, *_):
        for p in self.blocks:
            self.lib.cudaFree(p)


def _warm_up(gpu, profile, opts, sets):
    """Every kernel of the search by bounds and of the one that follows full lists, loaded while there is memory."""
    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, profile)
        gpu.cm_search_batch(ctx, sets * 20, opts)
        assert gpu.cm_last_stats(ctx)["repeated"] == 1
    finally:
        gpu.cm_destroy(ctx)


@pytest.mark.parametrize("leave,bounded", [(0, False), (4 << 20, None), (32 << 20, True)])
def test_workspaces_that_find_no_room(gpu, oracle_factory, leave, bounded):
    """A batch on a device that others have filled: all of the workspaces of the search by bounds find no room, all
    but one (if its 3 MB leave none for the other's), only the optional 57 MB of tiles' bounds.  The plans are the same, and a failure whose captured
    sequence was made before the workspaces moved still gets its own."""
    slow, opts = _slow_links(True, 8_000_000, 1)
    opts = W.SearchOptions(2, 2, 18, 21, opts.layer_mode, opts.batch_mode, opts.kappa_cap)
    only_minmax = W.SearchOptions(2, 2, 18, 21, opts.layer_mode, opts.batch_mode, 1)
    profile = _fast_links(slow)
    sets = [[3], [9]]
    orc = oracle_factory(profile, opts)
    want = [orc.search(f)[0] for f in sets]
    _warm_up(gpu, slow, opts, sets)
    ctx = gpu.cm_create(0)

    def search(many, **kw):
        for b, plan in enumerate(gpu.plans_from_array(gpu.cm_search_batch(ctx, many, opts, **kw)[0])):
            _same(plan, want[b % 2])
        return gpu.cm_last_stats(ctx)

    try:
        gpu.cm_load_profile(ctx, profile)
        for _ in range(3):   # (from the second on a replayed graph)
            st = search(sets, latency=True)
            assert st["plans_run"] < st["plans_simulated"]
        gpu.cm_search_batch(ctx, sets * 6500, only_minmax)   # the batch's own tables find their room here
        with _Hog(leave):
            st = search(sets * 6000)
            assert st["repeated"] == 0 and bounded in (None, st["plans_run"] < st["plans_simulated"])
        for _ in range(2):
            search(sets, latency=True)
        st = search(sets * 6000)
        assert st["plans_run"] < st["plans_simulated"]
    finally:
        gpu.cm_destroy(ctx)


def _many_sets(share):
    """Two pipelines of 20 and 21 stages over links about as slow as the stages: 10 k plans a set, so that the tables of
    tens of thousands of sets, and not their search, are what is large.  To be shared: small nodes and seven failures a
    set, which leave hardly two sets with the same boundaries."""
    L, pp, per_node = 44, 24 if share else 21, 2 if share else 8
    rng = np.random.default_rng(3)
    fwd = rng.uniform(5e6, 6e6, L).round()
    profile = W.make_profile_ns(L, 2, pp, 48, fwd, 2.0 * fwd, 1_000_000, 50_000_000, 300_000_000, 8_000_000,
                                [round(i * L / pp) for i in range(pp + 1)], 80_000_000_000, per_node, 1, 1)
    sets = [[b % (2 * pp)] if not share else sorted(rng.choice(2 * pp, 7, replace=False).tolist()) for b in range(60000)]
    return profile, W.SearchOptions(2, 2, 20, 21, W.LAYERS_REMAINDER, W.BATCH_REMAINDER, 1 << 16), sets


@pytest.mark.parametrize("share", [False, True])
def test_repeated_search_that_finds_no_room(gpu, oracle_factory, share):
    """A prepared batch whose lists are full and whose second set of tables, for the search of every plan, finds no
    room: an error that leaves the caller's arrays alone, and with room again the same batch can be searched."""
    profile, opts, sets = _many_sets(share)
    orc = oracle_factory(profile, opts)
    want = [orc.search(f)[0] for f in sets[:8]]
    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, profile)
        gpu.cm_set_sharing(ctx, share)
        gpu.cm_search_batch(ctx, sets[:600], opts)   # (loads the kernels)
        packed = gpu.PackedScenarios(sets)
        batch, _ = packed.prepare(ctx, opts)
        for array in (packed.best, packed.per_policy):
            C.memset(array, 0xa5, C.sizeof(array))
        with _Hog(0):
            for _ in range(2):
                with pytest.raises(gpu.ChameleonError) as e:
                    packed.search_prepared(ctx, batch)
                assert e.value.status == gpu.CM_ENOMEM
        for array in (packed.best, packed.per_policy):
            assert bytes(array) == b"\xa5" * C.sizeof(array)
        packed.search_prepared(ctx, batch)
        assert gpu.cm_last_stats(ctx)["repeated"] == 1
        for plan, w in zip(gpu.plans_from_array(packed.best), want):
            _same(plan, w)
        gpu.cm_batch_free(batch)
    finally:
        gpu.cm_destroy(ctx)


def _one_heavy_layer():
    """One layer takes nearly all of the time: a pipeline's is its micro-batches times that layer's, so that all
    strategies whose deepest pipeline is equally deep come out alike."""
    L, n_dp, n_pp = 14, 9, 7
    fwd = np.full(L, 1e3)
    fwd[5] = 5e7
    return W.make_profile_ns(L, n_dp, n_pp, 61, fwd, 2.0 * fwd, 1_000_000, 50_000_000, 300_000_000, 0,
                             [round(i * L / n_pp) for i in range(n_pp + 1)], 80_000_000_000, 4, 300, 20)


def _many_strategies():
    L, n_dp, n_pp = 32, 5, 8
    fwd = np.random.default_rng(11).uniform(2.5e6, 3.5e6, L).round()
    return W.make_profile_ns(L, n_dp, n_pp, 16, fwd, 2.0 * fwd, 1_000_000, 50_000_000, 300_000_000, 8_000_000,
                             [4 * i for i in range(9)], 80_000_000_000, 8, 300, 20)


@pytest.mark.parametrize("mode", [0, 1])
def test_more_strategies_within_reach_than_a_list_holds(gpu, oracle_factory, mode):
    """A scenario's strategies within reach are kept in a list of 14: here 15 and more have the same step time."""
    profile = _one_heavy_layer()
    opts = W.SearchOptions(10, 10, 2, 7, W.LAYERS_FULL, W.BATCH_REMAINDER, 1 << 14, mode)   # 61 survivors: 23 strategies
    sets = [[3, 4], [0, 17]]
    orc = oracle_factory(profile, opts)
    obj = W.ObjectiveOptions(topk=16)
    for f in sets:
        short = orc.search_objective(f, obj)[1].shortlist
        assert len({p.strategy for p in short}) > 14 and len({(p.cost, p.cost_ns) for p in short}) == 1
    want = [orc.search(f)[0] for f in sets]
    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, profile)
        best = gpu.plans_from_array(gpu.cm_search_batch(ctx, sets * 600, opts)[0])
        st = gpu.cm_last_stats(ctx)
        assert 0 < st["plans_run"] < st["plans_simulated"]
        for b, plan in enumerate(best):
            _same(plan, want[b % 2])
    finally:
        gpu.cm_destroy(ctx)


@pytest.mark.parametrize("topk", [1, 9])
def test_more_strategies_than_are_kept(gpu, oracle_factory, topk):
    """Step times from bounds of up to 2048 strategies are kept from the first look to the second."""
    profile = _many_strategies()
    opts = W.SearchOptions(4, 7, 2, 24, W.LAYERS_REMAINDER, W.BATCH_REMAINDER, 300)
    sets = [[3], [0, 17]]
    orc = oracle_factory(profile, opts)
    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, profile)
        if topk == 1:
            got = gpu.plans_from_array(gpu.cm_search_batch(ctx, sets * 300, opts)[0])
            want = [orc.search(f)[0] for f in sets]
        else:
            obj = W.ObjectiveOptions(topk=topk)
            got = gpu.plans_from_array(gpu.cm_search_objective(ctx, sets * 300, opts, obj, shortlist=True)[2])
            want = [p for f in sets for p in orc.search_objective(f, obj)[1].shortlist]
            assert len(want) == 2 * topk
        st = gpu.cm_last_stats(ctx)
        assert 0 < st["plans_run"] < st["plans_simulated"] and st["strategies"] > 2 * 2048   # (of two survivor counts)
        for b, plan in enumerate(got):
            _same(plan, want[b % len(want)])
    finally:
        gpu.cm_destroy(ctx)


@pytest.mark.parametrize("mode", [0, 1])
def test_shortlists_over_slow_links(gpu, oracle_factory, mode):
    """Results that come out later than their bounds: the strategies within reach of the bounds then hold too few step
    times for the shortlist, and all of them are looked at again."""
    profile, opts = _slow_links(True, 8_000_000, 3)
    opts = opts.with_cost_mode(mode)
    sets = [[3], [0, 9]]
    orc = oracle_factory(profile, opts)
    obj = W.ObjectiveOptions(topk=16)
    want = [orc.search_objective(f, obj) for f in sets]
    ctx = gpu.cm_create(0)
    try:
        gpu.cm_load_profile(ctx, profile)
        best, _, short, moved, _ = gpu.cm_search_objective(ctx, sets * 10, opts, obj, shortlist=True)
        st = gpu.cm_last_stats(ctx)
        assert 0 < st["plans_run"] < st["plans_simulated"]
        best, short = gpu.plans_from_array(best), gpu.plans_from_array(short)
        for b, plan in enumerate(best):
            _same(plan, want[b % 2][0])
            got = [short[16 * b + r] for r in range(16) if moved[b, r] >= 0]
            assert len(got) == len(want[b % 2][1].shortlist)
            for p, w in zip(got, want[b % 2][1].shortlist):
                _same(p, w)
    finally:
        gpu.cm_destroy(ctx)
