"""The search by bounds where its work lists, its workspaces or the device memory run out -- against the CPU
oracle: plan tuples bit-exact, costs equal."""
import copy

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
