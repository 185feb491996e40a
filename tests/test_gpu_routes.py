"""Which kernels a filter launch takes: what a caller asks for is what runs."""
import numpy as np
import pytest

import oracle
import workload as W
from tests._helpers import PRF, alloc_outs, from_dev, load_tables, oracle_group

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2209_03526_gb300")

ALWAYS = (1 << 64) - 1


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = P.Context(0, prf_keys=PRF)
    yield c
    c.close()


def _workload(n, bits=32, seed=5):
    g = W.rng(seed)
    wl = {"tables": [W.table(W.uniform_attrs(g, 2, n, bits), bits, g)]}
    v = wl["tables"][0]["values"]
    wl["preds"] = [W.eq_pred(0, 0, 0, int(v[0, n // 2])), W.range_pred(0, 1, 0, 5, (1 << bits) // 2, combine=P.COMBINE_OR),
                   W.range_pred(0, 0, 1, 9, (1 << bits) - 1)]
    return wl


def _shares(outs):
    return [np.stack([from_dev(t) for t in grp]) for grp in outs]


@pytest.mark.parametrize("setting", [0, ALWAYS])
@pytest.mark.parametrize("n", [1, 3333, 25000])
def test_a_caller_s_switch_over_is_followed(ctx, n, setting):
    """0: one thread per element for every batch, UINT64_MAX: walk-parallel; one launch either way,
    as a call and as a plan, and the shares of the library's own choice."""
    wl = _workload(n)
    load_tables(ctx, wl)
    toks = P.keygen(wl["preds"], 32, bytes(range(16)))
    own = alloc_outs(wl)
    ctx.filter_and_combine(7, toks, own)
    ctx.sync()
    prev = ctx.set_walk_parallel(setting)
    try:
        outs = alloc_outs(wl)
        before = ctx.launch_count()
        ctx.filter_and_combine(7, toks, outs)
        ctx.sync()
        assert ctx.launch_count() - before == 1
        planned = alloc_outs(wl)
        plan = ctx.plan_create([7], [toks], [planned])
        assert ctx.plan_describe(plan)["kernel"] == ("k_filter_wp" if setting else "k_filter")
        before = ctx.launch_count()
        ctx.plan_launch(plan)
        ctx.sync()
        assert ctx.launch_count() - before == 1
        ctx.plan_destroy(plan)
    finally:
        ctx.set_walk_parallel(prev)
    idx = np.unique([0, n // 2, n - 1])
    for grp, (a, b, c) in enumerate(zip(_shares(own), _shares(outs), _shares(planned))):
        assert np.array_equal(a, b) and np.array_equal(a, c), grp
        assert np.array_equal(a[:, idx], oracle_group(oracle, wl, toks, 7, grp, idx)), grp


def test_a_dense_column_is_weighed_by_what_it_costs(ctx):
    """Two equality predicates on 5,000 16-bit values: all 2^16 nodes of the last levels cost twice
    the walk-parallel kernel, though the sorted values alone, without their sort, would not."""
    n = 5000
    wl = {"tables": [W.table(W.uniform_attrs(W.rng(8), 2, n, 16), 16, W.rng(9))]}
    v = wl["tables"][0]["values"]
    wl["preds"] = [W.eq_pred(0, 0, 0, int(v[0, 1])), W.eq_pred(0, 1, 1, int(v[1, n - 1]))]
    load_tables(ctx, wl)
    toks = P.keygen(wl["preds"], 16, bytes(range(2, 18)))
    outs = alloc_outs(wl)
    before = ctx.launch_count()
    ctx.filter_and_combine(8, toks, outs)
    ctx.sync()
    assert ctx.launch_count() - before == 1
    for grp, got in enumerate(_shares(outs)):
        assert np.array_equal(got, oracle_group(oracle, wl, toks, 8, grp, np.arange(n))), grp


@pytest.mark.parametrize("sizes", [(2500, 2500), (2700, 2700), (3040, 1), (5200,), (9728,)])
def test_equality_groups_of_one_wave(ctx, sizes):
    """Groups of equality predicates alone, of more elements than 32 a CTA and at most 64: one wave of
    tiles, and the oracle's shares."""
    g = W.rng(sum(sizes))
    wl = {"tables": [W.table(W.uniform_attrs(g, 1, n, 24), 24, g) for n in sizes]}
    wl["preds"] = [W.eq_pred(t, 0, t, int(wl["tables"][t]["values"][0, -1])) for t in range(len(sizes))]
    load_tables(ctx, wl)
    toks = P.keygen(wl["preds"], 24, bytes(range(4, 20)))
    outs = alloc_outs(wl)
    plan = ctx.plan_create([9], [toks], [outs])
    shape = ctx.plan_describe(plan)
    before = ctx.launch_count()
    ctx.plan_launch(plan)
    ctx.sync()
    launches = ctx.launch_count() - before
    ctx.plan_destroy(plan)
    assert launches == 1 and shape["kernel"] == "k_filter_wp" and shape["items"] == shape["grid"]
    for grp, got in enumerate(_shares(outs)):
        assert np.array_equal(got, oracle_group(oracle, wl, toks, 9, grp, np.arange(sizes[grp]))), grp


def test_a_staged_plan_says_so(ctx):
    """What plan_describe reports of a staged plan and of a fused one is what a launch does."""
    for n, staged in ((60000, True), (1000, False)):
        wl = _workload(n)
        load_tables(ctx, wl)
        toks = P.keygen(wl["preds"], 32, bytes(16))
        plan = ctx.plan_create([3], [toks], [alloc_outs(wl)])
        d = ctx.plan_describe(plan)
        before = ctx.launch_count()
        ctx.plan_launch(plan)
        ctx.sync()
        assert ctx.launch_count() - before == d["launches"]
        ctx.plan_destroy(plan)
        assert d["staged"] == staged and (d["launches"] > 10) == staged and (d["rounds"] == 1) == staged
        # at least the columns' sorted keys, element numbers and ranks, twice and once, for two columns
        assert d["scratch"] >= 2 * 20 * n if staged else d["scratch"] == 0


def test_a_small_call_is_weighed_as_a_call(ctx):
    """An equality and a range on 3,200 12-bit values each: a staged call would allocate and upload for
    longer than the walk-parallel kernel runs."""
    n = 3200
    wl = {"tables": [W.table(W.uniform_attrs(W.rng(12), 2, n, 12), 12, W.rng(13))]}
    v = wl["tables"][0]["values"]
    wl["preds"] = [W.eq_pred(0, 0, 0, int(v[0, 0])), W.range_pred(0, 1, 1, 100, 2000)]
    load_tables(ctx, wl)
    toks = P.keygen(wl["preds"], 12, bytes(range(6, 22)))
    outs = alloc_outs(wl)
    before = ctx.launch_count()
    ctx.filter_and_combine(11, toks, outs)
    ctx.sync()
    assert ctx.launch_count() - before == 1
    for grp, got in enumerate(_shares(outs)):
        assert np.array_equal(got, oracle_group(oracle, wl, toks, 11, grp, np.arange(n))), grp
