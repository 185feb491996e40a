"""The staged evaluation's limits: no memory for its scratch (what then runs instead), more predicates
than a round takes, more distinct values than a chunk takes.  The limits are set small, so that
the sizes need not follow the defaults, and each test asserts that it met the limit; one case
meets the default chunk.  Shares are integers: equal bit for bit."""
import numpy as np
import pytest

import oracle
import workload as W
from tests._helpers import PRF, alloc_outs, from_dev, load_tables, oracle_group, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2209_03526_gb300")

AND, XOR, OR = P.COMBINE_AND, P.COMBINE_XOR, P.COMBINE_OR


@pytest.fixture()
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = P.Context(0, prf_keys=PRF)
    yield c
    c.close()


def _workload(n, bits, n1=9001, seed=3):
    """a uniform and a skewed column of one table, one column of another; six predicates in three groups"""
    g = W.rng(seed + n + bits)
    v0 = np.stack([W.uniform_attrs(g, 1, n, bits)[0], W.zipf_attrs(g, 1, n, 1.2, bits)[0]])
    wl = {"tables": [W.table(v0, bits, g), W.table(W.uniform_attrs(g, 1, n1, bits), bits, g)]}
    top = (1 << bits) - 1
    wl["preds"] = [W.range_pred(0, 0, 0, top // 5, top // 2), W.eq_pred(0, 1, 0, int(v0[1, 7]), combine=OR),
                   W.range_pred(0, 1, 0, 0, 3, combine=XOR), W.eq_pred(0, 0, 1, int(v0[0, n - 1])),
                   W.range_pred(1, 0, 2, 0, top - 1), W.range_pred(0, 0, 0, 9, top, combine=OR)]
    return wl


def _stack(outs):
    torch.cuda.synchronize()
    return [np.stack([from_dev(t) for t in grp]) for grp in outs]


def _run(ctx, wl, toks, qid=5, plan=False):
    outs = alloc_outs(wl)
    if not plan:
        before = ctx.launch_count()
        ctx.filter_and_combine(qid, toks, outs)
        ctx.sync()
        return _stack(outs), ctx.launch_count() - before
    p = ctx.plan_create([qid], [toks], [outs])
    d = ctx.plan_describe(p)
    for _ in range(2):
        ctx.plan_launch(p)
    ctx.sync()
    ctx.plan_destroy(p)
    return _stack(outs), d


def _check(wl, toks, got, qid=5):
    for grp in range(3):
        t = next(p["table"] for p in wl["preds"] if p["group"] == grp)
        vals = wl["tables"][t]["values"]
        n = vals.shape[1]
        assert np.array_equal(oracle.reconstruct(got[grp]), oracle.plain_group(wl["preds"], grp, vals)), grp
        idx = np.unique(np.concatenate([[0, 1023, 1024, n - 1], W.rng(n).integers(0, n, 24)]))
        assert np.array_equal(got[grp][:, idx], oracle_group(oracle, wl, toks, qid, grp, idx, threads=16)), grp


@pytest.mark.parametrize("n,bits", [(60001, 32), (60001, 16), (12000, 16)])
def test_no_scratch_runs_the_fused_kernels(ctx, n, bits):
    """Above and below the walk-parallel switch-over, sorted and dense columns; calls and plans."""
    wl = _workload(n, bits, n1=min(9001, n // 4))
    load_tables(ctx, wl)
    toks = P.keygen(wl["preds"], bits, bytes(range(16)))
    want, launches = _run(ctx, wl, toks)
    assert launches > 3
    _check(wl, toks, want)
    ctx.test_staged_limits(scratch_bytes=0)
    got, launches = _run(ctx, wl, toks)
    assert launches == 1
    planned, d = _run(ctx, wl, toks, plan=True)
    assert not d["staged"] and d["launches"] == 1 and d["scratch"] == 0
    for a, b, c in zip(want, got, planned):
        assert np.array_equal(a, b) and np.array_equal(a, c)
    ctx.test_staged_limits()
    again, launches = _run(ctx, wl, toks)
    assert launches > 3 and all(np.array_equal(a, b) for a, b in zip(want, again))


@pytest.mark.parametrize("kind,keys,points,bits", [(P.KEY_DCF, 9, 40001, 32), (P.KEY_DPF, 70, 20000, 9)])
def test_no_scratch_evaluates_per_item(ctx, kind, keys, points, bits):
    g = np.random.default_rng(points)
    draw = lambda n, top: g.integers(0, top, n, dtype=np.uint64).astype(np.uint32)  # noqa: E731
    L = 28 + (24 if kind == P.KEY_DCF else 20) * bits
    pairs = (keys + 1) // 2
    wire = torch.zeros(2 * pairs * L, dtype=torch.uint8, device="cuda")
    ctx.keygen_device(kind, bits, to_dev(draw(pairs, 1 << bits)), to_dev(draw(pairs, 1 << 32)), bytes(16), wire)
    pts = to_dev(draw(points, 1 << 32))
    got = []
    for scratch in ((1 << 64) - 1, 0):
        ctx.test_staged_limits(scratch_bytes=scratch)
        out = torch.full((keys * points,), -1, dtype=torch.int32, device="cuda")
        before = ctx.launch_count()
        ctx.eval_device_keys(kind, bits, wire, keys, pts, out, all_pairs=True)
        ctx.sync()
        got.append((from_dev(out), ctx.launch_count() - before))
    assert got[0][1] > 2 and got[1][1] == 2          # the keys' repacking and one evaluation
    assert np.array_equal(got[0][0], got[1][0])


def _fresh(ctx, wl, bits, sizes, toks, n_groups=3):
    ng = [next(p["table"] for p in wl["preds"] if p["group"] == g) for g in range(n_groups)]
    outs = [[torch.full((sizes[t],), -1, dtype=torch.int32, device="cuda") for _ in range(3)] for t in ng]
    before = ctx.launch_count()
    ctx.filter_fresh(4, toks, outs)
    ctx.sync()
    return _stack(outs), ctx.launch_count() - before


@pytest.mark.parametrize("n,bits", [(2000, 16), (1, 5), (1027, 32)])
def test_fresh_keys_without_scratch_and_in_rounds(ctx, n, bits):
    """filter_fresh: one thread per element where its sums find no room, and rounds of one predicate
    that hand a group's result on."""
    wl = _workload(n, bits, n1=max(1, n // 3)) if n > 7 else _workload(8, bits, n1=3)
    sizes = [t["values"].shape[1] for t in wl["tables"]]
    load_tables(ctx, wl)
    size = P.fresh_token_size(wl["preds"], bits, sizes)
    toks = [torch.zeros(size, dtype=torch.uint8, device="cuda") for _ in range(3)]
    ctx.keygen_fresh(wl["preds"], bits, sizes, bytes(range(5, 21)), toks)
    want, launches = _fresh(ctx, wl, bits, sizes, toks)
    assert launches == 2
    for grp in range(3):
        t = next(p["table"] for p in wl["preds"] if p["group"] == grp)
        vals = wl["tables"][t]["values"]
        assert np.array_equal(oracle.reconstruct(want[grp]), oracle.plain_group(wl["preds"], grp, vals)), grp
    ctx.test_staged_limits(scratch_bytes=0)
    alone, launches = _fresh(ctx, wl, bits, sizes, toks)
    assert launches == 1
    ctx.test_staged_limits(round_bytes=256)
    rounds, launches = _fresh(ctx, wl, bits, sizes, toks)
    assert launches == (2 * 6 if n > 16 else launches) and launches >= 2
    for a, b, c in zip(want, alone, rounds):
        assert np.array_equal(a, b) and np.array_equal(a, c)


@pytest.mark.parametrize("n,bits", [(30011, 32), (50000, 16)])
def test_groups_cross_rounds(ctx, n, bits):
    """A round holds one or two predicates: a group's fold goes on from its outputs."""
    wl = _workload(n, bits)
    load_tables(ctx, wl)
    toks = P.keygen(wl["preds"], bits, bytes(range(3, 19)))
    want, d = _run(ctx, wl, toks, plan=True)
    assert d["staged"] and d["rounds"] == 1
    _check(wl, toks, want)
    for round_bytes, least in ((1, 6), (d["scratch"] // 4, 2)):
        ctx.test_staged_limits(round_bytes=round_bytes)
        got, d2 = _run(ctx, wl, toks, plan=True)
        assert d2["staged"] and least <= d2["rounds"] <= 6
        called, launches = _run(ctx, wl, toks)
        assert launches == d2["launches"]
        for a, b, c in zip(want, got, called):
            assert np.array_equal(a, b) and np.array_equal(a, c)


@pytest.mark.parametrize("n,bits,chunk", [(30011, 32, 1024), (30011, 32, 16384), (24576, 17, 8192), (50000, 16, 1024),
                                          (20001, 13, 4096)])
def test_several_chunks_of_values(ctx, n, bits, chunk):
    """Sorted columns (whole and ragged last chunks, a skewed column with fewer chunks than the other)
    and dense ones; also with a round per predicate."""
    wl = _workload(n, bits)
    load_tables(ctx, wl)
    toks = P.keygen(wl["preds"], bits, bytes(range(9, 25)))
    want, d = _run(ctx, wl, toks, plan=True)
    assert d["staged"] and d["chunks"] == 1
    for round_bytes in (0, 1):
        ctx.test_staged_limits(chunk_values=chunk, round_bytes=round_bytes)
        got, d2 = _run(ctx, wl, toks, plan=True)
        assert d2["chunks"] >= 2 and d2["launches"] > d["launches"]
        for a, b in zip(want, got):
            assert np.array_equal(a, b)
    _check(wl, toks, got)


@pytest.mark.parametrize("kind,keys,points,bits,chunk", [(P.KEY_DCF, 9, 40001, 32, 4096), (P.KEY_DPF, 70, 40000, 14, 1024)])
def test_raw_evaluation_in_chunks_and_rounds(ctx, kind, keys, points, bits, chunk):
    g = np.random.default_rng(points + 1)
    draw = lambda n, top: g.integers(0, top, n, dtype=np.uint64).astype(np.uint32)  # noqa: E731
    L = 28 + (24 if kind == P.KEY_DCF else 20) * bits
    pairs = (keys + 1) // 2
    wire = torch.zeros(2 * pairs * L, dtype=torch.uint8, device="cuda")
    ctx.keygen_device(kind, bits, to_dev(draw(pairs, 1 << bits)), to_dev(draw(pairs, 1 << 32)), bytes(16), wire)
    pts = to_dev(draw(points, 1 << 32))
    got = []
    for limits in ({}, {"chunk_values": chunk}, {"chunk_values": chunk, "round_bytes": 1 << 20}):
        ctx.test_staged_limits(**limits)
        out = torch.full((keys * points,), -1, dtype=torch.int32, device="cuda")
        before = ctx.launch_count()
        ctx.eval_device_keys(kind, bits, wire, keys, pts, out, all_pairs=True)
        ctx.sync()
        got.append((from_dev(out), ctx.launch_count() - before))
    assert got[0][1] < got[1][1] < got[2][1]
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][0], got[2][0])


def test_more_values_than_the_default_chunk(ctx):
    """2^22 + 100,003 uniform 32-bit values: two chunks of distinct ones."""
    n, g = (1 << 22) + 100003, W.rng(22)
    v = W.uniform_attrs(g, 1, n, 32)
    wl = {"tables": [W.table(v, 32, g)]}
    wl["preds"] = [W.range_pred(0, 0, 0, 1 << 20, 3 << 30), W.eq_pred(0, 0, 0, int(v[0, n // 2]), combine=XOR)]
    load_tables(ctx, wl)
    toks = P.keygen(wl["preds"], 32, bytes(range(1, 17)))
    got, d = _run(ctx, wl, toks, plan=True)
    assert d["staged"] and d["chunks"] == 2
    assert np.array_equal(oracle.reconstruct(got[0]), oracle.plain_group(wl["preds"], 0, v))
    order = np.argsort((v[0].astype(np.uint64)), kind="stable")
    idx = np.unique(np.concatenate([[0, n - 1], order[[0, -1]], order[(1 << 22) - 2050:(1 << 22) + 2050:41],
                                    g.integers(0, n, 64)]))
    assert np.array_equal(got[0][:, idx], oracle_group(oracle, wl, toks, 5, 0, idx, threads=16))
