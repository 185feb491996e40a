"""The staged masked-mode evaluation (shared tree nodes) at the sizes where it can go wrong.

Large launches visit each tree node once instead of once per element: columns are sorted (or
dense, where the domain is about as small as the table), levels are cut into stages, and each
element looks its sums up.  Every element must reconstruct to the plaintext (Def. 2) and sampled
elements must equal the oracle share for share (integers: bit-exact).  The columns: uniform,
one value only, two values at both ends of the domain, consecutive values that wrap past 2^n
under the mask, skewed; sizes around the sort tile (4,096) and the run block (1,024), more
distinct values than one chunk holds (2^21), odd bit lengths, and groups of two tables.
"""
import numpy as np
import pytest

import oracle
import workload as W
from tests._helpers import PRF, alloc_outs, from_dev, load_tables, oracle_group

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2209_03526_gb300")

AND, XOR, OR = P.COMBINE_AND, P.COMBINE_XOR, P.COMBINE_OR


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = P.Context(0, prf_keys=PRF)
    yield c
    c.close()


def _column(kind, g, n, bits):
    top = 1 << bits
    if kind == "uniform":
        return W.uniform_attrs(g, 1, n, bits)[0]
    if kind == "one":
        return np.full(n, top // 3, dtype=np.uint32)
    if kind == "two_ends":
        return np.where(np.arange(n) % 2 == 0, 0, top - 1).astype(np.uint32)
    if kind == "consecutive":
        return (np.arange(n, dtype=np.uint64) % top).astype(np.uint32)
    return W.zipf_attrs(g, 1, n, 1.2, bits)[0]


def _check(ctx, wl, toks, qid, groups, launch):
    outs = alloc_outs(wl)
    launch(outs)
    torch.cuda.synchronize()
    ctx.sync()
    for grp, t in groups.items():
        vals = wl["tables"][t]["values"]
        n = vals.shape[1]
        got = np.stack([from_dev(x) for x in outs[grp]])
        assert np.array_equal(oracle.reconstruct(got), oracle.plain_group(wl["preds"], grp, vals)), grp
        fixed = [i for i in (0, 1, 31, 32, 1023, 1024, 4095, 4096, n // 2, n - 2, n - 1) if i < n]
        sample = np.unique(np.concatenate([fixed, W.rng(qid).integers(0, n, 64)]))
        assert np.array_equal(got[:, sample], oracle_group(oracle, wl, toks, qid, grp, sample, threads=16)), grp


@pytest.mark.parametrize("n,bits,kinds", [
    (40961, 32, ("uniform", "zipf")),            # ten sort tiles and one key
    (65536, 32, ("consecutive", "one")),
    (81919, 17, ("zipf", "uniform")),            # a tile short of a key; three sort passes, one of 1 bit
    (100003, 32, ("two_ends", "consecutive")),
    (50000, 16, ("uniform", "two_ends")),        # dense
    (60001, 1, ("two_ends", "one")),             # dense, one level
    (200001, 24, ("uniform", "consecutive")),
    ((1 << 21) + 4097, 32, ("uniform", "zipf")), # two chunks of distinct values
])
def test_columns_and_sizes(ctx, n, bits, kinds):
    g = W.rng(n + bits)
    vals = np.stack([_column(k, g, n, bits) for k in kinds])
    wl = {"tables": [W.table(vals, bits, g)]}
    top = (1 << bits) - 1
    mid = int(vals[0, n // 2])
    wl["preds"] = [W.eq_pred(0, 0, 0, mid), W.range_pred(0, 1, 0, top // 4, max(top // 4, top // 2), combine=XOR),
                   W.range_pred(0, 0, 0, 0, mid, combine=OR), W.eq_pred(0, 1, 0, int(vals[1, n - 1]), combine=XOR),
                   W.range_pred(0, 1, 1, max(0, top - 9), top)]
    load_tables(ctx, wl)
    toks = P.keygen(wl["preds"], bits, bytes(range(16)))
    _check(ctx, wl, toks, 5, {0: 0, 1: 0}, lambda outs: ctx.filter_and_combine(5, toks, outs))


def test_two_tables_in_rounds_plan_and_graph(ctx):
    """More predicates than one round's memory holds, over a sorted and a skewed table, launched
    as a plan twice and replayed from a CUDA graph; groups cross the rounds."""
    g = W.rng(77)
    n0, n1 = 600011, 150001
    wl = {"tables": [W.table(W.uniform_attrs(g, 3, n0, 32), 32, g), W.table(W.zipf_attrs(g, 2, n1, 1.2, 32), 32, g)]}
    v0 = wl["tables"][0]["values"]
    wl["preds"] = [W.range_pred(0, k % 3, 0, 1000 * k, (1 << 31) + 77 * k, combine=(AND, AND, OR, XOR)[k % 4]) for k in range(6)]
    wl["preds"] += [W.eq_pred(0, 0, 0, int(v0[0, 9]), combine=OR), W.range_pred(1, 0, 1, 0, 5),
                    W.eq_pred(1, 1, 1, 0, combine=OR), W.eq_pred(0, 2, 2, int(v0[2, n0 - 1]))]
    load_tables(ctx, wl)
    toks = P.keygen(wl["preds"], 32, bytes(range(3, 19)))
    groups = {0: 0, 1: 1, 2: 0}

    def twice_then_graph(outs):
        plan = ctx.plan_create([9], [toks], [outs])
        try:
            ctx.plan_launch(plan)
            ctx.plan_launch(plan)
            torch.cuda.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                ctx.plan_launch(plan, torch.cuda.current_stream())
            for grp in outs:
                for t in grp:
                    t.fill_(-1)
            graph.replay()
            torch.cuda.synchronize()
        finally:
            ctx.plan_destroy(plan)

    _check(ctx, wl, toks, 9, groups, twice_then_graph)


def test_two_streams_at_once(ctx):
    """Two launches on two streams share no scratch: both equal the call on its own."""
    g = W.rng(78)
    wl = {"tables": [W.table(W.uniform_attrs(g, 2, 120001, 32), 32, g)]}
    wl["preds"] = [W.range_pred(0, 0, 0, 5, 1 << 30), W.eq_pred(0, 1, 0, 7, combine=OR)]
    load_tables(ctx, wl)
    toks = P.keygen(wl["preds"], 32, bytes(16))
    want = [alloc_outs(wl) for _ in range(2)]
    for q in range(2):
        ctx.filter_and_combine(20 + q, toks, want[q])
    got = [alloc_outs(wl) for _ in range(2)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    for _ in range(3):
        for q, s in enumerate(streams):
            ctx.filter_and_combine(20 + q, toks, got[q], stream=s)
    torch.cuda.synchronize()
    for q in range(2):
        assert all(torch.equal(a, b) for a, b in zip(got[q][0], want[q][0]))


@pytest.mark.parametrize("dcf,keys,points,bits", [(False, 3, 200001, 32), (True, 70, 40001, 32), (True, 5, 50000, 9),
                                                  (False, 65, 100000, 17), (True, 2, 1, 32), (False, 129, 7, 4)])
def test_raw_evaluation_of_all_pairs(ctx, dcf, keys, points, bits):
    """Many keys at the same points: staged (sorted and dense points, more keys than a round
    takes) and, for the few points of the last two, the per-item kernel; keys read from the
    device and from the host; point bits above n are ignored."""
    g = np.random.default_rng(points)
    pairs = (keys + 1) // 2
    kind = P.KEY_DCF if dcf else P.KEY_DPF
    L = 28 + (24 if dcf else 20) * bits
    pts = g.integers(0, 1 << 32, points, dtype=np.uint64).astype(np.uint32)
    alpha = torch.from_numpy(g.integers(0, 1 << bits, pairs, dtype=np.uint64).astype(np.uint32).view(np.int32)).cuda()
    alpha[0] = int(pts[0].astype(np.uint64) & ((1 << bits) - 1)) - (1 << 32 if pts[0] >> 31 and bits == 32 else 0)
    beta = torch.arange(1, pairs + 1, dtype=torch.int32, device="cuda")
    wire = torch.zeros(2 * pairs * L, dtype=torch.uint8, device="cuda")
    ctx.keygen_device(kind, bits, alpha, beta, bytes(range(16)), wire)
    d_pts = torch.from_numpy(pts.view(np.int32)).cuda()
    out = torch.full((keys * points,), -1, dtype=torch.int32, device="cuda")
    ctx.eval_device_keys(kind, bits, wire, keys, d_pts, out, all_pairs=True)
    host = torch.full_like(out, -1)
    raw = bytes(wire.cpu().numpy().tobytes())[:keys * L]
    (ctx.eval_dcf_batch if dcf else ctx.eval_dpf_batch)(raw, keys, d_pts, host, all_pairs=True)
    torch.cuda.synchronize()
    ctx.sync()
    assert torch.equal(out, host)
    got = from_dev(out).reshape(keys, points)
    sample = np.unique(np.concatenate([[0, points - 1], g.integers(0, points, 32)]))
    x = pts[sample] & np.uint32((1 << bits) - 1)
    for k in {0, 1, keys // 2, keys - 1}:
        want = oracle.eval_many(raw[k * L:(k + 1) * L], x, oracle.KIND_DCF if dcf else oracle.KIND_DPF)
        assert np.array_equal(got[k, sample], want), k
    # a pair's two keys add up to beta [x == alpha] or beta [x < alpha] on every point
    full = pts.astype(np.uint64) & ((1 << bits) - 1)
    a0 = int(from_dev(alpha)[0])
    if keys >= 2:
        assert np.array_equal(got[0] + got[1], ((full < a0) if dcf else (full == a0)).astype(np.uint32))
