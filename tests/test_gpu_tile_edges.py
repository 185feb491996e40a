"""Kernels that pair lanes, share nodes or split words, at the sizes where that can go wrong, bit
for bit against the oracle."""
import numpy as np
import pytest

import oracle
import workload as W
from tests._helpers import PRF, from_dev, to_dev
from tests.test_gpu_keygen import SEED, _gen, _oracle_pair

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2209_03526_gb300")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = P.Context(0, prf_keys=PRF)
    yield c
    c.close()


@pytest.mark.parametrize("kind", [P.KEY_DPF, P.KEY_DCF])
@pytest.mark.parametrize("pairs", [1, 15, 16, 17, 33])
def test_keygen_warp_of_lane_pairs(ctx, kind, pairs):
    """A warp generates 16 key pairs: a single one, one short of a warp, whole, one more."""
    g = np.random.default_rng(pairs + 100 * kind)
    alpha = g.integers(0, 1 << 7, pairs, dtype=np.uint64).astype(np.uint32)
    beta = g.integers(0, 1 << 32, pairs, dtype=np.uint64).astype(np.uint32)
    keys, L = _gen(ctx, kind, 7, alpha, beta)
    raw = keys.cpu().numpy().tobytes()
    for i in range(pairs):
        k0, k1 = _oracle_pair(kind, 7, SEED, i, int(alpha[i]), int(beta[i]))
        assert raw[2 * i * L: (2 * i + 1) * L] == bytes(k0) and raw[(2 * i + 1) * L: (2 * i + 2) * L] == bytes(k1), i


@pytest.mark.parametrize("n", [1, 7, 8, 17, 65])
def test_fresh_tokens_warp_of_lane_pairs(ctx, n):
    g = W.rng(n)
    vals = W.uniform_attrs(g, 2, n, 6)
    preds = [W.eq_pred(0, 0, 0, int(vals[0, 0])), W.range_pred(0, 1, 0, 3, 40)]
    size = P.fresh_token_size(preds, 6, [n])
    toks = [torch.zeros(size, dtype=torch.uint8, device="cuda") for _ in range(3)]
    ctx.keygen_fresh(preds, 6, [n], SEED, toks)
    torch.cuda.synchronize()
    for got, want in zip(toks, oracle.keygen_fresh(preds, 6, [n], SEED)):
        assert got.cpu().numpy().tobytes() == want


@pytest.mark.parametrize("bits", [1, 3, 9, 32])
@pytest.mark.parametrize("tile", [1, 2, 31, 32, 33, 40])
def test_walk_parallel_shared_levels(ctx, bits, tile):
    """Tiles on both sides of a level of nodes, domains smaller than a tile (every level is shared)
    and ragged last tiles; a group of equality predicates, one of both kinds."""
    g = W.rng(bits * 64 + tile)
    n = 3 * tile + max(1, tile // 3)
    vals = W.uniform_attrs(g, 2, n, bits)
    tab = W.table(vals, bits, g)
    ctx.load_shares(0, [to_dev(s) for s in tab["shares"]], bits)
    top = (1 << bits) - 1
    preds = [W.eq_pred(0, 0, 0, int(vals[0, 0])), W.range_pred(0, 1, 1, top // 3, top),
             W.eq_pred(0, 0, 1, int(vals[0, -1]), W.COMBINE_OR), W.eq_pred(0, 1, 0, int(vals[1, 0]))]
    toks = P.keygen(preds, bits, bytes(range(3, 19)))
    prev, prev_tile = ctx.set_walk_parallel((1 << 64) - 1), ctx.set_walk_parallel_tile(tile)
    try:
        outs = [[torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(3)] for _ in range(2)]
        ctx.filter_and_combine(9, toks, outs)
        ctx.sync()
    finally:
        ctx.set_walk_parallel(prev)
        ctx.set_walk_parallel_tile(prev_tile)
    for grp in range(2):
        got = np.stack([from_dev(t) for t in outs[grp]])
        assert np.array_equal(got, oracle.filter_group(toks, 9, PRF, [(tab["shares"], bits)], grp, np.arange(n), threads=4))


@pytest.mark.parametrize("n,n_elems,n_preds", [(12, 1, 1), (13, 16, 2), (14, 17, 5), (15, 48, 3), (16, 331, 4)])
def test_onehot_halves_of_words(ctx, n, n_elems, n_preds):
    """Every width of the staged dot pass, CTAs with one half of an output word, tables that end
    inside either half."""
    g = W.rng(n)
    vals = W.uniform_attrs(g, 1, n_elems, n)
    tab = W.onehot_table(vals, n, g)
    ctx.load_onehot(0, [to_dev(s) for s in tab["shares"]], n)
    preds = [W.eq_pred(0, 0, p, int(vals[0, p % n_elems])) for p in range(n_preds)]
    toks = P.keygen_onehot(preds, n, bytes([n]) * 16)
    outs = [[torch.full(((n_elems + 31) // 32,), -1, dtype=torch.int32, device="cuda") for _ in range(3)] for _ in preds]
    ctx.filter_onehot(3, toks, outs)
    ctx.sync()
    for grp in (0, n_preds - 1):
        words = np.stack([from_dev(t) for t in outs[grp]])
        got = ((words[:, :, None] >> np.arange(32, dtype=np.uint32)) & 1).reshape(3, -1)
        idx = np.arange(n_elems) if n < 15 else np.unique([0, n_elems // 2, n_elems - 1])
        assert np.array_equal(got[:, idx], oracle.filter_onehot(toks, 3, PRF, [(tab["shares"], n)], grp, idx))
        assert np.array_equal(oracle.reconstruct_bits(got[:, :n_elems]), oracle.plain_group([preds[grp]], grp, vals))
        assert not got[:, n_elems:].any()


@pytest.mark.parametrize("n,attrs", [(1, []), (33, [0]), (1025, [1, 0]), (2048, [2, 1, 0]), (515, [0, 1, 2, 0, 1, 2, 0])])
def test_fetch_multi_record_widths(ctx, n, attrs):
    """Records of 2, 3, 4, 5 and 9 words (part of a 16-byte group, whole, several), row counts on
    both sides of an opening block."""
    g = W.rng(n)
    vals = W.uniform_attrs(g, 3, n, 16)
    tab = W.table(vals, 16, g)
    ctx.load_shares(0, [to_dev(s) for s in tab["shares"]], 16)
    flags = vals[0] % 3 == 0
    xs = W.table(flags.astype(np.uint32)[None], 32, g)["shares"]
    outs = [torch.zeros((n, 1 + len(attrs)), dtype=torch.int32, device="cuda") for _ in range(3)]
    m = ctx.fetch_multi(0, [to_dev(x[0]) for x in xs], attrs, bytes(range(100, 148)), outs)
    wm, want = oracle.fetch_multi([x[0] for x in xs], (tab["shares"], 16), attrs, bytes(range(100, 148)), cap=n)
    assert m == wm == int(flags.sum())
    for j in range(3):
        assert np.array_equal(from_dev(outs[j][:m]), want[j])


@pytest.mark.parametrize("bits,n", [(8, 257), (8, 9000), (13, 4097), (16, 12001), (24, 6000), (32, 5003)])
def test_small_launches_by_every_route(ctx, bits, n):
    """Launches of several walk-parallel waves may take the staged evaluation, with a unit per key in
    its last stage: the same shares as the walk-parallel and the per-element kernel, and as the
    oracle on a sample."""
    g = W.rng(bits + n)
    vals = W.uniform_attrs(g, 2, n, bits)
    vals[1, ::3] = vals[1, 0]                 # a value that many elements share
    tab = W.table(vals, bits, g)
    ctx.load_shares(0, [to_dev(s) for s in tab["shares"]], bits)
    top = (1 << bits) - 1
    preds = [W.eq_pred(0, 0, 0, int(vals[0, 1])), W.range_pred(0, 1, 0, top // 5, top // 2, W.COMBINE_OR),
             W.range_pred(0, 0, 1, 0, top - 1), W.eq_pred(0, 1, 2, int(vals[1, 0])),
             W.range_pred(0, 1, 2, int(vals[1, 0]), top, W.COMBINE_XOR)]
    toks = P.keygen(preds, bits, bytes(range(7, 23)))
    got = []
    default = ctx.set_walk_parallel((1 << 64) - 1)
    try:
        for route in (default, (1 << 64) - 1, 0):
            ctx.set_walk_parallel(route)
            outs = [[torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(3)] for _ in range(3)]
            ctx.filter_and_combine(5, toks, outs)
            ctx.sync()
            got.append([np.stack([from_dev(t) for t in grp]) for grp in outs])
    finally:
        ctx.set_walk_parallel(default)
    idx = np.unique(np.concatenate([np.arange(0, n, max(1, n // 200)), [n - 1]]))
    for grp in range(3):
        assert np.array_equal(got[0][grp], got[1][grp]) and np.array_equal(got[0][grp], got[2][grp]), grp
        want = oracle.filter_group(toks, 5, PRF, [(tab["shares"], bits)], grp, idx, threads=4)
        assert np.array_equal(got[0][grp][:, idx], want), grp


def test_small_staged_plan_under_capture(ctx):
    """A prepared plan of a small staged launch, captured into a CUDA graph (its kernels are
    programmatic dependents), replays to the shares of the direct call."""
    g = W.rng(77)
    n, bits = 9000, 16
    vals = W.uniform_attrs(g, 2, n, bits)
    tab = W.table(vals, bits, g)
    ctx.load_shares(0, [to_dev(s) for s in tab["shares"]], bits)
    preds = [W.eq_pred(0, 0, 0, int(vals[0, 1])), W.range_pred(0, 1, 0, 100, 9000)]
    toks = P.keygen(preds, bits, bytes(16))
    outs = [[torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(3)]]
    ctx.filter_and_combine(5, toks, outs)
    ctx.sync()
    want = [t.clone() for t in outs[0]]
    plan = ctx.plan_create([5], [toks], [outs])
    for t in outs[0]:
        t.zero_()
    torch.cuda.synchronize()
    graph, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=s):
        ctx.plan_launch(plan, stream=s.cuda_stream)
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    ctx.plan_destroy(plan)
    for a, b in zip(outs[0], want):
        assert torch.equal(a, b)


@pytest.mark.parametrize("dcf", [False, True])
@pytest.mark.parametrize("points", [1, 64, 65, 152 * 64 + 1, 152 * 768, 152 * 768 + 1, 2 * 152 * 768 + 33])
def test_per_item_evaluation_in_even_waves(ctx, dcf, points):
    """Points with a key each, around one item per warp and per thread of every SM and two full
    waves: a sample against the oracle, and on every point the pair's two keys add up to beta where
    x = alpha or x < alpha."""
    g, bits = np.random.default_rng(points), 9
    kind, L = (P.KEY_DCF, 28 + 24 * bits) if dcf else (P.KEY_DPF, 28 + 20 * bits)
    x = g.integers(0, 1 << bits, points, dtype=np.uint64).astype(np.uint32)
    alpha, beta = int(x[points // 2]), 0x9E3779B1
    keys = torch.zeros(2 * L, dtype=torch.uint8, device="cuda")
    ctx.keygen_device(kind, bits, to_dev(np.uint32([alpha])), to_dev(np.uint32([beta])), SEED, keys)
    raw, got = keys.cpu().numpy().tobytes(), []
    idx = np.unique([0, points - 1, points // 2, *g.integers(0, points, 16)])
    for k in range(2):
        out = torch.full((points,), -1, dtype=torch.int32, device="cuda")
        of = torch.full((points,), k, dtype=torch.int32, device="cuda")
        ctx.eval_device_keys(kind, bits, keys, 2, to_dev(x), out, key_of_point=of)
        ctx.sync()
        got.append(from_dev(out))
        want = oracle.eval_many(raw[k * L:(k + 1) * L], x[idx], oracle.KIND_DCF if dcf else oracle.KIND_DPF)
        assert np.array_equal(got[k][idx], want)
    hit = x < alpha if dcf else x == alpha
    assert np.array_equal(got[0] + got[1], np.where(hit, np.uint32(beta), np.uint32(0)))


@pytest.mark.parametrize("bits", [4, 29])
@pytest.mark.parametrize("groups", [((0, 0, 0, 1, 1, 1, 1, 1),), ((0, 1, 0), (1, 0, 1, 1, 1)), ((0, 0, 0, 0, 1), (1, 1))])
def test_walk_parallel_keys_up_to_the_end_of_shared_memory(ctx, bits, groups):
    """66 keys, the most that a launch keeps in shared memory, in groups of both kinds whose last
    predicate is an equality: its walks' idle slots have no key of their own there."""
    g, n = W.rng(bits + len(groups)), 207
    vals = W.uniform_attrs(g, 2, n, bits)
    tab = W.table(vals, bits, g)
    ctx.load_shares(0, [to_dev(s) for s in tab["shares"]], bits)
    top, preds = (1 << bits) - 1, []
    for grp, kinds in enumerate(groups):
        for k, eq in enumerate(kinds):
            op = (W.COMBINE_AND, W.COMBINE_OR, W.COMBINE_XOR)[k % 3] if k else W.COMBINE_AND
            preds.append(W.eq_pred(0, k % 2, grp, int(vals[k % 2, k]), op) if eq else
                         W.range_pred(0, k % 2, grp, k, top // 2 + k, op))
    assert sum(6 if p["kind"] == W.PRED_EQ else 12 for p in preds) == 66
    toks = P.keygen(preds, bits, bytes(range(5, 21)))
    prev = ctx.set_walk_parallel((1 << 64) - 1)
    try:
        outs = [[torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(3)] for _ in groups]
        ctx.filter_and_combine(9, toks, outs)
        ctx.sync()
    finally:
        ctx.set_walk_parallel(prev)
    for grp in range(len(groups)):
        got = np.stack([from_dev(t) for t in outs[grp]])
        want = oracle.filter_group(toks, 9, PRF, [(tab["shares"], bits)], grp, np.arange(n), threads=4)
        assert np.array_equal(got, want), grp
