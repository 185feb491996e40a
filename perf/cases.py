"""What is timed of this library: one pass of each thing that its users have it do.

A case is a dict of plain values; "kind" names the public call and the rest its sizes.
The sizes are those of the repository's workloads (the 1k / 4k path query, the 1,048,576-vertex
filter, the triangle + pendant query on a 1M / 10M graph, the 107,614-vertex one-hot table, the
1M-candidate fetches and shuffle) and generic ragged ones between them.  Values are drawn as the
workloads draw them: vertex attributes uniform on [0, 2^n), edge attributes bounded Zipf (1.1 at
n <= 16, 1.2 above); equality values and range bounds lie around the values of elements of the
table, so predicates have matches.  Everything is made on the GPU from the seed.
"""
import math
import random

import torch

import paper_2209_03526_gb300 as P

DEV = "cuda:0"
PRF = bytes(range(48))
U32 = 0xFFFFFFFF


def listed():
    return [
        # The smallest call: the 3-vertex path query on 1,000 vertices / 4,000 edges with 16-bit
        # attributes (one equality, one range), asked once, tokens in hand: latency counts.
        {"name": "path_1k_4k", "kind": "filter", "vertices": 1000, "edges": 4000, "bits": 16,
         "spec": "ve0 er1"},
        # The same query as a standing one: a prepared plan launched again.
        {"name": "path_1k_4k_plan", "kind": "plan", "vertices": 1000, "edges": 4000, "bits": 16,
         "spec": "ve0 er1"},
        # An ordinary filter of a mid-size ragged table: equality OR range, AND a range, n = 32.
        {"name": "filter_100003", "kind": "filter", "vertices": 100003, "edges": 0, "bits": 32,
         "spec": "ve0 vr0| vr0&"},
        # The headline: 8 predicates (4 equality, 4 range) ANDed on 1,048,576 vertices, n = 32.
        {"name": "bulk_1m_8pred", "kind": "filter", "vertices": 1 << 20, "edges": 0, "bits": 32,
         "spec": "ve0 ve0& ve0& ve0& vr0& vr0& vr0& vr0&"},
        # The largest: triangle + pendant, 6 predicates in 6 groups on 1M vertices / 10M edges.
        {"name": "triangle_1m_10m", "kind": "plan", "vertices": 1000000, "edges": 10000000, "bits": 32,
         "spec": "ve0 er1 ve2 er3 ve4 er5"},
        # Several users' queries in one launch on a small graph: 12 mixed queries, n = 32.
        {"name": "batch_12q_20k_80k", "kind": "batch", "vertices": 20000, "edges": 80000, "bits": 32,
         "queries": 12},
        # The paper's secEval as written: one-hot shares of 16-bit values, the paper's vertex
        # count, 4 predicates on one column in 3 groups.
        {"name": "onehot_107614_n16", "kind": "onehot", "elems": 107614, "bits": 16,
         "spec": "ve0 vr0& ve1 vr2"},
        # Fresh masks and keys per element, the servers' side: an equality AND a range, n = 32.
        {"name": "fresh_filter_131071", "kind": "fresh_filter", "elems": 131071, "bits": 32},
        # ... and the client's side: the three servers' tokens for 50,000 elements.
        {"name": "fresh_keygen_50000", "kind": "fresh_keygen", "elems": 50000, "bits": 32},
        # The raw primitive: a few comparison keys evaluated at every point of a column.
        {"name": "eval_dcf_12x65537", "kind": "eval", "dcf": True, "keys": 12, "points": 65537, "bits": 32},
        # secFetch case I: index and 4 attributes of the one match among 1,048,576 candidates.
        {"name": "fetch_unique_1m_4attr", "kind": "fetch_unique", "elems": 1 << 20, "attrs": 4},
        # secFetch case II: shuffle 1,048,576 candidates and fetch the 1 % that match.
        {"name": "fetch_multi_1m_4attr", "kind": "fetch_multi", "elems": 1 << 20, "attrs": 4},
    ]


def _log_int(rng, lo, hi):
    """log-uniform, odd and ragged values among them"""
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))


def _spec(rng, preds, with_edges):
    words, group, table = [], -1, "v"
    for _ in range(preds):
        op = ""
        if group < 0 or rng.random() < 0.4:
            group += 1
            table = "e" if with_edges and rng.random() < 0.5 else "v"
        else:
            op = rng.choice("&&|^")
        words.append(table + rng.choice("er") + str(group) + op)
    return " ".join(words)


def _batch_specs(case):
    """the queries' shapes, 1 to 6 predicates each: a part of the case, the same for every seed"""
    rng = random.Random(case["vertices"] * 64 + case["queries"])
    return [_spec(rng, rng.randint(1, 6), True) for _ in range(case["queries"])]


def draw(rng):
    kind = rng.choice(["filter", "filter", "plan", "batch", "onehot", "fresh_filter", "fresh_keygen", "keygen",
                       "eval", "fetch_unique", "fetch_multi", "shuffle"])
    if kind in ("filter", "plan"):
        nv = _log_int(rng, 1000, 1 << 20)
        ne = _log_int(rng, 4000, 3000000) if rng.random() < 0.5 else 0
        return {"kind": kind, "vertices": nv, "edges": ne, "bits": rng.choice([8, 16, 24, 32, 32]),
                "spec": _spec(rng, rng.randint(1, 6), ne > 0)}
    if kind == "batch":
        nv = _log_int(rng, 1000, 50000)
        return {"kind": kind, "vertices": nv, "edges": 4 * nv, "bits": rng.choice([16, 32]),
                "queries": rng.randint(2, 20)}
    if kind == "onehot":
        bits = rng.randint(6, 16)
        top = min(500000, (107614 << 16) >> bits)
        return {"kind": kind, "elems": _log_int(rng, 1000, top), "bits": bits, "spec": _spec(rng, rng.randint(1, 5), False)}
    if kind == "fresh_filter":
        return {"kind": kind, "elems": _log_int(rng, 1000, 150000), "bits": rng.choice([16, 32])}
    if kind == "fresh_keygen":
        return {"kind": kind, "elems": _log_int(rng, 1000, 60000), "bits": rng.choice([16, 32])}
    if kind == "keygen":
        return {"kind": kind, "dcf": rng.random() < 0.5, "pairs": _log_int(rng, 1000, 150000), "bits": rng.choice([16, 32])}
    if kind == "eval":
        return {"kind": kind, "dcf": rng.random() < 0.5, "keys": rng.randint(1, 24), "points": _log_int(rng, 1000, 300000),
                "bits": rng.choice([8, 16, 32])}
    if kind == "shuffle":
        return {"kind": kind, "elems": _log_int(rng, 1000, 1 << 20), "width": rng.randint(1, 12)}
    return {"kind": kind, "elems": _log_int(rng, 1000, 1 << 20), "attrs": rng.randint(1, 8)}


# ------------------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _i32(x):
    """int64 values mod 2^32 as int32 bit patterns"""
    return (((x + (1 << 31)) & U32) - (1 << 31)).to(torch.int32)


def _uniform(g, shape, bits):
    return torch.randint(0, 1 << bits, shape, dtype=torch.int64, device=DEV, generator=g)


def _zipf(g, n, s, bits):
    """bounded Zipf(s) ranks less one, by rejection from the Pareto envelope"""
    top, b = float(1 << bits), 2.0 ** (s - 1.0)
    parts, have = [], 0
    while have < n:
        m = 2 * (n - have) + 1024
        u = 1.0 - torch.rand(m, dtype=torch.float64, device=DEV, generator=g)
        v = torch.rand(m, dtype=torch.float64, device=DEV, generator=g)
        x = torch.floor(u ** (-1.0 / (s - 1.0)))
        t = (1.0 + 1.0 / x) ** (s - 1.0)
        x = x[(v * x * (t - 1.0) / (b - 1.0) <= t / b) & (x <= top)]
        parts.append(x[: n - have].to(torch.int64) - 1)
        have += len(parts[-1])
    return torch.cat(parts)


def _share3(g, x, bits):
    """three additive shares of int64 values mod 2^bits, as int32 tensors"""
    a, b = _uniform(g, x.shape, bits), _uniform(g, x.shape, bits)
    return [_i32(a), _i32(b), _i32((x - a - b) & ((1 << bits) - 1))]


def _graph(case, seed):
    """attribute values of the vertex table (uniform) and the edge table (Zipf)"""
    g, bits = _gen(seed), case["bits"]
    tabs = [_uniform(g, (4 if bits > 16 else 2, case["vertices"]), bits)]
    if case["edges"]:
        s = 1.1 if bits <= 16 else 1.2
        tabs.append(torch.stack([_zipf(g, case["edges"], s, bits) for _ in range(2 if bits > 16 else 1)]))
    return g, tabs


def _preds(spec, tabs, bits, rng):
    """a predicate per word: table (v, e), kind (e, r), group, fold; attributes in turn"""
    out, seen = [], {}
    ops = {"": P.COMBINE_AND, "&": P.COMBINE_AND, "|": P.COMBINE_OR, "^": P.COMBINE_XOR}
    for word in spec.split():
        t = 1 if word[0] == "e" else 0
        group, op = (word[2:], "") if word[-1].isdigit() else (word[2:-1], word[-1])
        attr = seen.get(word[:2], 0) % tabs[t].shape[0]
        seen[word[:2]] = attr + 1
        v = int(tabs[t][attr, rng.randrange(tabs[t].shape[1])])
        p = {"kind": P.PRED_EQ, "table": t, "attr": attr, "group": int(group), "lo": v, "hi": v, "combine": ops[op]}
        if word[1] == "r":
            top = (1 << bits) - 1
            width = max(1, int(rng.uniform(0.02, 0.6) * (top + 1)))
            lo = max(0, v - rng.randrange(width))
            p.update(kind=P.PRED_RANGE, lo=lo, hi=max(v, min(top, lo + width - 1)))
        out.append(p)
    return out


def _outs(preds, sizes):
    table = {p["group"]: p["table"] for p in preds}
    return [[torch.zeros(sizes[table[k]], dtype=torch.int32, device=DEV) for _ in range(3)] for k in sorted(table)]


def prepare(case, seed):
    kind, rng = case["kind"], random.Random(seed)
    s = {"kind": kind, "qid": rng.randrange(1 << 32)}
    seed16 = bytes(rng.randrange(256) for _ in range(16))
    ctx = s["ctx"] = P.Context(0, prf_keys=PRF)
    if kind in ("filter", "plan", "batch"):
        g, tabs = _graph(case, seed)
        for t, x in enumerate(tabs):
            ctx.load_shares(t, _share3(g, x, case["bits"]), case["bits"])
        sizes = [x.shape[1] for x in tabs]
        if kind == "batch":
            qs = [_preds(spec, tabs, case["bits"], rng) for spec in _batch_specs(case)]
        else:
            qs = [_preds(case["spec"], tabs, case["bits"], rng)]
        s["qids"] = [(s["qid"] + i) & U32 for i in range(len(qs))]
        s["toks"] = [P.keygen(q, case["bits"], bytes([i]) + seed16[1:]) for i, q in enumerate(qs)]
        s["outs"] = [_outs(q, sizes) for q in qs]
        if kind == "plan":
            s["plan"] = _Plan(ctx, s)
    elif kind == "onehot":
        g, bits, n = _gen(seed), case["bits"], case["elems"]
        x = _uniform(g, (1, n), bits)
        words = max(1, (1 << bits) // 32)
        low = 32 if bits >= 5 else 1 << bits
        sh = [_i32(_uniform(g, (1, n, words), low)) for _ in range(2)]
        e = sh[0] ^ sh[1]
        at = (x // 32).unsqueeze(2)
        e.scatter_(2, at, e.gather(2, at) ^ _i32(1 << (x % 32)).unsqueeze(2))
        ctx.load_onehot(0, sh + [e], bits)
        preds = [dict(p, attr=0) for p in _preds(case["spec"], [x], bits, rng)]
        s["toks"] = P.keygen_onehot(preds, bits, seed16)
        s["outs"] = _outs(preds, [(n + 31) // 32])
    elif kind in ("fresh_filter", "fresh_keygen"):
        g, bits, n = _gen(seed), case["bits"], case["elems"]
        x = _uniform(g, (2, n), bits)
        s["preds"] = _preds("ve0 vr0&", [x], bits, rng)
        s["bits"], s["elems"], s["seed"] = bits, n, seed16
        size = P.fresh_token_size(s["preds"], bits, [n])
        s["toks"] = [torch.zeros(size, dtype=torch.uint8, device=DEV) for _ in range(3)]
        if kind == "fresh_filter":
            ctx.load_shares(0, _share3(g, x, bits), bits)
            ctx.keygen_fresh(s["preds"], bits, [n], seed16, s["toks"])
            s["outs"] = _outs(s["preds"], [n])
    elif kind in ("keygen", "eval"):
        g, bits = _gen(seed), case["bits"]
        s["dcf"], s["bits"], s["seed"] = case["dcf"], bits, seed16
        pairs = case["pairs"] if kind == "keygen" else (case["keys"] + 1) // 2
        s["alpha"], s["beta"] = _i32(_uniform(g, (pairs,), bits)), _i32(_uniform(g, (pairs,), 32))
        s["keys"] = torch.zeros(2 * pairs * (28 + (24 if case["dcf"] else 20) * bits), dtype=torch.uint8, device=DEV)
        if kind == "eval":
            ctx.keygen_device(P.KEY_DCF if case["dcf"] else P.KEY_DPF, bits, s["alpha"], s["beta"], seed16, s["keys"])
            s["n_keys"] = case["keys"]
            s["wire"] = s["keys"].cpu().numpy().tobytes()[: case["keys"] * (s["keys"].numel() // (2 * pairs))]
            s["points"] = _i32(_uniform(g, (case["points"],), bits))
            s["out"] = torch.zeros(case["keys"] * case["points"], dtype=torch.int32, device=DEV)
    elif kind in ("fetch_unique", "fetch_multi"):
        g, n, a = _gen(seed), case["elems"], case["attrs"]
        ctx.load_shares(0, _share3(g, _uniform(g, (a, n), 32), 32), 32)
        s["attrs"] = list(range(a))
        x = torch.zeros(n, dtype=torch.int64, device=DEV)
        if kind == "fetch_unique":
            x[rng.randrange(n)] = 1
            s["out"] = torch.zeros(3 * (1 + a), dtype=torch.int32, device=DEV)
        else:
            x[torch.rand(n, device=DEV, generator=g) < 0.01] = 1
            s["seeds"] = bytes(rng.randrange(256) for _ in range(48))
            s["outs"] = [torch.zeros((n // 50 + 64, 1 + a), dtype=torch.int32, device=DEV) for _ in range(3)]
        s["x"] = _share3(g, x, 32)
    else:
        g = _gen(seed)
        s["ins"] = _share3(g, _uniform(g, (case["elems"], case["width"]), 32), 32)
        s["outs"] = [torch.zeros_like(t) for t in s["ins"]]
        s["seeds"] = bytes(rng.randrange(256) for _ in range(48))
    return s


class _Plan:
    """a prepared plan, freed with the state that holds it"""

    def __init__(self, ctx, s):
        self.ctx = ctx
        torch.cuda.synchronize()
        self.plan = ctx.plan_create(s["qids"], s["toks"], s["outs"])

    def __del__(self):
        if getattr(self.ctx, "_h", None):
            self.ctx.plan_destroy(self.plan)


def run(s):
    kind, ctx = s["kind"], s["ctx"]
    if kind == "filter":
        ctx.filter_and_combine(s["qids"][0], s["toks"][0], s["outs"][0])
    elif kind == "plan":
        ctx.plan_launch(s["plan"].plan)
    elif kind == "batch":
        ctx.filter_batch(s["qids"], s["toks"], s["outs"])
        flat = [t for q in s["outs"] for grp in q for t in grp]
        return [torch.cat(flat[j::3]) for j in range(3)]        # one tensor per share set
    elif kind == "onehot":
        ctx.filter_onehot(s["qid"], s["toks"], s["outs"])
    elif kind == "fresh_filter":
        ctx.filter_fresh(s["qid"], s["toks"], s["outs"])
    elif kind == "fresh_keygen":
        ctx.keygen_fresh(s["preds"], s["bits"], [s["elems"]], s["seed"], s["toks"])
        return s["toks"]
    elif kind == "keygen":
        ctx.keygen_device(P.KEY_DCF if s["dcf"] else P.KEY_DPF, s["bits"], s["alpha"], s["beta"], s["seed"], s["keys"])
        return s["keys"]
    elif kind == "eval":
        fn = ctx.eval_dcf_batch if s["dcf"] else ctx.eval_dpf_batch
        fn(s["wire"], s["n_keys"], s["points"], s["out"], all_pairs=True)
        return s["out"]
    elif kind == "fetch_unique":
        ctx.fetch_unique(s["qid"], 0, 0, s["x"], s["attrs"], s["out"])
        return s["out"]
    elif kind == "fetch_multi":
        return [ctx.fetch_multi(0, s["x"], s["attrs"], s["seeds"], s["outs"])] + s["outs"]
    else:
        ctx.shuffle(s["ins"], s["seeds"], s["outs"])
    return s["outs"]


# ------------------------------------------------------------------------------ work

def _spec_bytes(spec, sizes, bits, attrs):
    """masked filter: the columns read (three share sets), the tokens, the outputs"""
    cols, groups, seen, b = set(), {}, {}, 0
    for word in spec.split():
        t = 1 if word[0] == "e" else 0
        a = seen.get(word[:2], 0) % attrs[t]
        seen[word[:2]] = a + 1
        cols.add((t, a))
        groups[word[2:].rstrip("&|^")] = t
        b += 3 * (24 + (2 * (28 + 20 * bits) if word[1] == "e" else 4 * (28 + 24 * bits)))
    return b + 12 * sum(sizes[t] for t, _ in cols) + 12 * sum(sizes[t] for t in groups.values())


def work(case):
    """bytes: each input read once, each output written once.  The arithmetic is AES on
    integers, so there are no floating-point operations to count."""
    kind, bits = case["kind"], case.get("bits", 32)
    na = [4 if bits > 16 else 2, 2 if bits > 16 else 1]
    key = lambda dcf: 28 + (24 if dcf else 20) * bits  # noqa: E731
    if kind in ("filter", "plan"):
        b = _spec_bytes(case["spec"], [case["vertices"], case["edges"]], bits, na)
    elif kind == "batch":
        # each query's outputs and tokens, and the columns it reads
        b = sum(_spec_bytes(spec, [case["vertices"], case["edges"]], bits, na) for spec in _batch_specs(case))
    elif kind == "onehot":
        groups = len({w[2:].rstrip("&|^") for w in case["spec"].split()})
        b = 3 * case["elems"] * max(4, (1 << bits) // 8) + groups * 12 * ((case["elems"] + 31) // 32)
    elif kind in ("fresh_filter", "fresh_keygen"):
        # per element and server: two mask shares and two DPF keys; those, c beta' and four DCF keys
        tok = 3 * case["elems"] * (8 + 2 * (28 + 16 * bits) + 12 + 4 * (28 + 20 * bits))
        b = tok + (36 * case["elems"] if kind == "fresh_filter" else 0)
    elif kind == "keygen":
        b = case["pairs"] * (8 + 2 * key(case["dcf"]))
    elif kind == "eval":
        b = case["keys"] * key(case["dcf"]) + 4 * case["points"] * (1 + case["keys"])
    elif kind == "fetch_unique":
        b = 12 * case["elems"] * (1 + case["attrs"]) + 12 * (1 + case["attrs"])
    elif kind == "fetch_multi":
        b = 12 * case["elems"] * (1 + case["attrs"]) + 12 * (case["elems"] // 100) * (1 + case["attrs"])
    else:
        b = 24 * case["elems"] * case["width"]
    return {"bytes": b, "flops": 0}


def exact(case, seed):
    """Shares and keys are whole numbers made from AES streams: they have no 64-bit counterpart
    outside this library and have to be equal bit for bit."""
    return None
