"""The work that a user of the colour-coding library has it do, as cases that can be timed.

A case is a dict of plain values: a host graph family with its size, one or more patterns, the
number of colours and colourings, and how the library is asked (one call from host arrays, a
resident context, tables kept for enumeration, a captured batch, a running server).  Patterns are
texts: path6, cycle5, grid2x4, treeA (the 9-vertex tree with three joins), ktree10w3s7004 (random
partial 3-tree, 10 vertices, seed), er10q20s3 (G(10, 0.20), seed; its decomposition is left to the
library); cycle4! is a served query that wants embeddings too.  Everything random in a case's graph and colouring comes from prepare()'s seed.
"""
import math

import numpy as np

import paper_1908_11248_gb300 as cc

# ---- host graphs (CSR) ---------------------------------------------------------------------


def _csr(n, a, b):
    keep = a != b
    a, b = a[keep].astype(np.int64), b[keep].astype(np.int64)
    key = np.unique(np.concatenate([a * n + b, b * n + a]))
    row = np.zeros(n + 1, np.int64)
    row[1:] = np.cumsum(np.bincount(key // n, minlength=n))
    return row.astype(np.int32), (key % n).astype(np.int32)


def _er(n, deg, rng):
    """Erdos-Renyi, mean degree `deg`."""
    if n <= 2000:
        i, j = np.triu_indices(n, k=1)
        keep = rng.random(len(i)) < deg / (n - 1)
        return _csr(n, i[keep], j[keep])
    m = rng.binomial(n * (n - 1) // 2, deg / (n - 1))
    return _csr(n, rng.integers(0, n, m), rng.integers(0, n, m))


def _ba(n, m, rng):
    """Preferential attachment, m edges a vertex: an edge's second end copies a uniformly drawn
    earlier edge end (resolved by following the references), repeats dropped."""
    m0 = m + 1
    core = [(i, j) for i in range(m0) for j in range(i + 1, m0)]
    e0, total = len(core), len(core) + (n - m0) * m
    src = np.empty(total, np.int64)
    src[:e0] = [a for a, _ in core]
    src[e0:] = np.repeat(np.arange(m0, n), m)
    ref = (rng.random(total) * (2 * np.arange(total))).astype(np.int64)  # an end of an earlier edge
    known = np.full(total, -1, np.int64)
    known[:e0] = [b for _, b in core]
    at = ref[e0:].copy()
    dst = np.full(total - e0, -1, np.int64)
    todo = np.arange(total - e0)
    while len(todo):
        p = at[todo]
        e = p // 2
        even, core_end = p % 2 == 0, e < e0
        done = even | core_end
        dst[todo[done]] = np.where(even[done], src[e[done]], known[e[done]])
        todo, e = todo[~done], e[~done]
        at[todo] = ref[e]
    known[e0:] = dst
    return _csr(n, src, known)


def _pl(n, deg, rng):
    """Erased power-law configuration model, exponent 2.5."""
    d = np.minimum((deg / 3.0 + 0.4) * (1.0 - rng.random(n)) ** (-1 / 1.5), n ** (1 / 1.5))
    stubs = np.repeat(np.arange(n), np.maximum(1, d.astype(np.int64)))
    if len(stubs) % 2:
        stubs = stubs[:-1]
    rng.shuffle(stubs)
    s = stubs.reshape(-1, 2)
    return _csr(n, s[:, 0], s[:, 1])


def _graph(case, rng):
    return {"er": _er, "ba": _ba, "pl": _pl}[case["graph"]](case["n"], case["deg"], rng)


# ---- patterns: (n_F, edges, (bags, parent) or None) ----------------------------------------


def _chain(bags):
    return bags, [i + 1 for i in range(len(bags) - 1)] + [-1]


def _ktree(n, w, seed):
    rng = np.random.default_rng(seed)
    bags, parent = [list(range(w + 1))], [-1]
    edges = {(i, j) for i in range(w + 1) for j in range(i + 1, w + 1)}
    for v in range(w + 1, n):
        b = int(rng.integers(0, len(bags)))
        out_i = int(rng.integers(0, w + 1))
        kept = [u for i, u in enumerate(bags[b]) if i != out_i]
        bags.append(sorted(kept + [v]))
        parent.append(b)
        edges |= {(u, v) for u in kept}
    comp, out = list(range(n)), []
    edges = sorted(edges)
    for i in rng.permutation(len(edges)):  # a random spanning tree and half of the other edges
        a, b = edges[i]
        if comp[a] != comp[b]:
            old, new = comp[a], comp[b]
            comp = [new if x == old else x for x in comp]
            out.append((a, b))
        elif rng.random() < 0.5:
            out.append((a, b))
    return n, sorted(out), (bags, parent)


def _pattern(text):
    text = text.rstrip("!")
    if text.startswith("path"):
        n = int(text[4:])
        return n, [(i, i + 1) for i in range(n - 1)], _chain([[i, i + 1] for i in range(n - 1)])
    if text.startswith("cycle"):
        n = int(text[5:])
        return n, [(i, (i + 1) % n) for i in range(n)], _chain([[0, i, i + 1] for i in range(1, n - 1)])
    if text.startswith("grid"):  # r <= c: swept column by column
        r, c = (int(x) for x in text[4:].split("x"))
        e = [(i * c + j, i * c + j + 1) for i in range(r) for j in range(c - 1)]
        e += [(i * c + j, i * c + j + c) for i in range(r - 1) for j in range(c)]
        order = [i * c + j for j in range(c) for i in range(r)]
        return r * c, e, _chain([sorted(order[s:s + r + 1]) for s in range(r * c - r)])
    if text == "treeA":
        e = [(0, 1), (1, 2), (2, 3), (2, 4), (5, 4), (6, 4), (6, 7), (7, 8)]
        bags = [[0, 1], [1, 2], [2, 3], [2, 4], [4, 5], [4, 6], [6, 7], [7, 8]]
        return 9, e, (bags, [1, 3, 3, -1, 3, 3, 5, 6])
    if text.startswith("ktree"):
        n, rest = text[5:].split("w")
        w, s = rest.split("s")
        return _ktree(int(n), int(w), int(s))
    n, rest = text[2:].split("q")  # er<n>q<percent>s<seed>
    q, s = rest.split("s")
    rng = np.random.default_rng(int(s))
    n = int(n)
    e = [(i, j) for i in range(n) for j in range(i + 1, n) if rng.random() < int(q) / 100]
    return n, e, None


# ---- the cases -----------------------------------------------------------------------------


def listed():
    return [
        # one interactive query on a small graph: a colouring, the DP with its tables kept, the
        # count, every embedding (latency)
        dict(name="query_er200_c5", how="query", graph="er", n=200, deg=10, patterns="cycle5",
             spare=0, trials=1, limit=8192, arena_gb=1),
        # a caller with host arrays and no device allocator: the graph is checked, copied and
        # counted in one call, every table sized exactly; one colour more than vertices
        dict(name="oneshot_er997_c5", how="oneshot", graph="er", n=997, deg=6, patterns="cycle5",
             spare=1, trials=2, limit=0, arena_gb=0),
        # enumeration where there is much to enumerate: the first 100 000 of some 300 000 rows
        dict(name="enum_er1999_p4", how="query", graph="er", n=1999, deg=12, patterns="path4",
             spare=0, trials=1, limit=100_000, arena_gb=4),
        # one colouring of a path, the lightest pattern, on a large resident graph
        dict(name="count_ba200k_p6", how="count", graph="ba", n=200_000, deg=5, patterns="path6",
             spare=0, trials=1, limit=0, arena_gb=16),
        # one colouring of a short cycle on the same graph: hubs make its tables
        dict(name="count_ba200k_c4", how="count", graph="ba", n=200_000, deg=5, patterns="cycle4",
             spare=0, trials=1, limit=0, arena_gb=16),
        # many colourings at once of the 2x4 grid (64-bit keys)
        dict(name="grid2x4_ba20k_t64", how="count", graph="ba", n=20_000, deg=4,
             patterns="grid2x4", spare=0, trials=64, limit=0, arena_gb=40),
        # a ragged one of the same kind: odd sizes, few colourings, one colour more
        dict(name="grid2x4_ba4999_t13", how="count", graph="ba", n=4999, deg=4,
             patterns="grid2x4", spare=1, trials=13, limit=0, arena_gb=8),
        # the largest: 3x3 grid, width 3, 128-bit keys, tables kept and enumerated
        dict(name="grid3x3_er100k_t32", how="query", graph="er", n=100_000, deg=10,
             patterns="grid3x3", spare=0, trials=32, limit=100_000, arena_gb=80),
        # a tree whose decomposition branches: three joins
        dict(name="tree_ba20k_t4", how="count", graph="ba", n=20_000, deg=4, patterns="treeA",
             spare=0, trials=4, limit=0, arena_gb=32),
        # several patterns of one graph in one captured batch: partial 2- and 3-trees (joins,
        # wide bags) on a power-law graph
        dict(name="batch_pl2000_ktrees", how="batch", graph="pl", n=2000, deg=8,
             patterns="ktree10w2s7001 ktree9w2s7002 ktree7w3s7003 ktree8w2s7004 path8 cycle5",
             spare=0, trials=4, limit=0, arena_gb=48),
        # a random pattern in a random target, ten colourings: the phase-transition study
        dict(name="phase_er150_g10", how="count", graph="er", n=150, deg=9, patterns="er10q18s5",
             spare=0, trials=10, limit=0, arena_gb=8),
        # a server with a resident graph: 24 mixed queries submitted together, some of which want
        # embeddings
        dict(name="serve_ba20k_mix", how="serve", graph="ba", n=20_000, deg=5,
             patterns="path4 path5 cycle4! grid2x3 path7 ktree6w2s40 path8 cycle4 treeA "
                      "path6 ktree5w1s41 grid2x2! path4 path5 cycle4! grid2x3 path7 ktree6w2s40 "
                      "path8 cycle4 treeA path6 ktree5w1s41 grid2x2!",
             spare=0, trials=1, limit=1000, arena_gb=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    how = rng.choice(["query", "oneshot", "light", "grid", "wide", "tree", "batch", "phase",
                      "serve"])
    spare = rng.choice([0, 0, 0, 1, 2])
    if how == "query":
        return dict(how="query", graph="er", n=_log(rng, 50, 2000), deg=rng.randint(5, 12),
                    patterns=rng.choice(["cycle4", "cycle5", "path3", "path4", "grid2x2",
                                         "grid2x3"]),
                    spare=spare, trials=rng.randint(1, 3), limit=_log(rng, 1000, 100_000),
                    arena_gb=8)
    if how == "oneshot":
        return dict(how="oneshot", graph="er", n=_log(rng, 100, 1500), deg=rng.randint(3, 6),
                    patterns=rng.choice(["path4", "path5", "path6", "cycle4", "cycle5",
                                         "grid2x3"]),
                    spare=spare, trials=rng.randint(1, 3), limit=0, arena_gb=0)
    if how == "light":
        n = _log(rng, 2000, 200_000)
        return dict(how="count", graph="ba", n=n, deg=rng.randint(3, 5),
                    patterns=rng.choice(["path4", "path5", "path6", "path7", "cycle4", "grid2x2"]),
                    spare=spare, trials=rng.randint(1, max(1, min(16, 200_000 // n))), limit=0,
                    arena_gb=24)
    if how == "grid":
        n = _log(rng, 1500, 20_000)
        return dict(how="count", graph=rng.choice(["ba", "er"]), n=n, deg=rng.randint(3, 4),
                    patterns=rng.choice(["grid2x3", "grid2x4"]), spare=spare,
                    trials=_log(rng, 4, min(64, max(5, 1_000_000 // n))), limit=0, arena_gb=40)
    if how == "wide":
        return dict(how="query", graph="er", n=_log(rng, 5000, 100_000), deg=rng.randint(5, 9),
                    patterns="grid3x3", spare=spare % 2, trials=_log(rng, 2, 32), limit=100_000,
                    arena_gb=80)
    if how == "tree":
        return dict(how="count", graph="ba", n=_log(rng, 1000, 20_000), deg=rng.randint(3, 4),
                    patterns="treeA", spare=spare % 2, trials=rng.randint(1, 4), limit=0,
                    arena_gb=32)
    if how == "batch":
        two = ["ktree%dw2s%d" % (rng.randint(6, 9), rng.randint(1, 999)) for _ in range(2)]
        return dict(how="batch", graph="er", n=_log(rng, 200, 2000), deg=rng.randint(4, 7),
                    patterns=" ".join(two + ["path%d" % rng.randint(4, 8), "cycle4"]), spare=0,
                    trials=rng.randint(1, 4), limit=0, arena_gb=48)
    if how == "phase":
        return dict(how="count", graph="er", n=_log(rng, 60, 150), deg=rng.randint(4, 8),
                    patterns="er%dq%ds%d" % (rng.randint(7, 9), rng.randint(12, 20),
                                             rng.randint(1, 999)),
                    spare=0, trials=10, limit=0, arena_gb=24)
    few = [rng.choice(["path4", "path5", "path6", "cycle4!", "grid2x2", "ktree5w1s41",
                       "ktree6w1s42"]) for _ in range(rng.randint(6, 20))]
    return dict(how="serve", graph="ba", n=_log(rng, 2000, 20_000), deg=rng.randint(3, 5),
                patterns=" ".join(few), spare=0, trials=1, limit=rng.choice([100, 1000]),
                arena_gb=32)


class _State:
    """What a user's program keeps: the graph's arrays, a context with the graph and the patterns
    loaded (none for the one-call form), the colouring seed."""


def prepare(case, seed):
    s = _State()
    rng = np.random.default_rng([seed, case["n"]])
    s.case = case
    s.graph = _graph(case, rng)
    s.seed = int(rng.integers(1, 1 << 62))
    s.patterns = [_pattern(t) for t in case["patterns"].split()]
    s.ctx = None
    if case["how"] == "oneshot":
        return s
    s.ctx = cc.Context(arena_bytes=case["arena_gb"] << 30)
    cc.cc_load_graph(s.ctx.h, *s.graph)
    loaded = {}
    for text, p in zip(case["patterns"].split(), s.patterns):
        if text not in loaded:
            loaded[text] = cc.cc_load_pattern(s.ctx.h, *p)
    s.pids = [loaded[t] for t in case["patterns"].split()]
    s.limits = [case["limit"] if case["how"] == "query" or t.endswith("!") else 0
                for t in case["patterns"].split()]
    if case["how"] == "serve":
        cc.cc_serve_start(s.ctx.h, 0, 8)
    else:
        s.nodes = [cc.cc_pattern_info(s.ctx.h, pid)[0] for pid in s.pids]
        s.opts = cc.cc_default_opts(retain=int(case["how"] == "query"),
                                    use_graph=int(case["how"] == "batch"))
    return s


def _whole(rows, limit):
    """The rows in the array of `limit` rows that the caller set aside for them."""
    if len(rows) == limit:
        return rows
    out = np.zeros((limit, rows.shape[1]), np.int32)
    out[:len(rows)] = rows
    return out


def _serve(s):
    case, h, T = s.case, s.ctx.h, s.case["trials"]
    waiting, out = [], []
    for i, (pid, p, limit) in enumerate(zip(s.pids, s.patterns, s.limits)):
        waiting.append((cc.cc_serve_submit(h, pid, s.seed + i, T, p[0] + case["spare"], limit),
                        limit, p[0]))
    for ticket, limit, nF in waiting:
        while True:
            done, status, counts, exists, _, rows = cc.cc_serve_poll(h, ticket, T, limit, nF)
            if done:
                break
        if status:
            raise cc.CCError("cc_serve_poll", status)
        out += [counts.view(np.int64), exists] + ([_whole(rows, limit)] if limit else [])
    return out


def run(s):
    case, T = s.case, s.case["trials"]
    if case["how"] == "oneshot":
        nF, edges, td = s.patterns[0]
        counts, exists = cc.cc_count_noalloc(0, 0, *s.graph, nF, edges, td, s.seed, T,
                                             nF + case["spare"])
        return [counts.view(np.int64), exists]
    if case["how"] == "serve":
        return _serve(s)
    h, out = s.ctx.h, []
    cids = [cc.cc_color(h, s.seed + i, T, p[0] + case["spare"])
            for i, p in enumerate(s.patterns)]
    runs = cc.cc_run_batch(h, s.pids, cids, s.opts)
    for r, n_nodes, p in zip(runs, s.nodes, s.patterns):
        sizes, _ = cc.cc_table_stats(h, r, n_nodes)
        out += [cc.cc_count(h, r, T).view(np.int64), cc.cc_decide(h, r, T), sizes.view(np.int64)]
        if case["limit"]:
            rows, total = cc.cc_enumerate(h, r, case["limit"], p[0])
            out += [_whole(rows, case["limit"]), total]
        cc.cc_release(h, r)
    for cid in cids:
        cc.cc_release_colors(h, cid)
    return out


def work(case):
    """Bytes: the graph's CSR once for every pattern, every colour drawn and read once, the
    results.  The tables between are the method's own, and how many entries they hold depends on
    the graph."""
    n, T = case["n"], case["trials"]
    half = case["deg"] / 2 if case["graph"] != "ba" else case["deg"]
    per = 4 * (n + 1) + 8 * n * half + 2 * T * n + 9 * T
    return {"bytes": len(case["patterns"].split()) * per + 16 * case["limit"] * (case["n"] > 1000),
            "flops": 0}


def exact(case, seed):
    """None: every output is a whole number (counts mod 2^64, flags, sizes, vertex ids)."""
    return None
