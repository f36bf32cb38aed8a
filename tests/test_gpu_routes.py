"""The kernels' alternative routes against the oracle, at the sizes where each can go wrong.  Every
result is a whole number or a list of vertex ids: equality, no tolerance."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

cc = pytest.importorskip("paper_1908_11248_gb300")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__

    __graft_entry__.build()
    c = cc.Context(arena_bytes=8 << 30)
    yield c
    c.close()


def star_of_joins(n):
    """The star on n vertices with every leaf in a bag of its own below the first: n - 3 joins."""
    nF, e, _ = synth.star_pattern(n)
    return nF, e, ([[0, i] for i in range(1, n)], [-1] + [0] * (n - 2))


def test_enumeration_at_every_arena_size():
    """A reconstruction appends its states into two arrays of the counted size, or counts each
    step first when only exact room is left; its rows sort as records or by index.  Whatever the
    room, the rows are the oracle's or the call ends with CC_ENOMEM."""
    pat = star_of_joins(8)
    n = 60
    g = synth.erdos_renyi(n, 0.09, 4)
    z = oracle.colors(n, 2, 8, seed=3)
    want, total, _ = oracle.run_dp(g, pat, z, 8).enumerate(300)
    fitted = 0
    for kb in range(1024, 24 * 1024, 512):
        with cc.Context(arena_bytes=kb << 10) as c:
            cc.cc_load_graph(c.h, *g)
            pid = cc.cc_load_pattern(c.h, *pat)
            cid = cc.cc_set_colors(c.h, z, 8)
            try:
                run = cc.cc_run_dp(c.h, pid, cid, cc.cc_default_opts(retain=1))
                rows, got = cc.cc_enumerate(c.h, run, 300, 8)
            except cc.CCError as ex:
                assert ex.code == cc.CC_ENOMEM, kb
                continue
            fitted += 1
            assert got == total and np.array_equal(rows, want[:300]), kb
    assert 0 < fitted


@pytest.mark.parametrize("n", [1, 31, 33, 1025, 9001])
def test_enumeration_first_forget_over_all_vertices(ctx, n):
    """The last vertex forgotten has no neighbour left: its candidates are all n host vertices,
    shared by several warps."""
    g = synth.erdos_renyi(n, min(1.0, 3.0 / max(1, n - 1)), 5)
    for pat in (synth.path_pattern(1), synth.path_pattern(3)):
        nF = pat[0]
        z = oracle.colors(n, 2, nF, seed=9)
        want, total, _ = oracle.run_dp(g, pat, z, nF).enumerate(10 ** 6)
        cc.cc_load_graph(ctx.h, *g)
        pid = cc.cc_load_pattern(ctx.h, *pat)
        cid = cc.cc_set_colors(ctx.h, z, nF)
        run = cc.cc_run_dp(ctx.h, pid, cid, cc.cc_default_opts(retain=1))
        rows, got = cc.cc_enumerate(ctx.h, run, 10 ** 6, nF)
        assert got == total and np.array_equal(rows, want)


def rows_of(trial, phi, mask, cnt):
    """A table as sorted rows (trial, phi, colour set, count)."""
    cols = [np.asarray(trial, np.uint64)] + [np.asarray(p, np.uint64) for p in np.asarray(phi).T]
    cols += [np.asarray(mask, np.uint64), np.asarray(cnt, np.uint64)]
    return np.stack(cols)[:, np.lexsort(cols[::-1])]


def check_tables(ctx, g, pat, z, k, reps=2, **opt):
    """Counts, sizes and every stored table, of an exact and a planned run, against the oracle."""
    T = z.shape[0]
    ref = oracle.run_dp(g, pat, z, k)
    cc.cc_load_graph(ctx.h, *g)
    pid = cc.cc_load_pattern(ctx.h, *pat)
    N, _ = cc.cc_pattern_info(ctx.h, pid)
    nodes = cc.cc_pattern_nodes(ctx.h, pid, pat[0])
    cid = cc.cc_set_colors(ctx.h, z, k)
    for rep in range(reps):
        run = cc.cc_run_dp(ctx.h, pid, cid, cc.cc_default_opts(retain=1, **opt))
        assert cc.cc_run_mode(ctx.h, run) == ("planned" if rep else "exact")
        assert np.array_equal(cc.cc_count(ctx.h, run, T), ref.count)
        assert np.array_equal(cc.cc_decide(ctx.h, run, T), ref.exists)
        sizes = cc.cc_table_stats(ctx.h, run, N)[0]
        assert np.array_equal(sizes, ref.node_sizes.sum(axis=0))
        for x, nd in enumerate(nodes):
            b = len(nd[4])
            try:
                tr, phi, mask, cnt = cc.cc_table_dump(ctx.h, run, x, int(sizes[x]) + 1, b)
            except cc.CCError as ex:
                assert ex.code == cc.CC_EINVAL and nd[0] == cc.INTRODUCE
                continue
            got = rows_of(tr, phi, mask, cnt)
            want = [ref.table(t, x, b) for t in range(T)]
            want = rows_of(np.repeat(np.arange(T), [len(m) for _, m, _ in want]),
                           np.concatenate([np.reshape(p, (len(m), b)) for p, m, _ in want]),
                           np.concatenate([m for _, m, _ in want]),
                           np.concatenate([c for _, _, c in want]))
            assert np.array_equal(got, want), (rep, x)
        cc.cc_release(ctx.h, run)
    cc.cc_release_colors(ctx.h, cid)


# the join's bag is {0, 1}: k - 2 private colours.  One word of sums, several words, the most a warp
# keeps (11 private colours, k = 13; one more is below, with the routes); few entries (hash tables)
# and more than the 2^21 at which children are sorted and joined group by group
@pytest.mark.parametrize("k", [4, 6, 7, 12, 13])
@pytest.mark.parametrize("many", [0, 1])
def test_join_routes(ctx, k, many):
    n, trials = (8000, 3 + 36 // (k - 1)) if many else (70, 3)
    g = synth.erdos_renyi(n, 8 / n, 6)
    check_tables(ctx, g, star_of_joins(4), oracle.colors(n, trials, k, seed=k), k)


# the 4-cycle as the join of its two paths between opposite corners, bag {0, 2}: 64-bit keys, and
# 128-bit keys (20 bits a vertex)
@pytest.mark.parametrize("n,deg", [(1100, 37.0), (530_000, 2.0)])
def test_join_of_paths(ctx, n, deg):
    pat = (4, np.array([(0, 1), (1, 2), (2, 3), (0, 3)], np.int32),
           ([[0, 2], [0, 1, 2], [0, 2, 3]], [-1, 0, 0]))
    g = synth.erdos_renyi(n, deg / n, 8)
    check_tables(ctx, g, pat, oracle.colors(n, 2, 5, seed=8), 5)


def test_join_routes_hubs_and_empty(ctx):
    """Bags of up to three vertices over hubs, and a graph without an edge."""
    n = 150
    g = synth.power_law_config(n, 4.0, 2.5, 3)
    for pat in (synth.pattern_A(), synth.random_partial_ktree(8, 3, 7)):
        check_tables(ctx, g, pat, oracle.colors(n, 2, pat[0], seed=8), pat[0])
    e = synth.csr_from_edges(n, np.zeros((0, 2), np.int64))
    check_tables(ctx, e, synth.pattern_A(), oracle.colors(n, 2, 9, seed=1), 9)


# few entries go into the forget's hash table, more than 2^18 of an introduce are sorted and
# reduced; a 3x3 grid's first forget keeps its order for the chained pair above it either way
@pytest.mark.parametrize("pat,n,deg,trials", [
    (("cycle", 5), 3, 2.0, 1), (("cycle", 5), 30, 6.0, 2), (("cycle", 5), 500, 7.0, 2),
    (("cycle", 5), 1300, 8.0, 3), (("grid", 2, 3), 700, 6.0, 3), (("grid", 2, 4), 2000, 7.0, 6),
    (("grid", 3, 3), 90, 7.0, 3), (("grid", 3, 3), 2500, 9.0, 4), (("path", 6), 9000, 5.0, 5)])
def test_forget_routes(ctx, pat, n, deg, trials):
    p = synth.make_pattern(pat)
    k = p[0] + 1
    check_tables(ctx, synth.erdos_renyi(n, min(1.0, deg / n), 3), p,
                 oracle.colors(n, trials, k, seed=5), k)


@pytest.mark.parametrize("trials", [2, 40])
def test_hubs(ctx, trials):
    """Stars of the degrees at which a candidate list leaves its window (65) and is cut into parts
    (256), and of one far beyond, joined in a path: lists in parts, runs of equal keys longer than
    a reduce block's tile and range, in hash tables (few trials) and sorted."""
    edges, at, centres = [], 0, []
    for d in (63, 64, 65, 255, 256, 257, 513, 6000):
        centres.append(at)
        edges += [(at, at + 1 + i) for i in range(d - 2 if 0 < len(centres) - 1 < 7 else d - 1)]
        at += d
    edges += list(zip(centres, centres[1:]))
    g = synth.csr_from_edges(at, np.array(edges))
    for pat in (synth.path_pattern(4), synth.star_pattern(4)):
        check_tables(ctx, g, pat, oracle.colors(at, trials, 5, seed=2), 5)


def hub_graph(n, seed):
    return synth.barabasi_albert(n, 4, seed)


# introduces run by run need 8 trials, more than 2^18 entries (planned) and two entries a pair: one
# trial too few, the fewest, several bytes of trials; leaf, introduce and forget children; pairs
# that share their mapping (hubs); 64- and 128-bit keys; a vertex forgotten as it comes; joins above
# (one trial is enough where nothing is forgotten); a vertex without a bag neighbour
@pytest.mark.parametrize("pat,n,hubs,trials,spare", [
    (("grid", 2, 4), 1500, 1, 7, 0), (("grid", 2, 4), 1500, 1, 8, 0),
    (("grid", 2, 4), 400, 1, 33, 1), (("grid", 3, 3), 2500, 0, 9, 0),
    (("grid", 3, 3), 70_000, 0, 8, 0), (("cycle", 4), 4000, 1, 16, 2),
    (("path", 5), 9000, 0, 12, 0), (("star", 5), 3000, 0, 40, 0), (("A",), 1200, 0, 10, 0),
    (("ktree", 7, 2, 5), 700, 1, 9, 0), (("A",), 5000, 0, 1, 0), (("D",), 230, 0, 9, 0)])
def test_run_wise_introduces(ctx, pat, n, hubs, trials, spare):
    p = synth.make_pattern(pat)
    k = p[0] + spare
    deg = 2.0 if n > 50_000 else 6.0
    g = hub_graph(n, 3) if hubs else synth.erdos_renyi(n, deg / n, 3)
    check_tables(ctx, g, p, oracle.colors(n, trials, k, seed=5), k)


def test_run_wise_masks_filter_and_enumeration(ctx):
    """Allowed mappings and no degree filter; the rows reconstructed through tables in two
    regions."""
    n, T = 1500, 24
    g = hub_graph(n, 5)
    pat = synth.cycle_pattern(4)
    z = oracle.colors(n, T, 4, seed=7)
    allow = np.random.default_rng(2).integers(0, 16, n).astype(np.uint32)
    cc.cc_load_graph(ctx.h, *g)
    cid = cc.cc_set_colors(ctx.h, z, 4)
    for masks, df in ((None, 1), (None, 0), (allow, 1)):
        ref = oracle.run_dp(g, pat, z, 4, degree_filter=bool(df), allow=masks)
        pid = cc.cc_load_pattern_masked(ctx.h, *pat, masks) if masks is not None else \
            cc.cc_load_pattern(ctx.h, *pat)
        N, _ = cc.cc_pattern_info(ctx.h, pid)
        want, total, _ = ref.enumerate(50_000)
        for rep in range(2):
            run = cc.cc_run_dp(ctx.h, pid, cid, cc.cc_default_opts(retain=1, degree_filter=df))
            assert np.array_equal(cc.cc_count(ctx.h, run, T), ref.count)
            assert np.array_equal(cc.cc_table_stats(ctx.h, run, N)[0], ref.node_sizes.sum(axis=0))
            rows, got = cc.cc_enumerate(ctx.h, run, 50_000, 4)
            assert got == total and np.array_equal(rows, want[:50_000])
            cc.cc_release(ctx.h, run)


def theta(n_mid):
    """Two vertices joined through n_mid middle ones: every middle vertex is the others' twin."""
    e = [(u, 2 + i) for i in range(n_mid) for u in (0, 1)]
    bags = [[0, 1, 2 + i] for i in range(n_mid)]
    return 2 + n_mid, np.array(e, np.int32), (bags, [i + 1 for i in range(n_mid - 1)] + [-1])


# an entry alone with its mapping and trial has no candidate when a forgotten vertex could have
# been the candidate's (4-cycles, theta graphs, the first square of a grid; chained in the 3x3
# grid), and may have one when not (5-cycles, a triangle with a tail)
@pytest.mark.parametrize("name", ["C4", "theta3", "theta4", "grid24", "grid33", "C5", "B"])
@pytest.mark.parametrize("trials", [2, 9])
def test_twin_rule(ctx, name, trials):
    pat = {"C4": synth.cycle_pattern(4), "theta3": theta(3), "theta4": theta(4),
           "grid24": synth.grid_pattern(2, 4), "grid33": synth.grid_pattern(3, 3),
           "C5": synth.cycle_pattern(5), "B": synth.pattern_B()}[name]
    n = 2600 if trials == 2 else 700
    g = hub_graph(n, 9) if name not in ("grid33", "C5", "B") else \
        synth.erdos_renyi(n, 9.0 / n, 9)
    check_tables(ctx, g, pat, oracle.colors(n, trials, pat[0], seed=5), pat[0])


# routes with scratch beside the tables (introduces run by run, joins group by group) and hubs, kept
# and not, from rooms that hold little more than the graph to ones that hold everything twice
@pytest.mark.parametrize("pat,n,trials", [(("grid", 2, 4), 1500, 9), (("A",), 4000, 1)])
@pytest.mark.parametrize("retain", [0, 1])
def test_every_arena_size(pat, n, trials, retain):
    """Whatever the room, a run (planned from exact runs, or exact) counts what the oracle does or
    ends with CC_ENOMEM; only a run that keeps its tables, or a slice too many, ever does."""
    p = synth.make_pattern(pat)
    g = hub_graph(n, 3)
    z = oracle.colors(n, trials, p[0], seed=5)
    ref = oracle.run_dp(g, p, z, p[0])
    fitted = 0
    mb = 2.0
    while mb < 1024:
        with cc.Context(arena_bytes=int(mb * 2 ** 20)) as c:
            cc.cc_load_graph(c.h, *g)
            pid = cc.cc_load_pattern(c.h, *p)
            cid = cc.cc_set_colors(c.h, z, p[0])
            opts = cc.cc_default_opts(retain=retain, max_slices=8)
            for _ in range(3):
                try:
                    run = cc.cc_run_dp(c.h, pid, cid, opts)
                except cc.CCError as ex:
                    assert ex.code == cc.CC_ENOMEM, mb
                    break
                assert np.array_equal(cc.cc_count(c.h, run, trials), ref.count), mb
                assert np.array_equal(cc.cc_decide(c.h, run, trials), ref.exists), mb
                cc.cc_release(c.h, run)
            else:
                fitted += 1
        mb *= 1.2
    assert fitted


# entries of a mapping that one pair leads to are counted and not written, in runs that keep no
# tables, where the introduce above is a twin of the vertex forgotten; not under masks or the
# distance bound; few and many mappings with several origins; exact, planned and captured runs
@pytest.mark.parametrize("name,n,hubs,trials,spare,opt", [
    ("C4", 4000, 1, 16, 2, {}), ("grid24", 1500, 1, 8, 0, {}), ("grid24", 400, 1, 33, 1, {}),
    ("grid24", 1500, 1, 9, 0, {"chain": 0}), ("grid33", 2500, 0, 9, 0, {}),
    ("grid33", 70_000, 0, 8, 0, {}), ("theta3", 2600, 1, 9, 0, {}), ("theta4", 700, 1, 9, 0, {}),
    ("C5", 1500, 0, 24, 0, {}), ("grid24", 1500, 1, 9, 0, {"distance_prune": 1}),
    ("grid24", 1500, 1, 9, 0, {"masks": 1})])
def test_dropped_entries(ctx, name, n, hubs, trials, spare, opt):
    pat = {"C4": synth.cycle_pattern(4), "theta3": theta(3), "theta4": theta(4),
           "grid24": synth.grid_pattern(2, 4), "grid33": synth.grid_pattern(3, 3),
           "C5": synth.cycle_pattern(5)}[name]
    k, opt = pat[0] + spare, dict(opt)
    masks = opt.pop("masks", 0)
    deg = 2.0 if n > 50_000 else 6.0
    g = hub_graph(n, 3) if hubs else synth.erdos_renyi(n, deg / n, 3)
    z = oracle.colors(n, trials, k, seed=5)
    allow = np.random.default_rng(2).integers(0, 1 << 8, n).astype(np.uint32) if masks else None
    ref = oracle.run_dp(g, pat, z, k, allow=allow,
                        distance_prune=bool(opt.get("distance_prune", 0)))
    cc.cc_load_graph(ctx.h, *g)
    pid = cc.cc_load_pattern_masked(ctx.h, *pat, allow) if masks else \
        cc.cc_load_pattern(ctx.h, *pat)
    N, _ = cc.cc_pattern_info(ctx.h, pid)
    cid = cc.cc_set_colors(ctx.h, z, k)
    for rep in range(4):
        run = cc.cc_run_dp(ctx.h, pid, cid, cc.cc_default_opts(use_graph=int(rep > 1), **opt))
        assert np.array_equal(cc.cc_count(ctx.h, run, trials), ref.count), rep
        assert np.array_equal(cc.cc_decide(ctx.h, run, trials), ref.exists), rep
        assert np.array_equal(cc.cc_table_stats(ctx.h, run, N)[0], ref.node_sizes.sum(axis=0)), rep
        cc.cc_release(ctx.h, run)
    cc.cc_release_colors(ctx.h, cid)


def launched(ctx, g, pat, z, k, **opt):
    """Per run (exact, planned): the (node, kernel kind) pairs it launched, with repeats, and the
    number of its kernel launches.  Counts and sizes are checked."""
    T = z.shape[0]
    ref = oracle.run_dp(g, pat, z, k)
    cc.cc_load_graph(ctx.h, *g)
    pid = cc.cc_load_pattern(ctx.h, *pat)
    N, _ = cc.cc_pattern_info(ctx.h, pid)
    cid = cc.cc_set_colors(ctx.h, z, k)
    out = []
    for mode in ("exact", "planned"):
        before = cc.cc_context_stats(ctx.h)[0]
        run = cc.cc_run_dp(ctx.h, pid, cid, cc.cc_default_opts(profile=1, **opt))
        launches = cc.cc_context_stats(ctx.h)[0] - before
        assert cc.cc_run_mode(ctx.h, run) == mode
        assert np.array_equal(cc.cc_count(ctx.h, run, T), ref.count)
        assert np.array_equal(cc.cc_table_stats(ctx.h, run, N)[0], ref.node_sizes.sum(axis=0))
        node, kind, _, _ = cc.cc_run_timings(ctx.h, run)
        out.append(([(x, cc.KERNEL_KINDS[k2]) for x, k2 in zip(node.tolist(), kind.tolist())],
                    launches))
        cc.cc_release(ctx.h, run)
    cc.cc_release_colors(ctx.h, cid)
    return out, ref.node_sizes.sum(axis=0), cc.cc_pattern_nodes(ctx.h, pid, pat[0])


@pytest.mark.parametrize("k,groups", [(13, True), (14, False)])
def test_join_route_at_its_limit(ctx, k, groups):
    """Eleven private colours are joined group by group, twelve through hash tables."""
    n, trials = 8000, 6
    made, sizes, nodes = launched(ctx, synth.erdos_renyi(n, 8 / n, 6), star_of_joins(4),
                                  oracle.colors(n, trials, k, seed=k), k)
    x, = [i for i, nd in enumerate(nodes) if nd[0] == cc.JOIN]
    assert sizes[nodes[x][1]] + sizes[nodes[x][2]] >= 1 << 21 and len(nodes[x][4]) == 2
    planned = made[1][0]  # only joins by groups count in planned runs
    assert ((x, "join_count") in planned) == groups
    assert (x, "join_write") in planned


@pytest.mark.parametrize("over", [0, 1])
def test_forget_route_at_its_limit(ctx, over):
    """2^18 entries are added into the forget's hash table, two more are sorted: a properly coloured
    ring, both ends of every edge."""
    n = (1 << 17) + over
    z = (np.arange(n) % 2).astype(np.uint8)[None]
    if over:
        z[0, -1] = 2
    made, sizes, nodes = launched(ctx, synth.cycle_graph(n), synth.path_pattern(3), z, 3)
    assert sizes[1] == 2 * n and nodes[2][0] == cc.FORGET
    for kinds, _ in made:
        assert ((1, "intro_fused") in kinds) == (not over)
        assert ((2, "sort") in kinds) == bool(over)


@pytest.mark.parametrize("trials", [7, 8])
def test_run_wise_route_at_its_limit(ctx, trials):
    """Eight colourings are taken run by run below a forget (four timed launches an introduce)."""
    made, sizes, nodes = launched(ctx, hub_graph(1500, 3), synth.grid_pattern(2, 4),
                                  oracle.colors(1500, trials, 8, seed=5), 8)
    planned = made[1][0]
    large = [x for x, nd in enumerate(nodes) if nd[0] == cc.INTRODUCE and sizes[x] > 1 << 20]
    assert large and any((planned.count((x, "intro_write")) == 4) == (trials == 8) for x in large)
    assert trials == 8 or all(planned.count((x, "intro_write")) <= 1 for x in large)


def test_hub_route_at_its_limit(ctx):
    """A largest degree of 65 takes each expanding introduce's second kernel, 64 does not."""
    launches = []
    for d in (64, 65):
        g = synth.csr_from_edges(4 * (d + 1), np.array(
            [(c * (d + 1), c * (d + 1) + 1 + i) for c in range(4) for i in range(d)]))
        made, _, nodes = launched(ctx, g, synth.path_pattern(3),
                                  oracle.colors(4 * (d + 1), 1, 3, seed=1), 3)
        launches.append(made[1][1])
    assert launches[1] - launches[0] == sum(nd[0] == cc.INTRODUCE for nd in nodes)


@pytest.mark.parametrize("pat,n,trials,k,long", [("star", 12_000, 7, 5, False), ("A", 4000, 3, 9, True)])
def test_join_route_by_group_length(ctx, pat, n, trials, k, long):
    """More than 2^21 entries are joined group by group where a group has many pairs to test, and
    through hash tables where it has few, exactly and planned; introduces that the join stores go run
    by run where its groups are long."""
    p = star_of_joins(4) if pat == "star" else synth.pattern_A()
    g = synth.erdos_renyi(n, 8 / n, 6) if pat == "star" else synth.barabasi_albert(n, 4, 3)
    made, sizes, nodes = launched(ctx, g, p, oracle.colors(n, trials, k, seed=k), k)
    joins = [x for x, nd in enumerate(nodes) if nd[0] == cc.JOIN
             and sizes[nd[1]] + sizes[nd[2]] > 1 << 21]
    assert joins
    planned = made[1][0]  # only joins by groups count in planned runs
    for x in joins:
        assert ((x, "join_count") in planned) == long
    stored = [y for x in joins for y in nodes[x][1:3] if nodes[y][0] == cc.INTRODUCE
              and sizes[y] > 1 << 20]
    assert stored
    for y in stored:
        assert planned.count((y, "intro_write")) == (4 if long else 1)


def test_no_chain_over_an_introduce(ctx):
    """Two introduces over one whose table run by run comes sorted are not chained."""
    n, trials, k = 4000, 28, 6
    p = synth.random_partial_ktree(5, 3, 207)
    made, sizes, nodes = launched(ctx, synth.power_law_config(n, 7.0, 2.5, 3), p,
                                  oracle.colors(n, trials, k, seed=5), k)
    assert [nd[0] for nd in nodes[:4]] == [cc.LEAF] + [cc.INTRODUCE] * 3 and sizes[1] > 1 << 18
    planned = made[1][0]
    assert planned.count((1, "intro_write")) == 4
    assert not any(kind == "intro_chain" for _, kind in planned)


def test_few_pairs_stored_entry_by_entry(ctx):
    """Stored introduces of few (run, candidate) pairs are not taken run by run, however many entries
    a pair stands for."""
    made, sizes, nodes = launched(ctx, hub_graph(500, 3), synth.pattern_B(),
                                  oracle.colors(500, 64, 7, seed=5), 7)
    planned = made[1][0]
    stored = [x for x, nd in enumerate(nodes) if nd[0] == cc.INTRODUCE and sizes[x] > 1 << 18
              and (x, "intro_write") in planned]
    assert stored
    assert all(planned.count((x, "intro_write")) == 1 for x in stored)


def test_small_first_runs_try_nothing(ctx):
    """An exact run that expects few entries counts them once: no runs or pairs are listed first."""
    pat = (4, np.array([(0, 1), (1, 2), (2, 3), (0, 3)], np.int32),
           ([[0, 2], [0, 1, 2], [0, 2, 3]], [-1, 0, 0]))
    made, sizes, nodes = launched(ctx, hub_graph(171, 3), pat, oracle.colors(171, 9, 4, seed=5), 4)
    exact = made[0][0]
    for x, nd in enumerate(nodes):
        if nd[0] == cc.INTRODUCE:
            assert sizes[x] < 1 << 17 and exact.count((x, "intro_count")) == 1


@pytest.mark.parametrize("n,deg", [(1100, 37.0), (60_000, 5.0)])
def test_join_by_sampled_groups(ctx, n, deg):
    """Eight colours for the 4-cycle of two paths: a group could hold many colour sets; an exact run
    samples whether it does (dense graph) or not (sparse)."""
    pat = (4, np.array([(0, 1), (1, 2), (2, 3), (0, 3)], np.int32),
           ([[0, 2], [0, 1, 2], [0, 2, 3]], [-1, 0, 0]))
    check_tables(ctx, synth.erdos_renyi(n, deg / n, 8), pat, oracle.colors(n, 2, 8, seed=8), 8)
