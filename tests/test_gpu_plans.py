"""What a plan remembers: whether later runs of its key go the same way whatever colouring or room the
first ones had.  Results are whole numbers, compared for equality."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

cc = pytest.importorskip("paper_1908_11248_gb300")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()


def five_layers(size, deg, seed):
    """Five layers in a ring, every vertex with `deg` neighbours in the layer on either side: coloured
    by layer, half of an entry's candidates have a free colour."""
    rng = np.random.default_rng(seed)
    at, edges = np.arange(size), []
    for a in range(5):
        to = rng.permutation(size)
        for shift in rng.choice(size, deg, replace=False):
            edges.append(np.stack([a * size + at, (a + 1) % 5 * size + to[(at + shift) % size]], 1))
    return synth.csr_from_edges(5 * size, np.concatenate(edges))


def test_planned_when_pairs_yield_about_two_entries():
    """Two colourings of one key, one just below the two entries a (run, candidate) pair at which
    introduces are taken run by run and one at it: once planned, every run is."""
    size, trials = 2000, 8
    g = five_layers(size, 4, 1)
    layer = np.repeat(np.arange(5), size).astype(np.uint8)
    full = np.zeros((trials, 5 * size), np.uint8)
    full[:4] = layer
    fewer = full.copy()
    fewer[0, :200] = 4  # some of the first layer coloured as the last
    pat = synth.cycle_pattern(5)
    want = {w: oracle.run_dp(g, pat, z, 5) for w, z in (("full", full), ("fewer", fewer))}
    with cc.Context(arena_bytes=8 << 30) as c:
        cc.cc_load_graph(c.h, *g)
        pid = cc.cc_load_pattern(c.h, *pat)
        N, _ = cc.cc_pattern_info(c.h, pid)
        ids = {"full": cc.cc_set_colors(c.h, full, 5), "fewer": cc.cc_set_colors(c.h, fewer, 5)}
        modes = []
        for w in ("fewer", "full", "fewer", "fewer", "full"):
            run = cc.cc_run_dp(c.h, pid, ids[w], cc.cc_default_opts())
            modes.append(cc.cc_run_mode(c.h, run))
            assert np.array_equal(cc.cc_count(c.h, run, trials), want[w].count)
            assert np.array_equal(cc.cc_table_stats(c.h, run, N)[0],
                                  want[w].node_sizes.sum(axis=0))
            cc.cc_release(c.h, run)
        assert modes == ["exact"] + ["planned"] * 4


def candidates(g, pattern, ref, trials, nodes):
    """Per introduce of a vertex with one bag neighbour: the candidates examined when they are taken
    entry by entry, and when they are taken once for all entries of a mapping."""
    degree, out = np.diff(g[0]), {}
    for x, nd in enumerate(nodes):
        if nd[0] != cc.INTRODUCE:
            continue
        bag = nodes[nd[1]][4]
        near = [s for s, w in enumerate(bag)
                if any({w, nd[3]} == set(e) for e in np.asarray(pattern[1]).tolist())]
        if len(near) == 1:
            phi = np.concatenate([np.reshape(ref.table(t, nd[1], len(bag))[0], (-1, len(bag)))
                                  for t in range(trials)])
            out[x] = (int(degree[phi[:, near[0]]].sum()),
                      int(degree[np.unique(phi, axis=0)[:, near[0]]].sum()))
    return out


def kinds(c, pid, cid, trials, want, cand, **opt):
    """Mode of a run and the (node, kernel kind) list of its launches; its counts are checked, and
    that its candidates are those of one way to take them."""
    run = cc.cc_run_dp(c.h, pid, cid, cc.cc_default_opts(profile=1, max_slices=8, **opt))
    assert np.array_equal(cc.cc_count(c.h, run, trials), want.count)
    mode = cc.cc_run_mode(c.h, run)
    node, kind, _, seen = cc.cc_run_timings(c.h, run)
    chained = set(node[kind == cc.KERNEL_KINDS.index("intro_chain")].tolist())
    for x, v in zip(node.tolist(), seen.tolist()):
        assert v == 0 or x not in cand or x in chained or v in cand[x], (x, v, cand[x])
    cc.cc_release(c.h, run)
    return mode, list(zip(node.tolist(), kind.tolist()))


# many colourings: introduces run by run, which hold pairs beside the tables, and (in the partial
# 2-tree, where most mappings have several origins) more than the entry kernels would; one: forgets
# of few entries, whose hash tables are larger than sorted records
@pytest.mark.parametrize("pat,n,trials,retain,room_mb", [
    (("grid", 2, 4), 1500, 9, 0, 1024), (("ktree", 7, 2, 5), 700, 9, 0, 512),
    (("A",), 4000, 1, 1, 1024), (("path", 8), 3000, 1, 1, 128)])
def test_little_room_once_is_not_remembered(pat, n, trials, retain, room_mb):
    """A key whose first runs had only part of the arena (another colouring held the rest) runs, once
    that is given back, by the same kernels as a key that had all of it from the start."""
    p = synth.make_pattern(pat)
    g = synth.barabasi_albert(n, 4, 3) if pat[0] != "path" else synth.erdos_renyi(n, 6 / n, 3)
    z = oracle.colors(n, trials, p[0], seed=5)
    want = oracle.run_dp(g, p, z, p[0])
    with cc.Context(arena_bytes=room_mb << 20) as c:
        cc.cc_load_graph(c.h, *g)
        cid = cc.cc_set_colors(c.h, z, p[0])
        pid = cc.cc_load_pattern(c.h, *p)
        cand = candidates(g, p, want, trials, cc.cc_pattern_nodes(c.h, pid, p[0]))
        for _ in range(2):
            ref = kinds(c, pid, cid, trials, want, cand, retain=retain)
        assert ref[0] == "planned"
        _, used, size = cc.cc_context_stats(c.h)
        left, tight = size - used, 0
        while left > 4 << 20:
            left = int(left / 1.07)
            used = cc.cc_context_stats(c.h)[1]
            held = cc.cc_color(c.h, 1, (size - used - left) // n, p[0])
            pid = cc.cc_load_pattern(c.h, *p)  # a key of its own
            try:
                first = [kinds(c, pid, cid, trials, want, cand, retain=retain) for _ in range(2)]
            except cc.CCError as ex:
                assert ex.code == cc.CC_ENOMEM
                first = [("none", [])]
            cc.cc_release_colors(c.h, held)
            if first[0][0] == "exact":
                tight += first[-1] != ref
                for _ in range(3):
                    last = kinds(c, pid, cid, trials, want, cand, retain=retain)
                assert last == ref, left >> 20
        assert tight


def test_graphs_give_way_before_routes():
    """A run whose tables fit only without the routes that hold memory beside them, while a captured
    graph holds some, takes the graph's memory and keeps the routes."""
    p, n = synth.path_pattern(8), 3000
    g = synth.erdos_renyi(n, 6 / n, 3)
    z = oracle.colors(n, 1, 8, seed=5)
    want = oracle.run_dp(g, p, z, 8)
    with cc.Context(arena_bytes=256 << 20) as c:
        cc.cc_load_graph(c.h, *g)
        cid = cc.cc_set_colors(c.h, z, 8)
        ref = kinds(c, cc.cc_load_pattern(c.h, *p), cid, 1, want, {}, retain=1)
        other = cc.cc_load_pattern(c.h, *synth.path_pattern(6))
        many = cc.cc_color(c.h, 2, 8, 6)
        for mode in ("exact", "graph"):
            run = cc.cc_run_dp(c.h, other, many, cc.cc_default_opts(use_graph=1))
            assert cc.cc_run_mode(c.h, run) == mode
            cc.cc_release(c.h, run)
        _, used, size = cc.cc_context_stats(c.h)
        # (kept tables fit 19 MB without those routes and 23 MB with them)
        cc.cc_color(c.h, 1, (size - used - (41 << 19)) // n, 8)
        assert kinds(c, cc.cc_load_pattern(c.h, *p), cid, 1, want, {}, retain=1) == ref


def test_kept_tables_do_not_slow_runs_that_keep_none():
    """Kept tables fit only without the routes that hold memory beside them; runs of the same key that
    keep none do not go without."""
    p, n = synth.path_pattern(8), 3000
    g = synth.erdos_renyi(n, 6 / n, 3)
    z = oracle.colors(n, 1, 8, seed=5)
    want = oracle.run_dp(g, p, z, 8)
    with cc.Context(arena_bytes=256 << 20) as c:
        cc.cc_load_graph(c.h, *g)
        cid = cc.cc_set_colors(c.h, z, 8)
        _, used, size = cc.cc_context_stats(c.h)
        cc.cc_color(c.h, 1, (size - used - (41 << 19)) // n, 8)
        alone, both = cc.cc_load_pattern(c.h, *p), cc.cc_load_pattern(c.h, *p)
        for _ in range(2):
            ref = kinds(c, alone, cid, 1, want, {})
        assert ref[0] == "planned"
        kept = kinds(c, both, cid, 1, want, {}, retain=1)
        assert kept[0] == "exact" and kept[1] != kinds(c, alone, cid, 1, want, {})[1]
        assert kinds(c, both, cid, 1, want, {}) == ref


# the six-cycle: one introduce that is expected to yield just more than two entries a pair and yields
# just fewer, one that is expected to yield fewer; the partial 2-tree: most mappings have several origins
@pytest.mark.parametrize("pat,n,hubs,trials", [(("cycle", 6), 1500, 0, 8),
                                               (("ktree", 7, 2, 5), 700, 1, 9)])
def test_exact_runs_write_what_they_count(pat, n, hubs, trials):
    """An exact run lists and counts a node's (run, candidate) pairs, or sorts them, only where it also
    writes their entries: nothing is counted for the entry kernels to do again."""
    p = synth.make_pattern(pat)
    g = synth.barabasi_albert(n, 4, 3) if hubs else synth.erdos_renyi(n, 8 / n, 3)
    z = oracle.colors(n, trials, p[0], seed=100)
    want = oracle.run_dp(g, p, z, p[0])
    with cc.Context(arena_bytes=8 << 30) as c:
        cc.cc_load_graph(c.h, *g)
        pid = cc.cc_load_pattern(c.h, *p)
        N, _ = cc.cc_pattern_info(c.h, pid)
        nodes = cc.cc_pattern_nodes(c.h, pid, p[0])
        cid = cc.cc_set_colors(c.h, z, p[0])
        for mode in ("exact", "planned"):
            run = cc.cc_run_dp(c.h, pid, cid, cc.cc_default_opts(profile=1))
            assert cc.cc_run_mode(c.h, run) == mode
            assert np.array_equal(cc.cc_count(c.h, run, trials), want.count)
            assert np.array_equal(cc.cc_table_stats(c.h, run, N)[0], want.node_sizes.sum(axis=0))
            node, kind, _, _ = cc.cc_run_timings(c.h, run)
            cc.cc_release(c.h, run)
            if mode == "planned":
                break
            made = {(x, cc.KERNEL_KINDS[k]): int(((node == x) & (kind == k)).sum())
                    for x, k in zip(node.tolist(), kind.tolist())}
            for f, nd in enumerate(nodes):
                if nd[0] == cc.FORGET and nodes[nd[1]][0] == cc.INTRODUCE:
                    # pairs and side entries are sorted and reduced; else at most the runs are listed
                    # before the entries are counted
                    sorts, reduces = made.get((f, "sort"), 0), made.get((f, "reduce"), 0)
                    assert sorts == reduces, f
                    assert made.get((nd[1], "intro_count"), 0) <= (3 if sorts == 2 else 2), f


def test_join_without_room_to_sort():
    """A join of a large unsorted child with a small one (allowed mappings) where sorting the large one
    does not fit: it goes through hash tables, whose need is the small child's, in the same run."""
    n, trials, k = 16_000, 7, 6
    nF, edges, _ = synth.star_pattern(4)
    pat = nF, edges, ([[0, i] for i in range(1, 4)], [-1, 0, 0])
    g = synth.erdos_renyi(n, 8 / n, 6)
    z = oracle.colors(n, trials, k, seed=5)
    allow = np.full(n, 0b1011, np.uint32)
    allow[::1000] |= 0b0100  # vertex 2 on a few host vertices
    want = oracle.run_dp(g, pat, z, k, allow=allow)
    with cc.Context(arena_bytes=1 << 30) as c:
        cc.cc_load_graph(c.h, *g)
        cid = cc.cc_set_colors(c.h, z, k)
        pid = cc.cc_load_pattern_masked(c.h, *pat, allow)
        nodes = cc.cc_pattern_nodes(c.h, pid, nF)
        join = [x for x, nd in enumerate(nodes) if nd[0] == cc.JOIN]
        assert len(join) == 1
        sizes = want.node_sizes.sum(axis=0)
        large = max(int(sizes[nodes[join[0]][1]]), int(sizes[nodes[join[0]][2]]))
        assert large > 1 << 21
        _, used, size = cc.cc_context_stats(c.h)
        hashed, was_planned = 0, True
        parts = list(range(60, 19, -2))  # the room in tenths of the large table's records
        pids = [cc.cc_load_pattern_masked(c.h, *pat, allow) for _ in parts]  # a key each
        for part, pid in zip(parts, pids):
            left = 16 * large * part // 10
            used = cc.cc_context_stats(c.h)[1]
            held = cc.cc_color(c.h, 1, (size - used - left) // n, k)
            for rep in range(4):
                run = cc.cc_run_dp(c.h, pid, cid, cc.cc_default_opts(profile=1))
                mode = cc.cc_run_mode(c.h, run)
                assert np.array_equal(cc.cc_count(c.h, run, trials), want.count)
                assert np.array_equal(cc.cc_table_stats(c.h, run, len(nodes))[0], sizes)
                node, kind, _, _ = cc.cc_run_timings(c.h, run)
                cc.cc_release(c.h, run)
                assert mode in ("exact", "planned"), part
                groups = (node == join[0]) & (kind == cc.KERNEL_KINDS.index("join_count"))
                hashed += mode == "planned" and not groups.any()
            assert was_planned or mode == "exact", part  # planned down to some room
            was_planned = mode == "planned"
            cc.cc_release_colors(c.h, held)
        assert hashed


def test_what_fits_exactly_goes_on_fitting():
    """In every room in which a key's first run fits, its later ones do, though the planned
    capacities may not (kept tables of three joins: by groups they fit, as hash tables they would
    not)."""
    p, n, trials = synth.make_pattern(("A",)), 4000, 3
    g = synth.barabasi_albert(n, 4, 3)
    z = oracle.colors(n, trials, 9, seed=5)
    want = oracle.run_dp(g, p, z, 9)
    fitted = 0
    with cc.Context(arena_bytes=1024 << 20) as c:
        cc.cc_load_graph(c.h, *g)
        cid = cc.cc_set_colors(c.h, z, 9)
        size, left = cc.cc_context_stats(c.h)[2], 560 << 20
        while left > 320 << 20:
            left = int(left / 1.03)
            held = cc.cc_color(c.h, 1, (size - cc.cc_context_stats(c.h)[1] - left) // n, 9)
            pid = cc.cc_load_pattern(c.h, *p)
            for rep in range(3):
                try:
                    run = cc.cc_run_dp(c.h, pid, cid, cc.cc_default_opts(retain=1))
                except cc.CCError as ex:
                    assert ex.code == cc.CC_ENOMEM and rep == 0, (left >> 10, rep)
                    break
                fitted += 1
                assert np.array_equal(cc.cc_count(c.h, run, trials), want.count)
                cc.cc_release(c.h, run)
            cc.cc_release_colors(c.h, held)
    assert fitted


@pytest.mark.parametrize("retain", [0, 1])
@pytest.mark.parametrize("pat", [("A",), ("cycle", 5)])
def test_run_that_does_not_fit_is_tried_once(pat, retain):
    """A single trial too large for the room (and not to be sliced) ends with CC_ENOMEM after one
    attempt; a second one is made only where what the first held beside its tables is what it
    lacked, which is rare."""
    p = synth.make_pattern(pat)
    n = 20_000
    g = synth.barabasi_albert(n, 4, 3)
    z = oracle.colors(n, 1, p[0], seed=5)
    opts = cc.cc_default_opts(retain=retain, max_slices=1)
    full, spent = 0, []
    mb = 4096.0
    while mb > 8:
        with cc.Context(arena_bytes=int(mb * 2 ** 20)) as c:
            cc.cc_load_graph(c.h, *g)
            pid = cc.cc_load_pattern(c.h, *p)
            cid = cc.cc_set_colors(c.h, z, p[0])
            before = cc.cc_context_stats(c.h)[0]
            try:
                cc.cc_run_dp(c.h, pid, cid, opts)
                full = full or cc.cc_context_stats(c.h)[0] - before
            except cc.CCError as ex:
                assert ex.code == cc.CC_ENOMEM
                spent.append(cc.cc_context_stats(c.h)[0] - before)
        mb /= 1.2
    assert full and spent
    assert np.mean([s > full for s in spent]) < 0.25, (full, spent)


@pytest.mark.parametrize("limit", [0, 50])
def test_served_in_little_room(limit):
    """Queries of one key under budgets from one that holds its tables twice down to one that does not
    hold them: the oracle's counts (whole, or in slices), or CC_ENOMEM for kept tables."""
    p, n = synth.path_pattern(8), 3000
    g = synth.erdos_renyi(n, 6 / n, 3)
    want = [oracle.run_dp(g, p, oracle.colors(n, 1, 8, seed=s), 8) for s in range(3)]
    first = want[0].enumerate(limit)[0][:limit] if limit else None
    whole = 0
    with cc.Context(arena_bytes=256 << 20) as c:
        cc.cc_load_graph(c.h, *g)
        budget = 48 << 20
        while budget > 12 << 20:
            pid = cc.cc_load_pattern(c.h, *p)  # a key of its own
            cc.cc_serve_start(c.h, budget, 2)
            try:
                for s in (0, 1, 2, 0):
                    ticket = cc.cc_serve_submit(c.h, pid, s, 1, 8, limit)
                    done = False
                    while not done:
                        done, status, counts, _, _, rows = cc.cc_serve_poll(c.h, ticket, 1, limit, 8)
                    if status:
                        assert limit and status == cc.CC_ENOMEM, budget
                        continue
                    assert np.array_equal(counts, want[s].count), budget
                    if limit and s == 0:
                        assert np.array_equal(rows, first), budget
                whole += cc.cc_serve_stats(c.h)["sliced"] == 0 and not status
            finally:
                cc.cc_serve_stop(c.h)
            budget = int(budget / 1.08)
    assert whole
