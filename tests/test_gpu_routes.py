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
