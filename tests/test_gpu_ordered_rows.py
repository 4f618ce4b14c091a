"""Ordered mode, recoloring and peeling at the edges of their row classes against the oracle: rows one
lane, one warp or a whole block counts (32 / 33, 4,096 / 4,097 entries), more long rows than a block
keeps at a time, rows of one thread, an 8-lane group and one or several work items."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def _bipartite(a, b):
    u = np.repeat(np.arange(a), b)
    v = a + np.tile(np.arange(b), a)
    rows, cols = np.concatenate([u, v]), np.concatenate([v, u])
    order = np.lexsort((cols, rows))
    rowptr = np.searchsorted(rows[order], np.arange(a + b + 1)).astype(np.int32)
    return gg.Graph(a + b, rowptr, cols[order].astype(np.int32), f"K_{a},{b}")


def _dev(g):
    import torch
    return torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(g.colidx).cuda()


GRAPHS = [lambda: gg.star(9), lambda: gg.star(10), lambda: gg.star(33), lambda: gg.star(34), lambda: gg.star(66),
          lambda: gg.star(4097), lambda: gg.star(4098), lambda: gg.star(9000), lambda: _bipartite(200, 4200),
          lambda: _bipartite(65, 33), lambda: gg.complete(700), lambda: gg.rmat(13, 16, 2), lambda: gg.stencil27(8)]


@pytest.mark.parametrize("make", GRAPHS)
@pytest.mark.parametrize("priority", [0, 1])
def test_ordered_rows(gclib, make, priority):
    g = make()
    want = oracle.greedy_keyorder(g, 6, priority)[0]
    depth, rounds = oracle.keyorder_depth(g, 6, priority)
    r = gclib.color(*_dev(g), "ordered", 6, options=gclib.Options(priority=priority))
    np.testing.assert_array_equal(r.colors.cpu().numpy(), want)
    assert r.rounds == max(1, rounds)


@pytest.mark.parametrize("make", GRAPHS)
def test_recolor_and_levels(gclib, make):
    g = make()
    rp, ci = _dev(g)
    before = oracle.greedy(g)
    before = before[0] if isinstance(before, tuple) else before
    r = gclib.recolor(rp, ci, np.asarray(before, np.int32), 8)
    want = oracle.greedy_keyorder(g, 8, oracle.PRIORITY_RECOLOR, np.asarray(before, np.int32))[0]
    np.testing.assert_array_equal(r.colors.cpu().numpy(), want)
    level, _, degeneracy = gclib.smallest_last(rp, ci)
    ref, k = oracle.peel_levels(g)
    np.testing.assert_array_equal(level.cpu().numpy(), ref)
    assert degeneracy == k


@pytest.mark.parametrize("n", [40, 5000])
def test_malformed_long_row(gclib, n):
    import torch
    g = gg.star(n)
    for bad in (g.n, -1, 0):  # past the vertices, negative, the hub itself
        ci = g.colidx.copy()
        hub = int(np.argmax(np.diff(g.rowptr)))
        ci[g.rowptr[hub] + n // 2] = hub if bad == 0 else bad
        with pytest.raises(gclib.GCError) as e:
            gclib.color(torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(ci).cuda(), "ordered", 1)
        assert e.value.status == gclib.GC_ERR_INVALID_GRAPH
