"""The core phase at the edges of its decomposition, against the oracle or a closed form: rows of one and
of several pieces (pieces hold 2,048 entries), more vertices of several pieces than a block takes at a
time, and colors past the 8-bit and past the 512-color window in rows of several pieces."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def _color(gclib, g, seed, **kw):
    import torch
    rp, ci = torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(g.colidx).cuda()
    return gclib.color(rp, ci, "det", seed, stats=True, **kw)


@pytest.mark.parametrize("n", [2049, 2050, 2200])
def test_clique_of_several_pieces(gclib, n):
    # K_n: the vertex of rank k in key order gets color k, in n rounds with worklists n, n-1, ..., 1
    g = gg.complete(n)
    order = np.lexsort((np.arange(n), oracle.keys(5, n)))
    want = np.empty(n, np.int32)
    want[order] = np.arange(n)
    for opt in (gclib.Options(), gclib.Options(tail_vertices=-1)):
        r = _color(gclib, g, 5, options=opt)
        np.testing.assert_array_equal(r.colors.cpu().numpy(), want)
        assert (r.ncolors, r.rounds) == (n, n)
        np.testing.assert_array_equal(r.stats.wl_size, np.arange(n, 0, -1))


def test_more_large_rows_than_a_block_takes_at_once(gclib):
    g = gg.er(10000, 2700.0, 3)
    assert np.diff(g.rowptr).min() > 2048
    ref = oracle.det(g, 7)
    r = _color(gclib, g, 7)
    np.testing.assert_array_equal(r.colors.cpu().numpy(), ref.colors)
    assert (r.ncolors, r.rounds) == (ref.ncolors, ref.rounds)
    np.testing.assert_array_equal(r.stats.wl_size, ref.wl_size)


@pytest.mark.parametrize("extra", [0, 1, 3, 2047, 2048, 2049])
def test_row_lengths_around_a_piece(gclib, extra):
    # a hub over a random graph: its row has 2,048 + extra entries in round 1
    base = gg.er(6000, 30.0, 9)
    hub = np.arange(1, 2049 + extra, dtype=np.int64)
    src = np.repeat(np.arange(base.n, dtype=np.int64), np.diff(base.rowptr))
    keep = (src != 0) & (base.colidx != 0)
    u = np.concatenate([src[keep], np.zeros(len(hub), np.int64), hub])
    v = np.concatenate([base.colidx[keep].astype(np.int64), hub, np.zeros(len(hub), np.int64)])
    key = np.unique(u * base.n + v)
    rowptr = np.searchsorted(key, np.arange(base.n + 1) * base.n).astype(np.int32)
    g = gg.Graph(base.n, rowptr, (key % base.n).astype(np.int32), "hub")
    ref = oracle.det(g, 4)
    r = _color(gclib, g, 4)
    np.testing.assert_array_equal(r.colors.cpu().numpy(), ref.colors)
    assert (r.ncolors, r.rounds) == (ref.ncolors, ref.rounds)
