"""Graphs of hundreds of colors, on both sides of the limits of every window and saturated color: 127 (the
16-bit states), 255 (the core's bytes) and 512 (the windows; the row is read again past them)."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def _rank(g, seed):
    order = np.lexsort((np.arange(g.n), oracle.keys(seed, g.n)))
    want = np.empty(g.n, np.int32)
    want[order] = np.arange(g.n)
    return want


@pytest.mark.parametrize("n", [128, 129, 130, 254, 255, 256, 257, 258, 300, 511, 512, 513, 514, 770, 1026])
@pytest.mark.parametrize("how", ["default", "no core", "no tail", "full sweep", "ordered"])
def test_cliques(gclib, n, how):
    # the vertex of rank k in key order gets color k
    import torch
    g = gg.complete(n)
    opt = {"default": gclib.Options(), "no core": gclib.Options(core_vertices=-1),
           "no tail": gclib.Options(tail_vertices=-1), "full sweep": gclib.Options(flags=gclib.FLAG_FULL_SWEEP),
           "ordered": gclib.Options()}[how]
    rp, ci = torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(g.colidx).cuda()
    r = gclib.color(rp, ci, "ordered" if how == "ordered" else "det", 5, options=opt)
    np.testing.assert_array_equal(r.colors.cpu().numpy(), _rank(g, 5))
    assert (r.ncolors, r.rounds) == (n, n)


def test_an_inplace_clique_past_512_colors(gclib):
    import torch
    g = gg.complete(900)
    r = gclib.color(torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(g.colidx).cuda(), "inplace", 5)
    assert sorted(r.colors.cpu().tolist()) == list(range(900))


@pytest.mark.parametrize("how", ["default", "no core", "no tail"])
@pytest.mark.parametrize("n, degree", [(900, 1250.0), (2100, 9000.0)])
def test_dense_random_graphs(gclib, n, degree, how):
    # rows of one and of several pieces, hundreds of colors, worklists of many vertices
    import torch
    g = gg.er(n, min(degree, n - 2.0), 3)
    ref = oracle.det(g, 9)
    opt = {"default": gclib.Options(), "no core": gclib.Options(core_vertices=-1),
           "no tail": gclib.Options(tail_vertices=-1)}[how]
    r = gclib.color(torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(g.colidx).cuda(), "det", 9, options=opt)
    np.testing.assert_array_equal(r.colors.cpu().numpy(), ref.colors)
    assert (r.ncolors, r.rounds) == (ref.ncolors, ref.rounds)


def test_a_late_core_with_final_neighbours_past_255(gclib):
    # the core takes over when 300 of 900 vertices are left: most colors around them are final already
    import torch
    g = gg.complete(900)
    for core in (600, 300, 20):
        r = gclib.color(torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(g.colidx).cuda(), "det", 5,
                        options=gclib.Options(core_vertices=core, tail_vertices=-1))
        np.testing.assert_array_equal(r.colors.cpu().numpy(), _rank(g, 5))


def test_served_cliques(gclib):
    g = gg.complete(600)
    with gclib.Server(pool_vertices=2000, pool_entries=g.nnz * 2 + 64, mode="det") as srv:
        for _ in range(3):
            ids = [srv.submit(g.rowptr, g.colidx, seed=s) for s in (5, 6)]
            for s, rid in zip((5, 6), ids):
                colors, nc, rounds = srv.poll(rid)
                np.testing.assert_array_equal(colors, _rank(g, s))
                assert (nc, rounds) == (600, 600)
