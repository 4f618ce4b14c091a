"""Which calls take the core phase: the statistics tell, beside results equal to the oracle's."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def _core_round(gclib, g, **kw):
    import torch
    ref = oracle.det(g, 5)
    rp, ci = torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(g.colidx).cuda()
    r = gclib.color(rp, ci, "det", 5, options=gclib.Options(**kw), stats=True)
    np.testing.assert_array_equal(r.colors.cpu().numpy(), ref.colors)
    assert (r.ncolors, r.rounds) == (ref.ncolors, ref.rounds)
    return r.stats.core_round


@pytest.mark.parametrize("make, hubs", [(lambda: gg.rmat(15, 12, 3), True), (lambda: gg.rmat(14, 40, 2), True),
                                        (lambda: gg.er(30000, 20.0, 3), False), (lambda: gg.stencil27(30), False)])
def test_graphs_with_a_row_past_the_thread_bound_take_it(gclib, make, hubs):
    g = make()
    assert _core_round(gclib, g) == (1 if hubs else 0)
    assert _core_round(gclib, g, core_vertices=g.n) == 1
    assert _core_round(gclib, g, core_vertices=g.n // 2) > 1
    assert _core_round(gclib, g, core_vertices=-1) == 0


def test_a_batch_takes_it(gclib):
    import torch
    b = gg.pack([gg.rmat(14, 12, 3), gg.er(9000, 60.0, 1)])
    args = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (b.vtx_off, b.edge_off, b.rowptr, b.colidx)]
    assert gclib.color_batch(*args, "det", 3, stats=True)[3].core_round == 1


def test_a_servers_pool_hands_over_in_early_and_late_rounds(gclib):
    g = gg.rmat(14, 12, 3)
    ref = oracle.det(g, 7)
    with gclib.Server(pool_vertices=g.n + 64, pool_entries=g.nnz + 64, mode="det") as srv:
        seen = []
        for k in range(6):
            colors, nc, rounds = srv.poll(srv.submit(g.rowptr, g.colidx, seed=7))
            np.testing.assert_array_equal(colors, ref.colors)
            assert (nc, rounds) == (ref.ncolors, ref.rounds)
            st = srv.stats()
            assert st["core_handovers"] == k + 1
            seen.append(st["core_round"])
    # the pool's round numbers go on from request to request: both sides of the fused first round's limit
    assert seen == sorted(set(seen)) and seen[0] <= 63 < seen[-1]


@pytest.mark.parametrize("make, core", [(lambda: gg.er(2000, 90.0, 3), True), (lambda: gg.er(16384, 66.0, 3), True),
                                        (lambda: gg.er(16385, 66.0, 3), False), (lambda: gg.er(16384, 60.0, 3), False)])
def test_small_graphs_of_long_rows_take_it(gclib, make, core):
    g = make()
    assert g.max_degree <= 127
    assert _core_round(gclib, g) == (1 if core else 0)
