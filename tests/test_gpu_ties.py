"""Rows whose digests tie with a neighbour's: resolved by their own threads when many rows of a warp tie
(smallest last on grids and chains: neighbouring levels), by the warp when few do (stencil, hash key), with
colors past 126 and with malformed rows among them."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make", [lambda: gg.grid5(170, 101), lambda: gg.path(17001), lambda: gg.stencil27(27),
                                  lambda: gg.er(17000, 6.0, 1), lambda: gg.star(17000)])
@pytest.mark.parametrize("priority", [0, 2])
def test_ties(gclib, make, priority):
    import torch
    g = make()
    ref = oracle.det(g, 11, priority=priority)
    rp, ci = torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(g.colidx).cuda()
    r = gclib.color(rp, ci, "det", 11, options=gclib.Options(priority=priority, core_vertices=-1))
    np.testing.assert_array_equal(r.colors.cpu().numpy(), ref.colors)
    assert (r.ncolors, r.rounds) == (ref.ncolors, ref.rounds)


@pytest.mark.parametrize("k", [127, 128])
def test_equal_colors_up_to_the_largest_row(gclib, k):
    # rows of k - 1 entries: colors to 126 and to 127, where a state word saturates
    import torch
    g = gg.complete(k)
    ref = oracle.det(g, 3, priority=1)
    rp, ci = torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(g.colidx).cuda()
    r = gclib.color(rp, ci, "det", 3, options=gclib.Options(priority=1, core_vertices=-1))
    np.testing.assert_array_equal(r.colors.cpu().numpy(), ref.colors)


def test_self_loop_among_ties(gclib):
    import torch
    g = gg.grid5(170, 101)
    ci = g.colidx.copy()
    v = 9000
    ci[g.rowptr[v]] = v
    with pytest.raises(gclib.GCError) as e:
        gclib.color(torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(ci).cuda(), "det", 1,
                    options=gclib.Options(priority=1, core_vertices=-1))
    assert e.value.status == gclib.GC_ERR_INVALID_GRAPH
