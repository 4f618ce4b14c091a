"""The server's pool with the core phase: requests whose last rounds run in it, waves of requests after a
hand-over (the pool's round numbers go on, its counters start over), both sides of the 63-round limit of
the fused first core round, and a malformed request between them -- each result equal to the oracle's."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def test_waves_after_a_hand_over(gclib):
    waves = [[gg.rmat(13, 12, 1), gg.er(4000, 14.0, 2)], [gg.rmat(12, 16, 3)],
             [gg.er(9000, 8.0, 4), gg.rmat(14, 8, 5), gg.grid5(60, 50)], [gg.path(5)], [gg.rmat(13, 16, 6)]]
    total_n = sum(g.n for w in waves for g in w)
    total_m = sum(g.nnz for w in waves for g in w)
    with gclib.Server(pool_vertices=total_n, pool_entries=total_m, mode="det") as srv:
        for k in range(3):  # the same waves again, in a pool that has run
            for i, wave in enumerate(waves):
                ids = [srv.submit(g.rowptr, g.colidx, seed=7 + i) for g in wave]
                if i == 2:
                    bad = wave[0].colidx.copy()
                    bad[0] = wave[0].n
                    rid = srv.submit(wave[0].rowptr, bad)
                    with pytest.raises(gclib.GCError):
                        srv.poll(rid)
                for g, rid in zip(wave, ids):
                    colors, nc, rounds = srv.poll(rid)
                    ref = oracle.det(g, 7 + i)
                    np.testing.assert_array_equal(colors, ref.colors)
                    assert (nc, rounds) == (ref.ncolors, ref.rounds)
        assert srv.stats()["failed"] == 0


def test_default_without_large_rows_stays_in_the_round_kernel(gclib):
    # no row past 127 entries: the default leaves the core phase out; forcing it gives the same coloring
    import torch
    for g in (gg.er(30000, 20.0, 3), gg.stencil27(30)):
        rp, ci = torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(g.colidx).cuda()
        ref = oracle.det(g, 5)
        for opt in (None, gclib.Options(core_vertices=g.n), gclib.Options(core_vertices=-1)):
            r = gclib.color(rp, ci, "det", 5, options=opt)
            np.testing.assert_array_equal(r.colors.cpu().numpy(), ref.colors)
            assert (r.ncolors, r.rounds) == (ref.ncolors, ref.rounds)
