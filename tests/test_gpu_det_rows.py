"""The deterministic mode's thread-per-row sweep at its edges: rows around multiples of the eight-entry
group, windows of one, two and four words (rounds up to 32, 64 and beyond), color 127, colidx arrays at
every alignment, keys whose digests tie, and malformed entries anywhere in a row -- against the CPU
oracle, with the core phase off so that every round runs in the round kernel."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def _at(colidx, offset):
    """colidx on the device, `offset` entries past an aligned address (views of a larger array)."""
    import torch
    buf = torch.full((len(colidx) + offset,), -7, dtype=torch.int32, device="cuda")
    buf[offset:] = torch.from_numpy(np.ascontiguousarray(colidx)).cuda()
    return buf[offset:]


GRAPHS = [lambda: gg.path(2), lambda: gg.cycle(9), lambda: gg.star(8), lambda: gg.star(9), lambda: gg.star(16),
          lambda: gg.complete(8), lambda: gg.complete(9), lambda: gg.complete(10), lambda: gg.complete(34),
          lambda: gg.complete(66), lambda: gg.complete(128), lambda: gg.stencil27(7), lambda: gg.grid5(31, 17),
          lambda: gg.er(3000, 20.0, 3), lambda: gg.rmat(12, 16, 4)]


@pytest.mark.parametrize("make", GRAPHS)
@pytest.mark.parametrize("offset", [0, 1, 4, 7])
def test_rows_match_oracle(gclib, make, offset):
    import torch
    g = make()
    ref = oracle.det(g, 5)
    rp = torch.from_numpy(np.ascontiguousarray(g.rowptr)).cuda()
    ci = _at(g.colidx, offset)
    for opt in (gclib.Options(core_vertices=-1), gclib.Options(core_vertices=-1, flags=gclib.FLAG_FULL_SWEEP),
                gclib.Options(core_vertices=-1, small_max_degree=9, chunk=32)):
        r = gclib.color(rp, ci, "det", 5, options=opt, stats=True)
        np.testing.assert_array_equal(r.colors.cpu().numpy(), ref.colors)
        assert (r.ncolors, r.rounds) == (ref.ncolors, ref.rounds)
        np.testing.assert_array_equal(r.stats.wl_size, ref.wl_size)
        assert (r.stats.round_reads <= r.stats.wl_degsum).all()


@pytest.mark.parametrize("priority", ["PRIORITY_LARGEST_FIRST", "PRIORITY_SMALLEST_LAST"])
def test_tied_digests(gclib, priority):
    # a mesh under a degree or level key: nearly all digests are equal, so the full keys decide
    import torch
    g = gg.stencil27(11)
    ref = oracle.det(g, 3, priority=getattr(oracle, priority))
    rp, ci = torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(g.colidx).cuda()
    r = gclib.color(rp, ci, "det", 3, options=gclib.Options(priority=getattr(gclib, priority), core_vertices=-1))
    np.testing.assert_array_equal(r.colors.cpu().numpy(), ref.colors)
    assert (r.ncolors, r.rounds) == (ref.ncolors, ref.rounds)


@pytest.mark.parametrize("bad", [-1, -2**31, 2**31 - 1, "n", "self"])
@pytest.mark.parametrize("where", [0, 3, 7, 8, 12])
def test_malformed_entry_is_reported(gclib, bad, where):
    import torch
    g = gg.complete(14)  # rows of 13 entries
    ci = g.colidx.copy()
    v = 5
    ci[g.rowptr[v] + where] = g.n if bad == "n" else v if bad == "self" else bad
    for opt in (gclib.Options(core_vertices=-1), gclib.Options(core_vertices=-1, flags=gclib.FLAG_FULL_SWEEP)):
        with pytest.raises(gclib.GCError) as e:
            gclib.color(torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(ci).cuda(), "det", 1, options=opt)
        assert e.value.status == gclib.GC_ERR_INVALID_GRAPH
