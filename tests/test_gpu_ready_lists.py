"""Ordered mode and peeling with nearly all vertices ready in one round: the small ones fill the round's
array from the front, the medium-degree ones from the back."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def _hubs(leaves, mids, width):
    """Disjoint: a star of `leaves` leaves, and `mids` vertices joined to the same `width` hubs."""
    star = np.stack([np.zeros(leaves, np.int64), np.arange(1, leaves + 1)])
    h0 = leaves + 1
    m = np.arange(mids).repeat(width) + h0 + width
    h = np.tile(np.arange(width), mids) + h0
    src = np.concatenate([star[0], m])
    dst = np.concatenate([star[1], h])
    return gg.from_pairs(leaves + 1 + width + mids, src, dst)


@pytest.mark.parametrize("leaves, mids, width", [(5000, 5000, 9), (1, 9000, 32), (9000, 1, 16), (4097, 4095, 17), (3, 2, 9)])
def test_nearly_all_ready_at_once(gclib, leaves, mids, width):
    import torch
    g = _hubs(leaves, mids, width)
    rp, ci = torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(g.colidx).cuda()
    for prio in (gclib.PRIORITY_HASH, gclib.PRIORITY_LARGEST_FIRST, gclib.PRIORITY_SMALLEST_LAST):
        r = gclib.color(rp, ci, "ordered", 7, options=gclib.Options(priority=prio))
        np.testing.assert_array_equal(r.colors.cpu().numpy(), oracle.greedy_keyorder(g, 7, prio)[0])
    level, _, degen = gclib.smallest_last(rp, ci)
    ref, k = oracle.peel_levels(g)
    np.testing.assert_array_equal(level.cpu().numpy(), ref)
    assert degen == k


def test_a_batch_of_them(gclib):
    import torch
    gs = [_hubs(300, 300, 9), _hubs(40, 900, 32), gg.empty(3), _hubs(900, 2, 12)]
    b = gg.pack(gs)
    args = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (b.vtx_off, b.edge_off, b.rowptr, b.colidx)]
    colors = gclib.color_batch(*args, "ordered", 7, options=gclib.Options(priority=1))[0].cpu().numpy()
    for i, g in enumerate(gs):
        np.testing.assert_array_equal(colors[b.vtx_off[i]:b.vtx_off[i + 1]], oracle.greedy_keyorder(g, 7, 1)[0])


def test_scratch_of_the_ordered_mode(gclib):
    # state words (16 bytes a vertex), worklists (4 and 2 x 16), and what a coloring of any mode keeps
    import torch
    n = 4_000_000
    rp = torch.arange(0, 2 * n + 1, 2, dtype=torch.int32, device="cuda")
    v = torch.arange(n, dtype=torch.int32, device="cuda")
    ci = torch.stack([(v + 1) % n, (v - 1) % n], 1).reshape(-1).contiguous()
    gclib.release_scratch()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    gclib.color(rp, ci, "ordered", 1, out=torch.empty(n, dtype=torch.int32, device="cuda"))
    used = free0 - torch.cuda.mem_get_info()[0] - 4 * n
    gclib.release_scratch()
    assert used < 58 * n + (32 << 20)  # (allocations are rounded up to 2 MB)
