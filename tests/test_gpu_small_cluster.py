"""A small single graph on a cluster: round 1's results replace the initial states in the exchange
buffers whatever order the block's threads run in -- many calls in a row, each equal to the oracle's."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make", [lambda: gg.er(2049, 6.0, 1), lambda: gg.er(16384, 30.0, 2), lambda: gg.cycle(16001),
                                  lambda: gg.rmat(13, 12, 3)])
def test_every_call_gives_the_oracles_colors(gclib, make):
    import torch
    g = make()
    rp, ci = torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(g.colidx).cuda()
    for seed in range(4):
        ref = oracle.det(g, seed)
        want = torch.from_numpy(np.ascontiguousarray(ref.colors)).cuda()
        for _ in range(50):
            r = gclib.color(rp, ci, "det", seed)
            assert torch.equal(r.colors, want) and (r.ncolors, r.rounds) == (ref.ncolors, ref.rounds)
