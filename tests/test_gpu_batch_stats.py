"""gc_stats of a batch call that asks for nothing else (no flags): the rounds are the largest of the batch
whether the small-graph kernel, the round kernel or both colored it."""
import ctypes

import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mix", [
    lambda: [gg.er(300 + i, 9.0, i) for i in range(30)],                                  # all small
    lambda: [gg.complete(90)] + [gg.er(300 + i, 9.0, i) for i in range(600)] + [gg.path(5000)],  # most rounds in a small one
    lambda: [gg.rmat(14, 12, 3), gg.er(5000, 60.0, 1)],                                   # none small
    lambda: [gg.empty(4)],
])
def test_rounds_without_flags(gclib, mix):
    import torch
    from paper_1509_08267_gb300 import _Options, _Stats, load
    gs = mix()
    b = gg.pack(gs)
    refs = [oracle.det(g, 3) for g in gs]
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (b.vtx_off, b.edge_off, b.rowptr, b.colidx)]
    out = torch.empty(int(b.vtx_off[-1]), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    st, opt = _Stats(), _Options()
    rounds = np.zeros(len(gs), np.int32)
    p = [a.data_ptr() if a.numel() else None for a in dev]
    rc = load().gc_color_batch_ex(len(gs), *p, 0, 3, out.data_ptr(), None, rounds.ctypes.data, ctypes.byref(opt),
                                  ctypes.byref(st))
    assert rc == 0
    assert list(rounds) == [r.rounds for r in refs]
    assert st.rounds == max(r.rounds for r in refs)
    assert st.ncolors == sum(r.ncolors for r in refs) and st.max_color == max(int(r.colors.max()) for r in refs)
    assert st.grid_blocks >= 1 and st.block_size == 256
