"""The core phase from several threads at once: two servers with pools of different sizes (their core
kernels are launched with different amounts of shared memory) beside batch and single calls -- every
result equal to the oracle's, no request failed."""
import threading

import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def test_core_phase_from_four_threads(gclib):
    import torch
    big, small = gg.rmat(16, 12, 1), gg.rmat(11, 16, 2)
    pair = [gg.rmat(12, 16, 3), gg.rmat(15, 8, 4)]
    refs = {id(g): oracle.det(g, 7) for g in [big, small] + pair}
    b = gg.pack(pair)
    args = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (b.vtx_off, b.edge_off, b.rowptr, b.colidx)]
    rp, ci = torch.from_numpy(big.rowptr).cuda(), torch.from_numpy(big.colidx).cuda()
    torch.cuda.synchronize()
    errors = []

    def check(g, colors, nc, rounds):
        ref = refs[id(g)]
        assert np.array_equal(colors, ref.colors) and (nc, rounds) == (ref.ncolors, ref.rounds)

    def serve(g):
        with gclib.Server(pool_vertices=g.n + 64, pool_entries=g.nnz + 64, mode="det") as srv:
            for _ in range(60):
                check(g, *srv.poll(srv.submit(g.rowptr, g.colidx, seed=7)))
            assert srv.stats()["failed"] == 0

    def batches():
        for _ in range(60):
            colors, nc, rd = gclib.color_batch(*args, "det", 7)
            colors = colors.cpu().numpy()
            for i, g in enumerate(pair):
                check(g, colors[b.vtx_off[i]:b.vtx_off[i + 1]], int(nc[i]), int(rd[i]))

    def singles():
        for _ in range(60):
            r = gclib.color(rp, ci, "det", 7)
            check(big, r.colors.cpu().numpy(), r.ncolors, r.rounds)

    def run(f, *a):
        try:
            f(*a)
        except BaseException as e:  # noqa: BLE001 (reported below, from the main thread)
            errors.append(e)

    threads = [threading.Thread(target=run, args=a) for a in [(serve, big), (serve, small), (batches,), (singles,)]]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
