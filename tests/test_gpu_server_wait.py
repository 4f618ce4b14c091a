"""Requests that arrive while the resident batch is in the core phase: the core leaves its rounds for them, and
what was left goes on from the worklist -- colors, counts and rounds as the oracle's."""
import time

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


@pytest.mark.parametrize("mode", ["det", "inplace", "solo"])
def test_a_small_request_does_not_wait_for_the_batch(gclib, mode):
    big, small = gg.complete(2500), gg.er(3000, 20.0, 1)  # 2,500 rounds, some 200 ms
    ref = oracle.det(small, 3)
    with gclib.Server(pool_vertices=8000, pool_entries=big.nnz + small.nnz + 64, mode="det",
                      solo_entries=small.nnz if mode == "solo" else -1) as srv:
        if mode == "solo":  # (the clique must not be one)
            big = gg.complete(240)
        # (the first requests of a mode and size allocate, which waits for running kernels)
        srv.poll(srv.submit(small.rowptr, small.colidx, mode="inplace" if mode == "inplace" else "det", seed=1))
        srv.poll(srv.submit(big.rowptr, big.colidx, seed=1))
        a = srv.submit(big.rowptr, big.colidx, seed=5)
        time.sleep(0.05)  # the clique is in the core phase by now
        b = srv.submit(small.rowptr, small.colidx, seed=3, mode="inplace" if mode == "inplace" else "det")
        colors, nc, rounds = srv.poll(b)
        if mode != "solo":
            assert srv.poll(a, timeout_ms=0) is None  # the batch is not done
        if mode != "inplace":
            np.testing.assert_array_equal(colors, ref.colors)
            assert (nc, rounds) == (ref.ncolors, ref.rounds)
        colors, nc, rounds = srv.poll(a)
        np.testing.assert_array_equal(colors, _rank(big, 5))
        assert (nc, rounds) == (big.n, big.n)
        st = srv.stats()
        assert st["failed"] == 0
        if mode != "solo":
            assert st["core_handovers"] >= 2  # it left, and took over again


def test_the_first_requests_do_not_wait_either(gclib):
    # what a first submit sets up waits for running kernels
    big, small = gg.complete(2500), gg.er(3000, 20.0, 1)
    with gclib.Server(pool_vertices=8000, pool_entries=big.nnz + small.nnz + 64, mode="det", solo_entries=-1) as srv:
        a = srv.submit(big.rowptr, big.colidx, seed=5)
        time.sleep(0.05)
        srv.poll(srv.submit(small.rowptr, small.colidx, seed=3))
        assert srv.poll(a, timeout_ms=0) is None
        np.testing.assert_array_equal(srv.poll(a)[0], _rank(big, 5))


def test_many_arrivals(gclib):
    # power-law graphs (small and larger vertices, several work items) interrupted again and again
    gs = [gg.rmat(14, 16, 1), gg.rmat(13, 30, 2), gg.complete(400), gg.er(5000, 30.0, 3)]
    late = [gg.er(200 + 37 * i, 9.0, i) for i in range(40)]
    refs = [oracle.det(g, 7) for g in gs]
    late_refs = [oracle.det(g, 9) for g in late]
    with gclib.Server(pool_vertices=sum(g.n for g in gs + late) + 64, pool_entries=sum(g.nnz for g in gs + late) + 64,
                      mode="det") as srv:
        for _ in range(3):
            ids = [srv.submit(g.rowptr, g.colidx, seed=7) for g in gs]
            late_ids = []
            for g in late:
                late_ids.append(srv.submit(g.rowptr, g.colidx, seed=9))
                time.sleep(0.0005)
            for rid, ref in zip(ids + late_ids, refs + late_refs):
                colors, nc, rounds = srv.poll(rid)
                np.testing.assert_array_equal(colors, ref.colors)
                assert (nc, rounds) == (ref.ncolors, ref.rounds)
        st = srv.stats()
        assert st["failed"] == 0 and st["core_handovers"] > 3


def test_graphs_without_large_rows_stay_in_the_round_kernel(gclib):
    g = gg.stencil27(20)
    ref = oracle.det(g, 7)
    with gclib.Server(pool_vertices=g.n + 64, pool_entries=g.nnz + 64, mode="det") as srv:
        for _ in range(3):
            colors, nc, rounds = srv.poll(srv.submit(g.rowptr, g.colidx, seed=7))
            np.testing.assert_array_equal(colors, ref.colors)
            assert (nc, rounds) == (ref.ncolors, ref.rounds)
        assert srv.stats()["core_handovers"] == 0
