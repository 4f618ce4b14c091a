"""Offset tables of a batch: a row is accepted only if all of it lies inside the arrays."""
import ctypes
import itertools

import numpy as np
import pytest

import graphgen as gg
from hostcc import compile_shim

SHIM = """
extern "C" int row_ok(int g, long v0, long v1, long e0, long e1, long n, long nnz) {
    return gc::batch_row_ok(g, v0, v1, e0, e1, n, nnz);
}
"""


def test_every_accepted_row_lies_inside_the_arrays(tmp_path):
    lib = compile_shim(tmp_path, SHIM)
    lib.row_ok.argtypes = [ctypes.c_int] + [ctypes.c_long] * 6
    wrong = right = 0
    for t in itertools.product(range(-2, 5), repeat=3):  # interior values and total of a table of 3 graphs
        table, total = (0,) + t, t[-1]
        if total < 0:
            continue  # refused on the host
        rows = [lib.row_ok(g, table[g], table[g + 1], table[g], table[g + 1], total, total) for g in range(3)]
        for g, ok in enumerate(rows):
            assert not ok or 0 <= table[g] <= table[g + 1] <= total
        good = list(table) == sorted(table)
        assert all(rows) == good
        right += good
        wrong += not good
    assert right == 35 and wrong > 100
    # the tables of the vertices and of the entries are checked alike, and both start at 0
    assert not lib.row_ok(0, 1, 2, 0, 2, 9, 9) and not lib.row_ok(0, 0, 2, 1, 2, 9, 9)
    assert not lib.row_ok(1, 1, 2, -1, 2, 9, 9) and not lib.row_ok(1, 1, 2, 1, 10, 9, 9)


@pytest.mark.gpu
@pytest.mark.parametrize("table", ["vtx", "edge"])
@pytest.mark.parametrize("change", [(2, -4), (1, 10**6), (-1, 100), (0, 1)])
def test_malformed_tables_are_refused(gclib, table, change):
    # (the arrays are longer than any of these tables says)
    import torch
    gs = [gg.er(200, 8.0, i) for i in range(8)]
    b = gg.pack(gs)
    room = 2 * 10**6
    rp = torch.zeros(room, dtype=torch.int32, device="cuda")
    ci = torch.zeros(room, dtype=torch.int32, device="cuda")
    rp[:len(b.rowptr)] = torch.from_numpy(b.rowptr).cuda()
    ci[:len(b.colidx)] = torch.from_numpy(b.colidx).cuda()
    tabs = {"vtx": np.array(b.vtx_off), "edge": np.array(b.edge_off)}
    tabs[table][change[0]] = change[1]
    out = torch.full((room,), -5, dtype=torch.int32, device="cuda")
    args = [torch.from_numpy(tabs["vtx"]).cuda(), torch.from_numpy(tabs["edge"]).cuda(), rp, ci]
    with pytest.raises(gclib.GCError) as e:
        gclib.color_batch(*args, "det", 3, out=out)
    assert e.value.status == gclib.GC_ERR_INVALID_GRAPH and "offset tables" in str(e.value)
    assert bool((out == -5).all())
