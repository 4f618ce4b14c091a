"""A call on CUDA tensors comes after the work already queued on the current torch stream, which is
the default stream unless the caller chose another: each call's input is written by a copy that
waits behind a delay on that stream."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu

DELAY = 40_000_000  # clock cycles, about 20 ms


def _ring(n, step):
    """The cycle i - (i + step) mod n (step coprime to n): n rows of two entries each."""
    i = np.arange(n)
    ends = np.sort(np.stack([(i + step) % n, (i - step) % n], 1), 1)
    return gg.Graph(n=n, rowptr=np.arange(0, 2 * n + 1, 2, dtype=np.int32),
                  colidx=ends.reshape(-1).astype(np.int32), name=f"ring{n}")


def _late(value, before):
    """A CUDA tensor that holds `before` now and `value` once the current stream gets there."""
    import torch
    t = torch.from_numpy(np.ascontiguousarray(before)).cuda()
    v = torch.from_numpy(np.ascontiguousarray(value)).cuda()
    torch.cuda.synchronize()
    torch.cuda._sleep(DELAY)
    t.copy_(v, non_blocking=True)
    return t


@pytest.mark.parametrize("own_stream", [False, True])
@pytest.mark.parametrize("n", [1001, 20011])  # the small-graph kernel and the round kernel
@pytest.mark.parametrize("call", ["det", "ordered", "recolor", "batch", "det_round", "server"])
def test_calls_follow_the_current_stream(gclib, call, n, own_stream):
    import torch
    a, b = _ring(n, 2), _ring(n, 7)
    rp = torch.from_numpy(a.rowptr).cuda()
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream() if own_stream else torch.cuda.default_stream()):
        if call == "recolor":
            ci = torch.from_numpy(a.colidx).cuda()
            start = oracle.det(a, 5).colors
            got = gclib.recolor(rp, ci, _late(start, np.arange(n, dtype=np.int32)), 3).colors
            want, _ = oracle.greedy_keyorder(a, 3, oracle.PRIORITY_RECOLOR, start)
        elif call == "det_round":
            cur = torch.zeros(n, dtype=torch.int32, device="cuda")
            work = torch.arange(n, dtype=torch.int32, device="cuda")
            got, _ = gclib.det_round(rp, _late(a.colidx, b.colidx), 5, cur, work)
            torch.cuda.synchronize()
            want, _ = gclib.det_round(a.rowptr, a.colidx, 5, np.zeros(n, np.int32), np.arange(n, dtype=np.int32))
        elif call == "batch":
            off = np.array([0, n], np.int64), np.array([0, 2 * n], np.int64)
            got, _, _ = gclib.color_batch(*off, rp, _late(a.colidx, b.colidx), "det", 5)
            want = oracle.det(a, 5).colors
        elif call == "server":
            with gclib.Server(pool_vertices=1 << 16, pool_entries=1 << 18) as srv:
                got, _, _ = srv.poll(srv.submit(rp, _late(a.colidx, b.colidx), "det", 5))
            want = oracle.det(a, 5).colors
        else:
            got = gclib.color(rp, _late(a.colidx, b.colidx), call, 5).colors
            want = oracle.det(a, 5).colors if call == "det" else oracle.greedy_keyorder(a, 5)[0]
        got = got.cpu().numpy() if hasattr(got, "cpu") else got
    np.testing.assert_array_equal(got, want)
