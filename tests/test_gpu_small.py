"""Small graphs (one block, one cluster, or a block per graph of a batch) against the CPU oracle: sizes at
the limits of each path, row lengths around the thread / warp split, keys, alignments, host arrays,
mixed batches, and the calls that must fail."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def _dev(a, offset=0):
    import torch
    buf = torch.zeros(len(a) + offset, dtype=torch.int32, device="cuda")
    buf[offset:] = torch.from_numpy(np.ascontiguousarray(a)).cuda()
    return buf[offset:]


def _check(gclib, g, seed, **kw):
    opt = kw.pop("options", None)
    prio = opt.priority if opt else 0
    ref = oracle.det(g, seed, priority=prio)
    r = gclib.color(_dev(g.rowptr), _dev(g.colidx, kw.pop("offset", 0)), "det", seed, options=opt)
    np.testing.assert_array_equal(r.colors.cpu().numpy(), ref.colors)
    assert (r.ncolors, r.rounds) == (ref.ncolors, ref.rounds)


GRAPHS = [lambda: gg.path(2), lambda: gg.path(2048), lambda: gg.cycle(2049), lambda: gg.star(33), lambda: gg.star(34),
          lambda: gg.star(2000), lambda: gg.complete(3), lambda: gg.complete(33), lambda: gg.complete(65),
          lambda: gg.complete(200), lambda: gg.crown(40), lambda: gg.grid5(31, 17), lambda: gg.stencil27(9),
          lambda: gg.er(2047, 12.0, 3), lambda: gg.er(2048, 15.9, 3), lambda: gg.er(2048, 40.0, 4), lambda: gg.er(2049, 16.0, 3),
          lambda: gg.er(16383, 9.0, 3), lambda: gg.er(16384, 31.0, 5), lambda: gg.er(16385, 9.0, 3),
          lambda: gg.rmat(10, 12, 2), lambda: gg.rmat(13, 16, 2), lambda: gg.rmat(14, 16, 7)]


@pytest.mark.parametrize("make", GRAPHS)
@pytest.mark.parametrize("seed", [0, 7])
def test_small_graphs_match_oracle(gclib, make, seed):
    _check(gclib, make(), seed)


@pytest.mark.parametrize("make", [lambda: gg.er(900, 10.0, 3), lambda: gg.er(6000, 20.0, 3), lambda: gg.rmat(12, 8, 2)])
@pytest.mark.parametrize("offset", [1, 2, 3, 4])
def test_colidx_alignment(gclib, make, offset):
    _check(gclib, make(), 3, offset=offset)


@pytest.mark.parametrize("make", [lambda: gg.star(1000), lambda: gg.stencil27(9), lambda: gg.rmat(13, 12, 2),
                                  lambda: gg.grid5(100, 90)])
def test_largest_first(gclib, make):
    _check(gclib, make(), 5, options=gclib.Options(priority=gclib.PRIORITY_LARGEST_FIRST))


@pytest.mark.parametrize("make", [lambda: gg.er(1000, 8.0, 3), lambda: gg.er(9000, 16.0, 3)])
def test_host_arrays(gclib, make):
    g = make()
    ref = oracle.det(g, 9)
    r = gclib.color(g.rowptr, g.colidx, "det", 9)
    np.testing.assert_array_equal(r.colors, ref.colors)
    assert (r.ncolors, r.rounds) == (ref.ncolors, ref.rounds)


@pytest.mark.parametrize("n", [500, 9000])
@pytest.mark.parametrize("bad", ["entry", "negative", "self", "row", "end"])
def test_malformed(gclib, n, bad):
    import torch
    g = gg.er(n, 12.0, 3)
    rp, ci = g.rowptr.copy(), g.colidx.copy()
    v = n // 2
    if bad == "entry":
        ci[rp[v]] = n
    elif bad == "negative":
        ci[rp[v + 1] - 1] = -1
    elif bad == "self":
        ci[rp[v]] = v
    elif bad == "row":
        rp[v] = rp[v + 1] + 1
    else:
        rp[0] = 1
    out = torch.full((n,), -5, dtype=torch.int32, device="cuda")
    with pytest.raises(gclib.GCError) as e:
        gclib.color(_dev(rp), _dev(ci), "det", 1, out=out)
    assert e.value.status == gclib.GC_ERR_INVALID_GRAPH
    assert bool((out == -5).all())
    _check(gclib, g, 1)  # the next call works


@pytest.mark.parametrize("n", [500, 9000])
def test_round_cap(gclib, n):
    g = gg.er(n, 12.0, 3)
    rounds = oracle.det(g, 1).rounds
    with pytest.raises(gclib.GCError) as e:
        gclib.color(_dev(g.rowptr), _dev(g.colidx), "det", 1, options=gclib.Options(max_rounds=rounds - 1))
    assert e.value.status == gclib.GC_ERR_NO_CONVERGENCE
    r = gclib.color(_dev(g.rowptr), _dev(g.colidx), "det", 1, options=gclib.Options(max_rounds=rounds))
    assert r.rounds == rounds


def _batch(gclib, gs, seed, priority=0, host=False):
    import torch
    b = gg.pack(gs)
    arrays = [np.ascontiguousarray(a) for a in (b.vtx_off, b.edge_off, b.rowptr, b.colidx)]
    args = arrays if host else [torch.from_numpy(a).cuda() for a in arrays]
    opt = gclib.Options(priority=priority)
    colors, nc, rd = gclib.color_batch(*args, "det", seed, options=opt)
    colors = colors if host else colors.cpu().numpy()
    for i, g in enumerate(gs):
        ref = oracle.det(g, seed, priority=priority)
        np.testing.assert_array_equal(colors[b.vtx_off[i]:b.vtx_off[i + 1]], ref.colors, err_msg=f"graph {i} {g.name}")
        assert (nc[i], rd[i]) == (ref.ncolors, ref.rounds), i


MIXES = [
    lambda: [gg.er(100 + 37 * i, 4.0 + i % 9, i) for i in range(40)],                            # all small
    lambda: [gg.empty(3), gg.path(2), gg.rmat(11, 12, 5), gg.complete(150), gg.empty(1), gg.star(4096),
             gg.er(4096, 20.0, 2), gg.er(4097, 20.0, 2), gg.rmat(14, 12, 3), gg.workload("er10k")],  # both paths
    lambda: [gg.rmat(14, 12, 3), gg.er(5000, 60.0, 1)],                                          # none small
    lambda: [gg.empty(5)],
]


@pytest.mark.parametrize("mix", MIXES)
@pytest.mark.parametrize("host", [False, True])
def test_batches_match_oracle(gclib, mix, host):
    _batch(gclib, mix(), 3, host=host)


def test_batch_largest_first(gclib):
    _batch(gclib, MIXES[1](), 3, priority=1)


def test_batch_with_a_malformed_small_graph(gclib):
    import torch
    gs = [gg.er(300, 8.0, i) for i in range(20)] + [gg.rmat(14, 12, 3)]
    b = gg.pack(gs)
    ci = b.colidx.copy()
    ci[b.edge_off[7] + 3] = 300
    out = torch.full((int(b.vtx_off[-1]),), -5, dtype=torch.int32, device="cuda")
    args = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (b.vtx_off, b.edge_off, b.rowptr, ci)]
    with pytest.raises(gclib.GCError) as e:
        gclib.color_batch(*args, "det", 3, out=out)
    assert e.value.status == gclib.GC_ERR_INVALID_GRAPH
    assert bool((out == -5).all())
    _batch(gclib, gs, 3)
