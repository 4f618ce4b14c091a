"""Priority digests of the value keys (largest first, smallest last): in the keys' order for any table, and
rarely equal across an edge whatever the degrees are."""
import ctypes

import numpy as np
import pytest

import graphgen as gg
import oracle
from hostcc import compile_shim

SHIM = """
extern "C" int bins() { return gc::kDigestBins; }
extern "C" void digests(const unsigned *p31, const unsigned *weight, long n, unsigned *out) {
    unsigned long cnt[gc::kDigestBins] = {}, total = 0, before = 0;
    gc::DigestBin tab[gc::kDigestBins];
    for (long i = 0; i < n; ++i) cnt[gc::digest_bin(gc::kKeyCap - (p31[i] >> 11))] += weight[i], total += weight[i];
    for (int b = gc::kDigestBins - 1; b >= 0; --b) {
        tab[b] = gc::digest_range(before, cnt[b], total);
        before += cnt[b];
    }
    for (long i = 0; i < n; ++i) out[i] = gc::key_digest24(tab, p31[i]);
}
"""
CAP = (1 << 20) - 1


@pytest.fixture(scope="module")
def digests(tmp_path_factory):
    lib = compile_shim(tmp_path_factory.mktemp("digest"), SHIM)

    def f(p31, weight):
        p31, weight = np.ascontiguousarray(p31, np.uint32), np.ascontiguousarray(weight, np.uint32)
        out = np.empty(len(p31), np.uint32)
        lib.digests(p31.ctypes.data_as(ctypes.c_void_p), weight.ctypes.data_as(ctypes.c_void_p),
                    ctypes.c_long(len(p31)), out.ctypes.data_as(ctypes.c_void_p))
        return out

    return f


def test_in_the_keys_order(digests):
    rng = np.random.default_rng(1)
    value = np.concatenate([np.arange(4096), (2.0 ** rng.uniform(0, 20, 200000)).astype(np.int64), [CAP, CAP - 1, 1 << 19]])
    value = np.minimum(value, CAP)
    p31 = np.sort(((CAP - value).astype(np.uint32) << 11) | rng.integers(0, 2048, len(value)).astype(np.uint32))
    # (also a table made of other weights, of nothing, and of counts that have wrapped)
    for weight in (np.ones(len(p31)), rng.integers(0, 1 << 20, len(p31)), np.zeros(len(p31))):
        d = digests(p31, weight)
        assert (np.diff(d.astype(np.int64)) >= 0).all() and d.max() < 1 << 24


@pytest.mark.parametrize("make", [lambda: gg.stencil27(24), lambda: gg.grid5(150, 140), lambda: gg.er(20000, 60.0, 3),
                                  lambda: gg.rmat(14, 16, 2), lambda: gg.cycle(5000)])
def test_rarely_equal_across_an_edge(digests, make):
    g = make()
    deg = g.degrees().astype(np.int64)
    rng = np.random.default_rng(2)
    p31 = ((CAP - np.minimum(deg, CAP)).astype(np.uint32) << 11) | rng.integers(0, 2048, g.n).astype(np.uint32)
    d = digests(p31, deg)
    u = np.repeat(np.arange(g.n), deg)
    v = g.colidx
    # a hash key's pairs tie with 1/256 and 1/65,536; the value's hash has 11 bits
    assert np.mean((d >> 16)[u] == (d >> 16)[v]) < 2 / 256
    assert np.mean((d >> 8)[u] == (d >> 8)[v]) < np.mean(p31[u] == p31[v]) + 4 / 65536


@pytest.mark.gpu
@pytest.mark.parametrize("priority", [1, 2])
@pytest.mark.parametrize("make", [lambda: gg.stencil27(28), lambda: gg.grid5(160, 150), lambda: gg.cycle(20001),
                                  lambda: gg.er(17000, 70.0, 3), lambda: gg.rmat(15, 8, 2), lambda: gg.star(20000),
                                  lambda: gg.complete(300), lambda: gg.er(3000, 30.0, 3), lambda: gg.er(1500, 100.0, 3)])
def test_value_keys_match_oracle(gclib, make, priority):
    import torch
    g = make()
    ref = oracle.det(g, 5, priority=priority)
    rp, ci = torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(g.colidx).cuda()
    r = gclib.color(rp, ci, "det", 5, options=gclib.Options(priority=priority))
    np.testing.assert_array_equal(r.colors.cpu().numpy(), ref.colors)
    assert (r.ncolors, r.rounds) == (ref.ncolors, ref.rounds)


@pytest.mark.gpu
def test_value_keys_of_a_batch(gclib):
    import torch
    for gs in ([gg.er(300 + 7 * i, 9.0, i) for i in range(30)] + [gg.stencil27(12), gg.complete(200)],
               [gg.stencil27(20), gg.rmat(13, 16, 2), gg.grid5(90, 80), gg.empty(3), gg.er(200, 5.0, 1)]):
        b = gg.pack(gs)
        args = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (b.vtx_off, b.edge_off, b.rowptr, b.colidx)]
        colors, nc, rd = gclib.color_batch(*args, "det", 3, options=gclib.Options(priority=1))
        colors = colors.cpu().numpy()
        for i, g in enumerate(gs):
            ref = oracle.det(g, 3, priority=1)
            np.testing.assert_array_equal(colors[b.vtx_off[i]:b.vtx_off[i + 1]], ref.colors)
            assert (nc[i], rd[i]) == (ref.ncolors, ref.rounds)
