"""Short sorts (one thread-block cluster, one launch) against the plain
definition of the result: sizes at the edges of every launch shape and of the
shares that a cluster's CTAs hold, every key type and records, keys equal to the
padding (the largest key), unaligned buffers, pinned host keys, side streams
and graph capture."""
from __future__ import annotations

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ps():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2305_05245_gb300 as ps
    assert torch.cuda.is_available()
    return ps


def check(ps, ora, host, mode="exact", offset=0):
    import torch
    st = {"uint32": np.int32, "uint64": np.int64}.get(str(host.dtype), host.dtype)
    buf = torch.zeros(host.size + offset + 3, dtype=torch.from_numpy(host[:1].view(st)).dtype, device="cuda")
    x = buf[offset:offset + host.size]
    x.copy_(torch.from_numpy(host.view(st)))
    ps.sort(x.view(getattr(torch, str(host.dtype))) if st != host.dtype else x, mode)
    torch.cuda.synchronize()
    assert x.cpu().numpy().tobytes() == ora.reference_sort(host).tobytes()
    assert not buf[:offset].any() and not buf[offset + host.size:].any()


EDGES = [1024, 2048, 4096, 8192, 16384, 65536, 98304, 131072, 262144]
SIZES = sorted({2, 3, 31, 33, 100, 1000, 4 * 4096 - 3, 40961, 16 * 1028, 16 * 1028 + 1, 100003, 200001} |
               {e + d for e in EDGES for d in (-1, 0, 1)})


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("dtype", sorted(synth.DTYPES))
def test_sizes(ps, ora, dtype, n):
    check(ps, ora, synth.keys(n, dtype, "uniform", seed=synth.seed_for("cluster", n)), "regular" if n & 1 else "exact")


@pytest.mark.parametrize("n", [777, 9001, 50000, 131072])
@pytest.mark.parametrize("dtype", ["int32", "uint64", "float32", "float64"])
@pytest.mark.parametrize("dist", ["sorted", "reverse", "few_unique", "almost_sorted", "three_valued"])
def test_distributions(ps, ora, dtype, dist, n):
    check(ps, ora, synth.keys(n, dtype, dist, seed=n))


@pytest.mark.parametrize("n", [5, 1025, 16385, 70000])
@pytest.mark.parametrize("dtype", ["int32", "uint32", "int64", "uint64"])
def test_largest_keys(ps, ora, dtype, n):
    """Half the keys equal the largest one, which also pads short shares."""
    x = synth.keys(n, dtype, "uniform", seed=n)
    x[::2] = np.iinfo(dtype).max
    check(ps, ora, x)


@pytest.mark.parametrize("dtype,offset", [("int32", 1), ("float32", 3), ("int64", 1)])
@pytest.mark.parametrize("n", [1000, 8192, 30000])
def test_unaligned_buffers(ps, ora, dtype, offset, n):
    check(ps, ora, synth.keys(n, dtype, "uniform", seed=9), offset=offset)


@pytest.mark.parametrize("n", [2, 1023, 1025, 4097, 8193, 16385, 65536, 65537, 131071, 131072])
@pytest.mark.parametrize("few", [False, True])
def test_records(ps, n, few):
    import torch
    z = synth.splitmix64(n, 2 * n)
    k, p = z[:n].copy(), (z[n:] >> np.uint64(32)).astype(np.uint32)
    if few:
        k &= np.uint64(3)
    tk, tp = torch.from_numpy(k.view(np.int64).copy()).cuda(), torch.from_numpy(p.view(np.int32).copy()).cuda()
    ps.sort_pairs(tk, tp)
    torch.cuda.synchronize()
    o = np.lexsort((p, k))
    assert tk.cpu().numpy().view(np.uint64).tobytes() == k[o].tobytes()
    assert tp.cpu().numpy().view(np.uint32).tobytes() == p[o].tobytes()


@pytest.mark.parametrize("n", [1000, 20000, 100001])
def test_pinned_host_keys(ps, ora, n):
    import torch
    host = synth.keys(n, "int64", "uniform", seed=n)
    x = torch.from_numpy(host.copy()).pin_memory()
    ps.sort_host(x)
    assert x.numpy().tobytes() == ora.reference_sort(host).tobytes()


def test_streams_and_capture(ps, ora):
    """Eight clusters' sorts at once on four streams, then one replayed from a graph."""
    import torch
    hosts = [synth.keys(60000 + 7 * i, "int32", "uniform", seed=i) for i in range(8)]
    xs = [torch.from_numpy(h.copy()).cuda() for h in hosts]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(4)]
    for i, x in enumerate(xs):
        ps.sort(x, stream=streams[i % 4])
    torch.cuda.synchronize()
    for h, x in zip(hosts, xs):
        assert x.cpu().numpy().tobytes() == ora.reference_sort(h).tobytes()
    x = torch.from_numpy(hosts[0].copy()).cuda()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ps.sort(x)
    for h in hosts[1:3]:
        x.copy_(torch.from_numpy(h[:x.numel()]))
        g.replay()
        torch.cuda.synchronize()
        assert x.cpu().numpy().tobytes() == ora.reference_sort(h[:x.numel()]).tobytes()


@pytest.mark.parametrize("n,nb,np_", [(64 * 8192, 64, 16), (64 * 8192 + 1, 64, 64), (100 * 16384 - 7, 100, 7), (16385 * 32, 32, 5),
                                      (65537 * 8, 8, 8), (131072 * 4, 4, 3), (131073 * 4, 4, 3), (70001, 129, 200), (50, 64, 64),
                                      (300007, 128, 129)])
@pytest.mark.parametrize("dtype", ["int32", "float64"])
@pytest.mark.parametrize("mode", ["exact", "regular"])
def test_blocks_given_by_the_caller(ps, ora, dtype, mode, n, nb, np_):
    """Blocks sorted by clusters (up to 131072 keys each) and the sample pool in
    shared memory (up to 128 blocks): output and intermediates of the four steps."""
    import torch
    host = synth.keys(n, dtype, "few_unique" if nb == 100 else "uniform", seed=n + nb)
    x = torch.from_numpy(host.copy()).cuda()
    tr = ps.sort(x, mode, n_blocks=nb, n_parts=np_, trace=True)
    torch.cuda.synchronize()
    ref = ora.sort(host, ora.EXACT if mode == "exact" else ora.REGULAR, nb, np_)
    assert x.cpu().numpy().tobytes() == ref.out.tobytes()
    assert tr.pivots.cpu().numpy()[:np_ - 1].tobytes() == ref.pivots.tobytes()
    assert np.array_equal(tr.splits.cpu().numpy(), ref.splits)
    assert np.array_equal(tr.offsets.cpu().numpy(), ref.offsets)


@pytest.mark.parametrize("n,nb,np_", [(64 * 8192 + 5, 64, 16), (40000, 3, 9), (20000, 128, 60)])
@pytest.mark.parametrize("mode", ["exact", "regular"])
def test_record_blocks_given_by_the_caller(ps, n, nb, np_, mode):
    import torch
    z = synth.splitmix64(n, 2 * n)
    k, p = z[:n] & np.uint64(0xFFFF), (z[n:] >> np.uint64(32)).astype(np.uint32)
    tk, tp = torch.from_numpy(k.view(np.int64).copy()).cuda(), torch.from_numpy(p.view(np.int32).copy()).cuda()
    ps.sort_pairs(tk, tp, mode, nb, np_)
    torch.cuda.synchronize()
    o = np.lexsort((p, k))
    assert tk.cpu().numpy().view(np.uint64).tobytes() == k[o].tobytes()
    assert tp.cpu().numpy().view(np.uint32).tobytes() == p[o].tobytes()


@pytest.mark.parametrize("dtype,n", [("int32", 262144), ("int32", 262145), ("float32", 1 << 20), ("int64", 131072),
                                     ("int64", 131073), ("float64", 1 << 20), ("uint64", 999999)])
def test_noalloc(ps, ora, dtype, n):
    import torch
    host = synth.keys(n, dtype, "uniform", seed=n)
    st = {"uint64": np.int64}.get(dtype, host.dtype)
    x = torch.from_numpy(host.view(st).copy()).cuda()
    for _ in range(2):
        x.copy_(torch.from_numpy(host.view(st)))
        ps.sort_noalloc(x.view(getattr(torch, dtype)))
        torch.cuda.synchronize()
        assert x.cpu().numpy().tobytes() == ora.reference_sort(host).tobytes()
