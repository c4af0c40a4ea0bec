"""The radix block sort (one block, keys only) against the plain definition of
the result (the unique ascending order of the keys' bits, oracle.reference_sort):
sizes around its tiles and its smallest size, every key type, distributions
that leave digits out (all keys equal, one varying byte, few values) or that
fill a digit with one value, unaligned buffers, and repeated runs."""
from __future__ import annotations

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

T32, T64 = 512 * 24, 384 * 24  # keys per tile of a digit pass (large sorts; smaller ones: 4096, 8192)
MIN = 131073                   # smallest size the radix block sort takes


@pytest.fixture(scope="module")
def ps():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2305_05245_gb300 as ps
    assert torch.cuda.is_available()
    return ps


def check(ps, ora, host, mode="exact", offset=0, **kw):
    """Sort host on the device (starting `offset` elements into a buffer)."""
    import torch
    st = {"uint32": np.int32, "uint64": np.int64}.get(str(host.dtype), host.dtype)
    buf = torch.zeros(host.size + offset + 3, dtype=torch.from_numpy(host[:1].view(st)).dtype, device="cuda")
    x = buf[offset:offset + host.size]
    x.copy_(torch.from_numpy(host.view(st)))
    y = x.view(getattr(torch, str(host.dtype))) if st != host.dtype else x
    ps.sort(y, mode, **kw)
    torch.cuda.synchronize()
    got = x.cpu().numpy().view(host.dtype)
    want = ora.reference_sort(host)
    assert got.tobytes() == want.tobytes()
    assert not buf[:offset].any() and not buf[offset + host.size:].any()


SIZES = [MIN, MIN + 1, 683 * T32 - 1, 683 * T32, 683 * T32 + 1, 43 * T64 - 1, 43 * T64,
         43 * T64 + 1, 38 * 4096 + 1, 1 << 18, (1 << 18) + 1, 1 << 20, (1 << 23) + 1,
         3000017]


@pytest.mark.parametrize("dtype", sorted(synth.DTYPES))
@pytest.mark.parametrize("n", SIZES)
def test_sizes(ps, ora, dtype, n):
    check(ps, ora, synth.keys(n, dtype, "uniform", seed=synth.seed_for("radix", n)))


@pytest.mark.parametrize("dtype", sorted(synth.DTYPES))
@pytest.mark.parametrize("dist", ["sorted", "reverse", "few_unique", "gaussian", "almost_sorted", "three_valued"])
def test_distributions(ps, ora, dtype, dist):
    if dist == "gaussian" and not dtype.startswith("float"):
        pytest.skip("gaussian keys are floating point")
    check(ps, ora, synth.keys(400003, dtype, dist, seed=synth.seed_for("radix", dist)), mode="regular")


@pytest.mark.parametrize("dtype", ["int32", "uint32", "int64", "uint64"])
@pytest.mark.parametrize("bytes_", [(), (0,), (1,), (0, 3), (1, 2, 3), (-1,), (2, -1)])
def test_varying_bytes(ps, ora, dtype, bytes_):
    """Only the named bytes of the keys vary: none to three passes have work."""
    width = np.dtype(dtype).itemsize
    z = synth.splitmix64(7, 270001)
    u = np.full(z.size, 0x0123456789ABCDEF, dtype=np.uint64)
    for b in bytes_:
        s = np.uint64(8 * (b % width))
        u = (u & ~(np.uint64(255) << s)) | (((z >> s) & np.uint64(255)) << s)
    host = (u & np.uint64(0xFFFFFFFF)).astype(np.uint32).view(dtype) if width == 4 else u.view(dtype)
    check(ps, ora, np.ascontiguousarray(host))


@pytest.mark.parametrize("dtype", ["float32", "float64"])
def test_float_specials(ps, ora, dtype):
    x = synth.keys(270001, dtype, "gaussian", seed=5)
    info = np.finfo(dtype)
    sp = np.array([0.0, -0.0, np.inf, -np.inf, info.max, info.min, info.tiny, -info.tiny,
                   info.smallest_subnormal, -info.smallest_subnormal], dtype=dtype)
    x[::17] = sp[np.arange(x[::17].size) % sp.size]
    check(ps, ora, x)


@pytest.mark.parametrize("dtype,offset", [("int32", 1), ("float32", 3), ("int64", 1), ("float64", 1)])
def test_unaligned_buffers(ps, ora, dtype, offset):
    check(ps, ora, synth.keys(270007, dtype, "uniform", seed=9), offset=offset)


def test_one_block_given_by_the_caller(ps, ora):
    check(ps, ora, synth.keys(300007, "int32", "uniform", seed=3), n_blocks=1, n_parts=1)


def test_repeated_runs_are_identical(ps, ora):
    host = synth.keys(1 << 20, "int64", "few_unique", seed=11)
    for _ in range(10):
        check(ps, ora, host)


def clustered(n, sizes, top, seed):
    """n uniform uint64 keys, of which sizes[c] share the leading `top` bytes of
    one key and differ in the others (runs that the leading bytes alone leave in
    input order)."""
    u = synth.splitmix64(seed, n)
    place = np.argsort(synth.splitmix64(seed + 1, n))[:sum(sizes)]
    low = np.uint64((1 << (64 - 8 * top)) - 1)
    at = 0
    for c, m in enumerate(sizes):
        idx = place[at:at + m]
        u[idx] = (u[idx[0]] & ~low) | (u[idx] & low)
        at += m
    return u


@pytest.mark.parametrize("n,sizes,top", [
    (1 << 20, (2, 63, 64, 65, 66, 127, 128, 129), 5),   # around the length a run is ranked in place
    (1 << 20, (700, 40, 300, 2, 3), 4),
    (1 << 20, (300,) * 2, 7),
    (1 << 25, (9000,), 5),                              # runs over several tiles of the fix kernel
    (1 << 25, (5000, 70), 6),
    (1 << 18, (1 << 18,), 3),                           # one run: the sample sees it
    (300001, (100000, 50000), 6),
])
def test_runs_of_equal_leading_bytes(ps, ora, n, sizes, top):
    u = clustered(n, sizes, top, seed=n + top)
    check(ps, ora, u)
    if n < (1 << 25):
        check(ps, ora, u.view(np.int64), mode="regular")


def test_runs_of_equal_keys(ps, ora):
    """Long runs of identical keys among distinct ones (never out of order)."""
    u = synth.splitmix64(3, 1 << 20)
    u[::5] = u[0]
    u[1::5] = u[0] ^ np.uint64(1)  # and a neighbour that differs in the last byte only
    check(ps, ora, u)
    u[1::5] = u[0]
    check(ps, ora, u)


@pytest.mark.parametrize("n", [36 * 4096 - 1, 36 * 4096, 36 * 4096 + 1, 36 * 4096 + 64, 36 * 4096 + 65])
def test_fix_tile_edges(ps, ora, n):
    """Keys of 24 leading bits that come in pairs and triples, sizes around the
    fix kernel's tiles of 4096 positions."""
    z = synth.splitmix64(n, n)
    check(ps, ora, ((z >> np.uint64(44)) << np.uint64(44)) | (z & np.uint64(255)))


def check_records(ps, k, p, mode="exact"):
    """Records against numpy's order by (key, payload)."""
    import torch
    tk = torch.from_numpy(k.view(np.int64).copy()).cuda()
    tp = torch.from_numpy(p.view(np.int32).copy()).cuda()
    ps.sort_pairs(tk, tp, mode)
    torch.cuda.synchronize()
    o = np.lexsort((p, k))
    assert tk.cpu().numpy().view(np.uint64).tobytes() == k[o].tobytes()
    assert tp.cpu().numpy().view(np.uint32).tobytes() == p[o].tobytes()


@pytest.mark.parametrize("n", [MIN, MIN + 1, 43 * 6144 - 1, 43 * 6144, 43 * 6144 + 1, 1000003])
@pytest.mark.parametrize("kind", ["uniform", "index", "few", "few_index", "one_key", "all_equal"])
def test_records(ps, n, kind):
    """Payloads that are the input position, or random, or few; keys distinct,
    few or all equal: passes over key bytes, payload bytes, both or none."""
    z = synth.splitmix64(n, 2 * n)
    k, p = z[:n].copy(), (z[n:] >> np.uint64(32)).astype(np.uint32)
    if kind in ("index", "few_index"):
        p = np.arange(n, dtype=np.uint32)
    if kind in ("few", "few_index"):
        k = z[:16][(z[:n] >> np.uint64(60)).astype(np.int64)]
    if kind == "one_key":
        k[:] = k[0]
    if kind == "all_equal":
        k[:], p[:] = k[0], p[0]
    check_records(ps, k, p, "regular" if n & 1 else "exact")


@pytest.mark.parametrize("sizes,top", [((2, 63, 64, 65, 66, 129), 5), ((700, 300, 3), 4), ((300, 300), 7)])
def test_record_runs_of_equal_leading_bytes(ps, sizes, top):
    n = 1 << 20
    k = clustered(n, sizes, top, seed=top)
    k[5::1000] = k[5]  # some equal keys, ordered by payload
    check_records(ps, k, (synth.splitmix64(9, n) >> np.uint64(40)).astype(np.uint32))


def check_batch(ps, ora, lens, dtype, dist, how, seed=1):
    """Every segment of a batch against the plain definition; `how`: the
    batched call, a plan run twice, or the sort server (own buffers)."""
    import torch
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    host = np.concatenate([synth.keys(int(n), dtype, dist, seed=synth.seed_for(seed, i)) for i, n in enumerate(lens)])
    want = np.concatenate([ora.reference_sort(host[a:b]) for a, b in zip(off[:-1], off[1:])])
    x = torch.from_numpy(host.copy()).cuda()
    if how == "call":
        ps.sort_batch(x, torch.from_numpy(off).cuda())
    elif how == "plan":
        plan = ps.BatchPlan(off, getattr(torch, dtype))
        plan.run(x)
        x.copy_(torch.from_numpy(host))
        plan.run(x)
        torch.cuda.synchronize()
        plan.close()
    else:
        parts = [x[int(a):int(b)].clone() for a, b in zip(off[:-1], off[1:])]
        torch.cuda.synchronize()
        srv = ps.Server(budget_bytes=4 << 30)
        left = {srv.submit(p) for p in parts}
        while left:
            for rid, status in srv.poll():
                assert status == 0
                left.discard(rid)
        srv.close()
        x = torch.cat(parts)
    torch.cuda.synchronize()
    assert x.cpu().numpy().tobytes() == want.tobytes()


L32, L64 = 1 << 18, 1 << 17  # segments longer than this take the radix block sort


@pytest.mark.parametrize("how", ["call", "plan", "server"])
@pytest.mark.parametrize("dtype,edge", [("int32", L32), ("float32", L32), ("int64", L64), ("float64", L64)])
@pytest.mark.parametrize("dist", ["uniform", "few_unique", "sorted"])
def test_batch_segments(ps, ora, how, dtype, edge, dist):
    """Segments on both sides of the shortest radix length, of one and several
    tiles more, empty and tiny ones between; their digits (and the digits left
    out of 64-bit keys) are chosen segment by segment."""
    lens = [edge + 1, 0, edge, 3 * T32 * 8 + 5, 1, 700, edge + 4096 * 3, 5000, 2 * edge - 1]
    check_batch(ps, ora, lens, dtype, dist, how)


@pytest.mark.parametrize("dtype,n", [("int32", L32 + 5), ("int64", L64 + 5), ("int32", 20000)])
@pytest.mark.parametrize("how", ["call", "plan"])
def test_batch_of_one_long_segment(ps, ora, how, dtype, n):
    """No short segments: the instance table starts with the long bin."""
    check_batch(ps, ora, [n], dtype, "uniform", how)


def test_batch_long_runs_per_segment(ps):
    """64-bit segments with runs that leading bytes do not tell apart, longer
    than the fix kernel ranks, in segments of their own buffers and shared ones."""
    import torch
    segs = [clustered(200003, (300, 70, 2), 5, 1), clustered(150001, (150001,), 4, 2), clustered(300000, (65, 64, 500), 6, 3)]
    off = np.concatenate([[0], np.cumsum([s.size for s in segs])]).astype(np.int64)
    want = np.concatenate([np.sort(s) for s in segs])
    x = torch.from_numpy(np.concatenate(segs).view(np.int64)).cuda().view(torch.uint64)
    ps.sort_batch(x, torch.from_numpy(off).cuda())
    torch.cuda.synchronize()
    assert x.view(torch.int64).cpu().numpy().view(np.uint64).tobytes() == want.tobytes()


@pytest.mark.parametrize("how", ["call", "plan", "server"])
@pytest.mark.parametrize("dtype", ["int32", "float64"])
@pytest.mark.parametrize("lens", [
    [8193, 16384, 9000],                                # one small bin: a cluster per segment
    [16385, 65536, 30000, 8193, 131072],                # three and more small bins: one radix run
    [8193, 20000, 12289, 9216, 9217, 300000, 40000],    # a long segment takes the small bins along
    [8193 + 7 * i for i in range(300)],                 # one bin too large for clusters
    [70000, 500, 1025],
])
def test_batch_small_bins(ps, ora, how, dtype, lens):
    check_batch(ps, ora, lens, dtype, "uniform", how)


@pytest.mark.parametrize("dtype,n", [("int32", 300000), ("float64", 200001), ("int32", (3 << 24) - 1), ("float32", 3 << 24),
                                     ("int64", (3 << 23) + 5), ("float64", (1 << 26) + 1)])
@pytest.mark.parametrize("mode", ["exact", "regular"])
def test_pinned_host_keys(ps, ora, dtype, n, mode):
    """Automatic sorts of pinned host keys around the smallest size that is
    copied in groups, with a short last block."""
    import torch
    if n >= (1 << 26) and mode == "regular":
        pytest.skip("one large case")
    src = synth.keys_torch(n, dtype, "uniform", seed=n)
    h = torch.empty_like(src, device="cpu", pin_memory=True)
    h.copy_(src)
    ps.sort_host(h, mode)
    want = torch.sort(src)[0]
    assert torch.equal(h.cuda(), want)


def test_pinned_host_keys_short_last_block(ps, ora):
    """Copy groups whose last block ends a fix tile before the others, with runs
    longer than a thread orders in every block."""
    import torch
    L = 6144 * 1024 + 1                     # 4 blocks of L keys; the last has L - 3
    n = 4 * L - 3
    u = synth.splitmix64(77, n)
    top = u & ~np.uint64(0xFFFFFFFF)
    for b in range(4):                      # 90 keys of one leading half in every block
        at = b * L + 1000 * np.arange(90)
        top[at] = top[b * L]
    u = (top | (u & np.uint64(0xFFFFFFFF))).view(np.int64)
    h = torch.from_numpy(u.copy()).pin_memory()
    ps.sort_host(h)
    assert torch.equal(h.cuda(), torch.sort(torch.from_numpy(u).cuda())[0])
