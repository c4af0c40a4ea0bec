"""Inputs whose runs of equal leading bytes the sample misjudges: one value that
makes up most of a run, and a few neighbours of the same leading bytes that put
the run out of order unseen.  Results against the plain definition (the unique
order of the keys' bits; records by key and payload), and a bound on the time."""
from __future__ import annotations

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

TILE, TASK, ALONE = 4096, 8192, 16384  # fix tile, keys of a task, longest run of one CTA


@pytest.fixture(scope="module")
def ps():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2305_05245_gb300 as ps
    assert torch.cuda.is_available()
    return ps


def heavy(n, runs, rare, seed, low=16):
    """n uniform uint64 keys; runs[i] of them (at random places) are one value
    each, of which `rare` per run differ in the lowest `low` bits."""
    u = synth.splitmix64(seed, n)
    place = np.argsort(synth.splitmix64(seed + 1, n), kind="stable")
    bits = synth.splitmix64(seed + 2, len(runs) * rare) & np.uint64((1 << low) - 1)
    at = 0
    for i, m in enumerate(runs):
        idx = np.sort(place[at:at + m])
        u[idx] = u[idx[0]]
        odd = idx[(synth.splitmix64(seed + 3 + i, rare) % np.uint64(m)).astype(np.int64)]
        u[odd] ^= bits[i * rare:(i + 1) * rare]
        at += m
    return u


def sparse(n, share, seed, low=16):
    """Zeros but for a share of small values."""
    z = synth.splitmix64(seed, n)
    return np.where((z >> np.uint64(40)).astype(np.float64) < share * 2.0 ** 24, z & np.uint64((1 << low) - 1), np.uint64(0))


def check(ps, u, view=np.int64):
    import torch
    host = u.view(view)
    x = torch.from_numpy(host.copy()).cuda()
    ps.sort(x)
    torch.cuda.synchronize()
    got = x.cpu().numpy()
    if view == np.float64:  # order of the bits: negative values reversed, below the others
        s = np.int64(np.iinfo(np.int64).min)
        o = np.where(u.view(np.int64) < 0, ~u.view(np.int64), u.view(np.int64) ^ s).view(np.uint64)
        want = u[np.argsort(o, kind="stable")].view(view)
    else:
        want = np.sort(host, kind="stable")
    assert got.tobytes() == want.tobytes()


EDGES = [(65,), (TILE - 1,), (TILE,), (TILE + 1,), (ALONE - 1,), (ALONE,), (ALONE + 1,), (3 * TASK - 1,), (3 * TASK,),
         (3 * TASK + 1,), (9 * TASK + 77,), (200000, 100000, 33000, 16384, 5000, 100, 70)]


@pytest.mark.parametrize("runs", EDGES)
@pytest.mark.parametrize("view", [np.int64, np.float64])
@pytest.mark.parametrize("low", [3, 16, 30])
def test_one_value_and_rare_neighbours(ps, runs, view, low):
    check(ps, heavy((1 << 20) + 5, runs, 3, seed=sum(runs) + low, low=low), view)


@pytest.mark.parametrize("n,share", [(131073, 1e-3), (1 << 20, 1e-4), (1 << 20, 1e-6), ((1 << 23) + 1, 1e-5), (1 << 24, 0.0)])
@pytest.mark.parametrize("low", [8, 24])
def test_sparse(ps, n, share, low):
    check(ps, sparse(n, share, n, low))


def test_many_short_runs(ps):
    """Every tile holds runs longer than a thread orders, some out of order."""
    n = 1 << 21
    z = synth.splitmix64(5, n)
    u = ((z >> np.uint64(50)) << np.uint64(40)) ^ np.where(z & np.uint64(0xFFF), np.uint64(0), (z >> np.uint64(12)) & np.uint64(0xFFFF))
    check(ps, u)


@pytest.mark.parametrize("payload", ["index", "random"])
@pytest.mark.parametrize("runs,low", [((100,), 16), ((TILE + 1, 300), 16), ((ALONE,), 8), ((ALONE + 1, 40000), 24), ((300000,), 16)])
def test_records(ps, runs, low, payload):
    import torch
    n = (1 << 20) + 3
    k = heavy(n, runs, 3, seed=low + runs[0], low=low)
    p = np.arange(n, dtype=np.uint32) if payload == "index" else (synth.splitmix64(1, n) >> np.uint64(33)).astype(np.uint32)
    tk = torch.from_numpy(k.view(np.int64).copy()).cuda()
    tp = torch.from_numpy(p.view(np.int32).copy()).cuda()
    ps.sort_pairs(tk, tp)
    torch.cuda.synchronize()
    o = np.lexsort((p, k))
    assert tk.cpu().numpy().view(np.uint64).tobytes() == k[o].tobytes()
    assert tp.cpu().numpy().view(np.uint32).tobytes() == p[o].tobytes()


@pytest.mark.parametrize("how", ["call", "server"])
def test_segments(ps, how):
    """Segments of a batch (one buffer, and buffers of their own), several of them misjudged."""
    import torch
    segs = [sparse(400001, 1e-4, 1), heavy(300000, (100000, 5000, 90), 2, 2), synth.splitmix64(3, 140000), sparse(1 << 20, 1e-5, 4)]
    want = [np.sort(s.view(np.int64)) for s in segs]
    if how == "call":
        off = np.concatenate([[0], np.cumsum([s.size for s in segs])]).astype(np.int64)
        x = torch.from_numpy(np.concatenate(segs).view(np.int64)).cuda()
        ps.sort_batch(x, torch.from_numpy(off).cuda())
    else:
        parts = [torch.from_numpy(s.view(np.int64).copy()).cuda() for s in segs]
        torch.cuda.synchronize()
        srv = ps.Server(budget_bytes=1 << 30)
        left = {srv.submit(p) for p in parts}
        while left:
            for rid, status in srv.poll():
                assert status == 0
                left.discard(rid)
        srv.close()
        x = torch.cat(parts)
    torch.cuda.synchronize()
    assert x.cpu().numpy().tobytes() == np.concatenate(want).tobytes()


@pytest.mark.parametrize("share", [1e-4, 1e-6])
def test_pinned_host_keys(ps, share):
    """Blocks sorted by radix that stay order keys."""
    import torch
    n = (3 << 23) + 9
    u = sparse(n, share, 7).view(np.int64).copy()
    u[::2] = -u[::2]
    h = torch.from_numpy(u.copy()).pin_memory()
    ps.sort_host(h)
    assert torch.equal(h.cuda(), torch.sort(torch.from_numpy(u).cuda())[0])


def test_time_is_bounded(ps):
    """One value and rare neighbours: within a small factor of uniform keys' time
    (a run of this length sorted by one CTA alone takes thousands of times as long)."""
    import torch
    n = 1 << 22
    ms = []
    for u in (synth.splitmix64(1, n), sparse(n, 1e-4, 2), heavy(n, (n // 3,), 40, 3)):
        src = torch.from_numpy(u.view(np.int64).copy()).cuda()
        best = 1e9
        for _ in range(4):
            x = src.clone()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            ps.sort(x)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        ms.append(best)
    assert max(ms[1:]) < 20 * ms[0], ms
