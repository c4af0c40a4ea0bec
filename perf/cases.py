"""Performance cases: the work that users of the library have it do.

Every case is one call (for the server: one burst of requests) through the
package's public entry points, on keys that were not sorted before: a pass
first copies the pristine keys into the buffer that the call sorts in place,
as a program does that keeps its input.  Sizes, types and distributions are
those of the repository's benchmark configurations and tests: single sorts of
a thousand to 2^30 keys, key + payload records, fixed-size records with an
embedded key, batches of segments with log-uniform lengths, keys in pinned
host memory, and a burst of mixed requests to the sort server.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2305_05245_gb300 as ps

KEY_BYTES = {"int32": 4, "uint32": 4, "float32": 4, "int64": 8, "uint64": 8, "float64": 8}
SIGNED = {"uint32": torch.int32, "uint64": torch.int64}
DISTS = ("uniform", "sorted", "reverse", "few_unique", "gaussian", "almost_sorted", "three_valued")


def listed():
    return [
        # a short request on its own, where the call's latency is all there is
        dict(name="sort_1k_f32", op="sort", n=1000, dtype="float32", dist="uniform", mode="exact"),
        # a middling request of odd length, several tiles long
        dict(name="sort_41k_i64", op="sort", n=40961, dtype="int64", dist="uniform", mode="exact"),
        # the paper's shape: 64 blocks and 64 partitions given by the caller,
        # regular sampling, with the record of pivots, splits and offsets
        dict(name="method_1m_i32", op="sort", n=1 << 20, dtype="int32", dist="uniform", mode="regular",
             n_blocks=64, n_parts=64, trace=True),
        # an ordinary sort of many equal keys (categories), odd length
        dict(name="sort_3m_f32_few", op="sort", n=3000001, dtype="float32", dist="few_unique", mode="regular"),
        # 2^26 keys, the middle of the benchmark's single sorts
        dict(name="sort_64m_i32", op="sort", n=1 << 26, dtype="int32", dist="uniform", mode="exact"),
        dict(name="sort_64m_f64", op="sort", n=1 << 26, dtype="float64", dist="gaussian", mode="exact"),
        # the largest single sort, the benchmark's default workload
        dict(name="sort_1g_i64", op="sort", n=1 << 30, dtype="int64", dist="uniform", mode="exact"),
        # key + payload records (payload = original index): an argsort
        dict(name="pairs_256m", op="pairs", n=1 << 28, dist="uniform", mode="exact"),
        # Table 1's Particle: 96-byte records with an embedded key
        dict(name="particle_10m", op="struct", n=10000000, record_bytes=96, key_offset=0, dist="uniform",
             mode="exact"),
        # thousands of segments of very different lengths in one call
        dict(name="batch_4k_i32", op="batch", segs=4000, lo=6, hi=22, dtype="int32", dist="uniform", mode="exact"),
        # keys in pinned host memory, sorted where they lie
        dict(name="host_64m_i32", op="host", n=1 << 26, dtype="int32", dist="uniform", mode="exact"),
        # a burst of requests of mixed sizes and types at the sort server
        dict(name="server_burst", op="server", reqs=60, lo=10, hi=23, mode="exact"),
    ]


def _log_int(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    op = rng.choice(["sort"] * 6 + ["pairs", "struct", "batch", "batch", "plan", "host", "server", "noalloc"])
    mode = rng.choice(["exact", "exact", "regular"])
    dtype = rng.choice(sorted(KEY_BYTES))
    dists = [d for d in DISTS if d != "gaussian" or dtype.startswith("float")]
    if op in ("pairs", "struct", "server"):
        dists.remove("gaussian") if "gaussian" in dists else None
    dist = rng.choice(["uniform"] + dists)
    if op in ("sort", "noalloc", "host"):
        top = {"sort": 1 << 28, "noalloc": 1 << 20, "host": 1 << 26}[op]
        n = _log_int(rng, 100, top) if rng.random() < 0.8 else 1 << rng.randint(8, top.bit_length() - 1)
        c = dict(op=op, n=n, dtype=dtype, dist=dist, mode=mode)
        if op == "sort" and rng.random() < 0.2:
            c["n_blocks"] = rng.choice([1, 3, 16, 48, 128])
            c["n_parts"] = rng.choice([1, 16, 48, 128])
            c["trace"] = rng.random() < 0.5
        return c
    if op == "pairs":
        return dict(op=op, n=_log_int(rng, 1000, 1 << 27), dist=dist, mode=mode)
    if op == "struct":
        rb = 8 * rng.choice([2, 2, 3, 5, 12, 16])
        return dict(op=op, n=_log_int(rng, 1000, (1 << 31) // rb), record_bytes=rb,
                    key_offset=8 * rng.randint(0, rb // 8 - 1), dist=dist, mode=mode)
    if op in ("batch", "plan"):
        hi = rng.randint(10, 22)
        return dict(op=op, segs=_log_int(rng, 20, min(20000, (1 << 31) >> hi)), lo=rng.randint(4, hi - 2), hi=hi,
                    dtype=dtype, dist=dist, mode=mode)
    return dict(op="server", reqs=rng.randint(8, 60), lo=rng.randint(8, 14), hi=rng.randint(16, 23), mode=mode)


def _lengths(count, lo, hi):
    """count lengths spread evenly over [2^lo, 2^hi] on a log scale."""
    u = (np.arange(count) + 0.5) / count
    return np.floor(2.0 ** (lo + (hi - lo) * u)).astype(np.int64)


def _bits(n, dtype, gen):
    """n uniform keys: integers over the full range, floats in [0, 1)."""
    if dtype in ("int32", "uint32"):
        return torch.randint(-(1 << 31), 1 << 31, (n,), dtype=torch.int32, device="cuda", generator=gen)
    if dtype in ("int64", "uint64"):
        return torch.randint(-(1 << 63), (1 << 63) - 1, (n,), dtype=torch.int64, device="cuda", generator=gen)
    return torch.rand(n, dtype=getattr(torch, dtype), device="cuda", generator=gen)


def _order(x, dtype):
    """Indices and values of x (signed storage) in ascending key order, stable."""
    if dtype in SIGNED:
        flip = torch.tensor(-(1 << (8 * KEY_BYTES[dtype] - 1)), dtype=x.dtype, device=x.device)
        v, i = torch.sort(x ^ flip, stable=True)
        return v ^ flip, i
    return torch.sort(x, stable=True)


def _keys(n, dtype, dist, gen):
    """n keys as a device tensor (unsigned types in signed storage)."""
    st = SIGNED.get(dtype, getattr(torch, dtype))
    if dist == "gaussian":
        return torch.randn(n, dtype=st, device="cuda", generator=gen)
    if dist == "few_unique":
        vals = _bits(16, dtype, gen)
        return vals[torch.randint(0, 16, (n,), device="cuda", generator=gen)]
    if dist == "three_valued":
        return torch.randint(0, 3, (n,), device="cuda", generator=gen).to(st)
    if dist == "almost_sorted":
        k = max(1, math.isqrt(n) // 2)
        a = (torch.arange(n, device="cuda") + int(torch.randint(0, 1000, (1,), device="cuda", generator=gen))).to(st)
        p = torch.randperm(n, device="cuda", generator=gen)[:2 * k] if n < (1 << 20) else \
            torch.unique(torch.randint(0, n, (2 * k,), device="cuda", generator=gen))
        h = p.numel() // 2
        q = torch.cat([p[h:2 * h], p[:h]])
        a[p[:2 * h]] = a[q].clone()
        return a
    x = _bits(n, dtype, gen)
    if dist in ("sorted", "reverse"):
        x = _order(x, dtype)[0]
        if dist == "reverse":
            x = torch.flip(x, [0])
    return x


def _typed(x, dtype):
    return x.view(getattr(torch, dtype)) if dtype in SIGNED else x


def _plain(x):
    """x with unsigned keys in signed storage again, as other tensor code takes them."""
    signed = {torch.uint32: torch.int32, torch.uint64: torch.int64}
    return x.view(signed[x.dtype]) if x.dtype in signed else x


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _requests(case, seed):
    """(keys, dtype) of every request of a burst: four types, four shapes of data."""
    gen = _gen(seed)
    lens = _lengths(case["reqs"], case["lo"], case["hi"])
    order = np.random.default_rng(case["reqs"]).permutation(case["reqs"])  # arrival order
    kinds = ("int32", "int64", "float32", "float64")
    dists = ("uniform", "few_unique", "sorted", "uniform", "reverse")
    return [(_keys(int(lens[i]), kinds[i % 4], dists[i % 5], gen), kinds[i % 4]) for i in order]


def _offsets(case, seed):
    lens = _lengths(case["segs"], case["lo"], case["hi"])
    lens = np.random.default_rng(seed).permutation(lens)
    return np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)


def _records(case, seed):
    gen = _gen(seed)
    words = case["record_bytes"] // 8
    r = torch.randint(0, 1 << 62, (case["n"], words), dtype=torch.int64, device="cuda", generator=gen)
    r[:, case["key_offset"] // 8] = _keys(case["n"], "uint64", case["dist"], gen)
    return r


def prepare(case, seed):
    op = case["op"]
    st = dict(case=case)
    if op == "server":
        st["src"] = [k for k, _ in _requests(case, seed)]
        st["work"] = [torch.empty_like(k) for k in st["src"]]
        st["server"] = ps.Server(budget_bytes=32 << 30, max_inflight=1024)
    elif op == "struct":
        st["src"] = _records(case, seed)
        st["work"] = torch.empty_like(st["src"])
    elif op in ("batch", "plan"):
        off = _offsets(case, seed)
        st["src"] = _typed(_keys(int(off[-1]), case["dtype"], case["dist"], _gen(seed)), case["dtype"])
        st["work"] = torch.empty_like(st["src"])
        if op == "batch":
            st["offsets"] = torch.from_numpy(off).cuda()
        else:
            st["plan"] = ps.BatchPlan(off, getattr(torch, case["dtype"]), case["mode"])
    elif op == "pairs":
        st["src"] = _keys(case["n"], "uint64", case["dist"], _gen(seed))
        st["pos"] = torch.arange(case["n"], dtype=torch.int64, device="cuda").to(torch.int32)
        st["work"] = torch.empty_like(st["src"])
        st["payload"] = torch.empty_like(st["pos"])
    else:
        st["src"] = _typed(_keys(case["n"], case["dtype"], case["dist"], _gen(seed)), case["dtype"])
        st["work"] = torch.empty_like(st["src"], device="cpu", pin_memory=True) if op == "host" else \
            torch.empty_like(st["src"])
    return st


def run(state):
    case = state["case"]
    op, mode = case["op"], case["mode"]
    if op == "server":
        for w, s in zip(state["work"], state["src"]):
            w.copy_(s)
        torch.cuda.current_stream().synchronize()  # keys have to be ready before they are submitted
        srv = state["server"]
        left = {srv.submit(w, mode) for w in state["work"]}
        while left:
            for rid, status in srv.poll():
                if status != 0:
                    raise RuntimeError("request %d failed: %d" % (rid, status))
                left.discard(rid)
        return list(state["work"])
    work = state["work"]
    work.copy_(state["src"], non_blocking=True)
    if op == "sort":
        tr = ps.sort(work, mode, n_blocks=case.get("n_blocks", 0), n_parts=case.get("n_parts", 0),
                     trace=case.get("trace", False))
        if tr is not None:
            return dict(keys=_plain(work), pivots=_plain(tr.pivots), c=tr.c, splits=tr.splits, offsets=tr.offsets)
    elif op == "noalloc":
        ps.sort_noalloc(work, mode)
    elif op == "pairs":
        state["payload"].copy_(state["pos"])
        ps.sort_pairs(work, state["payload"], mode)
        return [work, state["payload"]]
    elif op == "struct":
        ps.sort_struct(work, case["record_bytes"], case["key_offset"], mode)
    elif op == "batch":
        ps.sort_batch(work, state["offsets"], mode)
    elif op == "plan":
        state["plan"].run(work)
    else:
        ps.sort_host(work, mode)
    return _plain(work)


def work(case):
    """Every key (record) read once and written once; no arithmetic of its own."""
    op = case["op"]
    if op == "server":
        lens = _lengths(case["reqs"], case["lo"], case["hi"])
        b = sum(int(n) * (4, 8, 4, 8)[i % 4] for i, n in enumerate(lens))
    elif op in ("batch", "plan"):
        b = int(_lengths(case["segs"], case["lo"], case["hi"]).sum()) * KEY_BYTES[case["dtype"]]
    elif op == "struct":
        b = case["n"] * case["record_bytes"]
    elif op == "pairs":
        b = case["n"] * 12
    else:
        b = case["n"] * KEY_BYTES[case["dtype"]]
    return {"bytes": 2 * b, "flops": 0}


def _exact_keys(x, dtype):
    v = _order(x, dtype)[0]
    return v.double() if dtype.startswith("float") else v


def exact(case, seed):
    op = case["op"]
    if op == "server":
        return [_exact_keys(k, d) for k, d in _requests(case, seed)]
    if op == "struct":
        r = _records(case, seed)
        return r[_order(r[:, case["key_offset"] // 8].contiguous(), "uint64")[1]]
    if op == "pairs":
        v, i = _order(_keys(case["n"], "uint64", case["dist"], _gen(seed)), "uint64")
        return [v, i.to(torch.int32)]
    if op in ("batch", "plan"):
        off = _offsets(case, seed)
        x = _keys(int(off[-1]), case["dtype"], case["dist"], _gen(seed))
        parts = [_order(x[int(a):int(b)], case["dtype"])[0] for a, b in zip(off[:-1], off[1:])]
        x = torch.cat(parts)
        return x.double() if case["dtype"].startswith("float") else x
    x = _exact_keys(_keys(case["n"], case["dtype"], case["dist"], _gen(seed)), case["dtype"])
    if op == "host":
        x = x.cpu()
    if case.get("trace"):
        return dict(keys=x, pivots=None, c=None, splits=None, offsets=None)
    return x
