"""Measured cases: symbolic LU of seeded sparsity patterns through the package's public entry points.

A case names an entry point ("call") and a pattern ("kind" and its sizes):

  call    device   symbolic_device: device CSR in, device L/U CSR, fill counts and supernodes out
          host     symbolic_host: the same from and to host arrays, copies included
          batch    batch_device: many device CSRs in one call
          counts   row_counts_noalloc: per-row sizes into the caller's buffers
          served   Server: a burst of requests submitted at once and collected in order
  kind    grid2d   5-point stencil, natural row-major order          (w, h, keep)
          grid3d   7-point stencil plus one random entry per row     (w, h, d, keep, extra)
          nd2d     5-point stencil, nested dissection, leaves of 64  (w, h, keep)
          banded   4-12 entries per row within a band                (n, band)
          mix      log-uniform orders, alternately grid2d and banded (count, n_lo, n_hi); "big" of the
                   members are nd2d grids of side big_side

Every pattern is nonsymmetric in structure and drawn on the GPU from the seed alone.
"""
import functools
import math

import numpy as np
import torch

import paper_2007_00840_gb300 as gs

ROWS = ("L_rowptr", "U_rowptr", "fill_count")


def listed():
    return [
        # one very small pattern: call latency, allocations and launches
        dict(name="device_grid2d_24", call="device", kind="grid2d", w=24, h=24, keep=0.7, chunk=0),
        # a small system in natural order: a long chain of dependent rows and few of them
        dict(name="device_grid2d_64", call="device", kind="grid2d", w=64, h=64, keep=0.7, chunk=0),
        # a 3D problem in natural order: wide band, dense factors
        dict(name="device_grid3d_32", call="device", kind="grid3d", w=32, h=32, d=32, keep=0.6, extra=1024, chunk=0),
        # an irregular band of odd order; rows of more than eight neighbours; another supernode limit
        dict(name="device_banded_15013", call="device", kind="banded", n=15013, band=211, chunk=64),
        # a ragged 2D system in natural order, near the largest whose visited sets stay on chip
        dict(name="device_grid2d_317x293", call="device", kind="grid2d", w=317, h=293, keep=0.7, chunk=0),
        # the large patterns of the served stream: fill-reducing order, sparse factors
        dict(name="device_nd_512", call="device", kind="nd2d", w=512, h=512, keep=0.8, chunk=0),
        # the largest single system
        dict(name="device_nd_1024", call="device", kind="nd2d", w=1024, h=1024, keep=0.8, chunk=0),
        # a solver with host data: copies in and out count
        dict(name="host_nd_203x197", call="host", kind="nd2d", w=203, h=197, keep=0.8, chunk=0),
        # sizes of the factors, asked for where nothing may be allocated
        dict(name="counts_grid3d_27x25x29", call="counts", kind="grid3d", w=27, h=25, d=29, keep=0.6, extra=700),
        # a few dozen small systems at once
        dict(name="batch_mix_37", call="batch", kind="mix", count=37, n_lo=500, n_hi=3000, big=0, big_side=0, chunk=0),
        # the many-matrix workload at full size
        dict(name="batch_mix_512", call="batch", kind="mix", count=512, n_lo=500, n_hi=20000, big=0, big_side=0,
             chunk=0),
        # a burst at the server: small requests and a large one in the same queue
        dict(name="served_burst_60", call="served", kind="mix", count=60, n_lo=500, n_hi=20000, big=1, big_side=512),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["device", "device", "device", "device", "host", "counts", "batch", "batch", "served"])
    if call == "batch":
        lo = _log(rng, 300, 2000)
        return dict(call=call, kind="mix", count=_log(rng, 6, 360), n_lo=lo, n_hi=_log(rng, lo + 50, 20000), big=0,
                    big_side=0, chunk=rng.choice([0, 0, 64]))
    if call == "served":
        return dict(call=call, kind="mix", count=_log(rng, 8, 120), n_lo=500, n_hi=_log(rng, 2000, 20000),
                    big=rng.choice([0, 1, 1, 2]), big_side=rng.randint(350, 512))
    kind = rng.choice(["grid2d", "grid3d", "nd2d", "banded"])
    top = 60000 if call == "counts" else 90000
    if kind == "banded":
        c = dict(n=_log(rng, 500, 40000), band=_log(rng, 8, 256))
    elif kind == "grid3d":
        w, h, d = (_log(rng, 9, 33) for _ in range(3))
        c = dict(w=w, h=h, d=d, keep=rng.choice([0.5, 0.6, 0.8]), extra=_log(rng, 64, 1024))
    elif kind == "nd2d":
        w = _log(rng, 20, 240 if call == "counts" else 1000)
        c = dict(w=w, h=max(16, int(w * rng.uniform(0.7, 1.0))), keep=rng.choice([0.7, 0.8]))
    else:
        w = _log(rng, 20, 300)
        c = dict(w=w, h=min(top // w, max(16, int(w * rng.uniform(0.6, 1.3)))), keep=rng.choice([0.6, 0.7, 0.8]))
    if call != "counts":
        c["chunk"] = rng.choice([0, 0, 0, 64, 256])
    return dict(call=call, kind=kind, **c)


# ------------------------------------------------------------------ patterns

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed & 0x7FFFFFFFFFFFFFFF)
    return g


def _csr(n, rows, cols):
    """int32 CSR of (row, column) pairs: sorted, duplicates dropped, diagonal added."""
    i = torch.arange(n, device="cuda")
    key = torch.unique(torch.cat([rows * n + cols, i * n + i]))
    rowptr = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    rowptr[1:] = torch.cumsum(torch.bincount(key // n, minlength=n), 0)
    return rowptr, (key % n).to(torch.int32)


def _stencil(dims, keep, g):
    """Directed neighbour pairs of a grid (x fastest), each kept with probability `keep`."""
    n = math.prod(dims)
    v = torch.arange(n, device="cuda")
    rows, cols, step = [], [], 1
    for size in dims:
        x = (v // step) % size
        for d, inside in ((-step, x > 0), (step, x < size - 1)):
            m = inside & (torch.rand(n, generator=g, device="cuda") < keep)
            rows.append(v[m])
            cols.append(v[m] + d)
        step *= size
    return n, torch.cat(rows), torch.cat(cols)


@functools.lru_cache(maxsize=None)
def _nd_order(w, h):
    """Cells (y * 4096 + x) of a w x h box in nested-dissection order: the longer side is split, the two
    halves come first and the separator line last; boxes of at most 64 cells row by row."""
    if w <= 0 or h <= 0:
        return torch.empty(0, dtype=torch.int64)
    if w * h <= 64:
        return (torch.arange(h)[:, None] * 4096 + torch.arange(w)[None, :]).reshape(-1)
    if w >= h:
        m = (w - 1) // 2
        return torch.cat([_nd_order(m, h), _nd_order(w - m - 1, h) + (m + 1), torch.arange(h) * 4096 + m])
    m = (h - 1) // 2
    return torch.cat([_nd_order(w, m), _nd_order(w, h - m - 1) + (m + 1) * 4096, m * 4096 + torch.arange(w)])


def _grid2d(w, h, keep, g):
    return _csr(*_stencil((w, h), keep, g))


def _grid3d(w, h, d, keep, extra, g):
    n, r, c = _stencil((w, h, d), keep, g)
    off = torch.randint(1, extra + 1, (n,), generator=g, device="cuda")
    off *= torch.randint(0, 2, (n,), generator=g, device="cuda") * 2 - 1
    v = torch.arange(n, device="cuda")
    m = (v + off >= 0) & (v + off < n)
    return _csr(n, torch.cat([r, v[m]]), torch.cat([c, (v + off)[m]]))


def _nd2d(w, h, keep, g):
    n, r, c = _stencil((w, h), keep, g)
    o = _nd_order(w, h).cuda()
    perm = torch.empty(n, dtype=torch.int64, device="cuda")
    perm[(o // 4096) * w + o % 4096] = torch.arange(n, device="cuda")
    return _csr(n, perm[r], perm[c])


def _banded(n, band, g):
    v = torch.arange(n, device="cuda")
    k = torch.randint(3, 12, (n, 1), generator=g, device="cuda")
    d = torch.randint(-band, band + 1, (n, 11), generator=g, device="cuda")
    c = v[:, None] + d
    m = (torch.arange(11, device="cuda")[None, :] < k) & (c >= 0) & (c < n)
    return _csr(n, v[:, None].expand(n, 11)[m], c[m])


def _members(case):
    """Orders and bands of a mix's members: log-uniform, evenly spread over their ranges."""
    pairs = (case["count"] + 1) // 2
    for m in range(case["count"]):
        a = (m // 2 + 0.5) / pairs
        n = int(round(case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** a))
        if m < case["big"]:
            side = case["big_side"]
            yield dict(kind="nd2d", w=side, h=side, keep=0.8)
        elif m % 2 == 0:
            w = math.isqrt(n - 1) + 1
            yield dict(kind="grid2d", w=w, h=-(-n // w), keep=0.7)
        else:
            yield dict(kind="banded", n=n, band=int(round(8 * 32 ** ((m // 2 * 0.381966) % 1.0))))


def _pattern(c, g):
    if c["kind"] == "grid2d":
        return _grid2d(c["w"], c["h"], c["keep"], g)
    if c["kind"] == "grid3d":
        return _grid3d(c["w"], c["h"], c["d"], c["keep"], c["extra"], g)
    if c["kind"] == "nd2d":
        return _nd2d(c["w"], c["h"], c["keep"], g)
    return _banded(c["n"], c["band"], g)


def _room(c):
    """At most this many entries of L, U and the supernode list for any pattern of these sizes."""
    n = c["n"] if c["kind"] == "banded" else c["w"] * c["h"] * c.get("d", 1)
    if c["kind"] == "nd2d":
        return int(5 * n * math.log2(n)) + 64 * n + 2
    band = {"grid2d": c.get("w"), "grid3d": max(c.get("w", 1) * c.get("h", 1), c.get("extra", 0)),
            "banded": c.get("band")}[c["kind"]]
    return 2 * n * (band + 1) + 2


# ---------------------------------------------------------------------- runs

def prepare(case, seed):
    call, g = case["call"], _generator(seed)
    parts = list(_members(case)) if case["kind"] == "mix" else [case]
    st = {"call": call, "mats": [_pattern(c, g) for c in parts], "opts": None}
    if case.get("chunk"):
        st["opts"] = gs.options(chunk_size=case["chunk"])
    if call == "counts":
        n = st["mats"][0][0].numel() - 1
        st["out"] = [torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(3)]
        return st
    # the solver's arena: the index arrays of the factors go there, end to end, whatever their sizes
    st["arena"] = torch.zeros(sum(_room(c) for c in parts), dtype=torch.int32, device="cuda")
    if call == "host":
        st["mats"] = [tuple(t.cpu().numpy() for t in m) for m in st["mats"]]
        st["arena"] = st["arena"].cpu().numpy()
    elif call == "served":
        st["server"] = gs.Server(streams=2, max_batch=512)
    return st


def _factor(st):
    if st["call"] == "device":
        return [gs.symbolic_device(*st["mats"][0], opts=st["opts"])]
    if st["call"] == "host":
        return [gs.symbolic_host(*st["mats"][0], opts=st["opts"])]
    if st["call"] == "batch":
        return gs.batch_device(st["mats"], opts=st["opts"])
    tickets = [st["server"].submit(rp, ci) for rp, ci in st["mats"]]
    return [st["server"].wait(t)[0] for t in tickets]


def run(st):
    if st["call"] == "counts":
        gs.row_counts_noalloc(*st["mats"][0], *st["out"])
        return dict(zip(("nnz_L", "nnz_U", "fill_count"), st["out"]))
    res = _factor(st)
    index = [getattr(r, f) for f in ("L_colidx", "U_colidx", "super_start") for r in res]
    used = sum(r.nnz_L + r.nnz_U + r.n_super + 1 for r in res)
    if st["call"] == "host":
        np.concatenate(index, out=st["arena"][:used])
        rows = {f: getattr(res[0], f) for f in ROWS}
    else:
        torch.cat(index, out=st["arena"][:used])
        rows = {f: getattr(res[0], f) if len(res) == 1 else torch.cat([getattr(r, f) for r in res]) for f in ROWS}
    return dict(rows, index=st["arena"])


def exact(case, seed):
    return None  # every output is a whole number


@functools.lru_cache(maxsize=None)
def _bytes(key):
    st = prepare(dict(key), 1)
    total = sum(a.nbytes for m in st["mats"] for a in m)
    if st["call"] == "counts":
        return total + sum(t.nbytes for t in st["out"])
    for r in _factor(st):
        total += 4 * (r.nnz_L + r.nnz_U) + 8 * 2 * (r.n + 1) + 4 * r.n + 4 * (r.n_super + 1)
    return total


def work(case):
    # a graph search on whole numbers: no floating-point operations. What has to move is the CSR, read once, and
    # the result, written once (its size is a property of the pattern: it is counted on one drawn pattern)
    return {"bytes": _bytes(tuple(sorted((k, v) for k, v in case.items() if k != "name"))), "flops": 0}
