"""The exchanges that programs run with this library, as measurable cases.

Every case builds a communication pattern, binds persistent requests to device buffers (what a
program does once), and measures one pass: start and wait (or start and a stream-ordered wait)
of those requests, through the Python binding.  Patterns are plain integer arrays that a program
keeps from step to step, so they are made once per process; payloads come from the seed.

Kinds:
  stencil     halo exchange of a structured 2D / 3D grid, or its gradient
  spmv        halo exchange of a row-partitioned sparse matrix-vector product, its gradient, or
              both through torch.autograd
  batch       many uneven SpMV halos started together
  alltoallw   stencil halo described by strided datatypes instead of send lists
  alltoallv   dense personalised exchange with uneven counts

"path" is "forward", "backward" (the reverse exchange alone) or "train" (both through autograd);
"alg" is the standard exchange or the locality-aware three-step one; "wait" is "host" (the call
returns when the exchange is done) or "stream" (later work on the stream waits for it).
"""
import functools
import math
import random

import numpy as np
import torch

import paper_2309_07337_gb300 as gbx
from paper_2309_07337_gb300 import autograd
from paper_2309_07337_gb300 import patterns as pt

TORCH = {"f64": torch.float64, "f32": torch.float32, "bytes": torch.uint8}
BYTES = {"f64": 8, "f32": 4, "bytes": 1}


def _stencil(name, block, ranks, comps, ppn, **kw):
    c = {"name": name, "kind": "stencil", "bx": block[0], "by": block[1], "bz": block[2], "rx": ranks[0],
         "ry": ranks[1], "rz": ranks[2], "comps": comps, "ppn": ppn, "dtype": "f64", "neighbors": "all",
         "path": "forward", "alg": "standard", "accumulate": False, "wait": "stream"}
    c.update(kw)
    return c


def _spmv(name, n, ranks, nnz, **kw):
    c = {"name": name, "kind": "spmv", "n": n, "ranks": ranks, "ppn": 32, "nnz": nnz, "dtype": "f64",
         "pattern": 2311, "path": "forward", "alg": "standard", "accumulate": False, "wait": "stream"}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: a 2D 5-point Laplacian on 256 x 256 points over 16 ranks, one value
        # per point (24 KB moved): launch and wait latency
        _stencil("stencil2d_256_small", (64, 64, 1), (4, 4, 1), 1, 4, neighbors="faces", wait="host"),
        # a ragged 3D block with three values per point (24-byte elements), a last node that is
        # only partly filled, through the locality-aware form: an ordinary small solver step
        _stencil("stencil3d_ragged_locality", (13, 11, 9), (6, 5, 4), 3, 7, alg="locality", wait="host"),
        # an ordinary 3D multi-component solver: 256^3 points, 8 values per point, 64 ranks per
        # node, locality-aware
        _stencil("stencil3d_256_locality", (32, 32, 32), (8, 8, 8), 8, 64, alg="locality"),
        # the large 3D solver: 512^3 points over 4096 ranks, standard exchange
        _stencil("stencil3d_512", (32, 32, 32), (16, 16, 16), 8, 64),
        # its reverse exchange: gradients of the halo summed back into the field
        _stencil("stencil3d_512_backward", (32, 32, 32), (16, 16, 16), 8, 64, path="backward"),
        # the halo of a 2^20-row sparse matrix over 1024 ranks, fp64: the iterative solver's
        # exchange before every matrix-vector product
        _spmv("spmv_2e20", 1 << 20, 1024, 20),
        # the same through the locality-aware form
        _spmv("spmv_2e20_locality", 1 << 20, 1024, 20, alg="locality"),
        # training through a distributed matrix-vector product: forward and gradient by
        # torch.autograd, fp32
        _spmv("spmv_2e20_train_f32", 1 << 20, 1024, 20, dtype="f32", path="train"),
        # an odd, middle-sized matrix: gradients accumulated into an existing buffer in the
        # node-blocked order of the locality-aware form
        _spmv("spmv_300k_accumulate", 300007, 509, 13, path="backward", alg="locality", accumulate=True, ppn=24,
              wait="host"),
        # a multigrid-like set of 16 uneven patterns, fp32 and fp64, started together
        {"name": "batch_16", "kind": "batch", "count": 16, "log_lo": 14, "log_hi": 20, "pattern": 7, "ppn": 32},
        # a component-major 3D field whose messages are strided datatypes
        {"name": "alltoallw_soa", "kind": "alltoallw", "bx": 24, "by": 20, "bz": 28, "rx": 6, "ry": 5, "rz": 4,
         "comps": 5, "ppn": 8, "dtype": "f64", "layout": "soa"},
        # a dense exchange (a distributed transpose) with uneven blocks of 24-byte records
        {"name": "alltoallv_dense", "kind": "alltoallv", "ranks": 256, "ppn": 16, "elem": 24, "count": 40,
         "dtype": "bytes", "pattern": 5, "alg": "standard", "wait": "host"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["stencil", "stencil", "stencil", "spmv", "spmv", "spmv", "batch", "alltoallw", "alltoallv"])
    common = {"path": rng.choice(["forward", "forward", "backward", "train"]),
              "alg": rng.choice(["standard", "locality"]), "wait": rng.choice(["host", "stream"]),
              "dtype": rng.choice(["f64", "f32"])}
    common["accumulate"] = common["path"] == "backward" and rng.random() < 0.3
    if kind == "stencil":
        two = rng.random() < 0.25
        while True:
            if two:
                block, ranks = (_log(rng, 5, 300), _log(rng, 5, 300), 1), (_log(rng, 2, 24), _log(rng, 2, 24), 1)
            else:
                block = tuple(_log(rng, 4, 40) for _ in range(3))
                ranks = tuple(_log(rng, 2, 14) for _ in range(3))
            comps = _log(rng, 1, 16)
            if np.prod(block) * np.prod(ranks) * comps * BYTES[common["dtype"]] <= 2 << 30:
                break
        return dict({k: v for k, v in _stencil("", block, ranks, comps, _log(rng, 1, np.prod(ranks)), **common,
                                               neighbors=rng.choice(["all", "faces"])).items() if k != "name"})
    if kind == "spmv":
        return {k: v for k, v in _spmv("", _log(rng, 5000, 1 << 20), _log(rng, 16, 1024), rng.randint(8, 24), **common,
                                       ppn=_log(rng, 4, 64), pattern=rng.randrange(1 << 20)).items() if k != "name"}
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(3, 16), "log_lo": 12, "log_hi": rng.randint(15, 20),
                "pattern": rng.randrange(1 << 20), "ppn": _log(rng, 4, 64)}
    if kind == "alltoallw":
        return {"kind": "alltoallw", "bx": _log(rng, 4, 32), "by": _log(rng, 4, 32), "bz": _log(rng, 4, 32),
                "rx": rng.randint(2, 6), "ry": rng.randint(2, 6), "rz": rng.randint(2, 6), "comps": _log(rng, 1, 8),
                "ppn": _log(rng, 2, 16), "dtype": common["dtype"], "layout": rng.choice(["soa", "aos"])}
    dtype = rng.choice(["bytes", "f32", "f64"])
    elem = rng.choice([3, 6, 12, 24, 40]) if dtype == "bytes" else BYTES[dtype] * rng.choice([1, 1, 2, 8])
    ranks = _log(rng, 8, 512)
    count = max(1, min(_log(rng, 1, 200), (300 << 20) // (ranks * ranks * elem)))
    return {"kind": "alltoallv", "ranks": ranks, "ppn": _log(rng, 2, 32), "elem": elem, "count": count,
            "dtype": dtype, "pattern": rng.randrange(1 << 20), "alg": common["alg"], "wait": common["wait"]}


# ------------------------------------------------------------------ the patterns

@functools.lru_cache(maxsize=2)
def _pattern_of(key):
    """The pattern(s) of a case and their index arrays on the device."""
    case = dict(key)
    if case["kind"] == "stencil":
        d = 2 if case["bz"] == 1 and case["rz"] == 1 else 3
        block, ranks = [case["b" + a] for a in "xyz"][:d], [case["r" + a] for a in "xyz"][:d]
        p = pt.stencil([b * r for b, r in zip(block, ranks)], ranks, case["ppn"], case["comps"], case["dtype"],
                       case["neighbors"])
    elif case["kind"] == "spmv":
        p = pt.spmv_halo_torch(case["n"], case["ranks"], case["ppn"], case["nnz"], case["pattern"], case["dtype"])
    elif case["kind"] == "batch":
        r = random.Random(case["pattern"])
        ps = [pt.spmv_halo_torch(_log(r, 1 << case["log_lo"], 1 << case["log_hi"]), r.randint(64, 1024), case["ppn"],
                                 r.randint(8, 32), r.randrange(1 << 20), r.choice(["f32", "f64"]), band=2048)
              for _ in range(case["count"])]
        return ps, [gbx.DevicePattern(p) for p in ps]
    elif case["kind"] == "alltoallw":
        block, ranks = [case["b" + a] for a in "xyz"], [case["r" + a] for a in "xyz"]
        w = pt.stencil_w([b * r for b, r in zip(block, ranks)], ranks, case["ppn"], case["comps"], case["dtype"],
                         layout=case["layout"])
        return w, gbx.DeviceWPattern(w)
    else:
        P = case["ranks"]
        rng = np.random.default_rng(case["pattern"])
        cnt = rng.integers(0, 2 * case["count"] + 1, size=(P, P))     # cnt[r, d]: elements r sends to d
        sd, rd = np.cumsum(cnt, 1) - cnt, np.cumsum(cnt.T, 1) - cnt.T
        sb = np.concatenate([[0], np.cumsum(cnt.sum(1))]) * case["elem"]
        rb = np.concatenate([[0], np.cumsum(cnt.sum(0))]) * case["elem"]
        host = {"cnt": cnt, "sd": sd, "rd": rd, "sb": sb, "rb": rb}
        i32 = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda()  # noqa: E731
        dev = {"sendcounts": i32(cnt), "sdispls": i32(sd), "recvcounts": i32(cnt.T), "rdispls": i32(rd),
               "send_base": torch.from_numpy(sb[:-1].copy()).cuda(), "recv_base": torch.from_numpy(rb[:-1].copy()).cuda()}
        return host, dev
    return p, gbx.DevicePattern(p)


def _pattern(case):
    return _pattern_of(tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "path", "alg", "wait", "accumulate"))))


def _source_of_slot(p):
    """Per receive slot, the element of the send buffer that it gets (its global index names it)."""
    s = p.elem_size
    rank = np.repeat(np.arange(p.P), np.diff(p.send_slot_ptr))
    el = np.asarray(p.send_base)[rank] // s + p.send_idx
    of = torch.full((int(p.global_sidx.max()) + 1,), -1, dtype=torch.int64)
    of[torch.from_numpy(p.global_sidx)] = torch.from_numpy(el)
    return of[torch.from_numpy(p.global_ridx)]


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _values(kind, n, dtype, g):
    """Field values of a stencil are uniform in (-1, 1); vectors and gradients are normal."""
    if dtype == torch.uint8:
        return torch.randint(0, 256, (n,), generator=g, device="cuda", dtype=torch.uint8)
    if kind in ("stencil", "alltoallw"):
        return torch.rand(n, generator=g, device="cuda", dtype=dtype).mul_(2).sub_(1)
    return torch.randn(n, generator=g, device="cuda", dtype=dtype)


def _payload(case, seed):
    """The random inputs of a case, the same for prepare() and exact()."""
    g, kind = _gen(seed), case["kind"]
    dt = TORCH[case["dtype"]] if "dtype" in case else None
    p, _ = _pattern(case)
    if kind == "batch":
        return {"x": [_values(kind, q.sendbuf_bytes // BYTES[q.dtype], TORCH[q.dtype], g) for q in p]}
    if kind == "alltoallv":
        return {"x": _values(kind, int(p["sb"][-1]) // BYTES[case["dtype"]], dt, g)}
    n, m = p.sendbuf_bytes // BYTES[case["dtype"]], p.recvbuf_bytes // BYTES[case["dtype"]]
    if kind == "alltoallw" or case["path"] == "forward":
        return {"x": _values(kind, n, dt, g)}
    out = {"grad": torch.randn(m, generator=g, device="cuda", dtype=dt)}
    if case["path"] == "train":
        out["x"] = _values(kind, n, dt, g)
    elif case["accumulate"]:
        out["old"] = torch.randn(n, generator=g, device="cuda", dtype=dt)
    return out


def prepare(case, seed):
    p, dp = _pattern(case)
    v, kind = _payload(case, seed), case["kind"]
    if kind == "batch":
        out = [torch.zeros(q.recvbuf_bytes // BYTES[q.dtype], dtype=TORCH[q.dtype], device="cuda") for q in p]
        ex = [gbx.Exchange(q, x, y, dp=d) for q, x, y, d in zip(p, v["x"], out, dp)]
        return {"batch": [e.request for e in ex], "keep": ex, "out": out}
    if kind == "alltoallv":
        out = torch.zeros(int(p["rb"][-1]) // BYTES[case["dtype"]], dtype=TORCH[case["dtype"]], device="cuda")
        comm = gbx.Comm(case["ranks"], case["ppn"])
        r = gbx.alltoallv_init(comm, v["x"], dp["send_base"], dp["sendcounts"], dp["sdispls"], out, dp["recv_base"],
                               dp["recvcounts"], dp["rdispls"], case["elem"], gbx.DTYPE_CODES[case["dtype"]],
                               info="algorithm=" + case["alg"])
        return {"request": r, "wait": case["wait"], "out": out}
    dt = TORCH[case["dtype"]]
    n, m = p.sendbuf_bytes // BYTES[case["dtype"]], p.recvbuf_bytes // BYTES[case["dtype"]]
    if kind == "alltoallw":
        out = torch.zeros(m, dtype=dt, device="cuda")
        ex = gbx.WExchange(p, v["x"], out, dw=dp)
        return {"request": ex.request, "keep": ex, "wait": "stream", "out": out}
    if case["path"] == "train":
        return {"halo": autograd.DistributedHalo(p, algorithm=case["alg"]), "x": v["x"].requires_grad_(True),
                "grad": v["grad"]}
    if case["path"] == "forward":
        out = torch.zeros(m, dtype=dt, device="cuda")
        ex = gbx.Exchange(p, v["x"], out, algorithm=case["alg"], dp=dp)
        return {"request": ex.request, "keep": ex, "wait": case["wait"], "out": out}
    ex = gbx.Exchange(p, torch.zeros(n, dtype=dt, device="cuda"), torch.zeros(m, dtype=dt, device="cuda"),
                      algorithm=case["alg"], dp=dp)
    out = v["old"] if case["accumulate"] else torch.zeros(n, dtype=dt, device="cuda")
    r = gbx.backward_init(ex.request, v["grad"], out, accumulate=case["accumulate"])
    return {"request": r, "keep": ex, "wait": case["wait"], "out": out}


def run(state):
    if "batch" in state:
        gbx.startall(state["batch"])
        gbx.waitall(state["batch"])
        return state["out"]
    if "halo" in state:
        x = state["x"]
        x.grad = None
        y = state["halo"](x)
        y.backward(state["grad"])
        return {"halo": y.detach(), "grad": x.grad}
    r = state["request"]
    r.start()
    if state["wait"] == "host":
        r.wait()
    else:
        r.wait_stream()
    return state["out"]


# ------------------------------------------------------------------ what a pass needs

def _exchange_work(p, path, accumulate):
    """Each input element read once and each output element written once; one addition for
    every gradient beyond the first that an element receives."""
    esz, s = BYTES[p.dtype], p.elem_size
    seen = np.zeros(int(p.global_sidx.max()) + 1, dtype=bool)
    seen[p.global_sidx] = True
    V, rows = p.volume, int(seen.sum())
    adds = (V - rows) * (s // esz)
    if path == "forward":
        return (rows + V) * s, 0
    if path == "backward":
        return (V + rows * (2 if accumulate else 1)) * s, adds + (rows * (s // esz) if accumulate else 0)
    return (rows + V) * s + V * s + p.sendbuf_bytes, adds


def work(case):
    p, _ = _pattern(case)
    if case["kind"] == "batch":
        return {"bytes": sum(_exchange_work(q, "forward", False)[0] for q in p), "flops": 0}
    if case["kind"] == "alltoallv":
        return {"bytes": 2 * int(p["sb"][-1]), "flops": 0}
    if case["kind"] == "alltoallw":
        return {"bytes": _exchange_work(p.meta["v_pattern"], "forward", False)[0], "flops": 0}
    b, f = _exchange_work(p, case["path"], case["accumulate"])
    return {"bytes": b, "flops": f}


def tolerance(case):
    # values are moved as they are, and sums run in a fixed order: every result is the same bits
    return "exact"


def _exact_v(p, v, path, accumulate):
    c, esz = p.elem_size // BYTES[p.dtype], BYTES[p.dtype]
    src = _source_of_slot(p).cuda()
    out = {}
    if "x" in v:
        out["halo"] = v["x"].double().view(-1, c)[src].view(-1)
    if "grad" in v:
        g = v["old"].double().view(-1, c).clone() if accumulate else \
            torch.zeros(p.sendbuf_bytes // esz // c, c, dtype=torch.float64, device="cuda")
        out["grad"] = g.index_add_(0, src, v["grad"].double().view(-1, c)).view(-1)
    return out if path == "train" else out["halo" if path == "forward" else "grad"]


def exact(case, seed):
    p, _ = _pattern(case)
    v = _payload(case, seed)
    if case["kind"] == "batch":
        return [_exact_v(q, {"x": x}, "forward", False) for q, x in zip(p, v["x"])]
    if case["kind"] == "alltoallw":
        q = p.meta["v_pattern"]
        npts = case["bx"] * case["by"] * case["bz"]
        x = v["x"].view(q.P, case["comps"], npts).transpose(1, 2).reshape(-1) if case["layout"] == "soa" else v["x"]
        return _exact_v(q, {"x": x}, "forward", False)
    if case["kind"] == "alltoallv":
        P, c = case["ranks"], case["elem"] // BYTES[case["dtype"]]
        cnt, e = p["cnt"], case["elem"]
        start = (p["sb"][:-1, None] // e + p["sd"]).T.reshape(-1)           # first element of block (d, r)
        n = cnt.T.reshape(-1)
        first = np.cumsum(n) - n
        idx = np.arange(int(n.sum())) + np.repeat(start - first, n)
        y = v["x"].view(-1, c)[torch.from_numpy(idx).cuda()].view(-1)
        return y if case["dtype"] == "bytes" else y.double()
    return _exact_v(p, v, case["path"], case["accumulate"])
