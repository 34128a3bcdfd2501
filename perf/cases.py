"""The workloads this library is measured on, each through its public entry points.

A case is a dict of plain values.  `listed` names the standing ones, `draw` gives others of the same
ranges, `prepare` makes what a program holds before the call, `run` is one pass, `work` what a pass
cannot do without, `exact` the same result in 64 bits.

Kinds of case:
  solve   one matrix on the device, in place (apsp_fw); the input is copied in first, as a program
          that keeps its graph does
  paths   the same with the stage record that paths are read from (apsp_fw_paths)
  host    one matrix in pinned host memory (apsp_fw_host)
  batch   many small graphs in one call (apsp_fw_batched)
  serve   requests of mixed sizes through a server (submit all, wait for all)
"""
import math
import random

import torch

from paper_1001_4108_gb300 import binding

INF_I32 = 1 << 29
INF_I16 = 16383
TORCH = {"f32": torch.float32, "i32": torch.int32, "i16": torch.int16}
SIZE = {"f32": 4, "i32": 4, "i16": 2}
# Largest n that plain 64-bit torch solves in a few seconds.
EXACT_MAX_N = 8192


def listed():
    return [
        # a small graph on its own: launches and latency are all there is
        {"name": "f32-100", "kind": "solve", "dtype": "f32", "n": 100, "ld": 100, "graph": "dense"},
        # the plain configuration: sparse directed graph, integer weights
        {"name": "i32-1024", "kind": "solve", "dtype": "i32", "n": 1024, "ld": 1024, "graph": "sparse30"},
        # a contiguous matrix of odd n: ragged tiles, rows that are not 16-byte aligned
        {"name": "f32-2047-odd", "kind": "solve", "dtype": "f32", "n": 2047, "ld": 2047, "graph": "dense"},
        # hop-like weights in the packed 16-bit form
        {"name": "i16-2048", "kind": "solve", "dtype": "i16", "n": 2048, "ld": 2048, "graph": "sparse10"},
        # middle sizes: complete fp32 graph, and integers with negative edges and a ragged last block
        {"name": "f32-4096", "kind": "solve", "dtype": "f32", "n": 4096, "ld": 4096, "graph": "dense"},
        {"name": "i32-6000", "kind": "solve", "dtype": "i32", "n": 6000, "ld": 6000, "graph": "negative"},
        # the headline size, and the largest 16-bit size its weight bound allows
        {"name": "f32-16384", "kind": "solve", "dtype": "f32", "n": 16384, "ld": 16384, "graph": "dense"},
        {"name": "i16-16000", "kind": "solve", "dtype": "i16", "n": 16000, "ld": 16000, "graph": "sparse10"},
        # thousands of small graphs, n uniform in 16..512, in one call
        {"name": "batch-i32-4096", "kind": "batch", "dtype": "i32", "count": 4096, "nmin": 16, "nmax": 512, "mix": 5},
        # distances with the record for path reconstruction, edges of both signs
        {"name": "paths-f32-2048", "kind": "paths", "dtype": "f32", "n": 2048, "ld": 2048, "graph": "negative"},
        # a program whose matrix lives in host memory
        {"name": "host-f32-4096", "kind": "host", "dtype": "f32", "n": 4096, "ld": 4096, "graph": "dense"},
        # a burst of requests, half int32 and half fp32, n log-uniform
        {"name": "serve-48", "kind": "serve", "count": 48, "nmin": 32, "nmax": 2048, "mix": 11},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 6 + ["paths", "host", "batch", "serve"])
    if kind == "batch":
        nmax = _log_uniform(rng, 48, 512)
        return {"kind": "batch", "dtype": rng.choice(["i32", "f32"]), "count": _log_uniform(rng, 16, 4096),
                "nmin": 16, "nmax": nmax, "mix": rng.randrange(1 << 20)}
    if kind == "serve":
        return {"kind": "serve", "count": rng.randrange(8, 57), "nmin": 32, "nmax": _log_uniform(rng, 256, 3000),
                "mix": rng.randrange(1 << 20)}
    if kind == "solve":
        dtype = rng.choice(["f32", "f32", "i32", "i32", "i16"])
        n = _log_uniform(rng, 40, 9000)
    else:
        dtype = rng.choice(["f32", "i32"])
        n = _log_uniform(rng, 200, 5000)
    # contiguous rows, rows padded to 16 bytes, or a block of a wider matrix
    q = 16 // SIZE[dtype]
    ld = rng.choice([n, -(-n // q) * q, -(-n // q) * q, n + 37])
    graph = "sparse10" if dtype == "i16" else rng.choice(["dense", "negative"] if dtype == "f32" else
                                                         ["sparse30", "sparse10", "negative"])
    return {"kind": kind, "dtype": dtype, "n": n, "ld": ld, "graph": graph}


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed & 0x7FFFFFFF)


def _weights(dtype, n, graph, g):
    """An n x n weight matrix on the GPU: 0 on the diagonal, the dtype's infinity where no edge is."""
    dev = "cuda"
    if dtype == "f32":
        if graph == "dense":  # complete, weights in (0, 1], each the nearest fp32 of a real number
            w = (1.0 - torch.rand((n, n), generator=g, device=dev, dtype=torch.float64)).to(torch.float32)
        else:  # complete, w + p_u - p_v in multiples of 2^-23: exact, both signs, no negative cycle
            w = torch.randint(1, (1 << 23) + 1, (n, n), generator=g, device=dev, dtype=torch.int32)
            p = torch.randint(0, (1 << 22) + 1, (n,), generator=g, device=dev, dtype=torch.int32)
            w = (w + p[:, None] - p[None, :]).to(torch.float32) * 2.0 ** -23
        w.fill_diagonal_(0)
        return w
    inf = INF_I16 if dtype == "i16" else INF_I32
    prob, hi = {"sparse30": (0.3, 1000), "sparse10": (0.1, 7), "negative": (0.2, 950)}[graph]
    if dtype == "i16":
        hi = max(1, min(hi, 16382 // max(1, n - 1)))
    w = torch.randint(0 if graph == "negative" else 1, hi + 1, (n, n), generator=g, device=dev, dtype=torch.int32)
    if graph == "negative":
        p = torch.randint(0, 51, (n,), generator=g, device=dev, dtype=torch.int32)
        w += p[:, None] - p[None, :]
    w.masked_fill_(torch.rand((n, n), generator=g, device=dev) >= prob, inf)
    w.fill_diagonal_(0)
    return w.to(TORCH[dtype])


def _block(case):
    """An uninitialised n x n device matrix with the case's leading dimension."""
    n, ld = case["n"], case["ld"]
    return torch.empty((n, ld), dtype=TORCH[case["dtype"]], device="cuda")[:, :n]


def _batch_shapes(case):
    """(n, leading dimension, offset) of each graph, and the buffer's elements: one device buffer, rows of
    16 bytes."""
    r = random.Random(case["mix"])
    out, at = [], 0
    for _ in range(case["count"]):
        n = r.randint(case["nmin"], case["nmax"])
        ld = -(-n // 4) * 4
        out.append((n, ld, at))
        at += n * ld
    return out, at


def _batch_weights(case, seed):
    """The whole batch in one buffer: each graph sparse (p = 0.2), weights of both signs, no negative cycle."""
    shapes, total = _batch_shapes(case)
    g = _gen(seed)
    dev = "cuda"
    ns = torch.tensor([s[0] for s in shapes], device=dev)
    lds = torch.tensor([s[1] for s in shapes], device=dev)
    at = torch.tensor([s[2] for s in shapes], device=dev)
    integer = case["dtype"] == "i32"
    w = torch.randint(0, 951, (total,), generator=g, device=dev, dtype=torch.int32)
    absent = torch.rand((total,), generator=g, device=dev) >= 0.2
    p = torch.randint(0, 51, (len(shapes), case["nmax"] + 4), generator=g, device=dev, dtype=torch.int32)
    step = max(1, len(shapes) // 16)
    for a in range(0, len(shapes), step):  # a slice of the batch at a time: the index vectors are 64-bit
        b = min(len(shapes), a + step)
        lo, hi = shapes[a][2], (shapes[b][2] if b < len(shapes) else total)
        graph = torch.repeat_interleave(torch.arange(a, b, device=dev), ns[a:b] * lds[a:b])
        e = torch.arange(lo, hi, device=dev) - at[graph]
        u = e // lds[graph]
        v = e - u * lds[graph]
        w[lo:hi] += p[graph, u] - p[graph, v]
        w[lo:hi].masked_fill_(u == v, 0)
        absent[lo:hi] &= u != v
    if integer:
        return w.masked_fill_(absent, INF_I32)
    return w.to(torch.float32).mul_(1.0 / 1024).masked_fill_(absent, math.inf)


def _views(case, buf):
    return [buf[at:at + n * ld].view(n, ld)[:, :n] for n, ld, at in _batch_shapes(case)[0]]


def _requests(case):
    r = random.Random(case["mix"])
    return [(_log_uniform(r, case["nmin"], case["nmax"]), "i32" if k % 2 == 0 else "f32")
            for k in range(case["count"])]


def _request_weights(case, seed):
    g = _gen(seed)
    return [_weights(dt, n, "sparse30" if dt == "i32" else "dense", g) for n, dt in _requests(case)]


class _Serving:
    """A server for the life of a state."""

    def __init__(self):
        self.server = binding.Server(max_inflight=64, hbm_budget_bytes=8 << 30, streams=4, max_n=4096)

    def __del__(self):
        self.server.close()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        w = _batch_weights(case, seed)
        d = torch.empty_like(w)
        return {"kind": kind, "w": w, "d": d, "mats": _views(case, d), "ns": [s[0] for s in _batch_shapes(case)[0]]}
    if kind == "serve":
        return {"kind": kind, "reqs": [w.cpu().numpy() for w in _request_weights(case, seed)], "serving": _Serving()}
    w = _weights(case["dtype"], case["n"], case["graph"], _gen(seed))
    if kind == "host":
        n, ld = case["n"], case["ld"]
        h = torch.empty((n, ld), dtype=TORCH[case["dtype"]], pin_memory=True)[:, :n]
        return {"kind": kind, "w": w, "h": h}
    d = _block(case)
    d.copy_(w)
    state = {"kind": kind, "w": w, "d": d}
    if kind == "paths":
        state["via"] = torch.empty((case["n"], case["n"]), dtype=torch.int16, device="cuda")
    return state


def run(state):
    kind = state["kind"]
    if kind == "solve":
        state["d"].copy_(state["w"])
        return binding.apsp_fw(state["d"])
    if kind == "paths":
        state["d"].copy_(state["w"])
        return list(binding.apsp_fw_paths(state["d"], state["via"]))
    if kind == "host":
        state["h"].copy_(state["w"], non_blocking=True)  # the program's producer fills the host matrix
        return binding.apsp_fw_host(state["h"])
    if kind == "batch":
        state["d"].copy_(state["w"])
        binding.apsp_fw_batched(state["mats"], ns=state["ns"])
        return state["d"]
    server = state["serving"].server
    tickets = [server.submit(w) for w in state["reqs"]]
    return [server.wait(t) for t in tickets]


def work(case):
    """Each matrix read once and written once (the stage record written once); an addition and a minimum
    per relaxation."""
    if case["kind"] == "batch":
        ns = [s[0] for s in _batch_shapes(case)[0]]
        return {"bytes": sum(8 * n * n for n in ns), "flops": sum(2 * n ** 3 for n in ns)}
    if case["kind"] == "serve":
        ns = [n for n, _ in _requests(case)]
        return {"bytes": sum(8 * n * n for n in ns), "flops": sum(2 * n ** 3 for n in ns)}
    n = case["n"]
    via = 2 * n * n if case["kind"] == "paths" else 0
    return {"bytes": 2 * SIZE[case["dtype"]] * n * n + via, "flops": 2 * n ** 3}


def _solve64(w):
    """Shortest distances in 64 bits: one rank-1 min-plus update per vertex.  w: (..., n, n)."""
    d = w.to(torch.float64)
    if w.dtype != torch.float32:
        d[w == (INF_I16 if w.dtype == torch.int16 else INF_I32)] = math.inf
    t = torch.empty_like(d)
    for k in range(d.shape[-1]):
        torch.add(d[..., :, k:k + 1], d[..., k:k + 1, :], out=t)
        torch.minimum(d, t, out=d)
    return d


def _like(d, dtype):
    if dtype == torch.float32:
        return d
    return torch.where(torch.isinf(d), torch.full_like(d, INF_I16 if dtype == torch.int16 else INF_I32), d).to(dtype)


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return [_like(_solve64(w), w.dtype).cpu() for w in _request_weights(case, seed)]
    if kind == "batch":
        w = _batch_weights(case, seed)
        out = w.to(torch.float64) if w.dtype == torch.float32 else w.clone()
        views, results = _views(case, w), _views(case, out)
        order = sorted(range(len(views)), key=lambda i: views[i].shape[0])
        inf = math.inf if w.dtype == torch.float32 else INF_I32
        for a in range(0, len(order), 256):  # graphs of about one size together, padded with lone vertices
            part = order[a:a + 256]
            m = views[part[-1]].shape[0]
            pad = torch.full((len(part), m, m), inf, dtype=w.dtype, device=w.device)
            for k, i in enumerate(part):
                n = views[i].shape[0]
                pad[k, :n, :n] = views[i]
            d = _like(_solve64(pad), w.dtype)
            for k, i in enumerate(part):
                n = views[i].shape[0]
                results[i].copy_(d[k, :n, :n])
        return out
    if case["n"] > EXACT_MAX_N:
        return [None, None] if kind == "paths" else None
    w = _weights(case["dtype"], case["n"], case["graph"], _gen(seed))
    d = _like(_solve64(w), w.dtype)
    if kind == "paths":
        return [d, None]
    return d.cpu() if kind == "host" else d
