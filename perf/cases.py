"""Timed cases of the library's public entry points: single solves of every element type, edge-list and
upper-triangular solves, batched solves, the request loop and the min-plus product.

listed() gives the fixed cases, draw(rng) one more of the same ranges; prepare() makes a case's inputs on the GPU
from a seed, run() is one pass, work() its unavoidable bytes and operations, exact() the result in 64 bits.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1902_04446_gb300 as apsp

INF32 = apsp.INF_I32
INF16 = 0x7FFF
DEV = "cuda:0"
TORCH_DT = {"int32": torch.int32, "auto": torch.int32, "u16": torch.int16, "fp32": torch.float32}
ESIZE = {"int32": 4, "auto": 4, "u16": 2, "fp32": 4}
# 64-bit Floyd-Warshall in torch stays below about 20 seconds up to this n
EXACT_MAX_N = 10000


def listed():
    return [
        # a small manifold graph (the 512-point Swiss roll): latency and launches count
        {"name": "solve_i32_roll512", "kind": "solve", "dtype": "int32", "graph": "roll", "n": 512, "ld": 512,
         "scale": 100.0},
        # a typical single request of the serving trace, undirected
        {"name": "solve_i32_er2048", "kind": "solve", "dtype": "int32", "graph": "er", "n": 2048, "ld": 2048,
         "scale": 1.0},
        # a directed graph of odd size in a contiguous matrix (rows not 16-byte aligned)
        {"name": "solve_i32_directed3001", "kind": "solve", "dtype": "int32", "graph": "directed", "n": 3001,
         "ld": 3001, "scale": 1.0},
        # automatic precision on a kNN graph of a Gaussian mixture (manifold learning)
        {"name": "solve_auto_gmm4096", "kind": "solve", "dtype": "auto", "graph": "gmm", "n": 4096, "ld": 4096,
         "scale": 50.0},
        # fp32 geodesic distances, ragged size in padded rows
        {"name": "solve_f32_gmm7900", "kind": "solve", "dtype": "fp32", "graph": "gmm", "n": 7900, "ld": 7904,
         "scale": 1.0},
        # the 16384-point Gaussian mixture in int32
        {"name": "solve_i32_gmm16k", "kind": "solve", "dtype": "int32", "graph": "gmm", "n": 16384, "ld": 16384,
         "scale": 50.0},
        # edge list to packed 16-bit distances, bound check included
        {"name": "edges_u16_roll12000", "kind": "edges", "dtype": "u16", "graph": "roll", "n": 12000, "ld": 12000,
         "scale": 20.0},
        # edge list to upper-triangular storage, solved and read back as the full matrix
        {"name": "tri_i32_roll25000", "kind": "tri", "dtype": "int32", "graph": "roll", "n": 25000, "ld": 25000,
         "scale": 8.0},
        # a large manifold in packed 16-bit, the fastest element type at scale
        {"name": "solve_u16_roll49152", "kind": "solve", "dtype": "u16", "graph": "roll", "n": 49152, "ld": 49152,
         "scale": 4.0},
        # many small graphs of uneven size in one launch
        {"name": "batch_i32_64", "kind": "batch", "dtype": "int32", "graph": "er", "count": 64, "lo": 128, "hi": 1024,
         "mix": 0},
        # a burst of solve requests, sizes as in the serving trace
        {"name": "serve_i32_24", "kind": "serve", "dtype": "int32", "graph": "er", "count": 24, "lo": 128, "hi": 4096,
         "mix": 1},
        # a ragged rectangular min-plus product
        {"name": "minplus_f32_3000", "kind": "minplus", "dtype": "fp32", "m": 3000, "k": 1777, "n": 5000},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "edges", "tri", "batch", "serve", "minplus"])
    if kind == "minplus":
        return {"kind": kind, "dtype": rng.choice(["int32", "u16", "fp32"]), "m": _log_int(rng, 64, 8192),
                "k": _log_int(rng, 64, 8192), "n": _log_int(rng, 64, 8192)}
    if kind in ("batch", "serve"):
        return {"kind": kind, "dtype": "int32", "graph": "er", "count": rng.randint(4, 64 if kind == "batch" else 32),
                "lo": 128, "hi": rng.randint(300, 1500 if kind == "batch" else 4096), "mix": rng.randint(2, 10**6)}
    dtype = rng.choice(["int32", "int32", "fp32", "u16"] if kind != "solve" else ["int32", "int32", "auto", "fp32", "u16"])
    graph = rng.choice(["er", "gmm", "roll"] if kind != "solve" or dtype == "auto" else ["er", "gmm", "roll", "directed"])
    n = _log_int(rng, 200, 20000 if graph == "directed" else 28000)
    # contiguous, padded to 16 bytes, or padded beyond that
    ld = rng.choice([n, n, (n + 7) // 8 * 8, (n + 7) // 8 * 8 + 64])
    scale = 1.0 if graph in ("er", "directed") else rng.choice([4.0, 10.0, 20.0])
    return {"kind": kind, "dtype": dtype, "graph": graph, "n": n, "ld": ld, "scale": scale}


def _sizes(case):
    rng = random.Random(case["mix"])
    return [_log_int(rng, case["lo"], case["hi"]) for _ in range(case["count"])]


def _points(kind, n, rng):
    """n points on a 3-D Swiss roll, or of a 10-D mixture of 8 Gaussians (float64, on the GPU)."""
    if kind == "roll":
        t = rng.uniform(1.5 * math.pi, 4.5 * math.pi, size=n)
        height = rng.uniform(0.0, 21.0, size=n)
        p = np.stack([t * np.cos(t), height, t * np.sin(t)], axis=1)
    else:
        means = rng.uniform(-10.0, 10.0, size=(8, 10))
        p = means[rng.integers(0, 8, size=n)] + rng.normal(0.0, 1.0, size=(n, 10))
    return torch.from_numpy(p).to(DEV)


def _edges(graph, n, scale, dtype, seed):
    """(src, dst, w) on the GPU: int64 vertex ids, float64 weights (whole numbers unless dtype is fp32)."""
    rng = np.random.default_rng([seed, n])
    if graph in ("er", "directed"):
        m = 8 * n
        perm = rng.permutation(n)
        src = np.concatenate([rng.integers(0, n, size=m), perm[:-1]])
        dst = np.concatenate([rng.integers(0, n, size=m), perm[1:]])
        w = rng.integers(1, 1001, size=src.shape[0]).astype(np.float64)
        keep = src != dst
        return tuple(torch.from_numpy(x[keep]).to(DEV) for x in (src, dst, w))
    k = 10 if n > 10 else n - 1
    p = _points(graph, n, rng)
    # neighbours by fp32 distance, their weights in float64
    p32 = p.to(torch.float32)
    idx = []
    for r0 in range(0, n, 4096):
        d = torch.cdist(p32[r0:r0 + 4096], p32, compute_mode="donot_use_mm_for_euclid_dist")
        r = torch.arange(d.shape[0], device=DEV)
        d[r, r + r0] = math.inf
        idx.append(torch.topk(d, k, dim=1, largest=False, sorted=False).indices)
    src = torch.arange(n, device=DEV).repeat_interleave(k)
    dst = torch.cat(idx).reshape(-1)
    w = (p[src] - p[dst]).square_().sum(dim=1).sqrt_()
    if dtype != "fp32":
        w = torch.round(w * scale).clamp_(min=1.0)
    return src, dst, w


def _dense(case, n, ld, seed):
    """The adjacency matrix as a (n, ld) buffer's first n columns: 0 on the diagonal, INF for no edge."""
    dtype = case["dtype"]
    src, dst, w = _edges(case["graph"], n, case.get("scale", 1.0), dtype, seed)
    inf = {"fp32": math.inf, "u16": INF16}.get(dtype, INF32)
    tdt = TORCH_DT[dtype]
    buf = torch.full((n, ld), inf, dtype=tdt, device=DEV)
    flat = buf.view(-1)
    if case["graph"] != "directed":
        src, dst, w = torch.cat([src, dst]), torch.cat([dst, src]), torch.cat([w, w])
    # the smallest weight of every pair
    pos = src * ld + dst
    key, inv = torch.unique(pos, return_inverse=True)
    best = torch.full((key.numel(),), math.inf, dtype=torch.float64, device=DEV)
    best.scatter_reduce_(0, inv, w, reduce="amin")
    flat[key] = best.to(tdt)
    flat[torch.arange(n, device=DEV) * (ld + 1)] = 0
    return buf


def _minplus_inputs(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    m, k, n, dtype = case["m"], case["k"], case["n"], case["dtype"]
    out = []
    for shape in ((m, k), (k, n), (m, n)):
        if dtype == "fp32":
            t = torch.rand(shape, generator=g, device=DEV) * 100.0
            missing = math.inf
        else:
            t = torch.randint(0, 1000, shape, generator=g, device=DEV, dtype=torch.int32)
            missing = INF16 if dtype == "u16" else INF32
        # a tenth of the entries are missing edges
        t[torch.rand(shape, generator=g, device=DEV) < 0.1] = missing
        out.append(t.to(TORCH_DT[dtype]))
    return out


def prepare(case, seed):
    kind, dtype = case["kind"], case["dtype"]
    st = {"case": case, "h": apsp.Handle(device=0)}
    if kind == "solve":
        st["W"] = _dense(case, case["n"], case["ld"], seed)
        st["D"] = torch.empty_like(st["W"])
    elif kind in ("edges", "tri"):
        n = case["n"]
        src, dst, w = _edges(case["graph"], n, case["scale"], dtype, seed)
        st["src"], st["dst"] = src.to(torch.int32), dst.to(torch.int32)
        st["w"] = w.to(TORCH_DT[dtype])
        st["D"] = torch.empty((n, case["ld"]), dtype=TORCH_DT[dtype], device=DEV)
        if kind == "tri":
            st["T"] = apsp.tri_empty(dtype, n, DEV)
    elif kind in ("batch", "serve"):
        st["W"] = [_dense(case, n, n, seed + i) for i, n in enumerate(_sizes(case))]
        st["D"] = [torch.empty_like(W) for W in st["W"]]
    else:
        st["A"], st["B"], st["C"] = _minplus_inputs(case, seed)
    torch.cuda.synchronize()
    return st


def run(st):
    case, h = st["case"], st["h"]
    kind, dtype = case["kind"], case["dtype"]
    if kind == "solve":
        return h.solve_t(dtype, st["W"], st["D"])[:, :case["n"]]
    if kind == "edges":
        return h.solve_edges(dtype, st["src"], st["dst"], st["w"], case["n"], st["D"])[:, :case["n"]]
    if kind == "tri":
        h.tri_from_edges(dtype, st["src"], st["dst"], st["w"], case["n"], st["T"])
        h.solve_tri(dtype, st["T"], case["n"])
        return apsp.tri_to_dense(dtype, st["T"], case["n"], st["D"])[:, :case["n"]]
    if kind == "batch":
        return h.solve_batch(st["W"], st["D"])
    if kind == "serve":
        tickets = [h.submit(W) for W in st["W"]]
        for t, D in zip(tickets, st["D"]):
            if h.wait(t) != 0:
                raise RuntimeError("request failed")
            h.fetch(t, D)
        # a request's matrix may go once its copy out has finished
        torch.cuda.current_stream().synchronize()
        for t in tickets:
            h.release(t)
        return st["D"]
    # C = min(C, A (x) B), in place: a second pass on the same state gives the same C
    return h.minplus(st["A"], st["B"], st["C"])


def work(case):
    """One add and one minimum per relaxation; an undirected graph needs the upper triangle's n^3 / 2 only."""
    kind, es = case["kind"], ESIZE[case["dtype"]]
    if kind == "minplus":
        m, k, n = case["m"], case["k"], case["n"]
        return {"bytes": (m * k + k * n + 2 * m * n) * es, "flops": 2.0 * m * k * n}
    if kind in ("batch", "serve"):
        ns = _sizes(case)
        return {"bytes": sum(2 * es * n * n for n in ns), "flops": float(sum(n**3 for n in ns))}
    n = case["n"]
    if kind in ("edges", "tri"):
        per = 8 if case["graph"] == "er" else 10
        return {"bytes": es * n * n + 12 * per * n, "flops": float(n)**3}
    return {"bytes": 2 * es * n * n, "flops": float(n)**3 * (2.0 if case["graph"] == "directed" else 1.0)}


def _exact_fw(W, dtype):
    """Textbook Floyd-Warshall in float64 / int64; a pair with no path keeps the element type's INF."""
    if dtype == "fp32":
        D = W.to(torch.float64)
    else:
        D = W.to(torch.int64)
    for t in range(D.shape[0]):
        torch.minimum(D, D[:, t:t + 1] + D[t:t + 1, :], out=D)
    return D


def exact(case, seed):
    kind, dtype = case["kind"], case["dtype"]
    if kind == "minplus":
        A, B, C = _minplus_inputs(case, seed)
        if float(case["m"]) * case["n"] * case["k"] > 1e11:
            return None
        wide = torch.float64 if dtype == "fp32" else torch.int64
        A, B, C = A.to(wide), B.to(wide), C.to(wide)
        for t in range(case["k"]):
            torch.minimum(C, A[:, t:t + 1] + B[t:t + 1, :], out=C)
        return C
    if kind in ("batch", "serve"):
        ns = _sizes(case)
        if max(ns) > 2048:
            return None
        return [_exact_fw(_dense(case, n, n, seed + i), dtype) for i, n in enumerate(ns)]
    n = case["n"]
    if n > EXACT_MAX_N:
        return None
    return _exact_fw(_dense(case, n, n, seed), dtype)
