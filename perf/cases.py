"""Timed cases of the 5-vertex census: what a program that uses this library has it do.

Every case is one pass through the public entry points of
``paper_1610_09411_gb300.escape`` on synthetic graphs of the kinds the
benchmark, the autotuner, the run-time model and the tests use: Erdos-Renyi,
Chung-Lu power laws, R-MAT, and batches of half G(n, p), half preferential
attachment.  Graphs are made on the GPU from the seed alone.

Counts come back as 64-bit words (low, high) of the 128-bit integers.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1610_09411_gb300 import escape as esc

PARTS = ("c3", "c4", "c5", "n3", "n4", "n5")


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # The smallest call: a host CSR of the ER(500, 0.012) workload, loaded,
        # counted and freed in one call.  Launches and host steps only.
        {"name": "er500_host", "kind": "count", "graph": "er", "n": 500, "p": 0.012},
        # A small dense graph held on the device (the autotuner's "small"
        # representative): cliques and common neighbours, no skew.
        {"name": "er800_dense", "kind": "census", "graph": "er", "n": 800, "p": 0.15},
        # The power-law workload (exponent 2.1, mean degree 16, ~2M edges).
        {"name": "cl21_262k", "kind": "census", "graph": "cl", "n": 262144, "gamma": 2.1, "mean": 16.0, "clip": 8192},
        # The largest serving request: Chung-Lu, exponent 2.3, ~5M edges.
        {"name": "cl23_5m", "kind": "census", "graph": "cl", "n": 625000, "gamma": 2.3, "mean": 16.0, "clip": 8192},
        # R-MAT of the run-time model's middle scale.
        {"name": "rmat16", "kind": "census", "graph": "rmat", "scale": 16, "ef": 16},
        # The headline generator at the largest scale whose census stays under two seconds.
        {"name": "rmat19", "kind": "census", "graph": "rmat", "scale": 19, "ef": 16},
        # A raw directed edge list on the device (duplicates, loops, one
        # direction) normalised, then its 3- and 4-vertex counts alone.
        {"name": "rmat18_raw4", "kind": "raw4", "graph": "rmat", "scale": 18, "ef": 16},
        # Per-vertex and per-edge counts beside the census, of an odd-sized power
        # law with a given number of edges.
        {"name": "cl21_elements", "kind": "elements", "graph": "cl", "n": 50021, "gamma": 2.1, "mean": 12.0,
         "clip": 4096, "m": 290017},
        # A batch of many small graphs (motif counts of a collection).
        {"name": "batch_small", "kind": "batch", "count": 256, "n_lo": 20, "n_hi": 200},
        # The batch workload's own size range.
        {"name": "batch_mixed", "kind": "batch", "count": 96, "n_lo": 20, "n_hi": 2000},
        # One step of the serving loop: resident requests of uneven size in one fused call.
        {"name": "serve_mix", "kind": "serve", "count": 8, "m_lo": 1000, "m_hi": 200000},
        # 4-cycles per vertex with no allocation, near that entry point's size limit.
        {"name": "noalloc_30k", "kind": "noalloc", "graph": "cl", "n": 30011, "gamma": 2.1, "mean": 16.0, "clip": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["count", "census", "census", "census", "raw4", "elements", "batch", "serve", "noalloc"])
    if kind == "batch":
        hi = _log_int(rng, 60, 2000)
        return {"kind": kind, "count": _log_int(rng, 3, 300 if hi < 400 else 90), "n_lo": 20, "n_hi": hi}
    if kind == "serve":
        return {"kind": kind, "count": rng.randint(2, 12), "m_lo": 1000, "m_hi": _log_int(rng, 4000, 300000)}
    if kind == "noalloc":
        n = _log_int(rng, 200, 32768)
        return {"kind": kind, "graph": "cl", "n": n, "gamma": rng.choice([2.1, 2.3, 2.5]),
                "mean": round(rng.uniform(4, 16), 2), "clip": max(16, n // rng.choice([4, 8, 16]))}
    if kind == "count":
        n = _log_int(rng, 30, 3000)
        return {"kind": kind, "graph": "er", "n": n, "p": round(min(0.3, rng.uniform(4, 30) / n), 5)}
    what = rng.choice(["er", "cl", "cl", "rmat"])
    if kind == "raw4":
        return {"kind": kind, "graph": "rmat", "scale": rng.randint(10, 18), "ef": rng.randint(4, 17)}
    if kind == "elements":
        n, mean = _log_int(rng, 500, 60000), round(rng.uniform(6, 16), 2)
        return {"kind": kind, "graph": "cl", "n": n, "gamma": rng.choice([2.1, 2.3, 2.6]), "mean": mean,
                "clip": max(16, min(4096, n // 8)), "m": int(n * mean * rng.uniform(0.35, 0.45))}
    if what == "er":
        n = _log_int(rng, 40, 20000)
        return {"kind": kind, "graph": "er", "n": n, "p": round(min(0.3, rng.uniform(2, 160) / n), 6)}
    if what == "cl":
        gamma = rng.choice([2.1, 2.2, 2.3, 2.6])
        n = _log_int(rng, 500, 270000 if gamma < 2.3 else 600000)
        return {"kind": kind, "graph": "cl", "n": n, "gamma": gamma, "mean": round(rng.uniform(6, 16), 2),
                "clip": max(16, min(8192, n // 4))}
    return {"kind": kind, "graph": "rmat", "scale": rng.randint(9, 18), "ef": rng.randint(6, 17)}


# ------------------------------------------------------------------ graphs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _csr(n, u, v, m=None, gen=None):
    """Simple symmetric CSR of the pairs (u, v); with m, of m of their distinct pairs."""
    keep = u != v
    u, v = u[keep], v[keep]
    if m is not None:
        one = torch.unique(torch.minimum(u, v) * n + torch.maximum(u, v))
        if one.numel() < m:
            raise ValueError("too few distinct pairs")
        one = one[torch.randperm(one.numel(), device="cuda", generator=gen)[:m]]
        u = torch.div(one, n, rounding_mode="floor")
        v = one - u * n
    keys = torch.unique(torch.cat([u * n + v, v * n + u]))
    rows = torch.div(keys, n, rounding_mode="floor")
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return row_ptr, (keys - rows * n).to(torch.int32)


def _er_edges(n, p, gen):
    """G(n, p) as vertex pairs: one draw per pair, in blocks of rows."""
    us, vs = [], []
    step = max(1, (1 << 24) // max(n, 1))
    for r0 in range(0, n, step):
        r = torch.arange(r0, min(n, r0 + step), device="cuda").unsqueeze(1)
        hit = torch.rand((r.shape[0], n), device="cuda", generator=gen) < p
        hit &= torch.arange(n, device="cuda").unsqueeze(0) > r
        i, j = hit.nonzero(as_tuple=True)
        us.append(i + r0)
        vs.append(j)
    return torch.cat(us), torch.cat(vs)


def _cl_edges(n, gamma, mean, clip, gen, more=1.0):
    """Edge-sampling Chung-Lu: both endpoints drawn by the clipped power-law
    weights, vertices permuted."""
    w = torch.arange(1, n + 1, dtype=torch.float64, device="cuda") ** (-1.0 / (gamma - 1.0))
    for _ in range(20):
        w = torch.clamp(w * (mean * n / w.sum()), max=float(clip))
    cum = torch.cumsum(w, 0)
    cnt = int(round(more * mean * n / 2.0))
    x = torch.rand(2 * cnt, dtype=torch.float64, device="cuda", generator=gen) * cum[-1]
    ids = torch.searchsorted(cum, x, right=True).clamp_(max=n - 1)
    ids = torch.randperm(n, device="cuda", generator=gen)[ids]
    return ids[:cnt], ids[cnt:]


def _rmat_edges(scale, ef, gen):
    """R-MAT (0.57, 0.19, 0.19, 0.05), vertices permuted."""
    cnt = int(ef) << scale
    u = torch.zeros(cnt, dtype=torch.int64, device="cuda")
    v = torch.zeros(cnt, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        x = torch.rand(cnt, device="cuda", generator=gen)
        u = u * 2 + (x >= 0.76)
        v = v * 2 + (((x >= 0.57) & (x < 0.76)) | (x >= 0.95))
    perm = torch.randperm(1 << scale, device="cuda", generator=gen)
    return perm[u], perm[v]


def _graph(case, seed):
    gen = _gen(seed)
    if case["graph"] == "er":
        n = case["n"]
        return (n,) + _csr(n, *_er_edges(n, case["p"], gen))
    if case["graph"] == "cl":
        n, m = case["n"], case.get("m")
        # with a given number of edges, twice the samples, so that enough are distinct
        u, v = _cl_edges(n, case["gamma"], case["mean"], case["clip"], gen, 1.0 if m is None else 2.0)
        return (n,) + _csr(n, u, v, m, gen)
    n = 1 << case["scale"]
    return (n,) + _csr(n, *_rmat_edges(case["scale"], case["ef"], gen))


def _ba_edges(sizes, attach, rng):
    """Preferential attachment, all graphs of the batch grown together: a seed
    clique of m + 1 vertices, then every vertex joins m earlier ones, each an
    endpoint of a uniformly drawn earlier edge (repeats dropped later)."""
    count, top = len(sizes), int(max(sizes))
    mmax = int(max(attach))
    cap = mmax * (mmax + 1) + 2 * mmax * top
    ends = np.zeros((count, cap), dtype=np.int64)
    used = np.zeros(count, dtype=np.int64)
    for k in range(count):
        i, j = np.triu_indices(min(int(attach[k]) + 1, int(sizes[k])), 1)
        ends[k, 0:2 * len(i):2], ends[k, 1:2 * len(i):2] = i, j
        used[k] = 2 * len(i)
    for t in range(2, top):
        live = np.nonzero((t > attach) & (t < sizes))[0]
        if len(live) == 0:
            continue
        base = used[live]
        pick = (rng.random((len(live), mmax)) * base[:, None]).astype(np.int64)
        to = ends[live[:, None], pick]
        for j in range(mmax):
            on = attach[live] > j
            at = live[on]
            ends[at, used[at]] = t
            ends[at, used[at] + 1] = to[on, j]
            used[at] += 2
    return [(ends[k, 0:used[k]:2], ends[k, 1:used[k]:2]) for k in range(count)]


def _union(parts):
    """Block-diagonal CSR with local ids from (n, row_ptr, col) of every member."""
    voff = np.zeros(len(parts) + 1, dtype=np.int64)
    voff[1:] = np.cumsum([p[0] for p in parts])
    base, rps = 0, []
    for _, rp, col in parts:
        rps.append(rp[:-1] + base)
        base += int(col.numel())
    rps.append(torch.tensor([base], dtype=torch.int64, device="cuda"))
    return torch.from_numpy(voff).cuda(), torch.cat(rps), torch.cat([p[2] for p in parts]).contiguous()


def _batch_sizes(case, rng):
    return np.array([rng.integers(case["n_lo"], case["n_hi"] + 1) for _ in range(case["count"])], dtype=np.int64)


def _batch(case, seed):
    """Half G(n, p) with p uniform in 0.01 .. 0.3, half preferential attachment with m of 2 .. 6."""
    rng = np.random.default_rng(seed)
    gen = _gen(seed)
    sizes = _batch_sizes(case, rng)
    odd = sizes[1::2]
    ba = _ba_edges(odd, rng.integers(2, 7, len(odd)), rng) if len(odd) else []
    parts = []
    for k, n in enumerate(int(x) for x in sizes):
        if k % 2 == 0:
            u, v = _er_edges(n, float(rng.uniform(0.01, 0.3)), gen)
        else:
            u, v = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in ba[k // 2])
        parts.append((n,) + _csr(n, u, v))
    return parts


def _serve_sizes(case):
    lo, hi, cnt = math.log(case["m_lo"]), math.log(case["m_hi"]), case["count"]
    return [math.exp(lo + (hi - lo) * (k + 0.5) / cnt) for k in range(cnt)]


def _serve(case, seed):
    """Requests of exponent 2.3 and mean degree 16, edge counts spread over the logarithm of the range."""
    gen = _gen(seed)
    rng = np.random.default_rng(seed)
    parts = []
    for m in _serve_sizes(case):
        n = max(8, int(m * float(rng.uniform(0.9, 1.1)) / 8))
        parts.append((n,) + _csr(n, *_cl_edges(n, 2.3, 16.0, max(16.0, min(8192.0, n / 4)), gen)))
    return parts


# ------------------------------------------------------------------ passes

class Handle:
    """A loaded graph that is freed with its owner."""

    def __init__(self, h):
        self.h = h

    def __del__(self):
        try:
            esc.escape_free(self.h)
        except Exception:
            pass


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind}
    if kind in ("batch", "serve"):
        st["voff"], st["rp"], st["col"] = _union(_batch(case, seed) if kind == "batch" else _serve(case, seed))
    elif kind == "raw4":
        # directed entries grouped by source, as an edge list file gives them
        u, v = _rmat_edges(case["scale"], case["ef"], _gen(seed))
        n = 1 << case["scale"]
        order = torch.sort(u, stable=True).indices
        st["n"] = n
        st["rp"] = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        st["rp"][1:] = torch.cumsum(torch.bincount(u, minlength=n), 0)
        st["col"] = v[order].to(torch.int32)
    else:
        n, rp, col = _graph(case, seed)
        st["n"] = n
        if kind == "count":
            st["rp"], st["col"] = rp.cpu().numpy(), col.cpu().numpy()
        elif kind == "noalloc":
            st["rp"], st["col"] = rp, col
            st["c4_v"] = torch.zeros(n, dtype=torch.int64, device="cuda")
            st["total"] = torch.zeros(1, dtype=torch.int64, device="cuda")
        else:
            torch.cuda.synchronize()
            st["graph"] = Handle(esc.escape_load_csr(n, rp, col))
            if kind == "elements":
                esc.escape_set_options(st["graph"].h, keep_per_element=True)
    torch.cuda.synchronize()
    return st


def _words(counts):
    """Python integers as an array of (low, high) 64-bit words."""
    return np.frombuffer(b"".join([c.to_bytes(16, "little") for c in counts]), dtype=np.int64).reshape(-1, 2)


def _result(r):
    return {k: _words(r[k]) for k in PARTS if k in r}


def run(st):
    kind = st["kind"]
    if kind == "census":
        return _result(esc.escape_census5(st["graph"].h))
    if kind == "count":
        return _result(esc.census(st["rp"], st["col"], n=st["n"]))
    if kind == "raw4":
        return _result(esc.census(st["rp"], st["col"], n=st["n"], flags=esc.ESCAPE_NORMALIZE, four_only=True))
    if kind == "elements":
        out = _result(esc.escape_census5(st["graph"].h))
        out.update({k: v.view(np.int64) for k, v in esc.escape_per_element(st["graph"].h).items()})
        return out
    if kind == "noalloc":
        esc.escape_cycles4_noalloc(st["n"], st["rp"], st["col"], st["c4_v"], st["total"])
        return {"c4_v": st["c4_v"], "total": st["total"]}
    res = esc.escape_census5_batch(st["voff"], st["rp"], st["col"])
    return {k: _words([c for r in res for c in r[k]]) for k in PARTS}


# ------------------------------------------------------------------ what a pass cannot do without

def _expected(case):
    """(graphs, vertices, adjacency entries) of a case, expected."""
    kind = case["kind"]
    if kind == "batch":
        n = (case["n_lo"] + case["n_hi"]) / 2.0
        n2 = (case["n_lo"] ** 2 + case["n_lo"] * case["n_hi"] + case["n_hi"] ** 2) / 3.0
        return case["count"], case["count"] * n, case["count"] * (0.5 * 0.155 * n2 + 0.5 * 8.0 * n)
    if kind == "serve":
        m = sum(_serve_sizes(case))
        return case["count"], m / 8.0, 2.0 * m
    if case["graph"] == "er":
        return 1, case["n"], case["p"] * case["n"] * (case["n"] - 1.0)
    if case["graph"] == "cl":
        return 1, case["n"], 2.0 * case["m"] if "m" in case else case["mean"] * case["n"]
    n = 1 << case["scale"]
    return 1, n, n * case["ef"] * (1.0 if kind == "raw4" else 2.0)


def work(case):
    """The CSR read once, the results written once.  The counting itself is
    integer work on the wedges and diamonds of the graph, which no formula in
    the sizes gives; one integer step for every adjacency entry stands in."""
    graphs, n, nnz = _expected(case)
    kind = case["kind"]
    out = graphs * 98 * 16.0
    if kind == "raw4":
        out = 30 * 16.0
    elif kind == "elements":
        out += 24.0 * (nnz + n)
    elif kind == "noalloc":
        out = 8.0 * (n + 1)
    return {"bytes": 8.0 * (n + graphs) + 4.0 * nnz + out, "flops": float(nnz)}


# ------------------------------------------------------------------ values from plain torch

def _dense(n, rp, col):
    a = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), rp[1:] - rp[:-1])
    a[rows, col.long()] = 1.0
    return a


def _four(a):
    """n3, c3, n4, c4 of a dense adjacency matrix, in Python integers."""
    n = a.shape[0]
    d = a.sum(1)
    i = lambda x: int(round(float(x)))  # noqa: E731  (every value here is far below 2^53)
    m = i(d.sum()) // 2
    w2 = a @ a
    t_e = w2 * a
    t_v = t_e.sum(1) / 2
    off = w2 - torch.diag(torch.diagonal(w2))
    W, S3 = i((d * (d - 1) / 2).sum()), i((d * (d - 1) * (d - 2) / 6).sum())
    T = i(t_e.sum()) // 6
    P4 = i((a * torch.outer(d - 1, d - 1)).sum()) // 2 - 3 * T
    TT = i((t_v * (d - 2)).sum())
    C4 = i((off * (off - 1) / 2).sum()) // 4
    D = i((t_e * (t_e - 1) / 2).sum()) // 2
    K4 = 0
    for v in range(n):
        nb = a[v].nonzero().squeeze(1)
        s = a[nb][:, nb]
        K4 += i(((s @ s) * s).sum()) // 6
    K4 //= 4
    c = math.comb
    n3 = [c(n, 3), m * (n - 2), W, T]
    i3 = [0, n3[1] - 2 * W + 3 * T, W - 3 * T, T]
    i3[0] = c(n, 3) - sum(i3)
    n4 = [S3, P4, TT, C4, D, K4, c(n, 4), m * c(n - 2, 2), c(m, 2) - W, W * (n - 3), T * (n - 3)]
    dia, tail = D - 6 * K4, TT - 4 * D + 12 * K4
    con = [S3 - TT + 2 * D - 4 * K4, P4 - 2 * TT - 4 * C4 + 6 * D - 12 * K4, tail, C4 - D + 3 * K4, dia, K4]
    two = n4[8] - con[1] - con[2] - 2 * con[3] - 2 * con[4] - 3 * con[5]
    tri = n4[10] - con[2] - 2 * con[4] - 4 * con[5]
    wed = n4[9] - 3 * con[0] - 2 * con[1] - 5 * con[2] - 4 * con[3] - 8 * con[4] - 12 * con[5] - 3 * tri
    one = (n4[7] - 3 * con[0] - 3 * con[1] - 4 * con[2] - 4 * con[3] - 5 * con[4] - 6 * con[5] - 2 * two - 2 * wed
           - 3 * tri)
    c4 = con + [0, one, two, wed, tri]
    c4[6] = c(n, 4) - sum(c4)
    return {"c3": _words(i3), "c4": _words(c4), "n3": _words(n3), "n4": _words(n4)}


def exact(case, seed):
    """The 3- and 4-vertex counts of small graphs and the 4-cycles per vertex,
    from dense matrices; the 5-vertex counts have no plain form."""
    kind = case["kind"]
    if kind in ("count", "census") and case.get("n", 1 << 30) <= 1500:
        out = _four(_dense(*_graph(case, seed)))
        return {k: out.get(k) for k in PARTS}
    if kind == "noalloc":
        n, rp, col = _graph(case, seed)
        a = torch.zeros((n, n), dtype=torch.float32, device="cuda")
        rows = torch.repeat_interleave(torch.arange(n, device="cuda"), rp[1:] - rp[:-1])
        a[rows, col.long()] = 1.0
        c4 = torch.zeros(n, dtype=torch.int64, device="cuda")
        for r0 in range(0, n, 4096):
            w = (a[r0:r0 + 4096] @ a).to(torch.int64)      # exact: entries are whole and below 2^24
            k = torch.arange(w.shape[0], device="cuda")
            w[k, k + r0] = 0
            c4[r0:r0 + 4096] = (w * (w - 1) // 2).sum(1)
        return {"c4_v": c4, "total": (c4.sum() // 4).reshape(1)}
    return None
