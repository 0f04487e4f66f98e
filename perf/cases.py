"""What this library is timed on: its entry points as an analysis of single cells calls them, from
the smallest dataset to a million cells.

The inputs stand in for PCA embeddings (cells x principal components): Gaussian mixtures with
cluster means N(0, 4 I) and noise N(0, 1/t) on component t, cells in random order, as in
`paper_2603_02402_gb300.synth`, drawn on the GPU with torch.  Graph inputs of the analysis steps
(connectivities, UMAP, Leiden) come from kNN lists inside blocks of cells, taken by brute force in
torch, with the ids of the cells shuffled.
"""
import math

import numpy as np
import torch

from paper_2603_02402_gb300 import rsc

K_CROSS = 3
UMAP_A, UMAP_B = 0.583, 1.334   # the curve of spread 1, min_dist 0.5 (scanpy's defaults)
EXACT_ROWS = 130_000        # brute force in 64 bits up to this many rows
EXACT_GRAPH_ROWS = 12_000   # beyond, a tie in the last bits may change a list and with it the CSR's layout


def listed():
    return [
        # a 2,700-cell dataset through the default options: launches and latency
        {"name": "graph_fp32_2700", "kind": "graph", "n": 2_700, "d": 50, "k": 15, "metric": "euclidean",
         "precision": "fp32", "comps": 9},
        # the plain exact graph of a 10,000-cell experiment (20 cell types)
        {"name": "graph_fp32_10k", "kind": "graph", "n": 10_000, "d": 50, "k": 15, "metric": "euclidean",
         "precision": "fp32", "comps": 20},
        # neighbours of an atlas-sized dataset with the default precision
        {"name": "knn_fp32_100k", "kind": "knn", "n": 100_003, "d": 50, "k": 15, "metric": "euclidean",
         "precision": "fp32", "comps": 60},
        # an ordinary experiment with the fast precision
        {"name": "graph_bf16_68k", "kind": "graph", "n": 68_579, "d": 50, "k": 15, "metric": "euclidean",
         "precision": "bf16", "comps": 40},
        # the headline graph: a million cells
        {"name": "graph_bf16_1m", "kind": "graph", "n": 1_000_000, "d": 50, "k": 15, "metric": "euclidean",
         "precision": "bf16", "comps": 100},
        # cosine neighbours with long lists
        {"name": "knn_cosine_k30", "kind": "knn", "n": 400_009, "d": 50, "k": 30, "metric": "cosine",
         "precision": "bf16", "comps": 100},
        # the fuzzy graph of lists that another search produced
        {"name": "connectivities_k30", "kind": "connectivities", "n": 300_007, "k": 30},
        # batch-balanced neighbours over the samples of a study
        {"name": "batched_32", "kind": "batched", "total": 600_000, "samples": 32, "d": 50, "k": 15, "comps": 30},
        # neighbours through a partitioner that the program keeps
        {"name": "partitioned_500k", "kind": "partitioned", "n": 500_000, "d": 50, "k": 15, "parts": 512, "probe": 8,
         "comps": 200},
        # the last epochs of a layout (a program that shows it as it goes asks for some at a time; in the
        # first ones, with their large steps, the last bits of a position grow to the size of the layout)
        {"name": "umap_300k", "kind": "umap", "n": 300_007, "k": 15, "dim": 2, "first": 187, "last": 200},
        # clustering at the default resolution
        {"name": "leiden_200k", "kind": "leiden", "n": 200_003, "k": 15, "resolution": 1.0},
        # energy distances of a perturbation screen
        {"name": "edistance_100k", "kind": "edistance", "n": 100_000, "groups": 700, "d": 50, "comps": 60},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["graph", "graph", "knn", "knn", "connectivities", "batched", "partitioned", "umap", "leiden",
                       "edistance"])
    if kind in ("graph", "knn"):
        precision = rng.choice(["fp32", "bf16"])
        metric = rng.choice(["euclidean", "euclidean", "cosine"])
        k = rng.randint(5, 30)
        top = 100_000 if precision == "fp32" else (400_000 if k > 16 or metric == "cosine" else 1_000_000)
        n = _log(rng, 2_000, top)
        return {"kind": kind, "n": n, "d": rng.randint(15, 50), "k": k, "metric": metric, "precision": precision,
                "comps": max(5, min(100, n // 500))}
    if kind == "connectivities":
        return {"kind": kind, "n": _log(rng, 2_000, 600_000), "k": rng.randint(5, 30)}
    if kind == "batched":
        samples = rng.randint(3, 32)
        return {"kind": kind, "total": max(samples * 2_500, _log(rng, 20_000, 600_000)), "samples": samples,
                "d": rng.randint(15, 50), "k": rng.randint(5, 15), "comps": 30}
    if kind == "partitioned":
        return {"kind": kind, "n": _log(rng, 50_000, 500_000), "d": rng.randint(15, 50), "k": rng.randint(5, 15),
                "parts": rng.choice([128, 256, 512]), "probe": rng.choice([2, 4, 8]), "comps": 200}
    if kind == "umap":
        first = rng.randint(187, 192)
        return {"kind": kind, "n": _log(rng, 3_000, 300_000), "k": rng.randint(8, 20), "dim": rng.choice([2, 2, 3]),
                "first": first, "last": first + rng.randint(4, 8)}
    if kind == "leiden":
        return {"kind": kind, "n": _log(rng, 3_000, 200_000), "k": rng.randint(8, 20),
                "resolution": rng.choice([0.5, 1.0, 2.0])}
    n = _log(rng, 4_000, 100_000)
    return {"kind": kind, "n": n, "groups": max(4, n // rng.randint(60, 400)), "d": rng.randint(15, 50), "comps": 60}


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _mixture(n, d, comps, g, means=None):
    if means is None:
        means = torch.randn((comps, d), generator=g, device="cuda") * 2.0
    scale = torch.arange(1, d + 1, device="cuda", dtype=torch.float32).rsqrt()
    label = torch.randint(0, len(means), (n,), generator=g, device="cuda")
    return (means[label] + torch.randn((n, d), generator=g, device="cuda") * scale).contiguous()


def _sizes(total, count, lo, hi, seed):
    r = np.random.default_rng(seed)
    s = np.exp(r.uniform(math.log(lo), math.log(hi), count))
    s = np.maximum(2, np.floor(s * (total / s.sum()))).astype(np.int64)
    s[int(np.argmax(s))] += total - s.sum()
    return s


def _lists(n, k, g, block=2_000):
    """kNN lists (int32 ids, float32 distances, the cell itself first) of n cells inside blocks of about
    `block` cells, each block a cluster of its own; ids shuffled.  Third, the block of each cell."""
    blocks = max(1, round(n / block))
    m = -(-n // blocks)
    scale = torch.arange(1, 51, device="cuda", dtype=torch.float32).rsqrt()
    ids = torch.randperm(n, generator=g, device="cuda")
    idx = torch.empty((n, k), dtype=torch.int32, device="cuda")
    dist = torch.empty((n, k), dtype=torch.float32, device="cuda")
    of = torch.empty(n, dtype=torch.int64, device="cuda")
    for s in range(0, n, m):
        c = min(m, n - s)
        x = (torch.randn((c, 50), generator=g, device="cuda") * scale).double()
        sq = (x * x).sum(1)
        d2 = sq[:, None] + sq[None, :] - 2.0 * (x @ x.T)
        d2.fill_diagonal_(-1.0)   # the cell itself comes first
        v, j = torch.topk(d2, k, largest=False)
        v[:, 0] = 0.0
        row = ids[s:s + c]
        idx[row] = row[j].int()
        dist[row] = v.clamp_min(0.0).sqrt().float()
        of[row] = s // m
    return idx, dist, of


def _graph(idx, dist):
    """(indptr, columns, values, rho, sigma): the fuzzy graph of kNN lists in 64 bits."""
    n, k = idx.shape
    i, d = idx.long(), dist.double()
    me = torch.arange(n, device=d.device)[:, None]
    valid = (i >= 0) & (i < n)
    rho = torch.where(d > 0, d, math.inf).min(1).values
    rho = torch.where(rho.isinf(), torch.zeros_like(rho), rho)
    gap = (d - rho[:, None]).clamp_min(0.0)
    target = math.log2(k)
    lo, hi = torch.zeros_like(rho), torch.full_like(rho, math.inf)
    sigma, done = torch.ones_like(rho), torch.zeros_like(rho, dtype=torch.bool)
    for _ in range(64):
        s = torch.exp(-gap[:, 1:] / sigma[:, None]).sum(1)
        done = done | ((s - target).abs() < 1e-5)
        big = s > target
        nhi = torch.where(big, sigma, hi)
        nlo = torch.where(big, lo, sigma)
        mid = torch.where(nhi.isinf(), 2.0 * sigma, 0.5 * (nlo + nhi))
        hi, lo = torch.where(done, hi, nhi), torch.where(done, lo, nlo)
        sigma = torch.where(done, sigma, mid)
    sigma = torch.maximum(sigma, 1e-3 * torch.where(rho > 0, d.mean(1), d.mean()))
    w = torch.where(gap <= 0, torch.ones_like(gap), torch.exp(-gap / sigma[:, None]))
    keep = valid & (i != me) & (w > 0)
    a = (me * n + i)[keep]
    b = (i * n + me)[keep]
    v = w[keep]
    keys, inv = torch.unique(torch.cat([a, b]), return_inverse=True)
    fwd = torch.zeros(len(keys), dtype=torch.float64, device=d.device)
    rev = torch.zeros_like(fwd)
    fwd[inv[:len(a)]] = v
    rev[inv[len(a):]] = v
    val = fwd + rev - fwd * rev
    indptr = torch.zeros(n + 1, dtype=torch.int64, device=d.device)
    indptr[1:] = torch.cumsum(torch.bincount(keys // n, minlength=n), 0)
    return indptr, keys % n, val, rho, sigma


def _symmetric_graph(n, k, g):
    idx, dist, of = _lists(n, k, g)
    indptr, col, val, _, _ = _graph(idx, dist)
    return indptr, col.int(), val.float(), of


def _csr_out(n, k):
    """Buffers that a program keeps for the graph (entries past indptr[n] stay zero)."""
    cap = rsc.rsc_connectivities_max_nnz(n, k)
    return (torch.empty(n + 1, dtype=torch.int64, device="cuda"), torch.zeros(cap, dtype=torch.int32, device="cuda"),
            torch.zeros(cap, dtype=torch.float32, device="cuda"), torch.empty(n, device="cuda"),
            torch.empty(n, device="cuda"))


def _embedding(case, seed):
    return _mixture(case["n"], case["d"], case["comps"], _gen(seed))


def _samples(case, seed):
    g = _gen(seed)
    sizes = _sizes(case["total"], case["samples"], 2e3, 2e5, seed)
    sizes = np.maximum(sizes, 100)   # each sample holds more cells than k
    means = torch.randn((case["comps"], case["d"]), generator=g, device="cuda") * 2.0
    X = torch.cat([_mixture(int(s), case["d"], 0, g,
                            means + torch.randn(case["d"], generator=g, device="cuda") * math.sqrt(0.5))
                   for s in sizes])
    return X, np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)


def _screen(case, seed):
    g = _gen(seed)
    sizes = _sizes(case["n"], case["groups"], 20, 2_000, seed)
    X = _mixture(int(sizes.sum()), case["d"], case["comps"], g)
    cells = torch.randperm(len(X), generator=g, device="cuda").int()
    return X, np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64), cells


def _layout(case, seed):
    g = _gen(seed)
    indptr, indices, data, of = _symmetric_graph(case["n"], case["k"], g)
    # a blob of positions for each block of cells
    centres = torch.rand((int(of.max()) + 1, case["dim"]), generator=g, device="cuda") * 20.0 - 10.0
    start = centres[of] + torch.randn((case["n"], case["dim"]), generator=g, device="cuda")
    return {"indptr": indptr, "indices": indices, "data": data, "start": start, "seed": seed, "nnz": len(indices)}


def _partitioner(case, X, g):
    """A network whose logits rank the parts' centres by distance (rows of X as centres): a stand-in for
    a trained one that is the same on every run."""
    d, parts, hidden = case["d"], case["parts"], 256
    centres = X[torch.randperm(len(X), generator=g, device="cuda")[:parts]].cpu().numpy()
    W1 = np.zeros((hidden, d), dtype=np.float32)
    W1[:d] = np.eye(d)
    W1[d:2 * d] = -np.eye(d)
    W2 = np.eye(hidden, dtype=np.float32)
    W3 = np.zeros((parts, hidden), dtype=np.float32)
    W3[:, :d], W3[:, d:2 * d] = 2.0 * centres, -2.0 * centres
    zero = np.zeros(hidden, dtype=np.float32)
    p = rsc.Partitioner(d, parts, hidden, seed=0)
    p.set_params(np.concatenate([W1.ravel(), zero, W2.ravel(), zero, W3.ravel(), -(centres ** 2).sum(1)]))
    p.build_index(X)
    return p


def prepare(case, seed):
    kind = case["kind"]
    if kind == "graph":
        return {"case": case, "X": _embedding(case, seed), "csr": _csr_out(case["n"], case["k"])}
    if kind == "knn":
        return {"case": case, "X": _embedding(case, seed)}
    if kind == "connectivities":
        idx, dist, _ = _lists(case["n"], case["k"], _gen(seed))
        return {"case": case, "idx": idx, "dist": dist, "csr": _csr_out(case["n"], case["k"])}
    if kind == "batched":
        X, off = _samples(case, seed)
        return {"case": case, "X": X, "off": off}
    if kind == "partitioned":
        X = _embedding(case, seed)
        return {"case": case, "X": X, "part": _partitioner(case, X, _gen(seed + 1))}
    if kind == "umap":
        return {"case": case, **_layout(case, seed)}
    if kind == "leiden":
        indptr, indices, data, _ = _symmetric_graph(case["n"], case["k"], _gen(seed))
        return {"case": case, "indptr": indptr, "indices": indices, "data": data}
    X, off, cells = _screen(case, seed)
    return {"case": case, "X": X, "off": off, "cells": cells}


# -------------------------------------------------------------------- a pass

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "graph":
        idx, dist = rsc.rsc_knn(state["X"], case["k"], case["metric"], case["precision"])
        return [idx, dist, *rsc.rsc_connectivities(idx, dist, out=state["csr"])]
    if kind == "knn":
        return list(rsc.rsc_knn(state["X"], case["k"], case["metric"], case["precision"]))
    if kind == "connectivities":
        return list(rsc.rsc_connectivities(state["idx"], state["dist"], out=state["csr"]))
    if kind == "batched":
        return list(rsc.rsc_knn_batched(state["X"], state["off"], case["k"], K_CROSS))
    if kind == "partitioned":
        return list(state["part"].knn(state["X"], k=case["k"], n_probe=case["probe"]))
    if kind == "umap":
        emb = state["start"].clone()
        rsc.rsc_umap_layout(state["indptr"], state["indices"], state["data"], emb, UMAP_A, UMAP_B,
                            n_epochs=200, epoch_first=case["first"], epoch_last=case["last"], seed=state["seed"],
                            nnz=state["nnz"])
        return [emb]
    if kind == "leiden":
        return list(rsc.rsc_leiden(state["indptr"], state["indices"], state["data"], resolution=case["resolution"]))
    return list(rsc.rsc_edistance(state["X"], state["off"], state["cells"]))


def work(case):
    """Inputs read once, outputs written once; operations of the definition on what is returned (a kNN
    list's own distances, not the search for them)."""
    kind = case["kind"]
    if kind in ("graph", "knn", "partitioned"):
        n, d, k = case["n"], case["d"], case["k"]
        bytes_, flops = 4 * n * d + 8 * n * k, 3 * n * k * d
        if kind == "graph":
            bytes_ += 8 * n * k + 8 * n + 8 * int(1.5 * n * k) + 8 * n
            flops += 60 * n * k
        return {"bytes": bytes_, "flops": flops}
    if kind == "connectivities":
        n, k = case["n"], case["k"]
        return {"bytes": 8 * n * k + 8 * n + 8 * int(1.5 * n * k) + 8 * n, "flops": 60 * n * k}
    if kind == "batched":
        n, per = case["total"], case["k"] + K_CROSS * case["samples"]
        return {"bytes": 4 * n * case["d"] + 8 * n * per, "flops": 3 * n * per * case["d"]}
    if kind == "umap":
        n, nnz, epochs = case["n"], int(1.5 * case["n"] * case["k"]), case["last"] - case["first"] + 1
        return {"bytes": epochs * (8 * nnz + 8 * n + 8 * n * case["dim"]), "flops": epochs * nnz * 40}
    if kind == "leiden":
        n, nnz = case["n"], int(1.5 * case["n"] * case["k"])
        return {"bytes": 8 * n + 8 * nnz + 4 * n, "flops": 20 * nnz}
    n, G, d = case["n"], case["groups"], case["d"]
    return {"bytes": 4 * n * d + 4 * n + 24 * G * G, "flops": n * (n - 1) // 2 * 3 * d}


# ------------------------------------------------------------- in 64 bits

def _exact_knn(X, k, metric, rows=None, cols=None):
    """The k smallest distances from `rows` of X to `cols` of X, ascending, with their ids."""
    x = X.double()
    if metric == "cosine":
        x = x / x.norm(dim=1, keepdim=True)
    q, y = (x if rows is None else x[rows]), (x if cols is None else x[cols])
    base = 0 if cols is None else cols.start
    sq = (y * y).sum(1)
    dist, ids = [], []
    for s in range(0, len(q), 4_096):
        c = q[s:s + 4_096]
        j = torch.topk(sq[None, :] - 2.0 * (c @ y.T), min(k + 4, len(y)), largest=False).indices
        v = ((c[:, None, :] - y[j]) ** 2).sum(2)
        v, o = torch.sort(v, 1)
        dist.append(v[:, :k])
        ids.append(torch.gather(j, 1, o)[:, :k] + base)
    dist, ids = torch.cat(dist), torch.cat(ids)
    return (0.5 * dist if metric == "cosine" else dist.sqrt()), ids


def _padded(val, size):
    out = torch.zeros(size, dtype=torch.float64, device=val.device)
    out[:len(val)] = val
    return out


def _mix64(z):
    """The output function of SplitMix64 on int64 bit patterns."""
    def shr(v, s):
        return (v >> s) & ((1 << (64 - s)) - 1)
    z = (z ^ shr(z, 30)) * (0xBF58476D1CE4E5B9 - (1 << 64))
    z = (z ^ shr(z, 27)) * (0x94D049BB133111EB - (1 << 64))
    return z ^ shr(z, 31)


def _exact_layout(case, s, neg=5):
    indptr, col, w = s["indptr"], s["indices"].long(), s["data"]
    n, nnz, a, b = case["n"], s["nnz"], float(np.float32(UMAP_A)), float(np.float32(UMAP_B))
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), indptr[1:] - indptr[:-1])
    f = w / w.max()   # the schedule is defined in 32 bits
    y = s["start"].double()
    half = (neg + 1) // 2
    for e in range(case["first"], case["last"] + 1):
        alpha = 1.0 - (e - 1) / 200
        on = torch.nonzero(torch.floor(f * float(e)) > torch.floor(f * float(e - 1))).squeeze(1)
        i, j = row[on], col[on]
        move = torch.zeros_like(y)
        diff = y[i] - y[j]
        d2 = (diff * diff).sum(1)
        p = torch.where(d2 > 0, d2, torch.ones_like(d2)) ** b
        c = torch.where(d2 > 0, -2.0 * a * b * p / (torch.where(d2 > 0, d2, torch.ones_like(d2)) * (1.0 + a * p)),
                        torch.zeros_like(d2))
        move.index_add_(0, i, 2.0 * alpha * (c[:, None] * diff).clamp(-4.0, 4.0))
        for q in range(neg):
            number = ((e - 1) * nnz + on) * half + q // 2 + 1
            z = _mix64(s["seed"] + number * (0x9E3779B97F4A7C15 - (1 << 64)))
            h = ((z >> 32) if q % 2 == 0 else z) & 0xFFFFFFFF
            v = (h * n) >> 32
            diff = y[i] - y[v]
            d2 = (diff * diff).sum(1)
            c = 2.0 * b / ((0.001 + d2) * (1.0 + a * d2 ** b))
            move.index_add_(0, i, alpha * (c[:, None] * diff).clamp(-4.0, 4.0))
        y = y + move
    return y


def _exact_energy(X, off, cells):
    G = len(off) - 1
    x = X.double()[cells.long()]
    size = torch.from_numpy(np.diff(off)).to("cuda")
    group = torch.repeat_interleave(torch.arange(G, device="cuda"), size)
    ends = torch.from_numpy(off[1:]).to("cuda") - 1   # every group holds at least two cells
    S = torch.zeros((G, G), dtype=torch.float64, device="cuda")
    sq = (x * x).sum(1)
    for s in range(0, len(x), 2_048):
        c = x[s:s + 2_048]
        dist = (sq[s:s + 2_048, None] + sq[None, :] - 2.0 * (c @ x.T)).clamp_min(0.0).sqrt()
        r = torch.arange(len(c), device="cuda")
        dist[r, s + r] = 0.0
        part = torch.diff(torch.cumsum(dist, 1)[:, ends], dim=1, prepend=torch.zeros_like(dist[:, :1]))
        S.index_add_(0, group[s:s + 2_048], part)
    S = torch.triu(S, 1) + torch.diag(S.diagonal() / 2)
    m = size.double()
    pairs = m[:, None] * m[None, :]
    pairs.diagonal().copy_((m * (m - 1) / 2).clamp_min(1.0))
    mean = (S + torch.triu(S, 1).T) / pairs
    within = mean.diagonal()
    return [S, mean, 2.0 * mean - within[:, None] - within[None, :]]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("graph", "knn") and case["n"] <= EXACT_ROWS:
        n, k = case["n"], case["k"]
        dist, ids = _exact_knn(_embedding(case, seed), k, case["metric"])
        if kind == "knn":
            return [None, dist]
        if n > EXACT_GRAPH_ROWS:
            return [None, dist, None, None, None, None, None]
        _, _, val, rho, sigma = _graph(ids, dist)
        return [None, dist, None, None, _padded(val, 2 * n * (k - 1)), rho, sigma]
    if kind == "connectivities":
        idx, dist, _ = _lists(case["n"], case["k"], _gen(seed))
        _, _, val, rho, sigma = _graph(idx, dist)
        return [None, None, _padded(val, 2 * case["n"] * (case["k"] - 1)), rho, sigma]
    if kind == "batched" and case["total"] <= EXACT_ROWS:
        X, off = _samples(case, seed)
        within, cross = [], []
        for s in range(len(off) - 1):
            own = slice(int(off[s]), int(off[s + 1]))
            within.append(_exact_knn(X, case["k"], "euclidean", own, own)[0])
            cross.append(_exact_knn(X, K_CROSS, "euclidean", None, own)[0])
        return [None, torch.cat(within), None, torch.sort(torch.cat(cross, 1), 1).values]
    if kind == "umap":
        return [_exact_layout(case, _layout(case, seed))]
    if kind == "edistance":
        return _exact_energy(*_screen(case, seed))
    return None
