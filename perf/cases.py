"""Workloads of the k-core library, each one call (or one request stream) that a
program makes through the public binding (`KCore`, `KCoreServer`).

listed() holds the fixed cases, draw(rng) gives another one of the same ranges,
prepare(case, seed) builds what a program has in hand before the call (a CSR or
an edge list on the GPU, or graphs in host memory, and the library handle),
run(state) makes the call, work(case) states the bytes the call cannot do
without, and exact(case, seed) computes the same outputs with plain torch in
64-bit integers. Every output is an integer (coreness, masks, CSR arrays).

Graphs are synthetic, of the shapes the benchmark uses: Erdos-Renyi, R-MAT
(0.57, 0.19, 0.19, 0.05; ids permuted), 10-nearest-neighbour graphs of points in
the unit square with planted cliques, and batches that mix ER and R-MAT.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2502_08042_gb300 import KCore, KCoreServer

DEV = "cuda:0"


def listed():
    return [
        # A single small graph: the latency of one call (10,000 vertices, 50,000 edges).
        {"name": "peel_er_10k", "kind": "peel", "graph": "er", "n": 10_000, "edges": 50_000},
        # A mid-size social graph from outside the library: the CSR is checked, then decomposed.
        {"name": "checked_rmat_20", "kind": "checked", "graph": "rmat", "n": 1 << 20, "edges": 1 << 24},
        # The largest single graph: R-MAT scale 24, edge factor 16 (the headline workload).
        {"name": "peel_rmat_24", "kind": "peel", "graph": "rmat", "n": 1 << 24, "edges": 1 << 28},
        # A spatial graph, low degrees and long cascades, with dense cliques (2^24 points).
        {"name": "peel_knn_24", "kind": "peel", "graph": "knn", "n": 1 << 24, "edges": 10 << 24},
        # A k'-core query (membership only) on the large R-MAT graph.
        {"name": "mask_rmat_24", "kind": "mask", "graph": "rmat", "n": 1 << 24, "edges": 1 << 28, "k": 128},
        # Edge list to CSR: a small ragged list (latency of the build's launches) ...
        {"name": "csr_er_100k", "kind": "csr", "graph": "er", "n": 99_991, "edges": 1_000_003},
        # ... and a large one with repeats and self-loops.
        {"name": "csr_rmat_22", "kind": "csr", "graph": "rmat", "n": 1 << 22, "edges": 1 << 26},
        # Edge lists of a batch of graphs to one segmented CSR.
        {"name": "csr_batch_256", "kind": "csr_batch", "graphs": 256, "lo": 1_000, "hi": 200_000},
        # A batch of small graphs: many independent requests decomposed in one launch.
        {"name": "batch_small_1000", "kind": "batch", "graphs": 1_000, "lo": 1_000, "hi": 8_000},
        # A mixed batch, 1k to 200k vertices, bound by its largest graphs.
        {"name": "batch_mixed_512", "kind": "batch", "graphs": 512, "lo": 1_000, "hi": 200_000},
        # End to end from pinned host buffers: copies in, decomposition, copies out.
        {"name": "host_rmat_20", "kind": "host", "graph": "rmat", "n": 1 << 20, "edges": 1 << 24},
        # A burst of requests to the server (host graphs in, coreness out), two of them large.
        {"name": "serve_192", "kind": "serve", "graphs": 192, "lo": 1_000, "hi": 200_000, "large": 2, "scale": 20},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng: random.Random) -> dict:
    kind = rng.choice(["peel", "peel", "checked", "mask", "csr", "csr_batch", "batch", "batch", "host", "serve"])
    if kind in ("batch", "csr_batch"):
        top = 512 if kind == "batch" else 256
        hi = _log_int(rng, 4_000, 200_000)
        return {"kind": kind, "graphs": _log_int(rng, 16, top), "lo": 1_000, "hi": hi}
    if kind == "serve":
        return {"kind": kind, "graphs": _log_int(rng, 8, 192), "lo": 1_000, "hi": _log_int(rng, 4_000, 200_000),
                "large": rng.randint(0, 2), "scale": 20}
    graph = rng.choice(["er", "rmat", "rmat", "knn"]) if kind == "peel" else rng.choice(["er", "rmat"])
    top = {"peel": 1 << 23, "mask": 1 << 23, "csr": 1 << 22}.get(kind, 1 << 20)
    n = _log_int(rng, 5_000, top)
    edges = 10 * n if graph == "knn" else int(n * rng.uniform(4, 16))
    c = {"kind": kind, "graph": graph, "n": n, "edges": edges}
    if kind == "mask":
        c["k"] = _log_int(rng, 4, 512)
    return c


# ------------------------------------------------------------------ generators
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _rmat_bits(bits, g, levels):
    """R-MAT ids of len(bits) edges: edge e takes bits[e] <= levels levels."""
    E = bits.numel()
    s = torch.zeros(E, dtype=torch.int32, device=DEV)
    d = torch.zeros(E, dtype=torch.int32, device=DEV)
    for level in range(levels):
        r = torch.rand(E, generator=g, device=DEV)
        on = (bits > level).to(torch.int32)
        sb = (r >= 0.76).to(torch.int32)
        db = ((r >= 0.57) & (r < 0.76) | (r >= 0.95)).to(torch.int32)
        s = (s << on) | (sb * on)
        d = (d << on) | (db * on)
    return s, d


def _rmat(n, E, g):
    bits = max(1, (n - 1).bit_length())
    perm = torch.randperm(n, generator=g, device=DEV, dtype=torch.int64).to(torch.int32)
    src, dst = [], []
    step = 1 << 26
    for e0 in range(0, E, step):
        m = min(step, E - e0)
        s, d = _rmat_bits(torch.full((m,), bits, dtype=torch.int32, device=DEV), g, bits)
        if n != 1 << bits:  # scale the ids to [0, n)
            s, d = ((x.to(torch.int64) * n >> bits).to(torch.int32) for x in (s, d))
        src.append(perm[s])
        dst.append(perm[d])
    return torch.cat(src), torch.cat(dst)


def _er(n, E, g):
    return (torch.randint(n, (E,), generator=g, device=DEV, dtype=torch.int32),
            torch.randint(n, (E,), generator=g, device=DEV, dtype=torch.int32))


def _knn(n, g, k=10):
    """Each point's k nearest among the points of the 3 x 3 cells around it
    (about five points per cell), plus cliques on random vertices."""
    p = torch.rand(n, 2, generator=g, device=DEV)
    w = max(3, int(math.sqrt(n / 5)))
    cell = (p * w).to(torch.int64).clamp_(0, w - 1)
    cid = cell[:, 0] * w + cell[:, 1]
    order = torch.argsort(cid)
    p, cid = p[order], cid[order]
    start = torch.searchsorted(cid, torch.arange(w * w + 1, device=DEV))
    span = 32  # candidates per row of three cells
    src, dst = [], []
    ar = torch.arange(span, device=DEV)
    for i0 in range(0, n, 1 << 21):
        i = torch.arange(i0, min(n, i0 + (1 << 21)), device=DEV)
        r, c = cid[i] // w, cid[i] % w
        cand = []
        for dr in (-1, 0, 1):
            rr = (r + dr).clamp(0, w - 1)
            a = start[rr * w + (c - 1).clamp(min=0)]
            b = start[rr * w + (c + 1).clamp(max=w - 1) + 1]
            j = a[:, None] + ar
            ok = (j < b[:, None]) & (r + dr == rr)[:, None] & (j != i[:, None])
            cand.append(torch.where(ok, j, -1))
        cand = torch.cat(cand, 1)
        q = p[cand.clamp(min=0)]
        dist = ((q - p[i][:, None]) ** 2).sum(2)
        dist[cand < 0] = 9.0
        near = torch.topk(dist, k, 1, largest=False, sorted=False).indices
        t = torch.gather(cand, 1, near)
        t = torch.where(t < 0, i[:, None], t)  # too few candidates: a self-loop, dropped by the build
        src.append(order[i].repeat_interleave(k).to(torch.int32))
        dst.append(order[t.reshape(-1)].to(torch.int32))
    for c in range(64):
        u = float(torch.rand(1, generator=g, device=DEV))
        size = min(n // 4, int(50 * (2000 / 50) ** u))
        v = torch.randint(n, (size,), generator=g, device=DEV, dtype=torch.int32)
        ij = torch.triu_indices(size, size, 1, device=DEV)
        src.append(v[ij[0]])
        dst.append(v[ij[1]])
    return torch.cat(src), torch.cat(dst)


def _edges(case, g):
    if case["graph"] == "er":
        return _er(case["n"], case["edges"], g)
    if case["graph"] == "rmat":
        return _rmat(case["n"], case["edges"], g)
    return _knn(case["n"], g)


def _sizes(case):
    """Vertices and edges of each graph of a batch (a property of the case:
    the seed changes the graphs, not their sizes)."""
    r = random.Random(case["graphs"] * 1_000_003 + case["hi"])
    ns = [_log_int(r, case["lo"], case["hi"]) for _ in range(case["graphs"])]
    return ns, [int(n * r.uniform(4, 64) / 2) for n in ns], [r.random() < 0.5 for _ in ns]


def _structure(case):
    """Generator of the graphs' structure where the seed only relabels and reorders them."""
    return _gen(case["edges"] if "edges" in case else case["graphs"] * 1_000_003 + case["hi"])


def _shuffled(s, d, g):
    """The same edges in another order, some of them the other way round."""
    p = torch.randperm(s.numel(), generator=g, device=DEV)
    s, d = s[p], d[p]
    turn = torch.rand(s.numel(), generator=g, device=DEV) < 0.5
    return torch.where(turn, d, s), torch.where(turn, s, d)


def _list_edges(case, seed):
    """The edge list of a build: the case fixes the graph up to its labels, the
    seed its labels and the list's order, so the number of arcs is the case's."""
    s, d = _edges(case, _structure(case))
    g = _gen(seed)
    perm = torch.randperm(case["n"], generator=g, device=DEV, dtype=torch.int64).to(torch.int32)
    return _shuffled(perm[s], perm[d], g)


def _batch_edges(case, g, labels=None):
    """Edge lists of a batch (graph-local ids); labels: the generator of the ids, if not g."""
    ns, es, rm = _sizes(case)
    n_g = torch.tensor(ns, device=DEV)
    e_g = torch.tensor(es, device=DEV)
    z = torch.zeros(1, dtype=torch.int64, device=DEV)
    gv, eo = torch.cat([z, n_g.cumsum(0)]), torch.cat([z, e_g.cumsum(0)])
    N, E = sum(ns), sum(es)
    gid = torch.repeat_interleave(torch.arange(len(ns), device=DEV), e_g)
    nn = n_g[gid]
    bits = torch.tensor([max(1, (n - 1).bit_length()) if x else 0 for n, x in zip(ns, rm)], device=DEV)[gid]
    s, d = _rmat_bits(bits.to(torch.int32), g, max(ns).bit_length())
    s, d = s.to(torch.int64) * nn >> bits, d.to(torch.int64) * nn >> bits
    er = bits == 0
    rs = (torch.rand(E, generator=g, device=DEV, dtype=torch.float64) * nn).to(torch.int64)
    rd = (torch.rand(E, generator=g, device=DEV, dtype=torch.float64) * nn).to(torch.int64)
    s, d = torch.where(er, rs, s), torch.where(er, rd, d)
    # ids permuted within each graph
    vid = torch.repeat_interleave(torch.arange(len(ns), device=DEV), n_g)
    key = vid + torch.rand(N, generator=labels or g, device=DEV, dtype=torch.float64)
    perm = torch.argsort(key) - gv[vid]
    return gv, eo, perm[gv[gid] + s].to(torch.int32), perm[gv[gid] + d].to(torch.int32), max(ns)


def _csr_of(case, seed):
    s, d = _edges(case, _gen(seed))
    with KCore(0) as k:
        off, adj = k.build_csr(case["n"], s, d)
        return off, adj.clone()


def _batch_csr_of(case, seed):
    gv, eo, s, d, top = _batch_edges(case, _gen(seed))
    with KCore(0) as k:
        off, adj = k.build_csr_batched(gv, eo, s, d, top)
        return gv, off, adj.clone()


def _pinned(t):
    return t.cpu().pin_memory()


def _served_graphs(case, seed):
    """Host graphs of a serve case (views of pinned tensors), the large ones last."""
    gv, off, adj = _batch_csr_of(case, seed)
    b = off[gv].tolist()
    v = gv.tolist()
    offs, adjs = [], []
    for i in range(case["graphs"]):
        offs.append(_pinned(off[v[i]:v[i + 1] + 1] - b[i]).numpy())
        adjs.append(_pinned(adj[b[i]:b[i + 1]]).numpy())
    for i in range(case["large"]):
        n = (1 << case["scale"]) + 1  # one vertex above the batched kernel's share of the requests
        o, a = _csr_of({"graph": "rmat", "n": n, "edges": 16 * n}, seed + 1 + i)
        offs.append(_pinned(o).numpy())
        adjs.append(_pinned(a).numpy())
    return offs, adjs


# ------------------------------------------------------------------ the calls
def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind}
    if kind == "serve":
        st["offs"], st["adjs"] = _served_graphs(case, seed)
        cut = np.cumsum([0] + [len(o) - 1 for o in st["offs"]])
        st["core"] = torch.empty(int(cut[-1]), dtype=torch.int32).pin_memory().numpy()
        st["outs"] = [st["core"][a:b] for a, b in zip(cut[:-1], cut[1:])]  # each request's part of the result
        st["server"] = KCoreServer(0, pool_bytes=8 << 30, max_requests=1024)
        return st
    st["k"] = KCore(0)
    if kind == "csr":
        st["n"] = case["n"]
        st["src"], st["dst"] = _list_edges(case, seed)
    elif kind == "csr_batch":
        st["gv"], st["eo"], st["src"], st["dst"], st["top"] = _batch_edges(case, _structure(case), _gen(seed))
    elif kind == "batch":
        st["gv"], st["off"], st["adj"] = _batch_csr_of(case, seed)
    else:
        st["off"], st["adj"] = _csr_of(case, seed)
        st["kprime"] = case.get("k", 0)
        if kind == "host":
            off, adj = st.pop("off"), st.pop("adj")
            st["off"], st["adj"] = _pinned(off).numpy(), _pinned(adj).numpy()
            st["core"] = torch.empty(case["n"], dtype=torch.int32).pin_memory().numpy()
            st["kmax"] = torch.zeros(1, dtype=torch.int32).pin_memory().numpy()
    return st


def run(state):
    kind = state["kind"]
    if kind == "serve":
        return _serve(state)
    k = state["k"]
    if kind == "peel":
        return k.decompose(state["off"], state["adj"])
    if kind == "checked":
        k.validate_csr(state["off"], state["adj"])
        return k.decompose(state["off"], state["adj"])
    if kind == "mask":
        return k.core_mask(state["off"], state["adj"], state["kprime"])
    if kind == "csr":
        return k.build_csr(state["n"], state["src"], state["dst"])
    if kind == "csr_batch":
        return k.build_csr_batched(state["gv"], state["eo"], state["src"], state["dst"], state["top"])
    if kind == "batch":
        return k.decompose_batched(state["gv"], state["off"], state["adj"])
    k.decompose_host_into(state["off"], state["adj"], state["core"], state["kmax"])
    return state["core"], state["kmax"]


def _serve(state):
    srv, offs, adjs, outs = state["server"], state["offs"], state["adjs"], state["outs"]
    ticket, kmax, left, nxt = {}, np.zeros(len(offs), np.int32), len(offs), 0
    while left:
        while nxt < len(offs):
            t = srv.submit(offs[nxt], adjs[nxt], outs[nxt])
            if t is None:
                break
            ticket[t] = nxt
            nxt += 1
        for t, km, status in srv.poll():
            if status != 0:
                raise RuntimeError(f"request failed with status {status}")
            kmax[ticket[t]] = km
            left -= 1
    return {"core": state["core"], "kmax": kmax}


# ------------------------------------------------------------------ work and exact results
def _arcs(case):
    if case["graph"] == "knn":
        return 14 * case["n"]  # about 14 neighbours once symmetrised
    return 2 * case["edges"]


def work(case):
    kind = case["kind"]
    if kind in ("batch", "csr_batch", "serve"):
        ns, es, _ = _sizes(case)
        n, e, G = sum(ns), sum(es), len(ns)
        if kind == "serve":
            n += case["large"] << case["scale"]
            e += 16 * (case["large"] << case["scale"])
        if kind == "csr_batch":
            return {"bytes": 8 * e + 16 * G + 8 * n + 8 * e, "flops": 0}
        return {"bytes": 8 * n + 8 * e + 12 * G + 4 * n, "flops": 0}
    n, m = case["n"], _arcs(case)
    if kind == "csr":
        return {"bytes": 8 * case["edges"] + 8 * (n + 1) + 4 * m, "flops": 0}
    return {"bytes": 8 * (n + 1) + 4 * m + 4 * n, "flops": 0}


def _peel(off, adj, only=None):
    """Coreness by Algorithm 1 in plain torch (int64); with `only`, one level: membership of the only-core."""
    n = off.numel() - 1
    deg = off[1:] - off[:-1]
    core = torch.zeros(n, dtype=torch.int64, device=off.device)
    left = torch.arange(n, device=off.device)
    lens, starts = deg.clone(), off[:-1]
    while left.numel():
        k = only - 1 if only is not None else int(deg[left].min())
        while True:
            out = deg[left] <= k
            f, left = left[out], left[~out]
            if not f.numel():
                break
            core[f] = k
            ln = lens[f]
            tot = int(ln.sum())
            base = torch.repeat_interleave(starts[f] - (ln.cumsum(0) - ln), ln, output_size=tot)
            u = adj[base + torch.arange(tot, device=off.device)].to(torch.int64)
            if tot > n // 8:
                deg -= torch.bincount(u, minlength=n)
            else:
                deg.index_add_(0, u, torch.full_like(u, -1))
        if only is not None:
            mask = torch.zeros(n, dtype=torch.int64, device=off.device)
            mask[left] = 1
            return mask
    return core


def _csr(n, s, d):
    """(offsets, keys source * n + target) of the simple undirected graph of an edge list, by sorting."""
    keep = s != d
    s, d = s[keep].to(torch.int64), d[keep].to(torch.int64)
    key = torch.unique(torch.cat([s * n + d, d * n + s]))
    return torch.searchsorted(key, torch.arange(n + 1, device=key.device) * n), key


def _plain_csr(case, edges):
    off, key = _csr(case["n"], *edges)
    return off, key % case["n"]


def _plain_batch(gv, eo, s, d, _):
    """A batch's edge lists as one disjoint union (global ids)."""
    base = torch.repeat_interleave(gv[:-1], eo[1:] - eo[:-1])
    off, key = _csr(int(gv[-1]), s + base, d + base)
    return gv, off, key % int(gv[-1])


def exact(case, seed):
    kind = case["kind"]
    if kind == "csr":
        return _plain_csr(case, _list_edges(case, seed))
    if kind in ("csr_batch", "batch", "serve"):
        g = _gen(seed)
        lists = _batch_edges(case, _structure(case), g) if kind == "csr_batch" else _batch_edges(case, g)
        gv, off, adj = _plain_batch(*lists)
        gid = torch.repeat_interleave(torch.arange(gv.numel() - 1, device=DEV), gv[1:] - gv[:-1])
        if kind == "csr_batch":
            return off, adj - torch.repeat_interleave(gv[gid], off[1:] - off[:-1])
        core = _peel(off, adj)
        kmax = torch.zeros(gv.numel() - 1, dtype=torch.int64, device=DEV).scatter_reduce_(0, gid, core, "amax")
        if kind == "batch":
            return core, kmax
        cores, kmaxs = [core], kmax.tolist()
        for i in range(case["large"]):
            n = (1 << case["scale"]) + 1
            big = {"graph": "rmat", "n": n, "edges": 16 * n}
            c = _peel(*_plain_csr(big, _edges(big, _gen(seed + 1 + i))))
            cores.append(c)
            kmaxs.append(int(c.max()))
        return {"core": torch.cat(cores).cpu().numpy(), "kmax": np.array(kmaxs)}
    off, adj = _plain_csr(case, _edges(case, _gen(seed)))
    if kind == "mask":
        mask = _peel(off, adj, case["k"])
        return mask, mask.sum().reshape(1)
    core = _peel(off, adj)
    km = core.max().reshape(1)
    return (core.cpu().numpy(), km.cpu().numpy()) if kind == "host" else (core, km)
