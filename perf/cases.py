"""The performance cases: what a user of the library has it do, from a graph of a thousand vertices, where a call is
all latency, to R-MAT scale 24 and a batch of hundreds of graphs.

A case names a path (scc, scc_host, reach, cc, lelists, batch, serve), a graph family and its sizes. Graph families are
the ones of the test suite and the benchmark (2D and 3D tori with independent arcs, R-MAT with a = .57, b = c = .19,
k-NN graphs of a Gaussian mixture); tori and R-MAT are drawn on the GPU here, from the seed alone, since the host
generators take seconds at these sizes. Every output is a whole number, so outputs are compared for equality.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2303_04934_gb300 import graphgen, scc

DEV = "cuda"


# ------------------------------------------------------------------ graphs --
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed & 0x7FFFFFFFFFFFFFFF)
    return g


def _csr(n, src, dst):
    """CSR (int32, on the GPU) of distinct arcs without self-loops."""
    key = torch.unique(src * n + dst)
    row = key // n
    adj = key - row * n
    loop = row == adj
    if bool(loop.any()):
        row, adj = row[~loop], adj[~loop]
    off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    return off.to(torch.int32), adj.to(torch.int32)


def _rmat(n, ef, seed):
    """R-MAT on ceil(log2 n) levels, ids of n and above dropped, the rest permuted."""
    gen = _gen(seed)
    levels = max(1, math.ceil(math.log2(n)))
    keys, left = [], ef << levels
    while left > 0:
        k = min(left, 1 << 26)
        src = torch.zeros(k, dtype=torch.int32, device=DEV)
        dst = torch.zeros(k, dtype=torch.int32, device=DEV)
        for _ in range(levels):
            r = torch.rand(k, generator=gen, device=DEV)
            down = r >= 0.76
            right = ((r >= 0.57) & ~down) | (r >= 0.95)
            src = src * 2 + down
            dst = dst * 2 + right
        keep = (src < n) & (dst < n)
        keys.append((src[keep], dst[keep]))
        left -= k
    perm = torch.randperm(n, generator=gen, device=DEV)
    src = torch.cat([perm[s] for s, _ in keys])
    dst = torch.cat([perm[d] for _, d in keys])
    del keys
    return _csr(n, src, dst)


def _torus(dims, side, p, seed):
    """Torus with `side` vertices an axis (3 or more); each of a vertex's 2 * dims arcs is present with probability p."""
    n = side ** dims
    v = torch.arange(n, device=DEV)
    nbr = []
    for d in range(dims):
        step = side ** d
        x = (v // step) % side
        nbr.append(v + torch.where(x == side - 1, step * (1 - side), step))
        nbr.append(v + torch.where(x == 0, step * (side - 1), -step))
    nbr = torch.stack(nbr, 1)
    there = torch.rand(nbr.shape, generator=_gen(seed), device=DEV) < p
    off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(there.sum(1), 0)
    return off.to(torch.int32), nbr[there].to(torch.int32)


def _n(c):
    return c["side"] ** 2 if c["graph"] == "torus2" else c["side"] ** 3 if c["graph"] == "torus3" else c["n"]


def _arcs(c):
    """Expected arcs (duplicates of R-MAT's draws not taken off)."""
    if c["graph"] == "torus2":
        return 2 * _n(c)
    if c["graph"] == "torus3":
        return int(1.8 * _n(c))
    return c["n"] * c["deg"]


def _entries(n):
    """The expected number of entries of the least-element lists of n vertices is at most this: n times the n-th
    harmonic number."""
    return int(n * (math.log(n) + 1))


def _graph(c, seed):
    """(n, offsets, targets) on the GPU."""
    if c["graph"] == "torus2":
        off, adj = _torus(2, c["side"], 0.5, seed)
    elif c["graph"] == "torus3":
        off, adj = _torus(3, c["side"], 0.3, seed)
    elif c["graph"] == "rmat":
        off, adj = _rmat(c["n"], c["deg"], seed)
    else:
        g = graphgen.knn(c["n"], c["deg"], seed)
        off, adj = torch.from_numpy(g.offsets).to(DEV), torch.from_numpy(g.targets).to(DEV)
    return _n(c), off, adj


# ------------------------------------------------------------------- cases --
def listed():
    return [
        # the smallest call: one small request, where launches and synchronisations are all there is
        {"name": "scc_torus2_1k", "path": "scc", "graph": "torus2", "side": 33},
        # the benchmark's small lattice: large diameter, L2-resident
        {"name": "scc_torus2_65k", "path": "scc", "graph": "torus2", "side": 256},
        # the benchmark's large-diameter lattice
        {"name": "scc_torus3_17m", "path": "scc", "graph": "torus3", "side": 256},
        # a point-cloud k-NN graph, the deepest of the families
        {"name": "scc_knn_1m", "path": "scc", "graph": "knn", "n": 1000003, "deg": 5},
        # the benchmark's flagship: a social-like graph of 16.8 M vertices, one step = create, run, destroy
        {"name": "scc_rmat_17m", "path": "scc", "graph": "rmat", "n": 1 << 24, "deg": 16},
        # the end-to-end call: page-locked host CSR in, host labels out, ragged size
        {"name": "scc_host_rmat_1.5m", "path": "scc_host", "graph": "rmat", "n": 1500007, "deg": 16},
        # reachability of the most sources one call takes, on a resident social-like graph, both directions
        {"name": "reach_rmat_4m_k64", "path": "reach", "graph": "rmat", "n": 1 << 22, "deg": 16, "k": 64},
        # a few sources on a resident lattice, both directions
        {"name": "reach_torus3_1m_k7", "path": "reach", "graph": "torus3", "side": 101, "k": 7},
        # connected components of a resident graph
        {"name": "cc_rmat_4m", "path": "cc", "graph": "rmat", "n": 1 << 22, "deg": 16},
        # least-element lists of a resident graph, computed and copied out
        {"name": "lelists_rmat_262k", "path": "lelists", "graph": "rmat", "n": 1 << 18, "deg": 16},
        # batched SCC: mixed lattices and R-MAT graphs of 1 k to 1 M vertices in one launch
        {"name": "batch_mixed_256", "path": "batch", "graphs": 256, "lo": 1000, "hi": 1000000},
        # a served burst: SCC requests of mixed sizes beside reachability queries on two resident graphs
        {"name": "serve_mixed_64", "path": "serve", "scc": 24, "reach": 40, "lo": 10000, "hi": 300000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["scc", "scc", "scc", "scc_host", "reach", "reach", "cc", "lelists", "batch", "serve"])
    if path == "batch":
        hi = _log(rng, 4000, 1000000)
        return {"path": path, "graphs": _log(rng, 8, 256), "lo": 1000, "hi": hi}
    if path == "serve":
        return {"path": path, "scc": _log(rng, 4, 24), "reach": _log(rng, 4, 40), "lo": 10000,
                "hi": _log(rng, 20000, 300000)}
    top = {"scc": 1 << 24, "scc_host": 1 << 22, "reach": 1 << 22, "cc": 1 << 23, "lelists": 1 << 18}[path]
    c = {"path": path, "graph": rng.choice(["torus2", "torus3", "rmat", "rmat", "knn"])}
    if c["graph"] == "torus2":
        c["side"] = _log(rng, 32, 1227 if path not in ("lelists", "reach") else 300)
    elif c["graph"] == "torus3":
        c["side"] = _log(rng, 10, int(top ** (1 / 3) + 0.01))
    elif c["graph"] == "rmat":
        c["n"] = _log(rng, 1000, top)
        c["deg"] = rng.randint(4, 16)
    else:
        c["n"] = _log(rng, 1000, min(top, 1000003))
        c["deg"] = rng.randint(3, 8)
    if path == "reach":
        c["k"] = rng.randint(1, 64)
    return c


# ------------------------------------------------------------ prepare, run --
class _State(dict):
    """A case's inputs and handles; the server is stopped with it."""

    def __del__(self):
        for h in ("server", "batch", "handle"):
            if h in self:
                self[h].close()


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)


def _mixed(count, lo, hi, seed):
    """`count` graphs (n, off, adj), alternately 2D tori and R-MAT of edge factor 8: sizes log-uniform, in an order
    that does not depend on the seed."""
    out = []
    sizes = np.exp(np.random.default_rng(count).uniform(math.log(lo), math.log(hi), count))
    for i, n in enumerate(sizes):
        s = seed * 1000003 + i
        if i % 2 == 0:
            side = int(math.ceil(math.sqrt(n)))
            out.append((side * side, *_torus(2, side, 0.5, s)))
        else:
            n = 1 << int(round(math.log2(n)))
            out.append((n, *_rmat(n, 8, s)))
    return out


def prepare(case, seed):
    path = case["path"]
    st = _State(case=case)
    if path == "batch":
        gs = _mixed(case["graphs"], case["lo"], case["hi"], seed)
        ns = torch.tensor([0] + [g[0] for g in gs], dtype=torch.int64)
        ms = torch.tensor([0] + [len(g[2]) for g in gs], dtype=torch.int64)
        p = graphgen.Packed(len(gs), torch.cumsum(ns, 0), torch.cumsum(ms, 0), torch.cat([g[1] for g in gs]),
                            torch.cat([g[2] for g in gs]), [])
        st["batch"] = scc.SccBatch(p)
        st["out"] = torch.empty(st["batch"].nv, dtype=torch.int32, device=DEV)
        return st
    if path == "serve":
        host = [(n, o.cpu().numpy(), t.cpu().numpy()) for n, o, t in
                _mixed(case["scc"] + 2, case["lo"], case["hi"], seed)]
        rng = np.random.default_rng(seed + 1)
        st["server"] = scc.SccServer()
        res = host[-2:]
        gids = [st["server"].add_graph(*g) for g in res]
        st["scc"] = [(g, np.zeros(g[0], np.int32)) for g in host[:-2]]
        st["reach"] = []
        for i in range(case["reach"]):
            n = res[i % 2][0]
            src = rng.integers(0, n, int(rng.integers(1, 65))).astype(np.int32)
            st["reach"].append((gids[i % 2], src, int(rng.integers(0, 2)), np.zeros(n, np.uint64)))
        return st
    n, off, adj = _graph(case, seed)
    if path == "scc":
        st.update(n=n, off=off, adj=adj, out=torch.empty(n, dtype=torch.int32, device=DEV))
    elif path == "scc_host":
        st.update(n=n, off=_pinned(off), adj=_pinned(adj), out=_pinned(torch.zeros(n, dtype=torch.int32)))
    else:
        st["handle"] = scc.SccGraph(n, off, adj)
        st["out"] = torch.empty(n, dtype=torch.int32, device=DEV)
        if path == "lelists":  # room for twice the entries expected of any graph, kept from call to call
            st["off"] = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
            st["entries"] = [torch.zeros(2 * _entries(n), dtype=torch.int32, device=DEV) for _ in range(2)]
        if path == "reach":
            st["src"] = torch.randint(n, (case["k"],), generator=_gen(seed + 1), device=DEV).to(torch.int32)
            st["masks"] = [torch.empty(n, dtype=torch.int64, device=DEV) for _ in range(2)]
    return st


def run(st):
    path = st["case"]["path"]
    if path in ("scc", "scc_host"):
        with scc.SccGraph(st["n"], st["off"], st["adj"]) as g:
            return g.labels(st["out"])
    if path == "reach":
        return [st["handle"].reach(st["src"], dir=d, out=st["masks"][d]) for d in range(2)]
    if path == "cc":
        scc.cc_run(st["handle"].h, st["out"])
        return st["out"]
    if path == "lelists":
        h = st["handle"].h
        total = scc.le_lists_run(h)
        scc.le_lists_get(h, st["out"], st["off"], *st["entries"], total)
        return [total, st["out"], st["off"], *st["entries"]]
    if path == "batch":
        return st["batch"].labels(st["out"])
    s = st["server"]
    ids = []
    reach = iter(st["reach"])
    every = max(1, len(st["reach"]) // max(1, len(st["scc"])))
    for (n, off, adj), lab in st["scc"]:
        ids.append(s.submit_scc(n, off, adj, lab))
        for _, (gid, src, d, out) in zip(range(every), reach):
            ids.append(s.submit_reach(gid, src, d, out))
    for gid, src, d, out in reach:
        ids.append(s.submit_reach(gid, src, d, out))
    for i in ids:
        if s.wait(i)[0] != 0:
            raise RuntimeError("a served request failed")
    return [lab for _, lab in st["scc"]] + [out for _, _, _, out in st["reach"]]


def work(case):
    """Bytes of one pass: the CSR (and, for a reachability call, the sources) read once, the results written once.
    There is no floating-point work."""
    path = case["path"]
    if path in ("batch", "serve"):
        count = case["graphs"] if path == "batch" else case["scc"]
        lo, hi = case["lo"], case["hi"]
        mean = (hi - lo) / math.log(hi / lo)
        nbytes = count * mean * (4 * 5 + 8)  # half the graphs have 2 arcs a vertex, half 8
        if path == "serve":
            nbytes += 2 * mean * 28 + case["reach"] * (mean * 8 + 130)
        return {"bytes": int(nbytes), "flops": 0}
    n, m = _n(case), _arcs(case)
    graph = 4 * (n + 1) + 4 * m
    if path == "reach":
        return {"bytes": 2 * (graph + 8 * n + 4 * case["k"]), "flops": 0}
    if path == "lelists":
        return {"bytes": graph + 4 * n + 8 * (n + 1) + 8 * _entries(n), "flops": 0}
    return {"bytes": graph + 4 * n, "flops": 0}


def _tarjan(n, off, adj):
    """Iterative Tarjan: the smallest id of each vertex's strongly connected component."""
    off, adj = off.tolist(), adj.tolist()
    num, low, lab = [0] * n, [0] * n, [-1] * n
    stack, count, pos = [], 0, off[:n]
    for root in range(n):
        if num[root]:
            continue
        count += 1
        num[root] = low[root] = count
        stack.append(root)
        call = [root]
        while call:
            v = call[-1]
            if pos[v] < off[v + 1]:
                w = adj[pos[v]]
                pos[v] += 1
                if not num[w]:
                    count += 1
                    num[w] = low[w] = count
                    stack.append(w)
                    call.append(w)
                elif lab[w] < 0:
                    low[v] = min(low[v], num[w])
                continue
            call.pop()
            if call:
                low[call[-1]] = min(low[call[-1]], low[v])
            if low[v] == num[v]:
                at = len(stack) - 1
                while stack[at] != v:
                    at -= 1
                least = min(stack[at:])
                for w in stack[at:]:
                    lab[w] = least
                del stack[at:]
    return torch.tensor(lab, dtype=torch.int64)


def exact(case, seed):
    """The result by a plain method where that is quick: Tarjan's for small graphs, a fixed point of the definition
    for components and reachability."""
    path = case["path"]
    if path in ("batch", "serve", "lelists") or (path.startswith("scc") and _n(case) + _arcs(case) > 300000):
        return None
    n, off, adj = _graph(case, seed)
    if path.startswith("scc"):
        return _tarjan(n, off, adj)
    src = torch.repeat_interleave(torch.arange(n, device=DEV), (off[1:] - off[:-1]).to(torch.int64))
    dst = adj.to(torch.int64)
    if path == "cc":
        lab = torch.arange(n, device=DEV)
        while True:
            low = lab.clone()
            low.scatter_reduce_(0, lab[src], lab[dst], "amin")
            low.scatter_reduce_(0, lab[dst], lab[src], "amin")
            low = low[low]
            low = torch.minimum(low[lab], low)
            if torch.equal(low, lab):
                return lab
            lab = low
    start = torch.randint(n, (case["k"],), generator=_gen(seed + 1), device=DEV)
    step = max(1, (1 << 28) // max(1, len(src)))  # sources searched together
    masks = []
    for a, b in ((src, dst), (dst, src)):
        mask = torch.zeros(n, dtype=torch.int64, device=DEV)
        for j in range(0, case["k"], step):
            some = start[j:j + step]
            bits = torch.arange(len(some), device=DEV)
            seen = torch.zeros((n, len(some)), dtype=torch.bool, device=DEV)
            seen[some, bits] = True
            have = -1
            while (now := int(seen.sum())) != have:
                have = now
                arc, bit = seen[a].nonzero(as_tuple=True)
                seen[b[arc], bit] = True
            mask |= (seen.to(torch.int64) << (bits + j)).sum(1)
        masks.append(mask)
    return masks
