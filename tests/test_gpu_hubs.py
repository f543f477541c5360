"""Graphs of low mean degree with hubs by out- or by in-degree: a hub of either
direction keeps its graph from the searches that only pull, which would read its
row in every pass: reach_multi's, and the grid-wide ones of batches and served
units. Results against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2303_04934_gb300 import graphgen as gg
from paper_2303_04934_gb300 import scc

from gpu_util import dev, ensure_lib, make_graph

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _csr(n, src, dst, name):
    order = np.argsort(src, kind="stable")
    off = np.zeros(n + 1, np.int32)
    off[1:] = np.cumsum(np.bincount(src, minlength=n))
    return gg.Graph(n, off, np.asarray(dst)[order].astype(np.int32), name)


def _hub(side, deg, into, seed=5):
    """A lattice and a vertex on a cycle of three with `deg` arcs from (or to) the lattice and one back."""
    g = gg.torus(2, side, 0.5, seed=seed)
    src = np.repeat(np.arange(g.n), np.diff(g.offsets.astype(np.int64)))
    leaf = np.random.default_rng(seed).choice(g.n, deg, replace=False)
    hub = np.full(deg, g.n)
    a, b = (leaf, hub) if into else (hub, leaf)
    one = ([g.n], leaf[:1]) if into else (leaf[:1], [g.n])
    ring = np.array([g.n, g.n + 1, g.n + 2]), np.array([g.n + 1, g.n + 2, g.n])
    return _csr(g.n + 3, np.concatenate([src, a, one[0], ring[0]]), np.concatenate([g.targets, b, one[1], ring[1]]),
                f"hub{deg}_{'in' if into else 'out'}")


def check_reach(G, g, src):
    import torch
    toff, tadj = oracle.transpose(g.n, g.offsets, g.targets)
    for d in (0, 1):
        o, a = (g.offsets, g.targets) if d == 0 else (toff, tadj)
        words = [oracle.reach_mask(g.n, o, a, src[i:i + 64]) for i in range(0, len(src), 64)]
        if len(src) <= 64:
            out = torch.full((g.n,), -1, dtype=torch.int64, device="cuda")
            scc.reach_multi(G.h, dev(src), len(src), d, out)
            assert np.array_equal(out.cpu().numpy().view(np.uint64), words[0]), (g.name, len(src), d)
        else:
            wide = torch.full((2 * g.n,), -1, dtype=torch.int64, device="cuda")
            scc.scc_debug_reach_multi_wide(G.h, dev(src), len(src), d, wide)
            got = wide.cpu().numpy().view(np.uint64)
            assert np.array_equal(got[0::2], words[0]) and np.array_equal(got[1::2], words[1]), (g.name, len(src), d)


@pytest.mark.parametrize("into", [False, True])
def test_reach_multi_does_not_pull_a_hubs_row(into):
    g = _hub(300, 30000, into)
    rng = np.random.default_rng(1)
    with make_graph(g) as G:
        for k in (1, 40, 128):
            check_reach(G, g, np.concatenate([[g.n - 1], rng.integers(0, g.n, k - 1)]).astype(np.int32))
            assert scc.scc_debug_forms(G.h)[1] == 0
    plain = gg.torus(2, 300, 0.5, seed=5)
    with make_graph(plain) as G:
        check_reach(G, plain, rng.integers(0, plain.n, 7).astype(np.int32))
        assert scc.scc_debug_forms(G.h)[1] == scc.FORM_PULL


def _mix():
    return [gg.torus(2, 300, 0.5, seed=31), _hub(250, 40000, True), gg.torus(2, 310, 0.5, seed=32),
            _hub(200, 20000, False), gg.from_edges(0, []), gg.torus(3, 40, 0.3, seed=33)]


def test_batch_leaves_hubs_of_either_direction_to_the_blocks():
    p = gg.pack(_mix())
    with scc.SccBatch(p) as B:
        lab = B.labels().cpu().numpy()
        rec = scc.scc_debug_batch_times(B.h, p.G)
    for g in range(p.G):
        h = p.graph(g)
        assert np.array_equal(p.labels_of(lab, g), oracle.scc_labels(h.n, h.offsets, h.targets)[0]), p.names[g]
        if h.n:  # the grid's graphs share the start of their launch in every field
            assert (rec[g, 1] == rec[g, 0]) == (g not in (1, 3)), p.names[g]


def test_served_unit_with_an_in_hub():
    gs = _mix()
    with scc.SccServer() as srv:
        outs = [np.full(max(g.n, 1), -5, np.int32) for g in gs]
        ids = [srv.submit_scc(g.n, np.ascontiguousarray(g.offsets), np.ascontiguousarray(g.targets), o)
               for g, o in zip(gs, outs)]
        for g, i, o in zip(gs, ids, outs):
            assert srv.wait(i)[0] == scc.SCC_OK
            assert np.array_equal(o[:g.n], oracle.scc_labels(g.n, g.offsets, g.targets)[0]), g.name
