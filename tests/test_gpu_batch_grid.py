"""Batches and served units whose graphs without hubs hold at least 2^17
vertices together: those run as one graph over the whole grid, the others a
block each. Labels equal the oracle's for every graph, with empty and one-vertex
graphs, self-loops, duplicates and graphs with hubs mixed in, for host and
device buffers, on replays, when nothing is left to the blocks, and when a
malformed request shares the unit."""
import numpy as np
import pytest

import oracle
from paper_2303_04934_gb300 import graphgen as gg
from paper_2303_04934_gb300 import scc

from gpu_util import ensure_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _mix():
    gs = [gg.torus(2, 40 + 13 * i, 0.5, seed=2000 + i) for i in range(24)]
    gs += [gg.rmat(12, 8, seed=2100), gg.from_edges(0, []), gg.from_edges(1, [(0, 0)]),
           gg.gnp(200, 0.02, seed=2101, allow_self=True), gg.knn(20000, 5, seed=2102), gg.torus(3, 30, 0.3, seed=2103),
           gg.rmat(10, 16, seed=2104), gg.from_edges(9, []),
           gg.from_edges(6, [(0, 1), (0, 1), (1, 0), (2, 2), (3, 4), (4, 5), (5, 3)])]
    return [gs[i] for i in np.random.default_rng(11).permutation(len(gs))]


def _check(p, labels):
    for g in range(p.G):
        h = p.graph(g)
        assert np.array_equal(p.labels_of(labels, g), oracle.scc_labels(h.n, h.offsets, h.targets)[0]), (g, p.names[g])


@pytest.mark.parametrize("host", [False, True])
def test_batch(host):
    import torch
    p = gg.pack(_mix())
    nv = int(p.vbase[-1])
    with scc.SccBatch(p) as B:
        for _ in range(2):
            out = np.full(nv, -5, np.int32) if host else torch.full((nv,), -5, dtype=torch.int32, device="cuda")
            scc.scc_batch_run(B.h, out)
            _check(p, out if host else out.cpu().numpy())
        scc.scc_batch_autotune(B.h, 2)  # tunes the graphs that the blocks take
        out = torch.full((nv,), -5, dtype=torch.int32, device="cuda")
        scc.scc_batch_run(B.h, out)
        _check(p, out.cpu().numpy())


def test_nothing_left_to_the_blocks():
    p = gg.pack([gg.torus(2, 300, 0.5, seed=2200 + i) for i in range(2)])
    with scc.SccBatch(p) as B:
        _check(p, B.labels().cpu().numpy())
        scc.scc_batch_autotune(B.h, 1)
        _check(p, B.labels().cpu().numpy())


@pytest.mark.parametrize("malformed", [False, True])
def test_served_unit(malformed):
    gs = _mix()
    with scc.SccServer() as srv:
        ids, outs = [], []
        for g in gs:
            out = np.full(max(g.n, 1), -5, np.int32)
            ids.append(srv.submit_scc(g.n, np.ascontiguousarray(g.offsets), np.ascontiguousarray(g.targets), out))
            outs.append(out)
        bad = None
        if malformed:
            bad = srv.submit_scc(3, np.array([0, 1, 2, 2], np.int32), np.array([0, 5], np.int32), np.zeros(3, np.int32))
        for g, i, out in zip(gs, ids, outs):
            assert srv.wait(i)[0] == scc.SCC_OK
            assert np.array_equal(out[:g.n], oracle.scc_labels(g.n, g.offsets, g.targets)[0]), g.name
        if bad is not None:
            assert srv.wait(bad)[0] == scc.SCC_ERR_INVALID_ARG


@pytest.mark.parametrize("copies", [1000, 1040])
def test_many_equal_graphs(copies):
    """Tori of 128^2 on either side of 2^24 vertices together, where the blocks take them over from the grid."""
    import torch
    g = gg.torus(2, 128, 0.5, seed=2300)
    p = gg.pack([g] * copies)
    with scc.SccBatch(p) as B:
        lab = B.labels().reshape(copies, g.n)
        assert torch.equal(lab, lab[:1].expand(copies, -1))
        assert np.array_equal(lab[0].cpu().numpy(), oracle.scc_labels(g.n, g.offsets, g.targets)[0])
