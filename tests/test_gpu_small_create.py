"""Graphs at the edges of the sizes that one block takes in: the transposed rows
and the labels against the oracle, long rows, self-loops (which take the general
path), and inputs that must be refused, from device and host arrays."""
import numpy as np
import pytest

import oracle
from paper_2303_04934_gb300 import graphgen as gg
from paper_2303_04934_gb300 import scc

from gpu_util import dev, ensure_lib, make_graph

pytestmark = pytest.mark.gpu

N, M = 8192, 65536  # the largest graph of the one-block path


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _graph(n, m, seed, hub=False, loops=0):
    rng = np.random.default_rng(seed)
    u, w = rng.integers(0, n, m), rng.integers(0, max(n - 1, 1), m)
    if hub:
        u[: m // 2] = n // 3
        w[m // 2:] = n // 5
    w = (u + 1 + (w % max(n - 1, 1))) % n  # no self-loops
    if loops:
        w[:loops] = u[:loops]
    return gg.from_edges(n, np.stack([u, w], 1), name=f"g{n}_{m}")


def _check(g, on_device):
    with make_graph(g, on_device=on_device) as G:
        lab = np.empty(g.n, np.int32)
        scc.scc_run(G.h, lab)
        assert np.array_equal(lab, oracle.scc_labels(g.n, g.offsets, g.targets)[0])
        toff, tadj = oracle.transpose(g.n, g.offsets, g.targets)
        src = np.arange(min(g.n, 64), dtype=np.int32)
        out = np.empty(g.n, np.uint64)
        scc.reach_multi(G.h, src, len(src), 1, out)  # searches the transposed rows
        assert np.array_equal(out, oracle.reach_mask(g.n, toff, tadj, src))


@pytest.mark.parametrize("on_device", [True, False])
@pytest.mark.parametrize("n,m,hub", [(2, 1, False), (31, 33, False), (1023, 1025, True), (1025, 4000, True),
                                     (N - 1, M - 1, False), (N, M, True), (N + 1, M, False), (N, M + 1, True)])
def test_sizes(n, m, hub, on_device):
    _check(_graph(n, m, n + m, hub), on_device)


@pytest.mark.parametrize("loops", [1, 500])
def test_self_loops(loops):
    for on_device in (True, False):
        _check(_graph(1000, 3000, loops, False, loops), on_device)


def test_refused_inputs():
    g = _graph(300, 900, 1)
    for what in range(6):
        off, adj = g.offsets.astype(np.int32).copy(), g.targets.astype(np.int32).copy()
        if what == 0:
            off[0] = 1
        elif what == 1:
            off[-1] -= 1
        elif what == 2:
            off[100], off[101] = off[101] + 1, off[100]
        elif what == 3:
            off[7] = -5
        elif what == 4:
            adj[-1] = 300
        else:
            adj[13] = -1
        for a, b in ((off, adj), (dev(off), dev(adj))):
            with pytest.raises(scc.SccError):
                scc.scc_graph_create(300, 900, a, b)
