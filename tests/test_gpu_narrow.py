"""Marking searches whose waves are a few vertices wide, which the warp that raised
them relaxes itself, up to 32 of them and 32 times in a row: layers of widths
around that bound, longer and shorter than that many hops, and a hub among them
whose row is left to its owner. reach_multi and SCC against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2303_04934_gb300 import graphgen as gg
from paper_2303_04934_gb300 import scc

from gpu_util import ensure_lib, labels_of, make_graph
from test_gpu_hubs import check_reach

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _layers(width, depth, hub, closed, seed):
    """`depth` layers of `width` vertices, each with arcs to two of the next one, under shuffled ids; every fifth layer
    also points at a hub of `hub` leaves (which keeps the graph from the pulling search); closed: the last layer
    points back at the first."""
    rng = np.random.default_rng(seed)
    i = np.arange(width * depth)
    lay, x = i // width, i % width
    n = width * depth + 1 + hub
    h = width * depth
    src, dst = [], []
    for step in (0, 1):
        to = (lay + 1) % depth * width + (x + step) % width
        keep = np.ones(len(i), bool) if closed else lay + 1 < depth
        src.append(i[keep])
        dst.append(to[keep])
    some = i[(lay % 5 == 0) & (x == 0)]
    src += [some, np.full(hub, h)]
    dst += [np.full(len(some), h), h + 1 + np.arange(hub)]
    p = rng.permutation(n)
    s, d = p[np.concatenate(src)], p[np.concatenate(dst)]
    order = np.argsort(s, kind="stable")
    off = np.zeros(n + 1, np.int32)
    off[1:] = np.cumsum(np.bincount(s, minlength=n))
    return gg.Graph(n, off, d[order].astype(np.int32), f"layers{width}x{depth}"), p


@pytest.mark.parametrize("width", [1, 2, 16, 31, 32, 33, 64, 65])
@pytest.mark.parametrize("depth", [3, 31, 33, 400])
def test_layers(width, depth):
    for hub, closed in ((70, False), (3000, True)):
        g, p = _layers(width, depth, hub, closed, seed=width * depth)
        rng = np.random.default_rng(depth)
        with make_graph(g) as G:
            assert np.array_equal(labels_of(G), oracle.scc_labels(g.n, g.offsets, g.targets)[0])
            for k in (1, 7, 64, 128):
                src = np.concatenate([p[:1], rng.integers(0, g.n, k - 1)]).astype(np.int32)
                check_reach(G, g, src)
            assert scc.scc_debug_forms(G.h)[1] == 0  # the searches mark
