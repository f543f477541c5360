"""GPU connected components where the passes of the union-find change over:
numbers of vertices at the edges of a thread's four and a block's 1024 walks,
one chain of every vertex in three numberings, rows at the edges of the pieces
of long rows outside the large tree, graphs without a large tree, and vertices
that only an arc into them, or out of them, ties to the large tree. Labels
against the oracle's union-find."""
import numpy as np
import pytest

import oracle
from paper_2303_04934_gb300 import graphgen as gg
from paper_2303_04934_gb300 import scc

from gpu_util import ensure_lib, make_graph

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _check(n, edges, name):
    g = gg.from_edges(n, edges, name=name)
    want, ncc = oracle.cc_labels(g.n, g.offsets, g.targets)
    out = np.empty(g.n, np.int32)
    with make_graph(g, on_device=False) as G:
        for _ in range(2):
            out.fill(-1)
            scc.cc_run(G.h, out)
            assert np.array_equal(out, want), name
        st = scc.cc_get_stats(G.h)
    assert st["components"] == ncc and ncc <= st["clusters"] <= n


def _path(n, order):
    p = np.arange(n)
    if order == "down":
        p = p[::-1]
    elif order == "mixed":
        p = np.random.default_rng(n).permutation(n)
    return np.stack([p[:-1], p[1:]], 1)


@pytest.mark.parametrize("order", ["up", "down", "mixed"])
@pytest.mark.parametrize("n", [2, 3, 4, 5, 1023, 1024, 1025, 1500007])
def test_one_chain(n, order):
    _check(n, _path(n, order), f"chain_{n}_{order}")


@pytest.mark.parametrize("deg", [31, 32, 33, 34, 1023, 1024, 1025, 3073, 40001])
@pytest.mark.parametrize("into", [False, True])
def test_long_rows_outside_the_large_tree(deg, into):
    """A large tree (a cycle of 2/3 of the vertices), a hub outside it whose row
    of deg arcs ends at leaves, and a second hub sharing only its last leaf."""
    big = 2 * (deg + 4)
    c = np.arange(big)
    hub, leaf = big, big + 2 + np.arange(deg)
    e = [np.stack([c, (c + 1) % big], 1)]
    star = np.stack([np.full(deg, hub), leaf], 1)
    e.append(star[:, ::-1] if into else star)
    e.append(np.array([[leaf[-1], hub + 1]] if into else [[hub + 1, leaf[-1]]]))
    _check(big + 2 + deg, np.concatenate(e), f"star_{deg}_{into}")


@pytest.mark.parametrize("size", [1, 2, 7, 40])
def test_no_large_tree(size):
    n = 4000 * size
    v = np.arange(n)
    e = np.stack([v, v + 1], 1)[(v + 1) % size != 0] if size > 1 else np.zeros((0, 2), np.int64)
    perm = np.random.default_rng(size).permutation(n)
    _check(n, perm[e], f"parts_{size}")


@pytest.mark.parametrize("into", [False, True])
def test_ties_beyond_the_sample(into):
    """Vertices tied to the large tree only by the last arc of a hub's long row,
    or by their own only arc, numbered below and above the hub."""
    k = 3000
    hub = k
    v = np.concatenate([np.arange(k), np.arange(k + 1, 2 * k)])
    tie = np.stack([np.full(len(v), hub), v], 1)
    ring = np.arange(2 * k, 4 * k)
    e = [np.stack([ring, np.roll(ring, 1)], 1), np.array([[hub, 2 * k], [2 * k + 5, hub]]),
         tie[:, ::-1] if into else tie]
    _check(4 * k, np.concatenate(e), f"ties_{into}")
