"""GPU least-element lists where the walk of a level changes over: rows at the
edges of the pieces in which long rows are queued, a queue of pieces that is too
short for a level (rows walked whole), frontiers at the edges of a warp's 32
items and of the grid, and a log and a table that must grow in the middle of
such a level. Lists against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2303_04934_gb300 import graphgen as gg
from paper_2303_04934_gb300 import scc

from gpu_util import ensure_lib, make_graph
from test_gpu_lelists import _check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _stars(hubs, deg):
    """`hubs` hubs of deg leaves each (every leaf of all the hubs' rows is shared
    by the next hub), the hubs in a ring."""
    h = np.arange(hubs)
    leaf = hubs + np.arange(hubs * deg).reshape(hubs, deg)
    e = [np.stack([np.repeat(h, deg), leaf.ravel()], 1), np.stack([h, (h + 1) % hubs], 1),
         np.stack([leaf.ravel(), np.repeat((h + 1) % hubs, deg)], 1)]
    return hubs + hubs * deg, np.concatenate(e)


@pytest.mark.parametrize("small", [False, True])
@pytest.mark.parametrize("hubs,deg", [(1, 253), (1, 254), (1, 255), (1, 256), (2, 126), (2, 127), (3, 300), (40, 129),
                                      (6, 2000), (1, 70000)])
def test_long_rows(hubs, deg, small):
    n, e = _stars(hubs, deg)
    _check(gg.from_edges(n, e, name=f"stars_{hubs}_{deg}"), small=small)


@pytest.mark.parametrize("n", [31, 32, 33, 4863, 4865, 20000])
def test_wide_frontiers(n):
    """Many short rows at once: a path of cliques of two, numbered at random."""
    rng = np.random.default_rng(n)
    p = rng.permutation(n)
    e = np.concatenate([np.stack([p[:-1], p[1:]], 1)[::2], rng.integers(0, n, (n // 2, 2))])
    _check(gg.from_edges(n, e, name=f"wide_{n}"), small=n > 1000)


def test_queue_of_pieces_too_short():
    """1000 vertices of 300 arcs each (two pieces a row), all in one level's
    frontier, with a table of 2048 slots, whose queue holds 1536 pieces."""
    a, b = np.meshgrid(np.arange(1000), 1000 + np.arange(300), indexing="ij")
    g = gg.from_edges(1300, np.stack([a.ravel(), b.ravel()], 1), name="bipartite")
    _check(g, small=True)
    _check(g)
