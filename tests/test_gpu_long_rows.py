"""Rows far longer than the mean in the searches: a vertex's row is never left to
one thread. Results against the oracle, and the time of the searches against
what one thread needs for such a row (90 ns an arc, two dependent loads)."""
import numpy as np
import pytest

import oracle
from paper_2303_04934_gb300 import graphgen as gg

from gpu_util import ensure_lib, labels_of, make_graph

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _csr(n, src, dst, name):
    order = np.argsort(src, kind="stable")
    off = np.zeros(n + 1, np.int32)
    off[1:] = np.cumsum(np.bincount(src, minlength=n))
    return gg.Graph(n, off, np.asarray(dst)[order].astype(np.int32), name)


def _late_hub(ring, leaves, into):
    """A dense ring, whose SCC comes first, and a vertex on a cycle of two whose
    row of `leaves` trimmed vertices has no other neighbour in its class."""
    i, h = np.arange(ring), ring
    leaf = np.arange(ring + 2, ring + 2 + leaves)
    hub = np.full(leaves, h)
    a, b = (leaf, hub) if into else (hub, leaf)
    return _csr(ring + 2 + leaves, np.concatenate([i, i, [h, h + 1], a]),
                np.concatenate([(i + 1) % ring, (i + 7) % ring, [h + 1, h], b]), f"late_hub_{'in' if into else 'out'}")


@pytest.mark.parametrize("into", [False, True])
def test_trimming_of_a_hub_whose_neighbours_are_finished(into):
    leaves = 1 << 20
    g = _late_hub(60000, leaves, into)
    want, _ = oracle.scc_labels(g.n, g.offsets, g.targets)
    with make_graph(g) as G:
        for _ in range(2):
            assert np.array_equal(labels_of(G), want)
        st = G.stats()
    assert st["n_trimmed"] == leaves and st["first_scc_size"] == 60000
    assert st["ms_multi_search"] * 1e6 < 40 * leaves
