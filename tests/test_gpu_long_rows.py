"""Rows far longer than the mean in the searches: a vertex's row is never left to
one thread, nor a hub's to one warp. Results against the oracle, and the time of
a hub's trimming and searches against what one thread needs for its row (90 ns
an arc, two dependent loads)."""
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


def _stars(n, k, two_way=True, into=False):
    """k disjoint stars on n vertices, centres 0 .. k - 1; one-way stars have a centre on a cycle of two."""
    leaf = np.arange(2 * k, n)
    c = leaf % k
    ring = np.arange(k)
    a, b = (leaf, c) if into else (c, leaf)
    src, dst = [a, ring, k + ring], [b, k + ring, ring]
    if two_way:
        src.append(b)
        dst.append(a)
    p = np.random.default_rng(k).permutation(n)
    return _csr(n, p[np.concatenate(src)], p[np.concatenate(dst)], f"stars{k}_{two_way}_{into}")


# rows just below, at and above the bound from which they are shared (4096 arcs), pieces (512) and their remainders,
# more shared rows than there are slots (24), and one row of everything
@pytest.mark.parametrize("n, k", [(2050, 1), (4096, 1), (4097, 1), (4098, 1), (4099, 1), (4100, 1), (4700, 1), (10000, 2),
                                  (40000, 7), (300_000, 64), (900_000, 200), (1_000_000, 3), (3_000_000, 1)])
@pytest.mark.parametrize("two_way, into", [(True, False), (False, False), (False, True)])
def test_stars(n, k, two_way, into):
    g = _stars(n, k, two_way, into)
    rng = np.random.default_rng(n)
    want, _ = oracle.scc_labels(g.n, g.offsets, g.targets)
    with make_graph(g) as G:
        for _ in range(2):
            assert np.array_equal(labels_of(G), want), g.name
        for ns in (1, 64, 128):
            check_reach(G, g, rng.integers(0, n, ns).astype(np.int32))


def _clusters(n, k, extra, seed):
    """k clusters joined by mutual arcs (each one node when contracted) with one-way arcs between vertices of any."""
    rng = np.random.default_rng(seed)
    of = np.sort(rng.integers(0, k, n) ** 2 // k)  # sizes from large to none
    i = np.arange(n)
    first = np.searchsorted(of, of)
    j = first + rng.integers(0, 1 << 30, n) % np.maximum(i - first, 1)
    m = i != first
    x = rng.integers(0, n, extra)
    y = x + (rng.random(extra) * (n - x)).astype(np.int64)
    keep = x != y
    p = rng.permutation(n)
    src, dst = np.concatenate([i[m], j[m], x[keep]]), np.concatenate([j[m], i[m], y[keep]])
    return _csr(n, p[src], p[dst], f"clusters{k}")


@pytest.mark.parametrize("n, k, extra", [(70_000, 3, 60_000), (300_000, 40, 300_000), (1_500_000, 1000, 3_000_000)])
def test_giant_nodes_of_a_contracted_graph(n, k, extra):
    g = _clusters(n, k, extra, seed=k)
    want, _ = oracle.scc_labels(g.n, g.offsets, g.targets)
    with make_graph(g) as G:
        for _ in range(2):
            assert np.array_equal(labels_of(G), want), g.name
        assert scc.scc_debug_forms(G.h)[0] == scc.FORM_CONTRACTED


@pytest.mark.parametrize("deg", [62, 63, 64, 65, 66, 128, 300, 1000])
@pytest.mark.parametrize("into", [False, True])
def test_trimming_around_the_first_arcs_of_a_row(deg, into):
    """Vertices on cycles of two whose rows (long in either direction) begin with trimmed leaves, with the other vertex
    of the cycle before, at and past the 64 arcs that a thread looks at, and chains of two that do get trimmed; the
    first SCC is a dense ring."""
    ring, k = 20000, 40
    i = np.arange(ring)
    src, dst = [i, i], [(i + 1) % ring, (i + 7) % ring]
    at = ring
    for j in range(k):
        a, b = at, at + 1
        leaf = np.arange(at + 2, at + 2 + deg)
        pos = (j * 7) % (deg + 1)
        row = np.insert(leaf, pos, b)  # b among the leaves
        src += [np.full(len(row), a), [b]] if not into else [row, [a]]
        dst += [row, [a]] if not into else [np.full(len(row), a), [b]]
        if j % 3 == 0:  # without the way back: a chain
            src.pop()
            dst.pop()
        at += 2 + deg
    g = _csr(at, np.concatenate([np.asarray(x) for x in src]), np.concatenate([np.asarray(x) for x in dst]), "first_arcs")
    want, _ = oracle.scc_labels(g.n, g.offsets, g.targets)
    with make_graph(g) as G:
        assert np.array_equal(labels_of(G), want)
