"""GPU parity of signature propagation (the whole SCC of a graph without hubs,
and the batches after the first SCC of one with hubs) against the oracle, where
its forms meet: bitmap words that are not full, one word a warp and several,
searches that only pull and searches that mark (the latter from about 7 arcs a
thread), rows at the bound of the warp-wide loop, long cycles, the head start
of a million vertices and more, and a hub in either direction."""
import numpy as np
import pytest

import oracle
from paper_2303_04934_gb300 import graphgen as gg
from paper_2303_04934_gb300 import scc

from gpu_util import config, ensure_lib, labels_of, make_graph

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _csr(n, src, dst, name):
    order = np.argsort(src, kind="stable")
    off = np.zeros(n + 1, np.int32)
    off[1:] = np.cumsum(np.bincount(src, minlength=n))
    return gg.Graph(n, off, dst[order].astype(np.int32), name)


def _cycles(lengths, seed):
    """Disjoint directed cycles under shuffled ids."""
    n = int(sum(lengths))
    p = np.random.default_rng(seed).permutation(n)
    src, dst, at = [], [], 0
    for k in lengths:
        i = np.arange(k)
        src.append(at + i)
        dst.append(at + (i + 1) % k)
        at += k
    return _csr(n, p[np.concatenate(src)], p[np.concatenate(dst)], f"cycles{len(lengths)}_{n}")


def _rows(deg, k, seed):
    """k vertices of `deg` out-arcs each into a ring of 16 * k vertices, and back."""
    rng = np.random.default_rng(seed)
    ring = 16 * k
    src = [k + np.arange(ring), np.repeat(np.arange(k), deg), k + rng.integers(0, ring, 2 * k)]
    dst = [k + (np.arange(ring) + 1) % ring, k + rng.integers(0, ring, k * deg), rng.integers(0, k, 2 * k)]
    return _csr(k + ring, np.concatenate(src), np.concatenate(dst), f"rows{deg}")


def _check(g, cfg=None):
    want, _ = oracle.scc_labels(g.n, g.offsets, g.targets)
    with make_graph(g, cfg) as G:
        for _ in range(2):  # the state of one run must not reach the next
            assert np.array_equal(labels_of(G), want), g.name
        st = G.stats()
    trimmed = oracle.trim(g.n, g.offsets, g.targets)
    assert st["n_trimmed"] == int(trimmed.sum())
    return st


@pytest.mark.parametrize("side", [5, 6, 8, 16, 17, 63, 64, 181, 393, 394, 395, 530, 800])
def test_lattices_across_words_and_forms(side):
    for p in (0.5, 0.65):
        _check(gg.torus(2, side, p, seed=side))


@pytest.mark.parametrize("n, k", [(33, 2), (1000, 3), (160_000, 7), (300_000, 6), (700_000, 3)])
def test_knn_graphs(n, k):
    _check(gg.knn(n, k, seed=n))


@pytest.mark.parametrize("deg", [3, 4, 5, 8, 63, 64, 65, 97, 130])
def test_rows_at_the_bounds_of_the_loops(deg):
    _check(_rows(deg, 400, seed=deg))
    _check(_rows(deg, 20000, seed=deg + 1))


def test_long_cycles():
    _check(_cycles([100_000], 1))
    _check(_cycles([1, 2, 3, 31, 32, 33, 5000, 70_000], 2))
    _check(_cycles([1_200_000, 300_000, 7], 3))


@pytest.mark.parametrize("make", [
    lambda: gg.torus(2, 1100, 0.6, seed=11),   # a giant SCC, flooded by the head start
    lambda: gg.torus(2, 1100, 0.45, seed=12),  # none: the head start ends early
    lambda: gg.torus(3, 110, 0.3, seed=13),
    lambda: gg.paper_lattice(1300, 1200, 1, seed=14),
], ids=["giant", "none", "torus3", "rec_prime"])
def test_head_start(make):
    for seed in (0x5CC00, 77):
        _check(make(), config(seed=seed))


@pytest.mark.parametrize("into", [False, True])
def test_hub_and_the_batches_after_its_scc(into):
    """A hub (in one direction only) beside a lattice: the first SCC by its own
    search, the lattice's classes by propagation."""
    g = gg.torus(2, 300, 0.5, seed=21)
    src = np.repeat(np.arange(g.n), np.diff(g.offsets.astype(np.int64)))
    leaf = np.random.default_rng(5).choice(g.n, 5000, replace=False)
    hub = np.full(5000, g.n)
    a, b = (leaf, hub) if into else (hub, leaf)
    ring = np.array([g.n, g.n + 1, g.n + 2]), np.array([g.n + 1, g.n + 2, g.n])
    _check(_csr(g.n + 3, np.concatenate([src, a, ring[0]]), np.concatenate([g.targets, b, ring[1]]), "hub"))


def _mutual(n, extra, share, seed):
    """A ring of random blocks of mutual arcs (chains and cliques of ids far apart
    and close by) with one-way arcs between them."""
    rng = np.random.default_rng(seed)
    a = rng.integers(0, n, int(share * n))
    b = np.where(rng.random(len(a)) < 0.5, (a + 1) % n, rng.integers(0, n, len(a)))
    x, y = rng.integers(0, n, extra), rng.integers(0, n, extra)
    keep, keep2 = a != b, x != y
    a, b, x, y = a[keep], b[keep], x[keep2], y[keep2]
    return _csr(n, np.concatenate([a, b, x]), np.concatenate([b, a, y]), f"mutual{n}_{share}")


@pytest.mark.parametrize("n", [65535, 65536, 65537, 70001, 400_000, 1_300_000])
@pytest.mark.parametrize("share", [0.3, 0.6, 1.0])
def test_contraction_along_mutual_arcs(n, share):
    """Graphs around the size from which mutual arcs are contracted, with too few
    of them, enough, and so many that a giant node remains."""
    _check(_mutual(n, n, share, seed=n + int(10 * share)))


def test_contraction_extremes():
    n = 100_000
    i = np.arange(n)
    _check(_csr(n, np.concatenate([i, (i + 1) % n]), np.concatenate([(i + 1) % n, i]), "two_way_ring"))  # one node
    star = np.arange(1, 60)  # many small stars: every node's rows meet in its centre
    c = np.repeat(np.arange(0, n, 60)[:-1], 59)
    leaf = c + np.tile(star, len(c) // 59)
    _check(_csr(n, np.concatenate([c, leaf, c[:-60]]), np.concatenate([leaf, c, c[60:]]), "stars"))
