"""The forms of signature propagation on graphs that take them for certain (the
form is read back): the head start of a million vertices and more without mutual
arcs, with a giant SCC, with none and with one beside others; searches that pull
and that mark on either side of 7 arcs a thread of the launch; contracted
graphs, one of them to a single node. Labels against the oracle, and the batches
that a run reports are those that ran."""
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
    return gg.Graph(n, off, np.asarray(dst)[order].astype(np.int32), name)


def _one_way(side, p, seed):
    """Torus whose arcs go right and down, each there with probability p: no two are mutual."""
    n = side * side
    v = np.arange(n)
    x, y = v % side, v // side
    to = np.stack([y * side + (x + 1) % side, (y + 1) % side * side + x], 1)
    there = np.random.default_rng(seed).random((n, 2)) < p
    return _csr(n, np.repeat(v, 2).reshape(n, 2)[there], to[there], f"one_way{side}_{p}")


def _spread(n, deg, seed):
    """Every vertex has arcs to `deg` others far ahead of it, in a ring: none mutual, no hubs."""
    v = np.arange(n)
    step = np.unique(np.random.default_rng(seed).integers(1, n // 3, 4 * deg))[:deg]
    assert len(step) == deg
    return _csr(n, np.repeat(v, deg), (v[:, None] + step[None, :]).reshape(-1) % n, f"spread{n}_{deg}")


def _check(g, form, seeds=(0x5CC00,)):
    want, _ = oracle.scc_labels(g.n, g.offsets, g.targets)
    for seed in seeds:
        with make_graph(g, config(seed=seed)) as G:
            for _ in range(2):
                assert np.array_equal(labels_of(G), want), g.name
            assert scc.scc_debug_forms(G.h)[0] == form, g.name
            st = G.stats()
    return st, want


@pytest.mark.parametrize("make, giant", [
    (lambda: _one_way(1100, 0.9, 1), True), (lambda: _one_way(1100, 0.5, 2), False),
    (lambda: gg.torus(3, 110, 0.3, seed=3), True), (lambda: gg.torus(3, 110, 0.2, seed=4), False)],
    ids=["one_way_giant", "one_way_none", "torus3_giant", "torus3_none"])
def test_head_start(make, giant):
    g = make()
    _, want = _check(g, scc.FORM_HEAD_START, seeds=(0x5CC00, 77))
    assert (np.bincount(want).max() > g.n // 4) == giant


# a launch has a thread a vertex, at most four blocks of 256 an SM: 155,648 on 152 SMs
@pytest.mark.parametrize("make, form", [
    (lambda: _spread(50_000, 6, 5), scc.FORM_PULL), (lambda: _spread(50_000, 8 - 1, 6), scc.FORM_PULL),
    (lambda: _spread(200_000, 5, 7), scc.FORM_PULL), (lambda: _spread(200_000, 6, 8), 0),
    (lambda: _one_way(720, 1.0, 9), scc.FORM_PULL), (lambda: _one_way(770, 1.0, 10), 0),
    (lambda: _one_way(760, 0.6, 11), scc.FORM_PULL)],
    ids=["50k_6", "50k_7", "200k_5", "200k_6", "one_way720", "one_way770", "one_way760_sparse"])
def test_pulling_and_marking(make, form):
    _check(make(), form)


def test_batches_are_those_that_ran():
    n = 100_000
    i = np.arange(n)
    ring = _csr(n, np.concatenate([i, (i + 1) % n]), np.concatenate([(i + 1) % n, i]), "two_way_ring")
    st, _ = _check(ring, scc.FORM_CONTRACTED | scc.FORM_PULL)  # one node, which is trimmed
    assert st["batches"] == 0 and st["first_scc_size"] == n
    st, _ = _check(_spread(30_000, 3, 12), scc.FORM_PULL)
    assert st["batches"] == 1
