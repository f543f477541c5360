"""GPU parity of reach_multi's forms against the oracle: searches that only pull
and searches that mark (the latter on large or skewed graphs), rows at the bound
of the warp-wide loop, two mask words, and a graph large and skewed enough that
the hub's own two sets come first, with sources that reach the hub, that only
the hub reaches, that lie in its component and that are outside of both."""
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
    return gg.Graph(n, off, dst[order].astype(np.int32), name)


def _check(G, g, src):
    import torch
    toff, tadj = oracle.transpose(g.n, g.offsets, g.targets)
    k = len(src)
    for d in (0, 1):
        o, a = (g.offsets, g.targets) if d == 0 else (toff, tadj)
        words = [oracle.reach_mask(g.n, o, a, src[i:i + 64]) for i in range(0, k, 64)]
        if k <= 64:
            out = torch.full((g.n,), -1, dtype=torch.int64, device="cuda")
            scc.reach_multi(G.h, dev(src), k, d, out)
            assert np.array_equal(out.cpu().numpy().view(np.uint64), words[0]), (g.name, k, d)
        wide = torch.full((2 * g.n,), -1, dtype=torch.int64, device="cuda")
        scc.scc_debug_reach_multi_wide(G.h, dev(src), k, d, wide)
        got = wide.cpu().numpy().view(np.uint64)
        assert np.array_equal(got[0::2], words[0]), (g.name, k, d)
        assert np.array_equal(got[1::2], words[1] if k > 64 else np.zeros(g.n, np.uint64)), (g.name, k, d)


@pytest.mark.parametrize("make", [
    lambda: gg.torus(2, 5, 0.5, seed=1), lambda: gg.torus(2, 64, 0.5, seed=2), lambda: gg.torus(3, 60, 0.3, seed=3),
    lambda: gg.knn(33, 2, seed=4), lambda: gg.knn(200_000, 8, seed=5), lambda: gg.rmat(15, 8, seed=6),
    lambda: gg.rmat(18, 16, seed=7), lambda: gg.torus(3, 120, 0.3, seed=8)],
    ids=["t5", "t64", "t3_60", "knn33", "knn200k", "rmat15", "rmat18", "t3_120"])
def test_forms(make):
    g = make()
    rng = np.random.default_rng(g.n)
    with make_graph(g) as G:
        for k in (1, 64, 65, 128):
            _check(G, g, rng.integers(0, g.n, k).astype(np.int32))


@pytest.mark.parametrize("deg", [3, 4, 5, 64, 65, 200])
def test_rows_at_the_bounds_of_the_loops(deg):
    rng = np.random.default_rng(deg)
    n, k = 20000, 300
    src = np.concatenate([np.repeat(np.arange(k), deg), np.arange(k, n)])
    dst = np.concatenate([rng.integers(0, n, k * deg), (np.arange(k, n) * 7 + 3) % n])
    g = _csr(n, src, dst, f"rows{deg}")
    with make_graph(g) as G:
        _check(G, g, rng.integers(0, k, 40).astype(np.int32))


def test_hub_first():
    base = gg.rmat(21, 16, seed=0x4B, a=0.57)
    n0 = base.n
    src0 = np.repeat(np.arange(n0), np.diff(base.offsets.astype(np.int64)))
    big = int(np.argmax(np.diff(base.offsets.astype(np.int64))))
    # into the hub's component (chain n0.. -> hub), out of it, and apart from both
    e = [(n0, n0 + 1), (n0 + 1, big), (big, n0 + 2), (n0 + 2, n0 + 3), (n0 + 4, n0 + 5), (n0 + 5, n0 + 4), (n0, n0 + 6)]
    g = _csr(n0 + 7, np.concatenate([src0, [a for a, _ in e]]), np.concatenate([base.targets, [b for _, b in e]]), "hub")
    assert g.m > 1 << 24 and g.m >= 8 * g.n  # the sizes from which the hub comes first
    rng = np.random.default_rng(9)
    src = np.concatenate([np.arange(n0, n0 + 7), [big], rng.integers(0, n0, 56)]).astype(np.int32)
    with make_graph(g) as G:
        _check(G, g, src)
        _check(G, g, np.array([n0 + 4], np.int32))


@pytest.mark.parametrize("shift", [0, 1, 2])
def test_wide_masks_at_any_word(shift):
    """Two-word masks into a device buffer that starts `shift` words after a 16-byte boundary."""
    import torch
    g = gg.torus(2, 60, 0.5, seed=9)
    src = np.random.default_rng(3).integers(0, g.n, 100).astype(np.int32)
    want = np.zeros(2 * g.n, np.uint64)
    want[0::2] = oracle.reach_mask(g.n, g.offsets, g.targets, src[:64])
    want[1::2] = oracle.reach_mask(g.n, g.offsets, g.targets, src[64:])
    buf = torch.full((2 * g.n + 4,), -1, dtype=torch.int64, device="cuda")
    with make_graph(g) as G:
        scc.scc_debug_reach_multi_wide(G.h, src, 100, 0, buf[shift:shift + 2 * g.n])
        torch.cuda.synchronize()
    got = buf.cpu().numpy().view(np.uint64)
    assert np.array_equal(got[shift:shift + 2 * g.n], want)
    assert (got[:shift] == ~np.uint64(0)).all() and (got[shift + 2 * g.n:] == ~np.uint64(0)).all()
