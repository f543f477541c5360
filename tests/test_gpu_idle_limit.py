"""Searches without a barrier on graphs that are one long chain: one warp works
while every other block waits. The wait's limit counts from the last time a
block found work, so a chain may be as long as it likes; results against the
oracle with a limit far below the time of the search."""
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


# a search that only pulls, and (above 7 arcs a thread of the chip) one that marks
@pytest.mark.parametrize("n, limit_ms", [(200_000, 4), (1_300_000, 40)])
@pytest.mark.parametrize("shuffled", [False, True])
def test_a_chain_longer_than_the_idle_limit(n, limit_ms, shuffled):
    import time

    import torch
    p = np.random.default_rng(n).permutation(n) if shuffled else np.arange(n)
    src, dst = p[:-1], p[1:]
    off = np.zeros(n + 1, np.int32)
    off[1:] = np.cumsum(np.bincount(src, minlength=n))
    g = gg.Graph(n, off, dst[np.argsort(src, kind="stable")].astype(np.int32), "chain")
    s = p[:1].astype(np.int32)
    out = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    with make_graph(g) as G:
        scc.scc_debug_idle_limit(G.h, limit_ms * 1_000_000)
        t = time.perf_counter()
        scc.reach_multi(G.h, dev(s), 1, 0, out)
        took = 1e3 * (time.perf_counter() - t)
        assert np.array_equal(out.cpu().numpy().view(np.uint64), oracle.reach_mask(n, g.offsets, g.targets, s))
        assert took > 2 * limit_ms  # else the limit was not put to the test
        scc.scc_debug_idle_limit(G.h, 0)
    with pytest.raises(scc.SccError):
        scc.scc_debug_idle_limit(None, 0)
