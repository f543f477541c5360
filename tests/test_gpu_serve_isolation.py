"""A malformed request leaves the other requests of its unit on the route they
would take without it: the groups that run over the whole GPU end before it and
begin after it. Seen in the launches of a unit, held together by a larger
request that is served first."""
import numpy as np
import pytest

import oracle
from paper_2303_04934_gb300 import graphgen as gg
from paper_2303_04934_gb300 import scc

from gpu_util import ensure_lib

pytestmark = pytest.mark.gpu

BAD = (3, np.array([0, 1, 2, 2], np.int32), np.array([0, 5], np.int32))


def _unit(srv, first, gs, bad_at):
    """Kernel launches and statuses of `first` alone and then the others as one unit; None if they were not one."""
    before, st0 = scc.scc_debug_launch_count(), srv.stats()
    outs = [np.full(g.n, -5, np.int32) for g in [first] + gs]
    ids = [srv.submit_scc(first.n, first.offsets, first.targets, outs[0])]
    bads = []
    for k, g in enumerate(gs):
        if k in bad_at:
            bads.append(srv.submit_scc(BAD[0], BAD[1], BAD[2], np.zeros(3, np.int32)))
        ids.append(srv.submit_scc(g.n, g.offsets, g.targets, outs[k + 1]))
    status = [srv.wait(i)[0] for i in ids + bads]
    assert status == [scc.SCC_OK] * len(ids) + [scc.SCC_ERR_INVALID_ARG] * len(bads)
    st = srv.stats()
    if st["batched_launches"] - st0["batched_launches"] != 1 or st["plain_scc"] - st0["plain_scc"] != 1:
        return None, outs[1:]
    return scc.scc_debug_launch_count() - before, outs[1:]


def test_a_malformed_request_does_not_change_the_others_route():
    ensure_lib()
    first = gg.rmat(20, 8, seed=41)  # too large for a unit: the others gather behind it
    gs = [gg.torus(2, 250 + i, 0.5, seed=4000 + i) for i in range(6)]
    want = [oracle.scc_labels(g.n, g.offsets, g.targets)[0] for g in gs]
    with scc.SccServer() as srv:
        count = {}
        for bad_at in ((), (3,), (0, 3)):
            for _ in range(20):
                launches, outs = _unit(srv, first, gs, bad_at)
                for o, w in zip(outs, want):
                    assert np.array_equal(o, w)
                if launches is not None:
                    count[bad_at] = launches
                    break
        assert set(count) == {(), (3,), (0, 3)}
        # the two halves hold 2^17 vertices each: two groups where there was one
        assert count[(3,)] > count[()] and count[(0, 3)] == count[(3,)]
