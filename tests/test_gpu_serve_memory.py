"""Admission under a tight memory cap: a request is admitted for what it needs
alone; what running a unit's graphs together over the whole GPU takes is used
only if there is room. Labels against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2303_04934_gb300 import graphgen as gg
from paper_2303_04934_gb300 import scc

from gpu_util import ensure_lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("left_mb", [5, 200])
def test_admission_does_not_count_the_units_temporaries(left_mb):
    """Room for three lattices of 65 k vertices (1.3 MB each), and with 200 MB also for their temporaries."""
    ensure_lib()
    gs = [gg.torus(2, 256, 0.5, seed=3000 + i) for i in range(3)]
    want = [oracle.scc_labels(g.n, g.offsets, g.targets)[0] for g in gs]
    need = [8 * (g.n + 1) + 4 * g.m + 4 * g.n + 4096 for g in gs]
    assert sum(need) < 5e6 < min(82 * g.n + 33 * g.m for g in gs)
    cfg = scc.scc_server_config_default()
    cfg.mem_cap_bytes = 4_000_000_000
    cfg.batch_vertices = 65536
    cfg.batch_min = 1
    with scc.SccServer(cfg) as srv:
        # a resident graph takes the rest: 18 bytes an arc and 360 a vertex and 64 MiB
        free = cfg.mem_cap_bytes - srv.stats()["mem_in_use"] - left_mb * 1_000_000
        n = (free - (64 << 20)) // 378
        i = np.arange(n + 1, dtype=np.int32)
        srv.add_graph(int(n), i, (i[:-1] + 1) % np.int32(n))
        before = srv.stats()["mem_in_use"]
        assert left_mb * 1e6 <= cfg.mem_cap_bytes - before < left_mb * 1e6 + 1000
        for _ in range(3):
            outs = [np.full(g.n, -5, np.int32) for g in gs]
            ids = [srv.submit_scc(g.n, g.offsets, g.targets, o) for g, o in zip(gs, outs)]
            for i, o, w in zip(ids, outs, want):
                assert srv.wait(i)[0] == scc.SCC_OK
                assert np.array_equal(o, w)
        srv.drain()
        st = srv.stats()
        assert st["failed"] == 0 and st["mem_peak"] <= cfg.mem_cap_bytes
        assert st["mem_in_use"] == before
