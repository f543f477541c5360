"""The symmetric CSR of the least-element lists has 32-bit offsets: a graph whose
arcs, taken both ways, are more than 2^31 - 1 is refused before anything is
built, and stays usable for the other calls."""
import pytest

from paper_2303_04934_gb300 import scc

from gpu_util import ensure_lib

pytestmark = pytest.mark.gpu


def test_too_many_arcs_for_the_symmetric_csr():
    import torch
    ensure_lib()
    n, deg = 1 << 20, 1032
    assert 2 * n * deg > 2**31 - 1
    off = torch.arange(n + 1, device="cuda", dtype=torch.int32) * deg
    adj = torch.empty((n, deg), device="cuda", dtype=torch.int32)
    j = torch.arange(1, deg + 1, device="cuda", dtype=torch.int32)
    for a in range(0, n, n // 8):
        v = torch.arange(a, a + n // 8, device="cuda", dtype=torch.int32)
        adj[a:a + n // 8] = (v[:, None] + j[None, :]) % n
    with scc.SccGraph(n, off, adj.reshape(-1)) as G:
        with pytest.raises(scc.SccError) as e:
            scc.le_lists_run(G.h)
        assert e.value.code == scc.SCC_ERR_CAPACITY
        out = torch.full((n,), -1, device="cuda", dtype=torch.int32)
        scc.cc_run(G.h, out)
        assert not bool(out.any())
