"""A server's resident graphs (add_graph) live by its own streams, also when no query ever ran on them."""
import pytest

from paper_2303_04934_gb300 import graphgen as gg
from paper_2303_04934_gb300 import scc

from gpu_util import ensure_lib

pytestmark = pytest.mark.gpu


def test_resident_graphs_that_were_never_queried():
    """Removed, or still there when the server ends."""
    ensure_lib()
    g = gg.torus(2, 40, 0.5, seed=3100)
    for _ in range(3):
        with scc.SccServer() as srv:
            ids = [srv.add_graph(g.n, g.offsets, g.targets) for _ in range(3)]
            srv.remove_graph(ids[1])
            assert srv.stats()["resident_graphs"] == 2
