"""The loop that walks a row's arcs (host only): every arc of the row once, none
outside it, also where the row ends at the largest arc count a graph may have
(2^31 - 1), where a signed place would wrap below the row's end."""
import pytest

from paper_2303_04934_gb300 import scc

TOP = 2**31 - 1


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2303_04934_gb300 import build
    build.build()


@pytest.mark.parametrize("lanes", [1, 32])
@pytest.mark.parametrize("end", [0, 1, 1000, TOP - 128, TOP - 1, TOP])
@pytest.mark.parametrize("length", [0, 1, 2, 3, 4, 5, 31, 64, 65, 127, 128, 129, 1000])
def test_every_arc_once(lanes, end, length):
    beg = max(0, end - length)
    length = end - beg
    seen = 0
    for lane in range(lanes):
        steps, places, first, last = scc.scc_debug_row_steps(beg, end, lane, lanes)
        assert steps == -(-length // (4 * lanes))
        assert places == len(range(beg + lane, end, lanes))
        if places:
            assert first == beg + lane and last == beg + lane + (places - 1) * lanes < end
        seen += places
    assert seen == length
