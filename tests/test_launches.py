"""What a call queues, on a runtime that runs nothing (tests/launch_util.py)."""
import pytest

import paper_0912_0947_gb300 as S
from launch_util import Launches

COVER, STEGO, MSG, RES = 1 << 40, 2 << 40, 3 << 40, 4 << 40


@pytest.fixture(scope="module")
def L():
    return Launches()


@pytest.mark.parametrize("C", [512 * 512 * 3, 8192 * 8192 * 3, 20 << 30])
@pytest.mark.parametrize("at", [0, 5])
def test_header_extract_is_one_wave(L, C, at):
    """The length of a headed message is known on the device alone: with a buffer for
    the cover's whole capacity no more CTAs than are resident together, whose
    first loads are all that is read before the header."""
    cap = C // 8 - 4
    q = L.queued("stego_extract", STEGO + at, C, MSG, cap, 0, None, S.HEADER_BE32, RES, 8)
    assert len(q) == 1 and "extract" in q[0][0]
    assert 1 <= q[0][1] <= L.wave


def test_known_length_extract_is_dealt_in_order(L):
    """Without a header the CTAs are as many as the message needs."""
    C = 8192 * 8192 * 3
    q = L.queued("stego_extract", STEGO, C, MSG, C // 8, C // 8, None, 0, RES, 8)
    assert len(q) == 1
    name, grid, block, _ = q[0]
    assert "extract_once" in name and grid == -(-(C // 16) // (4 * block))
    q = L.queued("stego_extract", STEGO, C, MSG, C // 8, 100, None, 0, RES, 8)
    assert q[0][1] == 1
