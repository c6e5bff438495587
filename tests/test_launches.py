"""What a call queues, on a runtime that runs nothing (tests/launch_util.py)."""
import ctypes

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


CALLS = {
    "one bit": (8192 * 64, 0, 0, 0, None),
    "one bit, same misalignment": (8192 * 64, 3, 3, 0, None),
    "one bit, other misalignment": (8192 * 64, 3, 0, 0, None),
    "one bit, a few bytes": (40, 3, 0, 0, None),
    "two bits": (8192 * 64, 0, 0, S.BITS(2), None),
    "two bits, odd": (8192 * 64, 3, 5, S.BITS(2), None),
    "one plane": (512 * 512 * 3, 0, 0, S.BITS(3) | S.PLANE_ONLY, (512, 512, 3, 1)),
    "one plane of two": (512 * 512 * 2, 0, 0, S.PLANE_ONLY, (512, 512, 2, 1)),
    "paper": (512 * 512 * 3, 0, 0, S.LAYOUT_PAPER2, (512, 512, 3, 1)),
    "paper, two channels": (512 * 512 * 2, 0, 0, S.LAYOUT_PAPER2, (512, 512, 2, 1)),
}


@pytest.mark.parametrize("inplace", [False, True])
@pytest.mark.parametrize("name", list(CALLS))
def test_embed_behind_a_memset_is_no_dependent(L, name, inplace):
    """Statistics without a slot (here: under capture) are zeroed by a memset right
    before the kernel that adds to them, which is then an ordinary launch."""
    C, at, out, flags, geom = CALLS[name]
    out = at if inplace else out
    g = S.Geom(*geom) if geom else None
    geom = ctypes.addressof(g) if g else None
    stego = COVER + out if inplace else STEGO + out
    q = L.queued("stego_embed", COVER + at, stego, C, MSG, 4, geom, flags | S.FUSE_STATS, RES, 8,
                 capturing=True)
    at = [i for i, e in enumerate(q) if e[0] == "memset"]
    assert len(at) == 1 and q[at[0]] == ("memset", 16)
    assert at[0] == len(q) - 2 and q[-1][3] == 0, q
    # with a slot: no memset, dependents only
    q = L.queued("stego_embed", COVER + C, STEGO + C, C, MSG, 4, geom, flags | S.FUSE_STATS, RES, 8)
    assert q and all(e[0] != "memset" and e[3] == 1 for e in q), q


@pytest.mark.parametrize("n", [0, 100, 1 << 20])
@pytest.mark.parametrize("at", [0, 5])
def test_comparison_behind_a_memset_is_no_dependent(L, n, at):
    q = L.queued("stego_changed_bytes", COVER + at, STEGO, n, RES, 8, capturing=True)
    assert q[0] == ("memset", 16) and len(q) == 1 + (n > 0) and all(e[3] == 0 for e in q[1:])
    if n:
        q = L.queued("stego_changed_bytes", COVER + at, STEGO, n, RES, 8)
        assert len(q) == 1 and q[0][3] == 1


def test_slots_are_the_statistics():
    """Embeds without statistics and comparisons on hundreds of streams leave every
    slot to embeds with statistics; those that use no slot do not ask for one."""
    L = Launches()  # slots are never handed back: a library of its own
    geom = S.Geom(512, 512, 3, 1)
    g = ctypes.addressof(geom)
    for s in range(1, 301):
        L.queued("stego_embed", COVER, STEGO, 1 << 30, MSG, 4, None, 0, None, s << 8)
        L.queued("stego_embed", COVER, STEGO, 512 * 512 * 3, MSG, 4, g, S.LAYOUT_PAPER2, None, s << 8)
        L.queued("stego_changed_bytes", COVER, STEGO, 1 << 20, RES, s << 8)
    for s in range(1001, 1257):
        q = L.queued("stego_embed", COVER, STEGO, 1 << 20, MSG, 4, None, S.FUSE_STATS, RES, s << 8)
        assert len(q) == 1, (s, q)
    q = L.queued("stego_embed", COVER, STEGO, 1 << 20, MSG, 4, None, S.FUSE_STATS, RES, 2000 << 8)
    assert q[0] == ("memset", 16)  # the 257th
    for C, flags, gm, asks in ((1 << 30, 0, None, 1), (1 << 20, 0, None, 0),
                               (1 << 30, S.BITS(2), None, 0),
                               (512 * 512 * 3, S.LAYOUT_PAPER2, g, 0),
                               (512 * 512 * 3, S.PLANE_ONLY, g, 0)):
        L.queued("stego_embed", COVER, STEGO, C, MSG, 4, gm, flags, None, 3000 << 8)
        assert L.lib.fake_id_queries() == asks, (C, flags)
