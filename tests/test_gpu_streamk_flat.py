"""The k-bit stream's units at any buffer addresses against the CPU oracle:
streams that end before, in and after the first and last units, covers of a
few vectors to several CTAs, cover and stego at equal and different addresses
mod 16, messages at odd addresses, bytes and statistics exactly equal."""
import numpy as np
import pytest

import oracle
from gpu_util import Guarded, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    return need_gpu()


@pytest.fixture(scope="module")
def O():
    return oracle.load()


# (cover, stego, message) bytes past a 256-byte boundary; equal and aligned
# covers with an odd message take the same kernels
OFFSETS = [(0, 0, 1), (0, 0, 2), (5, 5, 3), (13, 0, 0), (0, 7, 5), (3, 126, 6), (144, 48, 0)]
# pixels: one vector and less, around the head's 128 bytes and 16384 bytes,
# several CTAs of units
PIXELS = [40, 130, 301, 5500, 16411, 70003]


def _case(S, O, rng, k, pixels, channels, plane, header, offs, inplace, fill):
    geom = None if plane < 0 else (pixels, 1, channels, plane)
    C = pixels * channels
    flags = S.BITS(k) | (S.HEADER_BE32 if header else 0) | (S.PLANE_ONLY if geom else 0)
    cap = S.stego_capacity(C, flags, geom=geom)
    if header and (pixels if geom else C) * k < 32:
        return
    m = max(0, int(cap * fill))
    cover = rng.integers(0, 256, C, dtype=np.uint8)
    msg = rng.integers(0, 256, m, dtype=np.uint8)
    st, want = O.streamk_embed(cover, msg, k, header=header, geom=geom)
    assert st == oracle.OK
    gc = Guarded(C, offs[0], cover)
    gs = gc if inplace else Guarded(C, offs[1], 0x5A)
    gm, gx = Guarded(m, offs[2], msg), Guarded(m, offs[2], 0xEE)
    res, res2 = S.new_result(), S.new_result()
    S.stego_embed(gc.view, gs.view, gm.view, flags | S.FUSE_STATS, res, geom=geom)
    S.stego_extract(gs.view, gx.view, m, flags, res2, geom=geom)
    at = (k, pixels, channels, plane, header, offs, inplace, fill)
    assert np.array_equal(gs.host(), want), at
    assert np.array_equal(gx.host(), msg), at
    assert gs.canaries_intact() and gc.canaries_intact() and gx.canaries_intact(), at
    r, r2 = S.read_result(res), S.read_result(res2)
    assert (r["changed"], r["sse"]) == O.changed_bytes(cover, want), at
    assert r["msg_bytes"] == m and r2["msg_bytes"] == m and r2["status"] == 0, at


@pytest.mark.parametrize("k", [1, 2, 3, 4])
@pytest.mark.parametrize("offs", OFFSETS)
def test_any_alignment(S, O, k, offs):
    rng = np.random.default_rng(100 * k + sum(offs))
    for pixels in PIXELS:
        for channels, plane in ((1, -1), (3, -1), (1, 0), (3, 0), (3, 1), (3, 2), (4, 1), (4, 3)):
            if k == 1 and plane < 0:
                continue  # the one-bit stream's own kernels
            inplace = bool(rng.integers(2)) and offs[0] == offs[1]
            header = bool(rng.integers(2))
            for fill in (0.0, 0.02, 0.7, 1.0):
                _case(S, O, rng, k, pixels, channels, plane, header, offs, inplace, fill)
