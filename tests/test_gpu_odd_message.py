"""One-bit embeds of a message at an odd address into 16-byte aligned buffers, around
the size from which they run in the kernel for misaligned ones, the buffers on and
off a cache line's start, with a message that ends inside the cover or fills it."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import Guarded, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("inplace", [False, True])
@pytest.mark.parametrize("at,out", [(0, 0), (16, 16), (112, 48), (0, 96)])
@pytest.mark.parametrize("C", [(16 << 20) - 1, 16 << 20, (16 << 20) + 4099])
def test_odd_message(C, at, out, inplace):
    S, O = need_gpu(), oracle.load()
    out = at if inplace else out
    rng = np.random.default_rng(C + at + out)
    cover = rng.integers(0, 256, C, dtype=np.uint8)
    for header, room in ((True, 0), (True, 12345), (False, 7)):
        msg = rng.integers(0, 256, C // 8 - 4 - room, dtype=np.uint8)
        m = Guarded(msg.size, off=3, fill=msg)
        c = Guarded(C, off=at, fill=cover)
        s = c if inplace else Guarded(C, off=out, fill=0x5A)
        res = S.new_result()
        S.stego_embed(c.view, s.view, m.view, (S.HEADER_BE32 if header else 0) | S.FUSE_STATS, res)
        st, want = O.stream1_embed(cover, msg, header=header)
        assert st == oracle.OK
        assert np.array_equal(s.host(), want) and s.canaries_intact()
        r = S.read_result(res)
        assert (r["changed"], r["sse"]) == O.changed_bytes(cover, want)
