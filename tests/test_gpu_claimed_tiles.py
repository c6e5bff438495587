"""One-bit embeds whose CTAs claim their tiles (many tiles for each CTA: a launch
shape of one small CTA per SM), with and without statistics, in a row on one
stream with comparisons between them: the counter starts anew for each call."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import Guarded, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("at,out", [(0, 0), (13, 13), (13, 0), (0, 6)])
@pytest.mark.parametrize("inplace", [False, True])
def test_claimed_tiles(at, out, inplace):
    S, O = need_gpu(), oracle.load()
    old = S.stego_get_tune(S.OP_EMBED)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(at + out)
    stream = torch.cuda.Stream()
    out = at if inplace else out
    S.stego_set_tune(S.OP_EMBED, (64, 1, 1, 0))
    try:
        for C in (4 * 4096 * sms + 5000, 4 * 4096 * sms + 5000, 5 * 4096 * sms + 77, 9000):
            cover = rng.integers(0, 256, C, dtype=np.uint8)
            msg = rng.integers(0, 256, int((C // 8 - 4) * 0.9), dtype=np.uint8)
            st, want = O.stream1_embed(cover, msg, header=True)
            assert st == oracle.OK
            totals = O.changed_bytes(cover, want)
            m, ref = torch.from_numpy(msg).cuda(), torch.from_numpy(cover).cuda()
            for stats in (False, True, False):
                c = Guarded(C, off=at, fill=cover)
                s = c if inplace else Guarded(C, off=out, fill=0x5A)
                res, diff = S.new_result(), torch.zeros(2, dtype=torch.int64, device="cuda")
                torch.cuda.synchronize()
                S.stego_embed(c.view, s.view, m, S.HEADER_BE32 | (S.FUSE_STATS if stats else 0), res,
                              stream=stream)
                S.stego_changed_bytes(ref, s.view, diff, stream=stream)
                stream.synchronize()
                assert np.array_equal(s.host(), want) and s.canaries_intact()
                r = S.read_result(res)
                assert (r["changed"], r["sse"]) == (totals if stats else (0, 0))
                assert tuple(diff.tolist()) == totals
    finally:
        S.stego_set_tune(S.OP_EMBED, old)
