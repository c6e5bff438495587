"""Extraction of an aligned stego around the ends of its kernels' rounds: messages
of one round and a little more or less, of several rounds per warp, of any parity,
into buffers of their own size and of the cover's whole capacity, in every launch
shape, with and without the header."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import Guarded, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    S = need_gpu()
    old = S.stego_get_tune(S.OP_EXTRACT)
    yield S
    S.stego_set_tune(S.OP_EXTRACT, old)


@pytest.mark.parametrize("ctas", [0, 1])
@pytest.mark.parametrize("threads,vec", [(64, 1), (64, 2), (128, 4), (64, 8), (512, 4)])
def test_rounds(S, threads, vec, ctas):
    O = oracle.load()
    S.stego_set_tune(S.OP_EXTRACT, (threads, vec, ctas, 0))
    rng = np.random.default_rng(threads + vec)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    wave = 2 * sms * threads * vec  # message bytes of a round of a one-CTA-per-SM grid
    cover = rng.integers(0, 256, 8 * (2 * wave + 64) + 5, dtype=np.uint8)
    cap = cover.size // 8 - 4
    r = 64 * vec  # message bytes of a warp's round
    for i, m in enumerate((0, 1, 2, r - 1, r, r + 1, 2 * r, wave - 2, wave, wave + 1, wave + r + 3, cap)):
        msg = rng.integers(0, 256, m, dtype=np.uint8)
        for header in (True, False):
            st, stego = O.stream1_embed(cover, msg, header=header)
            assert st == oracle.OK
            d = torch.from_numpy(stego).cuda()
            for room in (m, cap):
                out = Guarded(room, off=i % 2, fill=0xEE)
                res = S.new_result()
                S.stego_extract(d, out.view, m, S.HEADER_BE32 if header else 0, res)
                got = S.read_result(res)
                assert got["status"] == 0 and got["msg_bytes"] == m
                h = out.host()
                assert np.array_equal(h[:m], msg) and np.all(h[m:] == 0xEE), (m, header, room)
                assert out.canaries_intact()


def test_refused_headers_leave_the_buffer(S):
    S.stego_set_tune(S.OP_EXTRACT, (128, 4, 0, 0))
    for fill, status in ((0xFF, S.E_BAD_HEADER), (None, S.E_MSG_TOO_SMALL)):
        C = 1 << 20
        stego = torch.zeros(C, dtype=torch.uint8, device="cuda")
        if fill is not None:
            stego.fill_(fill)
        else:
            stego[32 - 1 - 12] = 1  # 4096 bits
        out = Guarded(500 if fill is None else C // 8 - 4, fill=0xEE)
        res = S.new_result()
        S.stego_extract(stego, out.view, 0, S.HEADER_BE32, res)
        got = S.read_result(res)
        assert got["status"] == status and got["msg_bytes"] == 0
        assert np.all(out.host() == 0xEE) and out.canaries_intact()
