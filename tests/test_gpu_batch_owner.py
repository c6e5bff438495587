"""Which cover a tile belongs to: counts around the 32-way search's steps, covers
of one and of many tiles, and long runs of refused covers that own none."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", ["stream", "paper"])
@pytest.mark.parametrize("n", [2, 31, 34, 63, 64, 65, 1023, 1057])
def test_owner(n, layout):
    S, O = need_gpu(), oracle.load()
    rng = np.random.default_rng(n)
    paper = layout == "paper"
    h = np.where(rng.random(n) < 0.1, rng.integers(100, 300, n), 4)  # many tiles, or one
    refused = np.zeros(n, bool)
    refused[n // 3:n // 3 + n // 4] = True
    size = 64 * 3 * h
    at = np.concatenate([[0], np.cumsum(size)])
    cover = rng.integers(0, 256, int(at[-1]), dtype=np.uint8)
    msg = rng.integers(0, 256, int(at[-1]), dtype=np.uint8)
    # the paper layout holds a quarter byte a pixel, the stream an eighth a byte
    cap = (64 * h) // 4 if paper else size // 8 - 4
    mlen = np.where(refused, cap + 1, cap)
    tc, tm = torch.from_numpy(cover).cuda(), torch.from_numpy(msg).cuda()
    ts, tx = torch.full_like(tc, 0x5A), torch.full_like(tm, 0xEE)
    d = np.zeros(n, dtype=S.DESC_DTYPE)
    d["cover"], d["stego"] = tc.data_ptr() + at[:-1], ts.data_ptr() + at[:-1]
    d["msg"], d["cover_bytes"] = tm.data_ptr() + at[:-1], size
    d["msg_bytes"] = d["msg_len"] = mlen
    d["flags"] = S.LAYOUT_PAPER2 if paper else S.HEADER_BE32
    d["width"], d["height"], d["channels"], d["plane"] = 64, h, 3, 1
    ws = torch.full((S.stego_batched_workspace_bytes(n),), 0xCD, dtype=torch.uint8, device="cuda")
    res, res2 = S.new_result(n=n), S.new_result(n=n)
    tune = (0, 0, 0, 4096)
    S.stego_embed_batched(S.descs_to_device(d), n, res, S.FUSE_STATS, ws, tune=tune)
    x = d.copy()
    x["cover"], x["msg"], x["stego"] = d["stego"], tx.data_ptr() + at[:-1], 0
    x["msg_bytes"] = x["msg_len"] = cap
    if not paper:
        x = x[~refused]  # their covers hold no header
    res2 = S.new_result(n=len(x))
    S.stego_extract_batched(S.descs_to_device(x), len(x), res2, 0, ws, tune=tune)
    want, want_x = np.full_like(cover, 0x5A), np.full_like(msg, 0xEE)
    r = res.cpu().numpy()
    for j in range(n):
        a, b = int(at[j]), int(at[j + 1])
        if refused[j]:
            assert (r[j, 3] & 0xFFFFFFFF) == 0xFFFFFFFE, j  # capacity
            if paper:
                want_x[a:a + int(cap[j])] = 0xAA  # four pairs of 0x5A
            continue
        m = msg[a:a + int(cap[j])]
        st, w = (O.paper2_embed(cover[a:b], 64, int(h[j]), 3, 1, m) if paper else
                 O.stream1_embed(cover[a:b], m, header=True))
        assert st == 0
        want[a:b], want_x[a:a + m.size] = w, m
        diff = w.astype(np.int64) - cover[a:b]
        assert r[j].tolist() == [np.count_nonzero(diff), int((diff * diff).sum()), m.size, 0], j
    assert np.array_equal(ts.cpu().numpy(), want) and np.array_equal(tx.cpu().numpy(), want_x)
