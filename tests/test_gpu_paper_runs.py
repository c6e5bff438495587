"""Batched paper-layout calls on covers whose rows and quarters are whole vectors:
messages that end inside a run, at a row's end and a byte past it, in tiles of one
and of several rounds and in parts of a tile; outputs at even and odd addresses."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [4096, 65536, 4096 * 33])
@pytest.mark.parametrize("channels,plane", [(1, 0), (3, 0), (3, 2), (4, 1), (4, 3)])
def test_ends_of_aligned_runs(channels, plane, tile):
    S, O = need_gpu(), oracle.load()
    rng = np.random.default_rng(channels * 8 + plane)
    cases = []
    for W, H in ((64, 9), (128, 40), (320, 70), (1920, 33)):
        Q = W // 4
        for N in (1, 15, 16, Q - 1, Q, Q + 1, 3 * Q + 5, Q * (H - 1) + Q // 2, Q * H):
            cases.append((W, H, N, 0))
            cases.append((W, H, N, 5))  # the message at an odd address: no aligned runs
    n = len(cases)
    size = np.array([W * H * channels for W, H, _, _ in cases])
    at = np.concatenate([[0], np.cumsum(size)])
    mat = np.concatenate([[0], np.cumsum([(N + 31) // 16 * 16 for _, _, N, _ in cases])])
    moff = mat[:-1] + np.array([o for *_, o in cases])
    cover = rng.integers(0, 256, int(at[-1]), dtype=np.uint8)
    msg = rng.integers(0, 256, int(mat[-1]), dtype=np.uint8)
    tc, tm = torch.from_numpy(cover).cuda(), torch.from_numpy(msg).cuda()
    ts, tx = torch.full_like(tc, 0x5A), torch.full_like(tm, 0xEE)
    d = np.zeros(n, dtype=S.DESC_DTYPE)
    d["cover"], d["stego"], d["msg"] = tc.data_ptr() + at[:-1], ts.data_ptr() + at[:-1], tm.data_ptr() + moff
    d["cover_bytes"] = size
    d["msg_bytes"] = d["msg_len"] = [N for _, _, N, _ in cases]
    d["flags"], d["channels"], d["plane"] = S.LAYOUT_PAPER2, channels, plane
    d["width"], d["height"] = [c[0] for c in cases], [c[1] for c in cases]
    ws = torch.full((S.stego_batched_workspace_bytes(n),), 0xCD, dtype=torch.uint8, device="cuda")
    res, res2 = S.new_result(n=n), S.new_result(n=n)
    S.stego_embed_batched(S.descs_to_device(d), n, res, S.FUSE_STATS, ws, tune=(0, 0, 0, tile))
    x = d.copy()
    x["cover"], x["msg"], x["stego"] = d["stego"], tx.data_ptr() + moff, 0
    S.stego_extract_batched(S.descs_to_device(x), n, res2, 0, ws, tune=(0, 0, 0, tile))
    want, want_x, r = np.full_like(cover, 0x5A), np.full_like(msg, 0xEE), res.cpu().numpy()
    for j, (W, H, N, _) in enumerate(cases):
        m = msg[int(moff[j]):int(moff[j]) + N]
        c = cover[int(at[j]):int(at[j + 1])]
        st, w = O.paper2_embed(c, W, H, channels, plane, m)
        assert st == oracle.OK
        want[int(at[j]):int(at[j + 1])], want_x[int(moff[j]):int(moff[j]) + N] = w, m
        assert r[j].tolist() == [*O.changed_bytes(c, w), N, 0], cases[j]
    assert np.array_equal(ts.cpu().numpy(), want) and np.array_equal(tx.cpu().numpy(), want_x)
