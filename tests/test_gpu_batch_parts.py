"""Covers cut into parts of a tile whose size is 4096 bytes times an odd number:
the parts have to make up the tile, at any address and in either layout."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    return need_gpu()


@pytest.fixture(scope="module")
def O():
    return oracle.load()


@pytest.mark.parametrize("inplace", [False, True])
@pytest.mark.parametrize("off,stego_off", [(0, 0), (5, 5), (5, 0), (0, 9)])
@pytest.mark.parametrize("tile", [4096 * 257, 4096 * 513, 4096 * 1025])
def test_stream_parts_make_up_the_tile(S, O, tile, off, stego_off, inplace):
    if inplace:
        stego_off = off
    rng = np.random.default_rng(tile + 16 * off + stego_off)
    for C in (tile + 37, 4096 * 13 + 5):
        cover = rng.integers(0, 256, C, dtype=np.uint8)
        msg = rng.integers(0, 256, C // 8 - 4, dtype=np.uint8)
        tc = torch.full((C + 64,), 0x3C, dtype=torch.uint8, device="cuda")
        tc[off:off + C] = torch.from_numpy(cover)
        ts = tc if inplace else torch.full_like(tc, 0x5A)
        around = int(ts[-1])
        tm = torch.from_numpy(msg).cuda()
        tx = torch.full((msg.size + 8,), 0xEE, dtype=torch.uint8, device="cuda")
        item = dict(cover=tc[off:off + C], stego=ts[stego_off:stego_off + C], msg=tm,
                    cover_bytes=C, msg_bytes=msg.size, flags=S.HEADER_BE32)
        ws = torch.empty(S.stego_batched_workspace_bytes(1), dtype=torch.uint8, device="cuda")
        res, res2 = S.new_result(n=1), S.new_result(n=1)
        tune = (0, 0, 0, tile)
        S.stego_embed_batched(S.descs_to_device(S.pack_descs([item])), 1, res, S.FUSE_STATS, ws,
                              tune=tune)
        item.update(cover=ts[stego_off:stego_off + C], stego=0, msg=tx[:msg.size])
        S.stego_extract_batched(S.descs_to_device(S.pack_descs([item])), 1, res2, 0, ws, tune=tune)
        st, want = O.stream1_embed(cover, msg, header=True)
        assert st == 0
        got = ts.cpu().numpy()
        assert np.array_equal(got[stego_off:stego_off + C], want), C
        assert np.all(got[:stego_off] == around) and np.all(got[stego_off + C:] == around), C
        out = tx.cpu().numpy()
        assert np.array_equal(out[:msg.size], msg) and np.all(out[msg.size:] == 0xEE), C
        r = S.read_result(res[0])
        assert r["status"] == 0 and (r["changed"], r["sse"]) == O.changed_bytes(cover, want), C


@pytest.mark.parametrize("channels", [1, 2, 3])
@pytest.mark.parametrize("tile", [4096 * 257, 4096 * 513])
def test_paper_parts_make_up_the_tile(S, O, tile, channels):
    W, H = 509, tile // 509 // channels + 3
    C = W * H * channels
    rng = np.random.default_rng(tile + channels)
    cover = rng.integers(0, 256, C, dtype=np.uint8)
    msg = rng.integers(0, 256, (W // 4) * H, dtype=np.uint8)
    tc, tm = torch.from_numpy(cover).cuda(), torch.from_numpy(msg).cuda()
    ts, tx = torch.full_like(tc, 0x5A), torch.full_like(tm, 0xEE)
    item = dict(cover=tc, stego=ts, msg=tm, cover_bytes=C, msg_bytes=msg.size, msg_len=msg.size,
                flags=S.LAYOUT_PAPER2, width=W, height=H, channels=channels,
                plane=channels - 1)
    ws = torch.empty(S.stego_batched_workspace_bytes(1), dtype=torch.uint8, device="cuda")
    res, res2 = S.new_result(n=1), S.new_result(n=1)
    tune = (0, 0, 0, tile)
    S.stego_embed_batched(S.descs_to_device(S.pack_descs([item])), 1, res, S.FUSE_STATS, ws, tune=tune)
    item.update(cover=ts, stego=0, msg=tx)
    S.stego_extract_batched(S.descs_to_device(S.pack_descs([item])), 1, res2, 0, ws, tune=tune)
    st, want = O.paper2_embed(cover, W, H, channels, channels - 1, msg)
    assert st == 0
    assert np.array_equal(ts.cpu().numpy(), want) and np.array_equal(tx.cpu().numpy(), msg)
    r = S.read_result(res[0])
    assert r["status"] == 0 and (r["changed"], r["sse"]) == O.changed_bytes(cover, want)
