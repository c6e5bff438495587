"""Batches around the limits of the preparation launch (one warp, one CTA, a
cluster, several descriptors per thread), tiny covers of every kind and refused
ones among them, and one cover cut into parts of a tile, against the CPU oracle."""
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


@pytest.mark.parametrize("n", [1, 32, 33, 1024, 1025, 2049, 8193, 20000])
def test_counts(S, O, n):
    rng = np.random.default_rng(n)
    slot = 96
    cover = rng.integers(0, 256, n * slot, dtype=np.uint8)
    msg = rng.integers(0, 256, n * 16, dtype=np.uint8)
    tc, tm = torch.from_numpy(cover).cuda(), torch.from_numpy(msg).cuda()
    ts, tx = torch.full_like(tc, 0x5A), torch.full_like(tm, 0xEE)
    d = np.zeros(n, dtype=S.DESC_DTYPE)
    i = np.arange(n)
    kind = i % 4  # aligned stream, stream at an odd address, paper layout, message too long
    off = np.where(kind == 1, 3, 0)
    d["cover"] = tc.data_ptr() + i * slot + off
    d["stego"] = ts.data_ptr() + i * slot + off
    d["msg"] = tm.data_ptr() + i * 16
    d["cover_bytes"] = 72
    d["msg_bytes"] = d["msg_len"] = np.where(kind == 3, 12, 5)
    d["flags"] = np.where(kind == 2, S.LAYOUT_PAPER2, np.where(kind == 0, S.HEADER_BE32, 0))
    d["width"], d["height"], d["channels"], d["plane"] = 8, 3, 3, 1
    res, res2 = S.new_result(n=n), S.new_result(n=n)
    ws = torch.full((S.stego_batched_workspace_bytes(n),), 0xCD, dtype=torch.uint8, device="cuda")
    S.stego_embed_batched(S.descs_to_device(d), n, res, S.FUSE_STATS, ws)
    x = d.copy()
    x["cover"], x["msg"], x["stego"] = d["stego"], tx.data_ptr() + i * 16, 0
    S.stego_extract_batched(S.descs_to_device(x), n, res2, 0, ws)
    r, r2 = res.cpu().numpy(), res2.cpu().numpy()
    got, out = ts.cpu().numpy(), tx.cpu().numpy()
    want, want_out = np.full_like(cover, 0x5A), np.full_like(msg, 0xEE)
    for j in range(n):
        a = j * slot + int(off[j])
        c, m = cover[a:a + 72], msg[j * 16:j * 16 + 5]
        if kind[j] == 3:
            assert (r[j, 3] & 0xFFFFFFFF) == 0xFFFFFFFE and r[j, 2] == 0, j  # capacity
            assert (r2[j, 3] & 0xFFFFFFFF) == 0xFFFFFFFE, j
            continue
        st, w = (O.paper2_embed(c, 8, 3, 3, 1, m) if kind[j] == 2 else
                 O.stream1_embed(c, m, header=bool(kind[j] == 0)))
        assert st == 0
        want[a:a + 72], want_out[j * 16:j * 16 + 5] = w, m
        diff = w.astype(np.int64) - c
        assert r[j].tolist() == [np.count_nonzero(diff), int((diff * diff).sum()), 5, 0], j
        assert r2[j].tolist() == [0, 0, 5, 0], j
    assert np.array_equal(got, want) and np.array_equal(out, want_out)


@pytest.mark.parametrize("off", [0, 5])
@pytest.mark.parametrize("tile", [4096, 12288, 65536, 1 << 20])
def test_one_cover_in_parts(S, O, off, tile):
    """Sizes around a part, a tile and both, each a batch of its own."""
    rng = np.random.default_rng(tile + off)
    for C in (33, 4095, 4096, 4097, 12300, 65535, 65537, 70001, 300007):
        cover = rng.integers(0, 256, C, dtype=np.uint8)
        msg = rng.integers(0, 256, C // 8 - 4, dtype=np.uint8)
        tc = torch.from_numpy(np.concatenate([np.zeros(off, np.uint8), cover])).cuda()
        ts, tm = torch.full_like(tc, 0x5A), torch.from_numpy(msg).cuda()
        tx = torch.full((msg.size + 8,), 0xEE, dtype=torch.uint8, device="cuda")
        item = dict(cover=tc[off:], stego=ts[off:], msg=tm, cover_bytes=C, msg_bytes=msg.size,
                    flags=S.HEADER_BE32)
        ws = torch.empty(S.stego_batched_workspace_bytes(1), dtype=torch.uint8, device="cuda")
        res, res2 = S.new_result(n=1), S.new_result(n=1)
        S.stego_embed_batched(S.descs_to_device(S.pack_descs([item])), 1, res, S.FUSE_STATS, ws,
                              tune=(0, 0, 0, tile))
        item.update(cover=ts[off:], stego=0, msg=tx[:msg.size])
        S.stego_extract_batched(S.descs_to_device(S.pack_descs([item])), 1, res2, 0, ws,
                                tune=(0, 0, 0, tile))
        st, want = O.stream1_embed(cover, msg, header=True)
        assert st == 0 and np.array_equal(ts[off:].cpu().numpy(), want), C
        assert np.array_equal(tx.cpu().numpy()[:msg.size], msg) and bool((tx[msg.size:] == 0xEE).all()), C
        r = S.read_result(res[0])
        assert (r["changed"], r["sse"]) == O.changed_bytes(cover, want), C
