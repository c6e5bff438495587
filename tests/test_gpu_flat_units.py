"""The paper layout's flat units and runs (any row length, any buffer
addresses) against the CPU oracle: row lengths around a unit, a quarter and a
vector, cover and stego at equal and different addresses mod 16, single-cover
and batched, bytes and statistics exactly equal."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import Guarded, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    return need_gpu()


@pytest.fixture(scope="module")
def O():
    return oracle.load()


# rows shorter than a unit, quarters shorter than a unit, W % 4 != 0, W % 16
# around a vector, rows longer than a warp's 512 pixels, whole vectors
WIDTHS = [4, 5, 7, 17, 31, 63, 64, 66, 100, 255, 1000, 2051, 528]
OFFSETS = [(0, 0, 0), (5, 5, 3), (13, 0, 1), (0, 7, 16), (3, 11, 6)]


def _cover(rng, n):
    return rng.integers(0, 256, n, dtype=np.uint8)


@pytest.mark.parametrize("channels", [1, 3, 4])
@pytest.mark.parametrize("offs", OFFSETS)
def test_single_cover(S, O, channels, offs):
    rng = np.random.default_rng(1000 * channels + offs[0] * 17 + offs[1])
    for W in WIDTHS:
        for H in (1, 2, 9, 40):
            plane = int(rng.integers(channels))
            cap = W // 4 * H
            for N in sorted({1, cap // 3, cap - 1, cap} - {0, -1}):
                if not 0 < N <= cap:
                    continue
                cover, msg = _cover(rng, W * H * channels), _cover(rng, N)
                st, want = O.paper2_embed(cover, W, H, channels, plane, msg)
                assert st == oracle.OK
                gc, gs = Guarded(cover.size, offs[0], cover), Guarded(cover.size, offs[1], 0x5A)
                gm, gx = Guarded(N, offs[2], msg), Guarded(N, offs[2], 0xEE)
                res, res2 = S.new_result(), S.new_result()
                geom = (W, H, channels, plane)
                S.stego_embed(gc.view, gs.view, gm.view, S.LAYOUT_PAPER2 | S.FUSE_STATS, res, geom=geom)
                S.stego_extract(gs.view, gx.view, N, S.LAYOUT_PAPER2, res2, geom=geom)
                at = (W, H, channels, plane, N, offs)
                assert np.array_equal(gs.host(), want), at
                assert np.array_equal(gx.host(), msg), at
                assert gs.canaries_intact() and gc.canaries_intact() and gx.canaries_intact(), at
                r = S.read_result(res)
                assert (r["changed"], r["sse"]) == O.changed_bytes(cover, want), at
                assert r["msg_bytes"] == N and S.read_result(res2)["msg_bytes"] == N


@pytest.mark.parametrize("tile", [4096, 65536])
def test_batched(S, O, tile):
    """Covers of every width and offset, out of place and in place, in one batch."""
    rng = np.random.default_rng(tile)
    items, keep, want = [], [], []
    for channels in (1, 2, 3, 4):
        for i, W in enumerate(WIDTHS):
            for inplace in (False, True):
                offs = OFFSETS[(i + channels) % len(OFFSETS)]
                H = int(rng.integers(1, 60))
                plane, N = int(rng.integers(channels)), int(rng.integers(0, W // 4 * H + 1))
                cover, msg = _cover(rng, W * H * channels), _cover(rng, N)
                gc = Guarded(cover.size, offs[0], cover)
                gs = gc if inplace else Guarded(cover.size, offs[1], 0x5A)
                gm, gx = Guarded(N, offs[2], msg), Guarded(N, offs[2], 0xEE)
                keep.append((gc, gs, gm, gx))
                want.append((cover, msg, O.paper2_embed(cover, W, H, channels, plane, msg)[1]))
                items.append(dict(cover=gc.view, stego=gs.view, msg=gm.view, cover_bytes=cover.size,
                                  msg_bytes=N, msg_len=N, flags=S.LAYOUT_PAPER2, width=W, height=H,
                                  channels=channels, plane=plane))
    n = len(items)
    ws = torch.empty(S.stego_batched_workspace_bytes(n), dtype=torch.uint8, device="cuda")
    res, res2 = S.new_result(n=n), S.new_result(n=n)
    tune = (0, 0, 0, tile)
    S.stego_embed_batched(S.descs_to_device(S.pack_descs(items)), n, res, S.FUSE_STATS, ws, tune=tune)
    for it, (gc, gs, gm, gx) in zip(items, keep):
        it.update(cover=gs.view, stego=0, msg=gx.view)
    S.stego_extract_batched(S.descs_to_device(S.pack_descs(items)), n, res2, 0, ws, tune=tune)
    for i, ((gc, gs, gm, gx), (cover, msg, stego)) in enumerate(zip(keep, want)):
        at = {k: items[i][k] for k in ("width", "height", "channels", "plane", "msg_len")}
        assert np.array_equal(gs.host(), stego), at
        assert np.array_equal(gx.host(), msg), at
        assert gs.canaries_intact() and gx.canaries_intact(), at
        r = S.read_result(res[i])
        assert r["status"] == 0 and (r["changed"], r["sse"]) == O.changed_bytes(cover, stego), at
        assert S.read_result(res2[i])["msg_bytes"] == msg.size
