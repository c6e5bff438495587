"""stego_changed_bytes at every pair of addresses mod 16 and at sizes around its
kernels' limits (bytes alone, one round, rounds and a rest), on random bytes
and on the largest differences, against numpy's integers."""
import numpy as np
import pytest
import torch

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    return need_gpu()


def _pair(rng, n, extreme):
    a = rng.integers(0, 256, n, dtype=np.uint8)
    if extreme:
        a = np.where(a < 128, 0, 255).astype(np.uint8)
        return a, (255 - a).astype(np.uint8)
    b = np.where(rng.random(n) < 0.5, a, rng.integers(0, 256, n, dtype=np.uint8)).astype(np.uint8)
    return a, b


@pytest.mark.parametrize("n", [1, 16, 1024, 1025, 1300, 4096, 70001, 2500003])
@pytest.mark.parametrize("extreme", [False, True])
def test_any_alignment(S, n, extreme):
    rng = np.random.default_rng(n)
    a, b = _pair(rng, n, extreme)
    d = a.astype(np.int64) - b.astype(np.int64)
    want = [int(np.count_nonzero(d)), int((d * d).sum())]
    offs = [(x, y) for x in range(16) for y in range(16)] if n < 5000 else [
        (0, 0), (0, 1), (13, 0), (5, 5), (3, 14), (15, 1), (7, 9), (4, 8)]
    fa = torch.zeros(n + 32, dtype=torch.uint8, device="cuda")
    fb = torch.zeros(n + 32, dtype=torch.uint8, device="cuda")
    out = torch.full((len(offs), 2), -1, dtype=torch.int64, device="cuda")
    ta, tb = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    for i, (x, y) in enumerate(offs):
        fa.fill_(1), fb.fill_(200)  # what lies around the arrays does not count
        fa[x:x + n], fb[y:y + n] = ta, tb
        S.stego_changed_bytes(fa[x:x + n], fb[y:y + n], out[i])
    got = out.cpu().tolist()
    for i, at in enumerate(offs):
        assert got[i] == want, (at, n)


def test_captured_and_repeated(S):
    """Under stream capture (no slot: zeroed words) and back to back on one stream."""
    a, b = (torch.randint(0, 256, (100003,), dtype=torch.uint8, device="cuda") for _ in range(2))
    d = a.to(torch.int64) - b.to(torch.int64)
    want = [int((d != 0).sum()), int((d * d).sum())]
    out = torch.zeros(3, 2, dtype=torch.int64, device="cuda")
    S.stego_changed_bytes(a[1:], b[1:], out[0])
    S.stego_changed_bytes(a, b, out[1])
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        S.stego_changed_bytes(a, b, out[2])
    for _ in range(3):
        g.replay()
    got = out.cpu().tolist()
    first = int((d[0] != 0)), int(d[0] * d[0])
    assert got == [[want[0] - first[0], want[1] - first[1]], want, want]
