"""CTAs per SM of the batched embed in launch shapes other than the default one, read
from a captured call (the grid of the aligned stream kernel is SMs times the CTAs
that fit): the tile loop must not cost the kernels the registers of a CTA."""
import ctypes

import pytest
import torch

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


class KernelParams(ctypes.Structure):
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3),
                ("smem", ctypes.c_uint), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def captured_shapes(call):
    """(CTAs, threads) of each kernel that call(stream) queues."""
    cu = ctypes.CDLL("libcuda.so.1")
    vp = ctypes.c_void_p
    for f, a in (("cuStreamBeginCapture_v2", [vp, ctypes.c_int]), ("cuStreamEndCapture", [vp, vp]),
                 ("cuGraphGetNodes", [vp, vp, vp]), ("cuGraphNodeGetType", [vp, vp]),
                 ("cuGraphKernelNodeGetParams_v2", [vp, vp]), ("cuGraphDestroy", [vp])):
        getattr(cu, f).argtypes = a
    stream, graph, n = torch.cuda.Stream(), vp(), ctypes.c_size_t()
    assert cu.cuStreamBeginCapture_v2(stream.cuda_stream, 2) == 0  # relaxed
    try:
        call(stream)
    finally:
        assert cu.cuStreamEndCapture(stream.cuda_stream, ctypes.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (vp * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    out = []
    for node in nodes:
        kind, p = ctypes.c_int(), KernelParams()
        assert cu.cuGraphNodeGetType(node, ctypes.byref(kind)) == 0
        if kind.value == 0:
            assert cu.cuGraphKernelNodeGetParams_v2(node, ctypes.byref(p)) == 0
            out.append((p.grid[0], p.block[0]))
    assert cu.cuGraphDestroy(graph) == 0
    return out


@pytest.mark.parametrize("threads,vec,stats,per_sm", [
    (256, 4, True, 3), (256, 4, False, 3), (512, 4, False, 2), (512, 2, True, 2), (512, 2, False, 3),
    (512, 1, False, 4), (256, 2, True, 4), (256, 2, False, 6), (256, 1, False, 8), (128, 4, True, 6)])
def test_ctas_per_sm(threads, vec, stats, per_sm):
    S = need_gpu()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    c, m = torch.zeros(4096, dtype=torch.uint8, device="cuda"), torch.zeros(16, dtype=torch.uint8, device="cuda")
    s = torch.zeros_like(c)
    d = S.descs_to_device(S.pack_descs([dict(cover=c, stego=s, msg=m, cover_bytes=4096, msg_bytes=16)]))
    res = S.new_result(n=1)
    ws = torch.empty(S.stego_batched_workspace_bytes(1), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    shapes = captured_shapes(lambda st: S.stego_embed_batched(
        d, 1, res, S.FUSE_STATS if stats else 0, ws, tune=(threads, vec, 0, 0), stream=st))
    assert len(shapes) == 4  # preparation, aligned stream, misaligned stream, paper layout
    grid, block = shapes[1]
    assert block == threads and grid >= sms * per_sm, shapes
