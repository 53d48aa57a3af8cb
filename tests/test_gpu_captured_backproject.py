"""ct_backproject in a caller's stream capture: kernel nodes only (memory nodes
would keep the caller's graph from being cloned, nested in another graph or
instantiated twice), with the bits of the uncaptured call, at sizes below and
above those that take scratch uncaptured and on rows of every length mod 4."""
import ctypes

import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu

KERNEL = 0   # CU_GRAPH_NODE_TYPE_KERNEL


@pytest.mark.parametrize("N,V,B,batch", [(64, 90, 95, 1), (64, 90, 96, 1), (128, 180, 185, 4), (128, 180, 186, 4),
                                         (256, 720, 367, 3), (256, 720, 368, 3)])
def test_captured_call_is_kernel_nodes(N, V, B, batch):
    P = need_gpu()
    import torch
    cu = ctypes.CDLL("libcuda.so.1")
    vp = ctypes.c_void_p
    g = P.Geometry(N, V, B)
    y = torch.randn(batch, V, B, device="cuda")
    ref = P.ct_backproject(g, y)
    out = torch.empty_like(ref)
    stream = torch.cuda.Stream()
    graph, clone, execs = vp(), vp(), [vp(), vp(), vp()]
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        s = vp(stream.cuda_stream)
        assert cu.cuStreamBeginCapture_v2(s, 2) == 0   # CU_STREAM_CAPTURE_MODE_RELAXED
        P.ct_backproject(g, y, out)
        assert cu.cuStreamEndCapture(s, ctypes.byref(graph)) == 0
        n = ctypes.c_size_t()
        assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0 and n.value >= 1
        nodes = (vp * n.value)()
        assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
        for node in nodes:
            kind = ctypes.c_int(-1)
            assert cu.cuGraphNodeGetType(vp(node), ctypes.byref(kind)) == 0 and kind.value == KERNEL
        assert cu.cuGraphClone(ctypes.byref(clone), graph) == 0
        for e, gr in zip(execs, (graph, graph, clone)):
            assert cu.cuGraphInstantiateWithFlags(ctypes.byref(e), gr, ctypes.c_ulonglong(0)) == 0
        for e in execs:
            out.zero_()
            assert cu.cuGraphLaunch(e, s) == 0
            stream.synchronize()
            assert torch.equal(out, ref)
    for e in execs:
        cu.cuGraphExecDestroy(e)
    for gr in (graph, clone):
        cu.cuGraphDestroy(gr)
