"""Kernels whose blocks touch another block's shared memory (thread-block
clusters) wait first until every block of the cluster runs: CUDA leaves an
access to a block that has not started undefined.  The order is checked in the
source, on the CPU; on the GPU, the step-size setup that relies on it gives the
same bits on a busy device, whose clusters start late, as on an idle one."""
import glob
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1609_06041_gb300", "csrc")


def kernels():
    """(name, body) of every __global__ function: up to the closing brace in the first column."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(", text):
            yield m.group(1), text[m.end():text.index("\n}", m.end())]


def test_remote_shared_memory_is_reached_after_the_cluster_has_started():
    users = {name: body for name, body in kernels() if "map_shared_rank" in body}
    assert {"k_lanczos_fused", "k_backproject_orbit_cl"} <= set(users)
    for name, body in users.items():
        before = body[:body.index("map_shared_rank")]
        assert "cl.sync()" in before or "cl.barrier_wait()" in before, name
        if "cl.barrier_wait()" in before:
            assert before.index("cl.barrier_arrive()") < before.index("cl.barrier_wait()"), name


@pytest.mark.gpu
@pytest.mark.parametrize("N,V,B", [(64, 90, 96), (128, 32, 184), (180, 60, 260)])
def test_norms_on_a_busy_device(N, V, B):
    from gpu_util import need_gpu, to_gpu
    P = need_gpu()
    import torch
    r = np.random.default_rng(3)
    b, w = to_gpu(r.uniform(0.0, 1.0, (V, B))), to_gpu(r.uniform(1.0, 9.0, (V, B)))
    g, prm = P.Geometry(N, V, B), P.PDTVParams(mode=0, iters=0, beta=0.01)
    ref = P.ct_pdtv_solve(g, b, w, prm)[1]
    torch.cuda.synchronize()
    a = torch.randn(4096, 4096, device="cuda")
    streams = [torch.cuda.Stream() for _ in range(3)]
    work = [P.workspace_for(g, prm) for _ in streams]
    out = [torch.empty(N, N, device="cuda") for _ in streams]
    torch.cuda.synchronize()
    for _ in range(5):
        a = torch.tanh(a @ a)   # fills the device while the setups start
        for s, ws, x in zip(streams, work, out):
            with torch.cuda.stream(s):
                P.ct_pdtv_solve(g, b, w, prm, x_out=x, workspace=ws, report=False)
    torch.cuda.synchronize()
    for s, ws in zip(streams, work):
        with torch.cuda.stream(s):
            rep = P.ct_pdtv_solve(g, b, w, P.PDTVParams(mode=0, iters=0, beta=0.01, resume=1), x_out=out[0],
                                  workspace=ws)[1]
        assert (rep["norm_ADA"], rep["norm_WDW"], rep["sigma"]) == (ref["norm_ADA"], ref["norm_WDW"], ref["sigma"])
