"""The solve's setup passes: their reductions and fills at ragged sizes, from
one element to more than one pass of the reduction's grid (311296 threads),
on workspaces that hold NaN."""
import numpy as np
import pytest

import oracle as O
import synth
from gpu_util import f32, need_gpu, to_gpu, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,sigma", [(0, 0.0), (0, 0.3), (1, 0.0)])
@pytest.mark.parametrize("N,V,B", [(1, 1, 1), (3, 5, 7), (16, 16, 16), (17, 9, 31), (40, 1, 57), (64, 720, 433)])
def test_setup(N, V, B, mode, sigma):
    P = need_gpu()
    import torch
    x = synth.ellipse_phantom(N, 4, 1) * (2.0 / N)
    b, w = (f32(a) for a in synth.poisson_data(O.project(x, V, B), 1e4, 2))
    g = P.Geometry(N, V, B)
    out = {}
    for fill in (0, 0xFF):   # 0xFF bytes: NaN in every float and double
        for iters in (0, 2):
            prm = P.PDTVParams(mode=mode, iters=iters, tv_iters=3, beta=0.01, sigma=sigma)
            ws = P.workspace_for(g, prm)
            ws.fill_(fill)
            xo = torch.full((N, N), float("nan"), device="cuda")
            xo, rep = P.ct_pdtv_solve(g, to_gpu(b), to_gpu(w) if mode == 0 else None, prm, x_out=xo, workspace=ws)
            out[fill, iters] = (to_np(xo), rep)
    assert (out[0xFF, 0][0] == 0.0).all()
    np.testing.assert_array_equal(out[0, 2][0], out[0xFF, 2][0])
    rep = out[0xFF, 2][1]
    if mode == 0:
        # a float sum of positive terms: two per thread and 8 + 5 + 8 tree and 5 + 8 + 8 final additions at most,
        # each within 2^-24, and the reciprocals' own rounding
        kappa = np.mean(1.0 / w)
        assert rep["kappa"] == pytest.approx(kappa, rel=45 * 2.0 ** -24)
        assert rep["tau"] == pytest.approx(np.pi * rep["kappa"] / (2 * V), rel=1e-12)
    else:
        assert rep["tau"] == 0.01
    assert np.isfinite(rep["sigma"]) and rep["sigma"] > 0.0
    if sigma > 0.0:
        assert rep["sigma"] == sigma
