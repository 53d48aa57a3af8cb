"""The step-size setup's Lanczos run on sinograms of whole 16-byte groups at the
size that one launch takes (32768 elements): just below, at and just above it.
(A sinogram of V B % 4 != 0 elements takes two launches a step whatever its
size, so only such sizes reach the one-launch step on this side.)  The default
estimate lies within its documented -0.25 .. 2.2 % of a deeper run's."""
import numpy as np
import pytest

import oracle as O
import synth
from gpu_util import f32, need_gpu, to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,V,B", [(32, 182, 180), (64, 128, 256), (32, 12, 2731), (16, 2, 2)])
def test_norms_at_the_limit_of_one_launch(N, V, B):
    P = need_gpu()
    x = synth.ellipse_phantom(N, 6, 1) * (2.0 / N)
    b, w = (to_gpu(f32(a)) for a in synth.poisson_data(O.project(x, V, B), 1e4, 2))
    g = P.Geometry(N, V, B)
    norms = [P.ct_pdtv_solve(g, b, w, P.PDTVParams(mode=0, iters=1, tv_iters=2, beta=0.01, norm_iters=k))[1]["norm_WDW"]
             for k in (0, 64)]
    assert 0.995 * norms[1] <= norms[0] <= 1.04 * norms[1]
    assert np.isfinite(norms[1]) and norms[1] > 0.0
