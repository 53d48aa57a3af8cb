"""The frequency-domain D at every transform length and at the edges of its
lengths, against the FP64 oracle: the filter itself, and the dual step through
a few iterations of a low-dose solve, on grids of few view pairs (whose blocks
stage the residual with extra threads) and of more pairs than SMs.

Tolerance of the filter: a float transform of P points is off by at most
about eps log2 P of its norm, twice per filter, and white taps spread |Hhat|
by a factor of four at most: 2 * 6e-8 * 13 * 4 = 6e-6 relative."""
import numpy as np
import pytest

import oracle as O
import synth
from gpu_util import f32, need_gpu, rel_l2, to_gpu, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 31, 32, 33, 64, 65, 128, 129, 256, 257, 512, 513, 1024, 1025, 2048, 2049, 4096])
@pytest.mark.parametrize("V", [1, 4, 9])
def test_filter_at_every_length(V, B):
    P = need_gpu()
    g = P.Geometry(8, V, B)
    half = B if B < 200 else B // 3
    t = f32(np.random.default_rng(B).standard_normal(2 * half - 1))   # not symmetric: Hhat is complex
    y = f32(np.stack([synth.random_sinogram(V, B, s) for s in (1, 2)]))
    got = to_np(P.ct_ramp_filter(g, to_gpu(t), to_gpu(y)))
    for k in range(2):
        assert rel_l2(got[k], O.filt(y[k], t)) <= 6e-6


@pytest.mark.parametrize("N,V,B", [(8, 7, 20), (16, 9, 64), (24, 7, 65), (32, 12, 250), (130, 9, 500), (40, 8, 1000),
                                   (24, 5, 2048), (24, 5, 4000),
                                   (16, 1230, 30), (16, 620, 60), (24, 308, 128), (24, 308, 200), (24, 307, 520),
                                   (160, 306, 1100)])
@pytest.mark.parametrize("mode", [0, 1])
def test_dual_step_at_every_length(N, V, B, mode):
    P = need_gpu()
    x = synth.ellipse_phantom(N, 6, 3) * (2.0 / N)
    if mode == 0:
        b, w = (f32(a) for a in synth.poisson_data(O.project(x, V, B), 1e4, 5))
        tau = O.default_tau(0, V, float(np.mean(1.0 / w)))
        taps = O.ramp_taps(0, V, B, tau, float(np.mean(1.0 / w)))
    else:
        b, w, tau = f32(O.project(x, V, B)), None, 0.01
        taps = O.ramp_taps(1, V, B, tau, 0.0)
    sigma = 0.1
    g = P.Geometry(N, V, B)
    prm = P.PDTVParams(mode=mode, iters=3, tv_iters=4, beta=0.01, tau=tau, sigma=sigma)
    xg, _ = P.ct_pdtv_solve(g, to_gpu(b), None if w is None else to_gpu(w), prm)
    st, _ = O.pdtv(b, w, taps, mode, 0.01, tau, sigma, 4, 3, N)
    assert rel_l2(to_np(xg), st.x) <= 1e-3
