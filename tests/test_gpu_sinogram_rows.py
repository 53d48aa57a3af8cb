"""A^T on detectors of every length mod 4 (its input's rows are padded to whole
16-byte pieces, views v and v + V/2 interleaved), from ones narrower than a staged window to past the
diagonal, against the FP64 oracle, and the solves that write padded rows: the
paper's D, the shift-variant D, the few-view forms and the direct convolution
above 4096 bins.

Tolerance of A^T: a weight is off by the rounding of its detector coordinate,
at most 2^-24 (N + B) bins, so a pixel's sum of random rows is off by less
than 2e-5 of its norm up to 300 pixels and bins."""
import numpy as np
import pytest

import oracle as O
import synth
from gpu_util import f32, need_gpu, rel_l2, to_gpu, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 2, 3, 4, 5, 29, 30, 31, 33, 34, 35, 93, 94, 95, 97, 139])
@pytest.mark.parametrize("N,V", [(2, 4), (34, 10), (64, 18)])
def test_backproject_rows(N, V, B):
    P = need_gpu()
    import torch
    g = P.Geometry(N, V, B)
    ys = np.stack([f32(synth.random_sinogram(V, B, s)) for s in (1, 2, 3)])
    yg = to_gpu(ys)
    out = P.ct_backproject(g, yg)
    for i in range(3):
        assert rel_l2(to_np(out[i]), O.backproject(ys[i], N)) <= 2e-5
        assert torch.equal(P.ct_backproject(g, yg[i].clone()), out[i])


@pytest.mark.parametrize("B", [1, 2, 3, 4, 30, 33, 35, 94, 95, 96, 97])
@pytest.mark.parametrize("N,V", [(34, 10), (64, 18)])   # odd V/2: a transform's two views lie in different halves
def test_interleaved_rows_equal_plain_rows(N, V, B):
    # a batch of more than 2.5e6 pixel views is interleaved first, one image is not: the same bits
    P = need_gpu()
    import torch
    g = P.Geometry(N, V, B)
    batch = int(2.5e6 / (N * N * V)) + 2
    gen = torch.Generator(device="cuda").manual_seed(B)
    y = torch.randn(batch, V, B, device="cuda", generator=gen)
    out = P.ct_backproject(g, y)
    for i in (0, 1, batch // 2, batch - 1):
        assert torch.equal(P.ct_backproject(g, y[i].clone()), out[i])


@pytest.mark.parametrize("B", [70, 71, 72, 73, 4201])
@pytest.mark.parametrize("mode,precond,eps", [(0, 1, 0.0), (0, 2, 0.0), (1, 1, 0.0), (1, 3, 0.0), (1, 0, 0.05), (1, 1, 0.05)])
def test_solves_on_padded_rows(B, mode, precond, eps):
    if B > 4096 and (precond == 2 or eps > 0.0):
        pytest.skip("these forms need n_bins <= 4096")
    P = need_gpu()
    N, V, iters, sigma = 24, 8, 3, 0.05
    x = synth.ellipse_phantom(N, 5, 3) * (2.0 / N)
    kappa, w, s, taps_hi = 0.0, None, None, None
    if mode == 0:
        b, w = (f32(a) for a in synth.poisson_data(O.project(x, V, B), 1e4, 5))
        kappa = float(np.mean(1.0 / w))
        tau = O.default_tau(0, V, kappa)
    else:
        b, tau = f32(O.project(x, V, B)), 0.01
        if precond == 3:
            kappa = tau * O.fewview_ell(N, V, B)
    if precond == 2:
        taps, taps_hi, s = O.ramp_taps(2, V, B, tau, kappa), O.ramp_taps(3, V, B, tau, kappa), np.sqrt(kappa * w)
    elif precond:
        taps = O.ramp_taps(0 if kappa else 1, V, B, tau, kappa)
    else:
        taps = np.ones(1)
    prm = P.PDTVParams(mode=mode, iters=iters, tv_iters=4, beta=0.01, tau=tau, sigma=sigma, precond=precond, eps=eps)
    xg, _ = P.ct_pdtv_solve(P.Geometry(N, V, B), to_gpu(b), None if w is None else to_gpu(w), prm)
    st, _ = O.pdtv(b, w, taps, mode, 0.01, tau, sigma, 4, iters, N, taps_hi=taps_hi, s=s, eps=eps)
    assert rel_l2(to_np(xg), st.x) <= 1e-3
