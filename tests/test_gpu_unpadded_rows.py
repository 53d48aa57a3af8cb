"""Geometries whose A^T takes no rotation orbits (custom angles, an odd number
of views, an odd side) keep their sinogram rows unpadded inside the library.
The unrolled form's checkpoints then hold rows of any length between fields
that its kernels read in pairs (even sides): batches of one to three slices of
odd rows, each slice against its own run, bit for bit."""
import numpy as np
import pytest

import oracle as O
import synth
from gpu_util import f32, need_gpu, rel_l2, to_gpu, to_np

pytestmark = pytest.mark.gpu

GOLDEN = (5.0 ** 0.5 - 1.0) / 2.0


@pytest.mark.parametrize("N,V,B,custom", [(34, 9, 25, False), (34, 9, 27, True), (34, 10, 25, True), (33, 10, 27, False),
                                          (64, 15, 93, False)])
@pytest.mark.parametrize("S", [1, 2, 3])
def test_unrolled_slices_of_odd_rows(N, V, B, custom, S):
    P = need_gpu()
    import torch
    K, ntv, half, tau, sigma, beta = 3, 6, 8, 1e-4, 0.3, 0.02
    angles = np.mod(np.arange(V) * (np.pi * GOLDEN), np.pi) if custom else None
    g = P.Geometry(N, V, B, angles=angles)
    r = np.random.default_rng(S)
    b = to_gpu(np.stack([O.project(synth.ellipse_phantom(N, 5, s) * (2.0 / N), V, B) for s in range(S)]))
    w, gx = to_gpu(r.uniform(500.0, 2000.0, (S, V, B))), to_gpu(r.standard_normal((S, N, N)))
    taps = to_gpu(O.ramp_taps(0, V, B, tau, 1e-3, half=half))

    def run(b, w, gx):
        n = b.shape[0]
        ws = torch.empty(P.ct_unrolled_workspace_bytes(g, n, half, K, ntv), dtype=torch.uint8, device="cuda")
        ws.fill_(0xFF)
        x = P.ct_unrolled_forward(g, b, w, taps, tau, sigma, beta, 0, K, ntv, ws)
        return x, P.ct_unrolled_backward(g, b, w, taps, tau, sigma, beta, 0, K, ntv, gx, ws)

    x, grad = run(b, w, gx)
    ones = [run(b[s:s + 1].contiguous(), w[s:s + 1].contiguous(), gx[s:s + 1].contiguous()) for s in range(S)]
    for s in range(S):
        assert torch.equal(x[s], ones[s][0][0])
    # the slices' gradients add up (their terms summed in another order)
    total = sum(to_np(o[1]) for o in ones)
    scale = sum(np.abs(to_np(o[1])) for o in ones)
    assert np.all(np.abs(to_np(grad) - total) <= 1e-5 * scale.max())


@pytest.mark.parametrize("B", [25, 26, 27, 28])
def test_solve_on_unpadded_rows(B):
    P = need_gpu()
    N, V, iters, tau, sigma = 34, 9, 3, 1e-4, 0.3
    x = synth.ellipse_phantom(N, 5, 3) * (2.0 / N)
    b, w = (f32(a) for a in synth.poisson_data(O.project(x, V, B), 1e4, 5))
    kappa = float(np.mean(1.0 / w))
    prm = P.PDTVParams(mode=0, iters=iters, tv_iters=4, beta=0.01, tau=tau, sigma=sigma)
    xg, _ = P.ct_pdtv_solve(P.Geometry(N, V, B), to_gpu(b), to_gpu(w), prm)
    st, _ = O.pdtv(b, w, O.ramp_taps(0, V, B, tau, kappa), 0, 0.01, tau, sigma, 4, iters, N)
    assert rel_l2(to_np(xg), st.x) <= 1e-3
