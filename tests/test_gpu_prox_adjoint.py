"""The adjoint of the TV prox, several steps per launch: one unrolled
iteration's gradients against automatic differentiation in FP64, at the edges
of its tiles (52 columns for five steps, 56 for three) and of its chunks."""
import numpy as np
import pytest

import oracle as O
import synth
from gpu_util import f32, need_gpu, to_gpu, to_np

torch = pytest.importorskip("torch")


def reference(bs, taps, tau, sigma, beta, ntv, N, gx):
    """(dL/dtaps, dL/dbeta, rms of the pixels' shares of the latter) for
    L = <gx, x_1>, x_1 = prox of z = tau sigma A^T D b, in FP64."""
    V, B = bs.shape[1:]
    half, lam0 = (taps.size + 1) // 2, tau * beta
    gt, gl = np.zeros(taps.size), []
    for s in range(bs.shape[0]):
        z = torch.tensor(tau * sigma * O.backproject(O.filt(bs[s], taps), N), requires_grad=True)
        lam = torch.full((N, N), lam0, dtype=torch.float64, requires_grad=True)   # each pixel's lambda
        px = torch.zeros(N, N, dtype=torch.float64)
        py = px.clone()

        def x_of(px, py):
            mx = torch.cat([px[:, :-1], px.new_zeros(N, 1)], 1)
            my = torch.cat([py[:-1], py.new_zeros(1, N)], 0)
            d = mx - torch.nn.functional.pad(mx, (1, 0))[:, :-1] + my - torch.nn.functional.pad(my, (0, 0, 1, 0))[:-1]
            return torch.relu(z + lam * d)

        for _ in range(ntv):
            x = x_of(px, py)
            gxx = torch.cat([x[:, 1:] - x[:, :-1], x.new_zeros(N, 1)], 1)
            gyy = torch.cat([x[1:] - x[:-1], x.new_zeros(1, N)], 0)
            qx, qy = px + gxx / (8 * lam), py + gyy / (8 * lam)
            m = torch.sqrt(torch.clamp(qx * qx + qy * qy, min=1.0))
            px, py = qx / m, qy / m
        (x_of(px, py) * torch.from_numpy(gx[s])).sum().backward()
        gl.append(lam.grad.numpy())
        g = tau * sigma * O.project(z.grad.numpy(), V, B)
        for j in range(taps.size):
            e = np.zeros(taps.size)
            e[j] = 1.0
            gt[j] += (g * O.filt(bs[s], e)).sum()
    gl = np.stack(gl) * tau
    return gt, gl.sum(), np.sqrt((gl ** 2).mean())


def case(N, S, V=24):
    B = int(np.ceil(1.5 * N)) | 1
    bs = np.stack([f32(O.project(synth.ellipse_phantom(N, 5, s) * (2.0 / N), V, B)) for s in range(S)])
    tau = O.default_tau(0, V, 1.0)
    taps = f32(O.ramp_taps(0, V, B, tau, 1.0, half=min(4, B)))
    return bs, taps, tau


def test_reference_matches_oracle_differences():
    N, S, ntv, sigma, beta = 20, 1, 4, 0.5, 0.02
    bs, taps, tau = case(N, S)
    gx = np.random.default_rng(1).standard_normal((S, N, N))

    def loss(tp, be):
        z = tau * sigma * O.backproject(O.filt(bs[0], tp), N)
        return float((O.tv_prox(z, tau * be, ntv)[0] * gx[0]).sum())

    gt, gb, _ = reference(bs, taps, tau, sigma, beta, ntv, N, gx)
    h = 1e-6 * beta
    assert gb == pytest.approx((loss(taps, beta + h) - loss(taps, beta - h)) / (2 * h), rel=1e-5)
    d = np.random.default_rng(2).standard_normal(taps.size) * np.abs(taps).max() * 1e-6
    assert gt @ d == pytest.approx((loss(taps + d, beta) - loss(taps - d, beta)) / 2, rel=1e-5)


@pytest.mark.gpu
@pytest.mark.parametrize("N,S,ntv", [
    (2, 3, 5), (5, 1, 2),        # smaller than a warp's columns
    (52, 2, 5), (53, 1, 10),     # one column tile exactly; one more, odd (pairs not aligned)
    (57, 2, 6), (104, 1, 5),     # 3 + 3 steps: 56 columns; two tiles exactly
    (168, 3, 11),                # 4 + 4 + 3 steps; tiles inside the image
    (161, 1, 1), (224, 9, 5),    # a single step; many blocks: the most rows per warp
])
def test_prox_adjoint(N, S, ntv):
    # Bound: the prox's adjoint jumps where |q| = 1 or s = 0, so FP32 rounding
    # may move single pixels' shares by their own size; six pixels of the rms
    # are allowed (rounding itself: 1e-6 N of one).  A wrong or missing halo
    # line would change N pixels, sqrt(N) of the rms each step, or more.
    P = need_gpu()
    bs, taps, tau = case(N, S)
    sigma, beta = 0.5, 0.02
    gx = f32(np.random.default_rng(N).standard_normal((S, N, N)))
    gt, gb, rms = reference(bs, taps, tau, sigma, beta, ntv, N, gx)
    V, B = bs.shape[1:]
    g = P.Geometry(N, V, B)
    half = (taps.size + 1) // 2
    wsp = torch.empty(P.ct_unrolled_workspace_bytes(g, S, half, 1, ntv), dtype=torch.uint8, device="cuda")
    ws = to_gpu(np.ones_like(bs))
    args = (g, to_gpu(bs), ws, to_gpu(taps), tau, sigma, beta, 0, 1, ntv)
    P.ct_unrolled_forward(*args, wsp)
    out = to_np(P.ct_unrolled_backward(*args, to_gpu(gx), wsp))
    # six pixels out of the N^2 S whose random shares make up the norm of dL/dtaps
    # (images of a few pixels: no kink is met, 1e-2 is far above rounding)
    bound = 6.0 / N / np.sqrt(S) if N > 8 else 1e-2
    assert np.linalg.norm(out[:-1] - gt) <= bound * np.linalg.norm(gt)
    assert abs(out[-1] - gb) <= 6.0 * rms
