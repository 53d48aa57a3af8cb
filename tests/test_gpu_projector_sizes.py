"""The mirrored projector over the sides and angles it serves: bands cut off
by the middle of the image, the middle line of an odd side, custom angles
(views without a mirror view), and the largest sides of each staging form,
against the FP64 oracle; and its forms and batches against one another bit for
bit.

Tolerance: a sample's weight is off by the rounding of its coordinate, at most
about 2^-24 (N + B) pixels, so a ray of random pixels is off by less than that
relative: 2e-5 up to 300 pixels and bins, 2.5e-4 at 4000."""
import numpy as np
import pytest

import oracle as O
import synth
from gpu_util import f32, need_gpu, rel_l2, to_gpu, to_np

pytestmark = pytest.mark.gpu


def angles_of(kind, V):
    if kind == "uniform":
        return None
    return np.mod(np.arange(V) * 1.9416, np.pi)


@pytest.mark.parametrize("kind", ["uniform", "custom"])
@pytest.mark.parametrize("N", [1, 2, 3, 15, 16, 17, 31, 32, 33, 34, 47, 63, 65, 96, 127, 130])
def test_sides(N, kind):
    P = need_gpu()
    import torch
    V, B, batch = 11, int(1.44 * N) + 1, 2
    ang = angles_of(kind, V)
    g = P.Geometry(N, V, B, angles=ang)
    xs = np.stack([f32(synth.random_image(N, 7 + i)) for i in range(batch)])
    xg = to_gpu(xs)
    out = P.ct_project(g, xg)
    for i in range(batch):
        assert rel_l2(to_np(out[i]), O.project(xs[i], V, B, angles=ang)) <= 2e-5
        assert torch.equal(P.ct_project(g, xg[i].clone()), out[i])
    for items, rows, form in [(4, 2, 1), (16, 2, 2), (12, 4, 1), (8, 4, 2)]:
        g.set_tuning(items_per_block=items, proj_rows=rows, proj_form=form)
        assert torch.equal(P.ct_project(g, xg), out)


@pytest.mark.parametrize("N,V,B,kind", [(904, 6, 1301, "uniform"), (905, 6, 1300, "uniform"), (905, 5, 700, "custom"),
                                        (1811, 4, 2600, "uniform"), (1812, 4, 2600, "uniform")])
def test_large_sides(N, V, B, kind):
    # 904: float4 entries; 905 .. 1811: raw pixel pairs; from 1812: unmirrored bands in column passes
    P = need_gpu()
    ang = angles_of(kind, V)
    g = P.Geometry(N, V, B, angles=ang)
    x = f32(synth.random_image(N, 3))
    assert rel_l2(to_np(P.ct_project(g, to_gpu(x))), O.project(x, V, B, angles=ang)) <= 2.5e-4


@pytest.mark.parametrize("N,V,B", [(47, 20, 70), (130, 40, 189), (905, 6, 1301)])
def test_solve_on_ragged_sides(N, V, B):
    # the band sums feed the dual step: a low-dose solve at the solves' parity bar
    P = need_gpu()
    x = synth.ellipse_phantom(N, 6, 1) * (2.0 / N)
    b, w = (f32(a) for a in synth.poisson_data(O.project(x, V, B), 1e4, 2))
    kappa = float(np.mean(1.0 / w))
    tau = O.default_tau(0, V, kappa)
    prm = P.PDTVParams(mode=0, iters=3, tv_iters=5, beta=0.01, tau=tau, sigma=0.05)
    xg, _ = P.ct_pdtv_solve(P.Geometry(N, V, B), to_gpu(b), to_gpu(w), prm)
    st, _ = O.pdtv(b, w, O.ramp_taps(0, V, B, tau, kappa), 0, 0.01, tau, 0.05, 5, 3, N)
    assert rel_l2(to_np(xg), st.x) <= 1e-3


@pytest.mark.parametrize("kind", ["uniform", "custom"])
@pytest.mark.parametrize("N,V,B,batch", [(1, 1, 1, 1), (5, 4, 9, 3), (17, 7, 24, 1), (32, 12, 47, 2), (33, 6, 340, 1),
                                         (64, 90, 95, 1), (64, 11, 96, 40), (65, 10, 93, 1), (96, 8, 139, 2),
                                         (96, 9, 341, 1)])
def test_small_images_in_one_launch(N, V, B, batch, kind):
    # up to three band pairs: ct_project adds the band sums itself, in band order, to the same bits (one launch, or
    # two past the sizes that a block or the batch allows)
    P = need_gpu()
    import torch
    ang = angles_of(kind, V)
    g = P.Geometry(N, V, B, angles=ang)
    xg = to_gpu(np.stack([f32(synth.random_image(N, 5 + i)) for i in range(batch)]))
    parts = P.ct_project_bands(g, xg)
    t = np.arange(V) * np.pi / V if ang is None else ang
    rows = (4 * np.arange(V) <= V) | (4 * np.arange(V) >= 3 * V) if ang is None else np.abs(np.cos(t)) >= np.abs(np.sin(t))
    scale = to_gpu(np.abs(1.0 / np.where(rows, np.cos(t), np.sin(t))))[:, None]
    acc = torch.zeros_like(parts[:, 0])
    for k in range(parts.shape[1]):
        acc = acc + parts[:, k]
    assert torch.equal(P.ct_project(g, xg), acc * scale)
