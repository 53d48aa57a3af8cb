"""The step-size setup's Lanczos runs on vectors below, at and above the size
that one launch takes (32768 elements), with whole and ragged 16-byte groups:
the report's norms against numpy's 2-norm of the explicit operators (small) or
against a deeper run of the same estimate, which the default lies within the
estimate's documented -0.25 .. 2.2 % of."""
import numpy as np
import pytest

import oracle as O
import synth
from gpu_util import f32, need_gpu, to_gpu

pytestmark = pytest.mark.gpu


def report(P, N, V, B, norm_iters=0, seed=1):
    x = synth.ellipse_phantom(N, 6, seed) * (2.0 / N)
    b, w = (f32(a) for a in synth.poisson_data(O.project(x, V, B), 1e4, 2))
    prm = P.PDTVParams(mode=0, iters=1, tv_iters=2, beta=0.01, norm_iters=norm_iters)
    _, rep = P.ct_pdtv_solve(P.Geometry(N, V, B), to_gpu(b), to_gpu(w), prm)
    return rep, w


@pytest.mark.parametrize("N,V,B", [(1, 1, 1), (2, 3, 3), (7, 5, 9), (10, 7, 13)])
def test_norms_of_explicit_operators(N, V, B):
    P = need_gpu()
    rep, w = report(P, N, V, B)
    A = np.stack([O.project(np.eye(N * N)[i].reshape(N, N), V, B).ravel() for i in range(N * N)], axis=1)
    taps = O.ramp_taps(0, V, B, rep["tau"], rep["kappa"])
    D = np.stack([O.filt(np.eye(V * B)[i].reshape(V, B), taps).ravel() for i in range(V * B)], axis=1)
    sw = 1.0 / np.sqrt(w.ravel())
    for got, ref in ((rep["norm_ADA"], np.linalg.norm(A.T @ D @ A, 2)),
                     (rep["norm_WDW"], np.linalg.norm(sw[:, None] * D * sw[None, :], 2))):
        assert 0.995 * ref <= got <= 1.03 * ref


@pytest.mark.parametrize("N,V,B", [(64, 90, 95), (128, 32, 185), (180, 60, 260), (181, 60, 261), (182, 181, 181),
                                   (183, 31, 1057)])
def test_norms_across_the_fused_limit(N, V, B):
    # image side N^2 = 4096 .. 33489 and sinogram side 5920 .. 32767: both sides of 32768
    P = need_gpu()
    rep, _ = report(P, N, V, B)
    deep, _ = report(P, N, V, B, norm_iters=64)
    for k in ("norm_ADA", "norm_WDW"):
        assert 0.995 * deep[k] <= rep[k] <= 1.04 * deep[k]
