"""The TV prox's tiles at their edges: every count of rows per warp (regions
of up to 16, 32, 48, 64 and 80 rows), images smaller than a tile and one past
a tile's multiple, both prox forms.  The tiling decides only which block holds
a pixel, so every tile height gives the same solve bit for bit; the solve
itself is compared with the FP64 oracle (1e-3 relative, the solves' parity
bar)."""
import numpy as np
import pytest

import oracle as O
import synth
from gpu_util import f32, need_gpu, rel_l2, to_gpu, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fgp", [0, 1])
@pytest.mark.parametrize("N,ntv", [(1, 3), (2, 10), (5, 1), (30, 16), (31, 16), (42, 10), (43, 10), (59, 2), (61, 1),
                                   (100, 5), (131, 10)])
def test_tile_shapes(N, ntv, fgp):
    P = need_gpu()
    V, B, iters, beta, sigma = 12, int(1.44 * N) + 2, 4, 0.3, 0.2
    x = synth.ellipse_phantom(N, 6, 1) * (2.0 / N)
    b, w = (f32(a) for a in synth.poisson_data(O.project(x, V, B), 1e4, 2))
    kappa = float(np.mean(1.0 / w))
    tau = O.default_tau(0, V, kappa)
    prm = P.PDTVParams(mode=0, iters=iters, tv_iters=ntv, beta=beta, tau=tau, sigma=sigma, tv_accel=fgp)
    g = P.Geometry(N, V, B)
    out = []
    for rows in (0, 4, 8, 16, 32, 64):
        g.set_tuning(tv_rows=rows)
        out.append(to_np(P.ct_pdtv_solve(g, to_gpu(b), to_gpu(w), prm)[0]))
    for o in out[1:]:
        assert np.array_equal(o, out[0])
    st, _ = O.pdtv(b, w, O.ramp_taps(0, V, B, tau, kappa), 0, beta, tau, sigma, ntv, iters, N, fgp=bool(fgp))
    assert rel_l2(out[0], st.x) <= 1e-3
