"""A^T of sinograms whose rows are whole 16-byte pieces (B % 4 == 0): all but
large ones are read in their own rows, large ones with their row pairs
interleaved first.  The same bits, on detectors from one narrower than a staged
window to past the diagonal."""
import numpy as np
import pytest

import oracle as O
from gpu_util import f32, need_gpu, rel_l2, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [4, 28, 32, 36, 40, 92, 96, 140])
@pytest.mark.parametrize("N,V", [(2, 4), (34, 10), (64, 18), (34, 90)])   # one slice and several; odd and even V/2
def test_own_rows_and_interleaved_rows(N, V, B):
    P = need_gpu()
    import torch
    g = P.Geometry(N, V, B)
    batch = min(int(1.2e8 / (N * N * V)) + 2, 65535)   # past 1.2e8 pixel views (but for the smallest image)
    y = torch.randn(batch, V, B, device="cuda", generator=torch.Generator(device="cuda").manual_seed(B))
    out = P.ct_backproject(g, y)
    for i in (0, 1, batch // 2, batch - 1):
        one = P.ct_backproject(g, y[i].clone())
        assert torch.equal(one, out[i])
        assert rel_l2(to_np(one), O.backproject(f32(to_np(y[i])), N)) <= 2e-5
