"""A^T of batches: up to the 65535 images that the entry point takes (a grid
past the device's limit goes in several launches), and at sizes where a tile's
base-view slices are shared by fewer blocks than slices, whose count follows
the launch's work.  Neither changes the order of any sum: every image of a
batch has the bits it has alone."""
import numpy as np
import pytest

import oracle as O
from gpu_util import f32, need_gpu, rel_l2, to_np

pytestmark = pytest.mark.gpu


def sinograms(batch, V, B):
    import torch
    return torch.randn(batch, V, B, device="cuda", generator=torch.Generator(device="cuda").manual_seed(batch + B))


@pytest.mark.parametrize("batch", [8191, 8192, 16384, 65535])
@pytest.mark.parametrize("N,V,B,slices", [(16, 40, 25, 0), (16, 40, 24, 8), (10, 14, 17, 7)])
def test_large_batches(N, V, B, slices, batch):
    P = need_gpu()
    import torch
    g = P.Geometry(N, V, B)
    g.set_tuning(orbit_slices=slices)
    y = sinograms(batch, V, B)
    out = P.ct_backproject(g, y)
    for i in sorted({min(i, batch - 1) for i in (0, 1, 8190, 8191, 8192, 9361, 9362, 16383, 65534)}):
        one = P.ct_backproject(g, y[i].clone())
        assert torch.equal(out[i], one)
        assert rel_l2(to_np(one), O.backproject(f32(to_np(y[i])), N)) <= 2e-5


# blocks of slices: 4, 2 and 1 of 8 (14 views: a slice of no base views), 2 and 1 of 4, 1 of 2
@pytest.mark.parametrize("N,V,batch", [(34, 14, 5), (64, 90, 16), (128, 180, 5), (34, 16, 16), (100, 16, 4), (34, 14, 16),
                                       (100, 14, 3), (100, 60, 16), (256, 32, 3), (320, 60, 2), (192, 16, 2),
                                       (256, 60, 4), (512, 60, 2), (34, 90, 64), (96, 60, 16), (192, 60, 4), (34, 180, 128),
                                       (100, 180, 32), (384, 90, 2), (320, 90, 3)])
@pytest.mark.parametrize("wide", [False, True])
def test_blocks_that_share_the_slices(N, V, batch, wide):
    P = need_gpu()
    import torch
    B = 1 + N + N // 2 if wide else N // 4 * 4   # odd and a multiple of 4
    g = P.Geometry(N, V, B)
    y = sinograms(batch, V, B)
    out = P.ct_backproject(g, y)
    for i in range(batch):
        assert torch.equal(out[i], P.ct_backproject(g, y[i].clone()))
    assert rel_l2(to_np(out[batch - 1]), O.backproject(f32(to_np(y[batch - 1])), N)) <= 2e-5 * max(1.0, N / 128.0)
