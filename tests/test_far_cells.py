"""Gaussians whose window lies far from their LR cell (a huge scale, offsets that
bring the centres back to the origin), 2^31 HR px and more: grid binning finds
them all, and its lists hold what the footprint pass counted."""
import numpy as np
import pytest

import gs_synthetic as S
from _util import device_gaussians, normwise

pytestmark = pytest.mark.gpu
SORT, GRID = 1, 2
TILE, PAIR = 1, 2


def _scene(scale, lr_w):
    """Every centre within 60 HR px of the origin, whatever its cell."""
    rng = np.random.default_rng(64)
    f32 = lambda a: np.asarray(a, np.float64).astype(np.float32).astype(np.float64)
    j = np.arange(lr_w, dtype=np.float64)
    # j + o is exact in float32 only where o = -j: the cells share one centre
    off = f32(np.stack([-j, rng.uniform(5, 50, lr_w) / scale], 1))
    sig = f32(rng.uniform(2.0, 9.0, (lr_w, 2)) / scale)
    g = S.GaussianSet(off, sig, f32(rng.uniform(-0.8, 0.8, lr_w)), f32(rng.uniform(0.1, 1, (lr_w, 3))),
                      f32(rng.uniform(0.1, 1, lr_w)), lr_h=1, lr_w=lr_w, ref_grid_m=1)
    return g, S.View(1, lr_w, 61, 77, scale, norm=S.NORM_PEAK)


@pytest.mark.parametrize("scale,lr_w", [(1e6, 40), (1.5e8, 14), (1e9, 5), (1e12, 70)])
@pytest.mark.parametrize("tile,batch,raster", [(8, 0, TILE), (8, 64, TILE), (16, 0, TILE), (16, 64, TILE),
                                               (16, 0, PAIR), (32, 0, TILE)])
def test_far_cells(scale, lr_w, tile, batch, raster):
    import torch
    import paper_2501_06838_gb300 as gs
    g, v = _scene(scale, lr_w)
    dg, imgs, grads = device_gaussians(g), [], []
    go = torch.from_numpy(S.grad_out(65, v.out_h, v.out_w)).cuda()
    for v.binning, v.raster in ((SORT, TILE), (GRID, raster)):
        out, ws = gs.render(dg, v, tile=tile, batch=batch, check=True)
        imgs.append(out.cpu().numpy())
        grads.append(gs.render_bwd(dg, v, go, ws, tile=tile, batch=batch, check=True).cpu().double().numpy())
    assert imgs[0].any() and np.array_equal(imgs[0], imgs[1])
    # the same lists: sums of the same terms, in any order of a tile's parts
    assert np.all(normwise(grads[1], grads[0], axis=0) < 1e-5)
