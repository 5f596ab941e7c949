"""Gaussians whose window lies far from their LR cell (a huge scale, offsets that
bring the centres back to the origin): grid binning either finds them or says
that its lists are incomplete; it never returns a wrong image with a clean
status."""
import numpy as np
import pytest

import gs_synthetic as S
from _util import device_gaussians

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
def test_far_cells_found_or_flagged(scale, lr_w, tile, batch, raster):
    import paper_2501_06838_gb300 as gs
    g, v = _scene(scale, lr_w)
    dg = device_gaussians(g)
    v.binning = SORT
    want, _ = gs.render(dg, v, tile=tile, batch=batch, check=True)
    v.binning, v.raster = GRID, raster
    got, ws = gs.render(dg, v, tile=tile, batch=batch)
    try:
        gs.sync_status(ws)
    except gs.GsError as e:
        assert e.status == 6   # GS_ERR_INTERNAL: the lists are not the footprint count's
        return
    assert np.array_equal(got.cpu().numpy(), want.cpu().numpy())
