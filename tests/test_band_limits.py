"""Row bands at the limits of the 16-bit windows that grid binning keeps: a
band holds at most 32767 rows, wherever in its image they lie. Bands that
straddle image row 32768, that end on it with a last tile reaching past it, or
that lie far below it, in every raster layout, against the sorted list (the
same bits) and the FP64 oracle (1e-5 normwise)."""
import functools

import numpy as np
import pytest

import gs_synthetic as S
import oracle
from _util import device_gaussians, normwise

pytestmark = pytest.mark.gpu
SORT, GRID = 1, 2
TILE, PAIR = 1, 2
BANDS = {"straddles": (32720, 100), "last_tile_past": (32760, 8), "ends_on_it": (32752, 16),
         "below": (32800, 61)}


@functools.lru_cache(None)
def _scene():
    """A column of 33,280 rows; 4 Gaussians per LR pixel."""
    g = S.draw_gaussians(61, 8320, 6, 4, (0.3, 1.5))
    v = S.View(8320, 6, S.out_size(8320, 4.0), S.out_size(6, 4.0), 4.0)
    go = S.grad_out(62, v.out_h, v.out_w)
    return g, v, go, oracle.render(g, v)


@functools.lru_cache(None)
def _adjoint(band):
    g, v, go, _ = _scene()
    r0, n = BANDS[band]
    part = np.zeros_like(go)
    part[:, r0:r0 + n] = go[:, r0:r0 + n]
    return oracle.adjoint(g, v, part)


@pytest.mark.parametrize("band", sorted(BANDS))
@pytest.mark.parametrize("tile,batch,raster", [(8, 0, TILE), (16, 0, TILE), (16, 64, TILE), (16, 0, PAIR),
                                               (32, 0, TILE)])
def test_bands_past_row_32767(band, tile, batch, raster):
    import torch
    import paper_2501_06838_gb300 as gs
    g, whole, go, image = _scene()
    r0, n = BANDS[band]
    v = S.View(whole.lr_h, whole.lr_w, n, whole.out_w, whole.scale)
    v.row0, dg = r0, device_gaussians(g)
    go_band = torch.from_numpy(np.ascontiguousarray(go[:, r0:r0 + n])).cuda()
    imgs = []
    for v.binning, v.raster in ((GRID, raster), (SORT, TILE)):
        out, ws = gs.render(dg, v, tile=tile, batch=batch, check=True)
        imgs.append(out.cpu().numpy())
        gr = gs.render_bwd(dg, v, go_band, ws, tile=tile, batch=batch, check=True)
        err = normwise(gr.cpu().double().numpy(), _adjoint(band), axis=0)
        assert np.all(err < 1e-5), err
    assert np.array_equal(imgs[0], imgs[1])
    assert np.all(normwise(imgs[0], image[:, r0:r0 + n], axis=(1, 2)) < 1e-5)


def test_band_of_four_million_rows():
    """Rows beyond 2^21, where a row's float32 quotient by the scale is no longer
    exact to a pixel: the candidates still hold every Gaussian of the band."""
    import paper_2501_06838_gb300 as gs
    g = S.draw_gaussians(63, 1 << 20, 1, 1, (0.1, 0.4))
    dg = device_gaussians(g)
    for s, r0, n in ((3.999, 4_190_000, 333), (15.99, 16_760_001, 257)):
        v = S.View(1 << 20, 1, n, S.out_size(1, s), s)
        v.row0 = r0
        imgs = []
        for v.binning in (GRID, SORT):
            out, _ = gs.render(dg, v, check=True)
            imgs.append(out.cpu().numpy())
        assert imgs[0].any() and np.array_equal(imgs[0], imgs[1])
