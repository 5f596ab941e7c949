"""The emit pass of sorted binning on both of its loops, chosen per warp by the
size of its Gaussians' tile rectangles (more or fewer than 32 tiles on average):
rectangles around that size, a few huge ones among empty and small ones, and a
last warp that is not full. The pair list gives the same image, bit for bit, as
grid binning's enumeration, and the same number of pairs."""
import numpy as np
import pytest

import gs_synthetic as S
from _util import device_gaussians

pytestmark = pytest.mark.gpu
SORT, GRID = 1, 2


def _sigmas(kind, n, rng):
    if kind == "around":      # windows of 24 to 60 px: 9 to 72 tiles of 8 px
        return rng.uniform(4.0, 10.0, (n, 2))
    if kind == "wide":        # most of the image
        return rng.uniform(40.0, 90.0, (n, 2))
    s = rng.uniform(0.3, 2.0, (n, 2))          # "mixed": one in nine is huge
    s[::9] = rng.uniform(60.0, 90.0, (len(s[::9]), 2))
    return s


@pytest.mark.parametrize("kind", ["around", "wide", "mixed"])
@pytest.mark.parametrize("h,w", [(1, 1), (1, 33), (17, 15), (20, 27)])
def test_emit_equals_enumeration(kind, h, w):
    import paper_2501_06838_gb300 as gs
    rng = np.random.default_rng(len(kind) + h * w)
    f32 = lambda a: np.asarray(a, np.float64).astype(np.float32).astype(np.float64)
    scale, n = 256.0 / max(h, w), h * w
    off = rng.uniform(-0.5, 0.5, (n, 2))
    off[3::7] += 1e4          # off the image: no pairs
    g = S.GaussianSet(f32(off), f32(_sigmas(kind, n, rng) / scale), f32(rng.uniform(-0.9, 0.9, n)),
                      f32(rng.uniform(0.1, 1, (n, 3))), f32(rng.uniform(0.1, 1, n)), lr_h=h, lr_w=w,
                      ref_grid_m=1)
    v = S.View(h, w, S.out_size(h, scale), S.out_size(w, scale), scale, norm=S.NORM_PEAK)
    dg, imgs, pairs = device_gaussians(g), [], []
    for v.binning in (SORT, GRID):
        out, ws = gs.render(dg, v, tile=8, check=True)
        imgs.append(out.cpu().numpy())
        pairs.append(gs.read_stats(ws)["tile_pairs"])
    assert pairs[0] == pairs[1] and np.array_equal(imgs[0], imgs[1])
