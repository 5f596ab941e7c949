"""The tile-16 forward, which walks a tile in strips of a few columns, at the
sizes where its batches, strips and stores have edges: 0 to 65 Gaussians in a
tile (batches of 32), windows that meet only some strips, widths around
multiples of 4 and 16, and an output that is not 16-byte aligned. Against the
FP64 oracle at the forward's bar (1e-5 normwise per channel)."""
import numpy as np
import pytest

import gs_synthetic as S
import oracle
from _util import absolute, device_gaussians, normwise

pytestmark = pytest.mark.gpu


def _scene(n, w, h, sig, seed):
    rng = np.random.default_rng(seed)
    mu = rng.uniform(0, 1, (n, 2)) * [w - 1, h - 1]
    return absolute(mu, rng.uniform(*sig, (n, 2)), rng.uniform(-0.9, 0.9, n),
                    rng.uniform(0.1, 1, (n, 3)), rng.uniform(0.1, 1, n), h, w)


@pytest.mark.parametrize("n", [0, 1, 2, 31, 32, 33, 63, 64, 65])
@pytest.mark.parametrize("batch", [0, 64])
def test_strip_batches(n, batch):
    import paper_2501_06838_gb300 as gs
    g = _scene(n, 16, 16, (0.2, 1.5), n)
    v = S.View(16, 16, 16, 16, 1.0)
    out, _ = gs.render(device_gaussians(g), v, batch=batch, check=True)
    ref = oracle.render(g, v)
    assert np.all(normwise(out.cpu().double().numpy(), ref, axis=(1, 2)) < 1e-5)


@pytest.mark.parametrize("w", [1, 3, 4, 5, 15, 16, 17, 18, 20, 31, 33, 36])
@pytest.mark.parametrize("offset", [0, 1])
def test_strip_columns_and_stores(w, offset):
    import torch
    import paper_2501_06838_gb300 as gs
    h = 19
    g = _scene(70, w, h, (0.15, 0.8), w)
    v = S.View(h, w, h, w, 1.0)
    buf = torch.full((offset + 3 * h * w + 8,), -7.0, device="cuda")
    out = buf[offset:offset + 3 * h * w].view(3, h, w)
    gs.render(device_gaussians(g), v, out=out, check=True)
    ref = oracle.render(g, v)
    assert np.all(normwise(out.cpu().double().numpy(), ref, axis=(1, 2)) < 1e-5)
    assert torch.all(buf[:offset] == -7.0) and torch.all(buf[offset + 3 * h * w:] == -7.0)


@pytest.mark.parametrize("w", [1, 4, 15, 16, 17, 20, 31, 32, 33, 47, 48, 50, 64])
@pytest.mark.parametrize("offset", [0, 1])
def test_pair_stores(w, offset):
    """Pairs of tiles go out in rows: the one-tile layout's bits, and nothing
    outside the image."""
    import torch
    import paper_2501_06838_gb300 as gs
    h = 21
    g = S.draw_gaussians(w, h, w, 4, (0.2, 2.0))
    v = S.View(h, w, h, w, 1.0)
    dg = device_gaussians(g)
    v.binning, v.raster = 2, 1
    want, _ = gs.render(dg, v, check=True)
    buf = torch.full((offset + 3 * h * w + 8,), -7.0, device="cuda")
    out = buf[offset:offset + 3 * h * w].view(3, h, w)
    v.raster = 2
    _, ws = gs.render(dg, v, out=out, check=True)
    assert gs.read_stats(ws)["raster"] == 2
    assert torch.equal(out, want)
    assert torch.all(buf[:offset] == -7.0) and torch.all(buf[offset + 3 * h * w:] == -7.0)
