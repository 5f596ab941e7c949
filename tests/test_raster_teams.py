"""The tile-16 forward by teams of warps and the segments a tile's list is
summed in. Long lists (Algorithm 1's window, whole-image windows, dense small
images) make the render take a team per tile; one warp per tile, pairs of
tiles and the sorted list sum the same segments in the same order, so every
route gives the same bits. Against the FP64 oracle at the forward's bar (1e-5
normwise per channel)."""
import numpy as np
import pytest

import gs_synthetic as S
import oracle
from _util import absolute, device_gaussians, normwise

pytestmark = pytest.mark.gpu
SORT, GRID = 1, 2
TILE, PAIR = 1, 2

CASES = {
    # lists of a whole image's Gaussians: one segment to several, ragged tiles
    "whole_512": (16, 8, 4, dict(scale=3.3, trunc_k=0.0)),
    "whole_1040": (13, 5, 16, dict(scale=4.1, trunc_k=0.0)),
    "whole_4608": (18, 16, 16, dict(scale=2.2, trunc_k=0.0)),
    "ratio_few_tiles": (40, 36, 16, dict(scale=2.0, trunc_k=0.2, window=S.WINDOW_RATIO)),
    "ratio_many_tiles": (48, 52, 9, dict(scale=9.3, trunc_k=0.25, window=S.WINDOW_RATIO)),
    "dense_sigma": (30, 34, 16, dict(scale=1.3)),
    "sparse_sigma": (20, 24, 4, dict(scale=4.6)),        # 45 Gaussians per tile: lists below a segment
    "thin_sigma": (24, 24, 1, dict(scale=4.0)),          # 16 per tile, lists of about 75
    "wide_sigma": (11, 14, 4, dict(scale=12.0)),         # 6 per tile, lists of about 130
    "many_tiles_sigma": (112, 113, 9, dict(scale=4.0)),  # 812 tiles, 140 per tile: one warp
    "many_tiles_team": (150, 151, 9, dict(scale=3.0)),   # 841 tiles, 242 per tile: teams again
}
TEAM = {"ratio_many_tiles": 4, "many_tiles_sigma": 1, "many_tiles_team": 4}   # the others: 8 warps


def _scene(case):
    h, w, m, kw = CASES[case]
    g = S.draw_gaussians(sum(map(ord, case)), h, w, m, (0.2, 3.0))
    s = kw["scale"]
    return g, S.View(h, w, S.out_size(h, s), S.out_size(w, s), **kw)


@pytest.mark.parametrize("case", sorted(CASES))
def test_teams_equal_other_layouts(case):
    import torch
    import paper_2501_06838_gb300 as gs
    g, v = _scene(case)
    dg = device_gaussians(g)
    imgs, grads = [], []
    go = torch.from_numpy(S.grad_out(3, v.out_h, v.out_w)).cuda()
    # batch 64: one warp per tile; pairs whose segments may end in the second half of a batch
    for binning, raster, batch in ((GRID, TILE, 0), (SORT, TILE, 0), (GRID, PAIR, 0), (GRID, TILE, 64),
                                   (GRID, PAIR, 64)):
        v.binning, v.raster = binning, raster
        out, ws = gs.render(dg, v, batch=batch, check=True)
        assert gs.read_stats(ws)["raster"] == raster
        layout = gs.query_layout([dg], [v], ws, batch=batch)
        assert layout["raster"] == raster
        assert layout["team"] == (1 if raster == PAIR or batch else TEAM.get(case, 8))
        imgs.append(out.cpu().numpy())
        # the list each route leaves for the adjoint
        grads.append(gs.render_bwd(dg, v, go, ws, batch=batch, check=True).cpu().double().numpy())
    for im in imgs[1:]:
        assert np.array_equal(imgs[0], im)
    assert np.all(normwise(imgs[0].astype(np.float64), oracle.render(g, v), axis=(1, 2)) < 1e-5)
    ref = oracle.adjoint(g, v, go.cpu().numpy())
    for gr in grads:
        assert np.all(normwise(gr, ref, axis=0) < 1e-5)


def test_team_image_alone_and_in_a_batch():
    """An image's bits do not depend on what else is in the batch (which decides
    whether teams run) nor on the pair capacity (a team enumerates its list
    itself when it does not fit)."""
    import paper_2501_06838_gb300 as gs
    g, v = _scene("dense_sigma")   # a team alone, not in the batch
    big = S.draw_gaussians(5, 200, 180, 1, (0.3, 2.0))
    bv = S.View(200, 180, 1000, 900, 5.0)
    dg, db = device_gaussians(g), device_gaussians(big)
    alone, ws = gs.render(dg, v, check=True)
    assert gs.query_layout([dg], [v], ws)["team"] == 8
    (together, _), ws = gs.render_batched([dg, db], [v, bv], check=True)
    assert gs.query_layout([dg, db], [v, bv], ws)["team"] == 1
    assert np.array_equal(alone.cpu().numpy(), together.cpu().numpy())
    for case in ("dense_sigma", "whole_4608"):
        g, v = _scene(case)
        dg = device_gaussians(g)
        want, _ = gs.render(dg, v, check=True)
        v.binning = GRID
        small = gs.Workspace(gs.workspace_bytes([dg], [v], 100))
        got, _ = gs.render(dg, v, ws=small)
        with pytest.raises(gs.GsError) as ei:
            gs.sync_status(small)
        assert ei.value.status == 2   # capacity: the adjoint's lists do not fit
        assert np.array_equal(got.cpu().numpy(), want.cpu().numpy())


@pytest.mark.parametrize("n", [0, 1, 511, 512, 513, 1025])
def test_team_absolute_centres_segment_edges(n):
    """The sorted list at the segments' edges: every Gaussian on one tile."""
    import paper_2501_06838_gb300 as gs
    rng = np.random.default_rng(n)
    g = absolute(rng.uniform(0, 11, (n, 2)), rng.uniform(0.3, 2.0, (n, 2)),
                 rng.uniform(-0.9, 0.9, n), rng.uniform(0.1, 1, (n, 3)), rng.uniform(0.1, 1, n),
                 12, 12)
    v = S.View(12, 12, 12, 12, 1.0)
    out, _ = gs.render(device_gaussians(g), v, check=True)
    err = normwise(out.cpu().double().numpy(), oracle.render(g, v), axis=(1, 2))
    assert np.all(err < 1e-5), err
