"""The tile and quadrant adjoints on images of few tiles, whose lists are cut
into parts of whole 32-entry chunks: lists of 0 to a few thousand entries
around the chunk and part edges, more and fewer chunks than parts. Against the
FP64 oracle at the gradients' bar (1e-5 normwise per field)."""
import numpy as np
import pytest

import gs_synthetic as S
import oracle
from _util import absolute, device_gaussians, normwise

pytestmark = pytest.mark.gpu
TILE, QUADRANT = 1, 3


@pytest.mark.parametrize("mode,tile", [(TILE, 8), (TILE, 16), (TILE, 32), (QUADRANT, 16)])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 65, 2047, 2049, 3000])
def test_split_lists(n, mode, tile):
    import torch
    import paper_2501_06838_gb300 as gs
    rng = np.random.default_rng(n)
    w, h = 40, 24
    mu = rng.uniform(0, 1, (n, 2)) * [14, h - 1]   # the right half's tiles stay empty or thin
    g = absolute(mu, rng.uniform(0.3, 1.5, (n, 2)), rng.uniform(-0.9, 0.9, n),
                 rng.uniform(0.1, 1, (n, 3)), rng.uniform(0.1, 1, n), h, w)
    v = S.View(h, w, h, w, 1.0)
    v.adjoint = mode
    go = S.grad_out(n, h, w)
    dg = device_gaussians(g)
    _, ws = gs.render(dg, v, tile=tile, check=True)
    parts = gs.query_layout([dg], [v], ws, tile=tile)["adjoint_parts"]
    assert parts > 1 or n < 2047
    got = gs.render_bwd(dg, v, torch.from_numpy(go).cuda(), ws, tile=tile, check=True)
    err = normwise(got.cpu().double().numpy(), oracle.adjoint(g, v, go), axis=0)
    assert np.all(err < 1e-5), err


@pytest.mark.parametrize("mode,tile,edge,longest,whole", [(TILE, 8, 46, 35, 1), (TILE, 8, 30, 59, 2),
                                                          (TILE, 16, 30, 23, 1), (TILE, 32, 30, 8, 1),
                                                          (QUADRANT, 16, 20, 23, 1)])
def test_short_lists_stay_whole(mode, tile, edge, longest, whole):
    """A part costs a CTA, so short lists are not cut for the chip's sake, or only
    as far as the CTAs are next to free; a larger workspace (whose capacity no
    longer tells the mean length) has them cut, with the same gradients to
    rounding."""
    import torch
    import paper_2501_06838_gb300 as gs
    rng = np.random.default_rng(tile)
    side = edge * tile
    n = edge * edge * longest // 3
    g = absolute(rng.uniform(0, side - 1, (n, 2)), rng.uniform(0.3, 0.6, (n, 2)), rng.uniform(-0.9, 0.9, n),
                 rng.uniform(0.1, 1, (n, 3)), rng.uniform(0.1, 1, n), side, side)
    v = S.View(side, side, side, side, 1.0)
    v.adjoint = mode
    dg, go = device_gaussians(g), torch.from_numpy(S.grad_out(tile, side, side)).cuda()
    pairs = gs.count_pairs([dg], [v], tile=tile)
    assert pairs < edge * edge * longest
    ref = oracle.adjoint(g, v, go.cpu().numpy())
    for capacity in (pairs, 40 * pairs):
        ws = gs.make_workspace([dg], [v], capacity, tile=tile)
        parts = gs.query_layout([dg], [v], ws, tile=tile)["adjoint_parts"]
        assert parts == whole if capacity == pairs else parts > whole
        gs.render(dg, v, ws=ws, tile=tile, check=True)
        got = gs.render_bwd(dg, v, go, ws, tile=tile, check=True).cpu().double().numpy()
        assert np.all(normwise(got, ref, axis=0) < 1e-5)
