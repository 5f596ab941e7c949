"""Block shapes of the deterministic adjoint on reference grids. The shape follows
from the images, their windows and the workspace's pair capacity (which tells
the windows' mean size); every shape sums each Gaussian in one order, so the
gradients are the same bits whatever the capacity, and the oracle's."""
import numpy as np
import pytest

import gs_synthetic as S
import oracle
from _util import device_gaussians, normwise

pytestmark = pytest.mark.gpu
GAUSSIAN = 2
RATIO = S.WINDOW_RATIO

# lr_h, lr_w, m, sigma, view -> blocks with a workspace of the exact pairs, and with much more
CASES = {
    "few_small": (120, 119, 1, (0.2, 2.0), dict(scale=4.0), (8, 8), (8, 8)),
    "few_large": (60, 61, 1, (0.2, 1.0), dict(scale=8.0), (4, 4), (4, 4)),
    "few_dense": (20, 31, 16, (0.2, 1.0), dict(scale=2.0), (4, 2), (4, 2)),
    "many_fit": (152, 155, 1, (0.2, 1.0), dict(scale=3.0), (8, 8), (8, 8)),
    "many_half": (150, 203, 1, (0.2, 2.0), dict(scale=5.0), (8, 4), (8, 8)),
    "many_ratio": (150, 203, 1, (0.2, 2.0), dict(scale=2.0, trunc_k=0.02, window=RATIO), (8, 8), (8, 8)),
    "many_wide": (150, 203, 1, (0.2, 2.0), dict(scale=2.0, trunc_k=0.1, window=RATIO), (8, 4), (8, 4)),
    "many_wider": (150, 203, 1, (0.2, 2.0), dict(scale=4.0, trunc_k=0.05, window=RATIO), (4, 4), (4, 4)),
    "many_dense": (216, 320, 4, (0.2, 0.8), dict(scale=1.5), (8, 4), (8, 4)),
    "many_dense_large": (216, 320, 4, (0.2, 2.0), dict(scale=6.0), (4, 4), (8, 4)),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_blocks_by_capacity(case):
    import torch
    import paper_2501_06838_gb300 as gs
    h, w, m, sigma, kw, exact, ample = CASES[case]
    g, s = S.draw_gaussians(len(case), h, w, m, sigma), kw["scale"]
    v = S.View(h, w, S.out_size(h, s), S.out_size(w, s), **kw)
    v.adjoint = GAUSSIAN
    dg, go = device_gaussians(g), torch.from_numpy(S.grad_out(9, v.out_h, v.out_w)).cuda()
    pairs, got = gs.count_pairs([dg], [v]), []
    for capacity, blocks in ((pairs, exact), (20 * pairs, ample)):
        ws = gs.make_workspace([dg], [v], capacity)
        layout = gs.query_layout([dg], [v], ws)
        assert (layout["block_x"], layout["block_y"]) == blocks
        gs.render(dg, v, ws=ws, check=True)
        got.append(gs.render_bwd(dg, v, go, ws, check=True).cpu().numpy())
    assert np.array_equal(got[0], got[1])
    if g.rho.shape[0] < 50_000:
        err = normwise(got[0], oracle.adjoint(g, v, go.cpu().numpy()), axis=0)
        assert np.all(err < 1e-5), err
