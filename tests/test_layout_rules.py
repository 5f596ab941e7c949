"""The library's choice of layout on either side of its lines, by gs_query_layout
(host only, no GPU): pairs of tiles, teams of warps, quadrants or whole tiles
for the adjoint, and its refusals."""
import ctypes

import pytest

import gs_synthetic as S
from paper_2501_06838_gb300 import _abi

TILE, PAIR = 1, 2
QUADRANT, WHOLE = 3, 1


@pytest.fixture(scope="module")
def lib():
    from paper_2501_06838_gb300 import build
    build.build()
    return _abi.load()


def _args(images, **kw):
    """ctypes arrays of (m, lr_h, lr_w, scale) images; the pointers are never read."""
    n = len(images)
    G = (_abi.GsGaussians * n)(*[(1, 1, 1, 1, 1, m * h * w, 0, m, None) for m, h, w, _ in images])
    V = (_abi.GsView * n)()
    for v, (_, h, w, s) in zip(V, images):
        v.lr_h, v.lr_w, v.out_h, v.out_w, v.scale = h, w, S.out_size(h, s), S.out_size(w, s), s
        v.trunc_k = 3.0
        for k, x in kw.items():
            setattr(v, k, x)
    return n, G, V


def layout(lib, images, per_gaussian=4.0, **kw):
    n, G, V = _args(images, **kw)
    ws = lib.gs_workspace_size(n, G, V, int(per_gaussian * sum(g.n for g in G)))
    assert ws > 0, lib.gs_last_error()
    lo = _abi.GsLayout()
    assert lib.gs_query_layout(n, G, V, ws, ctypes.byref(lo)) == 0
    return lo


@pytest.mark.parametrize("images,raster", [
    ([(1, 397, 397, 4.0)], PAIR),            # 100 x 50 = 5,000
    ([(1, 396, 396, 4.0)], TILE),            # 99 x 50 = 4,950
    ([(1, 410, 410, 3.9)], TILE),            # scale below 4
    ([(16, 400, 400, 4.0)], TILE),           # 256 Gaussians per tile: long lists
    ([(1, 77, 77, 10.0)], PAIR),             # 49 x 25 = 1,225 at scale 10
    ([(1, 76, 76, 10.0)], TILE),             # 48 x 24 = 1,152
    ([(16, 77, 77, 10.0)], TILE),            # 39 per tile
    ([(1, 20, 20, 6.0)], TILE),              # one small image
    ([(1, 20, 20, 6.0)] * 4, PAIR),          # a batch of small images, short lists
    ([(1, 20, 20, 5.9)] * 4, TILE),
])
def test_pairs_of_tiles(lib, images, raster):
    lo = layout(lib, images)
    assert lo.raster == raster
    if raster == PAIR:
        assert lo.team == 1


@pytest.mark.parametrize("images,team,kw", [
    ([(1, 40, 40, 4.0)], 8, {}),             # 100 tiles, lists of some 75
    ([(4, 100, 100, 4.0)], 4, {}),           # 625 tiles, 64 per tile
    ([(1, 100, 100, 4.0)], 1, {}),           # 625 tiles, 16 per tile
    ([(4, 120, 120, 4.0)], 1, {}),           # 900 tiles, 64 per tile
    ([(9, 150, 150, 3.0)], 4, {}),           # 841 tiles, 241 per tile
    ([(16, 250, 250, 4.0)], 4, dict(trunc_k=0.02, window=1)),   # lists of 2,900 on 3,969 tiles
    ([(1, 250, 250, 4.0)], 1, dict(trunc_k=0.04, window=1)),    # lists of 600
])
def test_teams_of_warps(lib, images, team, kw):
    lo = layout(lib, images, **kw)
    assert (lo.raster, lo.team) == (TILE, team)
    lo = layout(lib, images, batch=64, **kw)
    assert lo.team == 1


@pytest.mark.parametrize("images,adjoint", [
    ([(4, 150, 150, 9.9)], QUADRANT), ([(4, 150, 150, 10.0)], WHOLE), ([(1, 150, 150, 10.0)], QUADRANT),
    ([(1, 150, 150, 13.9)], QUADRANT), ([(1, 150, 150, 14.0)], WHOLE),
    ([(1, 20, 20, 4.0), (1, 20, 20, 14.0)], WHOLE),
])
def test_quadrants_or_whole_tiles(lib, images, adjoint):
    assert layout(lib, images).adjoint == adjoint
    assert layout(lib, images, trunc_k=0.0).adjoint == WHOLE
    assert layout(lib, images, tile=8).adjoint == WHOLE
    assert layout(lib, images, adjoint=2).adjoint == 2


def test_refusals(lib):
    n, G, V = _args([(1, 20, 20, 4.0)])
    lo, launches = _abi.GsLayout(), lib.gs_launch_count()
    assert lib.gs_query_layout(n, G, V, 1 << 20, None) == _abi.GS_ERR_INVALID
    assert lib.gs_query_layout(n, G, V, 100, ctypes.byref(lo)) == _abi.GS_ERR_INVALID
    assert b"too small" in lib.gs_last_error()
    V[0].tile, V[0].adjoint = 8, QUADRANT
    assert lib.gs_query_layout(n, G, V, 1 << 20, ctypes.byref(lo)) == _abi.GS_ERR_UNSUPPORTED
    assert lib.gs_launch_count() == launches
