"""gs_count_pairs' own counting kernel against the pairs a render emits and
against the window areas, for every storage type, reference grid, window,
alignment and a fused head, a band and a batch; and its device status."""
import ctypes

import numpy as np
import pytest

import gs_synthetic as S
from _util import device_gaussians

pytestmark = pytest.mark.gpu
SORT, GRID = 1, 2

CASES = {
    "f32_m1": (S.draw_gaussians(1, 37, 53, 1, (0.3, 2.0)), dict(scale=2.7)),
    "bf16_m4": (S.draw_gaussians(2, 16, 20, 4, (0.2, 3.0), dtype="bf16"), dict(scale=9.5)),
    "f16_m9_half": (S.draw_gaussians(3, 20, 24, 9, (0.2, 1.5), dtype="f16"), dict(scale=3.05, align=S.ALIGN_HALF)),
    "m16_ratio": (S.draw_gaussians(4, 12, 14, 16, (0.2, 3.0)), dict(scale=4.0, trunc_k=0.1, window=S.WINDOW_RATIO)),
    "whole": (S.draw_gaussians(5, 12, 10, 1, (0.3, 2.0)), dict(scale=3.5, trunc_k=0.0)),
    "head": (S.draw_raw_head(6, 18, 22, 4, S.Head(0.2, 2.8, 0.9, 1.0, 1), dtype="bf16"), dict(scale=3.3)),
}


def _view(g, scale, **kw):
    return S.View(g.lr_h, g.lr_w, S.out_size(g.lr_h, scale), S.out_size(g.lr_w, scale), scale, **kw)


@pytest.mark.parametrize("case", sorted(CASES))
@pytest.mark.parametrize("tile", [8, 16, 32])
def test_count_equals_render(case, tile):
    import paper_2501_06838_gb300 as gs
    g, kw = CASES[case]
    dg, v = device_gaussians(g), _view(g, **kw)
    n = gs.count_pairs([dg], [v], tile=tile)
    for binning in (SORT, GRID):
        v.binning = binning
        _, ws = gs.render(dg, v, tile=tile, check=True)
        assert gs.read_stats(ws)["tile_pairs"] == n


def test_count_batch_band_and_status():
    import importlib
    import paper_2501_06838_gb300 as gs
    R = importlib.import_module("paper_2501_06838_gb300.render")
    abi = importlib.import_module("paper_2501_06838_gb300._abi")
    names = sorted(CASES)
    dgs = [device_gaussians(CASES[k][0]) for k in names]
    views = [_view(CASES[k][0], **CASES[k][1]) for k in names]
    assert gs.count_pairs(dgs, views) == sum(gs.count_pairs([d], [v]) for d, v in zip(dgs, views))
    band = S.View(views[0].lr_h, views[0].lr_w, 16, views[0].out_w, views[0].scale)
    band.row0 = 16
    _, ws = gs.render(dgs[0], band, check=True)
    assert gs.count_pairs([dgs[0]], [band]) == gs.read_stats(ws)["tile_pairs"]
    # the workspace keeps the counters and, with no room for the pairs, says so
    n, G, V = R._arrays([dgs[1]], [views[1]])
    small = gs.Workspace(gs.workspace_bytes([dgs[1]], [views[1]], 0))
    got = ctypes.c_int64(0)
    assert abi.load().gs_count_pairs(n, G, V, small.ptr, small.nbytes, R._stream(), ctypes.byref(got)) == 0
    st = gs.read_stats(small)
    _, ws = gs.render(dgs[1], views[1], check=True)
    full = gs.read_stats(ws)
    assert st["tile_pairs"] == got.value == full["tile_pairs"] and st["pixel_pairs"] == full["pixel_pairs"]
    with pytest.raises(gs.GsError) as ei:
        gs.sync_status(small)
    assert ei.value.status == 2
    # an invalid parameter is the count's error
    bad = CASES["f32_m1"][0].with_dtype("f32")
    bad.sigma = bad.sigma.copy()
    bad.sigma[7, 0] = -1.0
    with pytest.raises(gs.GsError) as ei:
        gs.count_pairs([device_gaussians(bad)], [views[names.index("f32_m1")]])
    assert ei.value.status == 1


def test_count_is_timed_as_itself():
    """Per-kernel times: the counting pass under its own name, not the footprint pass's."""
    import paper_2501_06838_gb300 as gs
    g, kw = CASES["f32_m1"]
    dg, v = device_gaussians(g), _view(g, **kw)
    gs.timing_read()
    gs.timing_enable()
    try:
        gs.count_pairs([dg], [v])
        counted = gs.timing_read()
        gs.render(dg, v, check=True)   # counts, then renders
        rendered = gs.timing_read()
    finally:
        gs.timing_enable([])
    assert {k: n for k, (_, n) in counted.items()} == {"setup": 1, "count": 1}
    assert {k: n for k, (_, n) in rendered.items()} == {"setup": 2, "count": 1, "preprocess": 1, "raster_fwd": 1}
