"""GSRenderBatched's `sizes`: the rows of the concatenated parameters that belong to
each image, as slices take them (a last image shorter than its size, unused
rows at the end, any integer type, any iterable)."""
import importlib

import numpy as np
import pytest
import torch

import gs_synthetic as S

R = importlib.import_module("paper_2501_06838_gb300.render")


@pytest.mark.parametrize("sizes", [[5, 7], [5, 6], [5, 10], [0, 12], [12, 3], [20, 4], [], [3, -1, 4],
                                   np.array([5, 7]), torch.tensor([4, 4, 4]), (n for n in (6, 6))])
def test_cut_is_slicing(sizes):
    ts = [torch.arange(24.0).view(12, 2), torch.arange(12.0)]
    sizes = list(sizes)
    got, o = R._cut(ts, iter(sizes)), 0
    assert [len(g) for g in got] == [len(sizes)] * 2
    for i, n in enumerate(sizes):
        for t, g in zip(ts, got):
            want = t[o:o + n]
            assert torch.equal(g[i], want) and g[i].is_contiguous() == want.is_contiguous()
        o += n
    with pytest.raises(TypeError):
        R._cut(ts, [2.0])


@pytest.mark.gpu
def test_last_image_shorter_than_its_size():
    """Absolute centres: the last image takes the rows there are, and its
    gradients come back in the tensors' shapes."""
    import paper_2501_06838_gb300 as gs
    rng = np.random.default_rng(3)
    f = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")
    n = 50
    ts = [f(rng.uniform(0, 20, (n, 2))), f(rng.uniform(0.5, 2, (n, 2))), f(rng.uniform(-0.8, 0.8, n)),
          f(rng.uniform(0.1, 1, (n, 3))), f(rng.uniform(0.1, 1, n))]
    views = [gs.View(20, 20, 60, 60, 3.0), gs.View(20, 22, 40, 44, 2.0)]
    gos = [f(S.grad_out(i, v.out_h, v.out_w)) for i, v in enumerate(views)]
    res = []
    for sizes in ([30, 20], np.array([30, 1000])):
        leaves = [t.clone().requires_grad_() for t in ts]
        outs = gs.GSRenderBatched.apply(views, 0, sizes, None, *leaves)
        res.append((outs, torch.autograd.grad(outs, leaves, gos)))
    for a, b in zip(*[r[0] for r in res]):
        assert torch.equal(a, b)
    for a, b, t in zip(res[0][1], res[1][1], ts):
        assert a.shape == b.shape == t.shape
        assert torch.allclose(a, b, rtol=1e-4, atol=1e-5)
