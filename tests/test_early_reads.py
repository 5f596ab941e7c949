"""The footprint pass and the chain rule of one small image read parameters
before they wait for the kernel before them in the chain. Parameters, upstream
gradient and moments written by kernels still queued on the stream must be the
ones used: the same bits as when every step is waited for. Sizes: one block, a
few, and either side of the number of Gaussians whose blocks are all resident."""
import pytest

import gs_synthetic as S
from _util import device_gaussians

pytestmark = pytest.mark.gpu
GAUSSIAN, SORT, GRID = 2, 1, 2


@pytest.mark.parametrize("h,w,scale", [(7, 9, 3.0), (40, 41, 4.0), (456, 512, 1.5), (457, 512, 1.5)])
@pytest.mark.parametrize("binning", [SORT, GRID])
def test_queued_writes_are_seen(h, w, scale, binning):
    import torch
    import paper_2501_06838_gb300 as gs
    g = S.draw_gaussians(h, h, w, 1, (0.3, 1.2))
    v = S.View(h, w, S.out_size(h, scale), S.out_size(w, scale), scale)
    v.binning, v.adjoint = binning, GAUSSIAN   # no atomics: bitwise reproducible
    dg = device_gaussians(g)
    first = [t.clone() for t in dg.tensors()]
    go = torch.from_numpy(S.grad_out(3, v.out_h, v.out_w)).cuda()

    def steps(wait):
        got = []
        for t, f in zip(dg.tensors(), first):
            t.copy_(f)
        g2 = go.clone()
        _, ws = gs.render(dg, v)
        torch.cuda.synchronize()
        for _ in range(6):
            if not wait:
                torch.cuda._sleep(200000)     # the launches below queue up behind this
            dg.sigma.mul_(0.97)
            dg.rgb.mul_(0.97)
            dg.offset.mul_(0.9)
            if wait:
                torch.cuda.synchronize()
            out, _ = gs.render(dg, v, ws=ws)
            if wait:
                torch.cuda.synchronize()
            g2.mul_(0.95)
            gr = gs.render_bwd(dg, v, g2, ws)
            got += [out.clone(), gr.clone()]
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        return got

    for a, b in zip(steps(False), steps(True)):
        assert torch.equal(a, b)
