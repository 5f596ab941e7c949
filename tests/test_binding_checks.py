"""Host-side checks of the binding (no GPU): every caller-supplied buffer is
checked for device, dtype, shape and contiguity before its pointer reaches the
library, which trusts the pointers and sizes it is given; parameters off the
GPU are refused before any library call."""
import importlib

import pytest
import torch

R = importlib.import_module("paper_2501_06838_gb300.render")


def test_buffer_checks():
    cpu = torch.device("cpu")
    t = torch.zeros(3, 4, 5)
    assert R._need(t, (3, 4, 5), torch.float32, cpu, "output") is t
    with pytest.raises(ValueError, match="shape"):
        R._need(t, (3, 5, 4), torch.float32, cpu, "output")
    with pytest.raises(ValueError, match="contiguous"):
        R._need(t.transpose(1, 2).contiguous().transpose(1, 2), (3, 4, 5), torch.float32, cpu,
                "output")
    with pytest.raises(TypeError, match="float32"):
        R._need(t.double(), (3, 4, 5), torch.float32, cpu, "output")
    with pytest.raises(ValueError, match="meta"):
        R._need(t, (3, 4, 5), torch.float32, torch.device("meta"), "output")


def test_parameters_must_be_on_the_gpu():
    n = 4
    g = R.Gaussians(torch.zeros(n, 2), torch.ones(n, 2), torch.zeros(n), torch.zeros(n, 3),
                    torch.zeros(n))
    with pytest.raises(ValueError, match="CUDA"):
        R._device([g])
    with pytest.raises(ValueError, match="CUDA"):
        R._struct_g(g)
    v = R.View(2, 2, 4, 4, 2.0)
    with pytest.raises(ValueError, match="CUDA"):
        R.render(g, v)
    with pytest.raises(ValueError, match="one view per image"):
        R.render_batched([g], [v, v])


def test_heads_made_on_access(monkeypatch):
    """An image whose head is a fresh object every time it is read (a property) gets
    that head, not none and not another image's whose object had the same id."""
    class Head:
        def __init__(self, lo):
            self.sigma_lo, self.sigma_span, self.rho_scale = lo, 1.0, 0.5
            self.offset_scale, self.offset_tanh = 1.0, 0

    class Image:
        def __init__(self, lo):
            self.lo = lo

        @property
        def head(self):
            return None if self.lo is None else Head(self.lo)

    monkeypatch.setattr(R, "_fields_g", lambda g, hp: (1, 1, 1, 1, 1, 4, 0, 1, hp))
    los = [0.125 * i if i % 3 else None for i in range(12)]
    _, G, _ = R._arrays([Image(lo) for lo in los], [R.View(2, 2, 4, 4, 2.0)] * len(los))
    for g, lo in zip(G, los):
        assert bool(g.head) == (lo is not None)
        if lo is not None:
            assert g.head.contents.sigma_lo == lo
    shared = Head(0.75)
    images = [type("Same", (), {"head": shared})() for _ in range(3)]
    _, G, _ = R._arrays(images, [R.View(2, 2, 4, 4, 2.0)] * 3)
    assert len(G._head_keep) == 1 and all(g.head.contents.sigma_lo == 0.75 for g in G)
