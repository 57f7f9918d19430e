"""Particle states on the host: arrays whose views are made late are those of
the buffer that the state was made with (no GPU)."""
import copy

import pytest

torch = pytest.importorskip("torch")


def test_arrays_keep_their_buffer():
    from paper_1807_01341_gb300 import sim
    p = sim.Particles(7, device="cpu")
    base, size = p.storage.data_ptr(), p.storage.numel()
    p.x.fill_(1.0)
    first = p.struct().x
    p.storage = torch.zeros_like(p.storage)  # the user's attribute: the arrays stay
    p.m = p.m.clone()                        # (drops the cached structure)
    assert p.struct().x == first
    for name, t in p.arrays().items():
        if name != "m":
            assert base <= t.data_ptr() < base + size, name
    assert p.struct().vy == p.vy.data_ptr()
    p.storage = None
    assert p.curl_v.numel() == 7


def test_absent_arrays_and_copies():
    from paper_1807_01341_gb300 import sim
    p = sim.Particles(5, device="cpu", with_counts=False, with_gradients=False)
    assert p.ngb_density is None and p.div_v is None
    assert not hasattr(p, "nothing")
    q = copy.deepcopy(p)
    assert p.struct().ngb_force is None
    q.h.fill_(3.0)
    assert float(p.h.sum()) == 0.0 and float(q.h.sum()) == 15.0


@pytest.mark.parametrize("mode", [torch.inference_mode, torch.no_grad])
def test_first_use_inside_a_mode(mode):
    """An array first asked for inside inference mode is an ordinary tensor."""
    from paper_1807_01341_gb300 import sim
    p = sim.Particles(6, device="cpu")
    with mode():
        assert float(p.h.sum()) == 0.0
        p.x.fill_(2.0)
    assert not p.h.is_inference()
    p.h.copy_(torch.ones(6))
    p.x[0] = 5.0
    w = torch.ones(6, requires_grad=True)
    (p.h * w).sum().backward()
    assert torch.equal(w.grad, p.h) and float(p.x.sum()) == 15.0
