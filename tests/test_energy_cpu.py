"""What the differentiable energy asks its handle for and keeps: the potentials only
where a charge gradient is wanted, nothing at all without gradients."""
import pytest


class _Handle:
    """Stands in for RBE: E = sum of charges, F and phi recognisable."""

    def __init__(self, torch):
        self.torch, self.asked = torch, []

    def forces(self, pos_q, step, energy=True, phi=False):
        t = self.torch
        self.asked.append(phi)
        n = pos_q.shape[0]
        F = t.arange(4.0 * n).reshape(n, 4)
        return F, t.ones((1, 4), dtype=t.float64), (t.arange(1.0 * n) + 0.5 if phi else None)


@pytest.mark.parametrize("wpos,wq", [(True, True), (True, False), (False, True), (False, False)])
def test_asks_for_what_is_differentiated(wpos, wq):
    torch = pytest.importorskip("torch")
    from paper_2010_01559_gb300 import RBEEnergy
    h = _Handle(torch)
    pos = torch.zeros((3, 3), requires_grad=wpos)
    q = torch.ones(3, requires_grad=wq)
    with torch.no_grad():
        RBEEnergy.apply(pos, q, h, 0)
    assert h.asked == [False]                    # no gradient can be asked for
    e = RBEEnergy.apply(pos, q, h, 0)
    assert h.asked == [False, wq] and e.requires_grad == (wpos or wq)
    if not (wpos or wq):
        return
    kept = [t for t in e.grad_fn.saved_tensors if t is not None]
    # the inputs, F with positions and phi with charges
    assert sum(t.numel() for t in kept) <= 12 + (12 if wpos else 0) + (3 if wq else 0)
    (2.0 * e).backward()
    F = torch.arange(12.0).reshape(3, 4)[:, :3]
    assert pos.grad is None if not wpos else torch.equal(pos.grad, -2.0 * F)
    assert q.grad is None if not wq else torch.equal(q.grad, 2.0 * (torch.arange(3.0) + 0.5))
    assert len(h.asked) == 2
