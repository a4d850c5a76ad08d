"""The plan that FourierLaplace keeps belongs to the node tensor it was made from:
another tensor that comes to lie at the same address, or another view of the same
memory, gets a plan of its own.  Planning is replaced by a recorder (CPU)."""
import pytest

torch = pytest.importorskip("torch")


class _Plan:
    def __init__(self, N, nodes, eps, precision="fp32", q=0):
        self.nodes = nodes.clone()

    def close(self):
        pass


@pytest.fixture
def op(monkeypatch):
    from paper_1606_03255_gb300 import autograd
    monkeypatch.setattr(autograd.fl, "Plan", _Plan)
    return autograd.FourierLaplace(8)


def test_fresh_tensors_each_step(op):
    # the one before is freed first, as where nodes are recomputed from parameters
    for step in range(16):
        w = torch.full((200000, 2), float(step), dtype=torch.float64)
        assert torch.equal(op.plan_for(w).nodes, w)
        del w


def test_views_with_other_strides(op):
    base = torch.arange(16, dtype=torch.float64).reshape(4, 4)
    for w in (base[:2, :2], base.T[:2, :2], base[::2, :2], base[:2, ::2]):
        assert torch.equal(op.plan_for(w).nodes, w)


def test_reused_until_changed(op):
    w = torch.zeros(500, 2, dtype=torch.float64, requires_grad=True)
    first = op.plan_for(w)
    assert op.plan_for(w) is first and op.plan_for(w.detach()) is first
    with torch.no_grad():
        w += 1.0
    assert op.plan_for(w) is not first
