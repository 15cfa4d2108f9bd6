"""The autograd function around aaqaoa_grad_device, with a stand-in for the plan
that fills its output row on the CPU."""
import pytest

torch = pytest.importorskip("torch")


class RowPlan:
    """E = 3, dE/dgamma = (1, 2), dE/dbeta = (4, 5)."""
    p = 2

    def grad_device(self, g, b, out, observable):
        out.copy_(torch.tensor([3.0, 1.0, 2.0, 4.0, 5.0], dtype=torch.float64))


def _angles():
    return [torch.zeros(2, dtype=torch.float64, requires_grad=True) for _ in range(2)]


def test_gradients_are_tensors_of_their_own():
    from paper_2410_22247_gb300.api import energy
    g, b = _angles()
    (2.0 * energy(g, b, RowPlan())).backward()
    assert g.grad.tolist() == [2.0, 4.0] and b.grad.tolist() == [8.0, 10.0]
    dg, db = torch.autograd.grad(energy(g, b, RowPlan()), [g, b])
    for x, y in ((g.grad, b.grad), (dg, db)):
        assert x.untyped_storage().data_ptr() != y.untyped_storage().data_ptr()
        y.detach_()
        version = y._version
        x.mul_(0.0)
        assert y._version == version and y.abs().sum() > 0
        x.detach_().resize_(8)


def test_gradient_changed_in_place_leaves_the_other_usable():
    from paper_2410_22247_gb300.api import energy
    g, b = _angles()
    dg, db = torch.autograd.grad(energy(g, b, RowPlan()), [g, b])
    w = torch.ones(2, dtype=torch.float64, requires_grad=True)
    loss = (db * w).sum()  # saves db
    dg.mul_(3.0)
    loss.backward()
    assert w.grad.tolist() == [4.0, 5.0]
