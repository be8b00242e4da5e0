"""The differentiable potential asks for gradients only where autograd records
them (a stand-in for the library call notes what it is asked; no GPU)."""
import numpy as np
import pytest
import torch

from paper_1902_01061_gb300 import scgr


@pytest.fixture
def calls(monkeypatch):
    seen = []

    def fake(handle, pose7, want_grad=True, grad_xyz_out=None):
        seen.append((bool(want_grad), grad_xyz_out is not None))
        if grad_xyz_out is not None:
            grad_xyz_out.fill_(2.0)
        return float(pose7.sum()), (np.arange(7.0) if want_grad else None)

    monkeypatch.setattr(scgr, "scgr_potential", fake)
    return seen


def inputs(pose=False, y=False):
    return (torch.ones(7, dtype=torch.float64, requires_grad=pose),
            torch.ones((5, 3), dtype=torch.float32, requires_grad=y))


@pytest.mark.parametrize("mode", [torch.no_grad, torch.inference_mode])
def test_no_gradient_pass_outside_grad_mode(calls, mode):
    p, y = inputs(pose=True, y=True)
    with mode():
        assert scgr.potential(p, y, None).item() == 7.0
    assert calls == [(False, False)]


def test_no_gradient_pass_without_a_leaf(calls):
    scgr.potential(*inputs(), None)
    assert calls == [(False, False)]


@pytest.mark.parametrize("pose,y", [(True, False), (False, True), (True, True)])
def test_one_call_gives_value_and_gradients(calls, pose, y):
    p, y0 = inputs(pose, y)
    u = scgr.potential(p, y0, None)
    (3.0 * u).backward()
    assert calls == [(True, True)]
    assert (p.grad is None) == (not pose) and (y0.grad is None) == (not y)
    if pose:
        np.testing.assert_array_equal(p.grad.numpy(), 3.0 * np.arange(7.0))
    if y:
        np.testing.assert_array_equal(y0.grad.numpy(), np.full((5, 3), 6.0, np.float32))
