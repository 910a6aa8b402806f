"""The tensors that Env.step returns are the caller's own: over the same
buffers on every step, but with a shape, a gradient flag and an autograd state
that no other step's share, whatever mode the first step ran in.  Without a
GPU: the views are made over host buffers here."""
import pytest
import torch

import paper_2505_08222_gb300 as ut
from paper_2505_08222_gb300 import _abi

NAMES = ("reward", "done", "obs", "estx", "esty", "err", "actions")


@pytest.fixture
def step(monkeypatch):
    """One Env.step's views of a 3-environment handle without a policy."""
    bufs = {}

    def view(ptr, shape, dtype=torch.float32):
        return torch.as_tensor(bufs.setdefault(ptr, torch.zeros(shape, dtype=dtype)).numpy()) if ptr else None

    monkeypatch.setattr(ut, "device_view", view)
    env = ut.Env.__new__(ut.Env)
    env._views, env.E, env.NA, env.NS, env.F, env.h = (None, None), 3, 4, 5, 6, None
    env.params = type("Params", (), {"n_actions": 3})
    out = _abi.StepOut()
    for k, name in enumerate(NAMES):
        setattr(out, name, 256 * (k + 1))
    return lambda: env._step_views(out)


def test_first_step_in_inference_mode(step):
    with torch.inference_mode():
        step()
    out = step()
    out["reward"].add_(1.0)
    w = torch.ones(3, requires_grad=True)
    (w * out["reward"]).sum().backward()
    assert torch.equal(w.grad, torch.ones(3))


def test_a_callers_changes_stay_with_its_tensors(step):
    first = step()
    first["reward"].unsqueeze_(0)
    first["estx"].requires_grad_()
    first["err"].resize_(2, 3)
    first["estx"].owner = first
    out = step()
    assert out["reward"].shape == (3,) and out["err"].shape == (6,)
    assert not out["estx"].requires_grad and not hasattr(out["estx"], "owner")
    assert out["logits"] is None and set(out) == {*NAMES, "logits"}
    # the same memory all the same, each with a version of its own: a value that
    # autograd has saved is not marked stale by the next step's caller
    w = torch.ones(3, requires_grad=True)
    y = (w * out["reward"]).sum()
    nxt = step()
    nxt["reward"].fill_(2.0)
    assert nxt["reward"].data_ptr() == out["reward"].data_ptr()
    y.backward()
    assert torch.equal(w.grad, torch.full((3,), 2.0))
