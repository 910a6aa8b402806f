"""Waits that run out in the estimator's network kernels (est_forward,
est_loss_grad, est_train), by the test hook of test_gpu_failure.py: reported as
UT_ERR_TIMEOUT, nothing written, and the handle goes on as if the call had not
been made."""
import numpy as np
import pytest
import torch

import synth
from synth import preset

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2505_08222_gb300 as ut  # noqa: E402

POLLS = 2000
TIMEOUT = pytest.raises(ut.UtError, match="UT_ERR_TIMEOUT")


def _env():
    env = ut.Env(preset("fleet5", n_envs=2).replace(n_particles=64, d_model=0))
    env.est_set_weights(synth.mlp_params(seed=7, bias_scale=0.1))
    return env


def _rows(n):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    return torch.randn(n, 96, generator=g, device="cuda"), torch.randn(n, 2, generator=g, device="cuda")


def test_forward_reports_the_wait():
    env = _env()
    X, _ = _rows(300)
    want = env.est_forward(X).clone()
    env.test_wait_timeout(POLLS)
    env.est_forward(X)
    with TIMEOUT:
        env.metrics()
    env.test_wait_timeout(0)
    env.metrics_reset()
    assert torch.equal(env.est_forward(X), want)
    assert env.metrics()["device_status"] == 0
    env.close()


@pytest.mark.parametrize("n", [100, 5000])
def test_gradient_and_training_report_the_wait_and_change_nothing(n):
    env, twin = _env(), _env()
    X, Y = _rows(n)
    other, _ = _rows(n + 1)
    env.est_loss_grad(other[:n].contiguous(), Y)  # partial sums of another batch
    grad = torch.full((156930,), 7.0, device="cuda")
    kw = dict(steps=3, batch=64, lr=1e-3, seed=4)
    for e in (env, twin):
        e.est_train(X, Y, **kw)
    before = env.est_get_weights()
    env.test_wait_timeout(POLLS)
    with TIMEOUT:
        ut._check(ut.lib.est_loss_grad(env.h, X.data_ptr(), Y.data_ptr(), n, n, 0, 0, 0.0, grad.data_ptr(), None), env.h)
    assert bool((grad == 7.0).all())
    with TIMEOUT:
        env.est_train(X, Y, **kw)
    np.testing.assert_array_equal(env.est_get_weights(), before)
    env.test_wait_timeout(0)
    # weights, moments and step count are the twin's, which never waited
    a, b = (e.est_loss_grad(X, Y) for e in (env, twin))
    assert a[0] == b[0] and torch.equal(a[1], b[1])
    for e in (env, twin):
        e.est_train(X, Y, **kw)
    np.testing.assert_array_equal(env.est_get_weights(), twin.est_get_weights())
    assert not np.array_equal(env.est_get_weights(), before)
    env.close()
    twin.close()
