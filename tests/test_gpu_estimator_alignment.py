"""Feature rows that are not 16-byte aligned (the kernels read them 16 bytes at
a time) are refused by every call that takes them, before anything is launched;
rows at an offset that keeps the alignment are taken."""
import ctypes

import pytest
import torch

import synth
from paper_2505_08222_gb300 import _abi
from synth import preset

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2505_08222_gb300 as ut  # noqa: E402


@pytest.mark.parametrize("offset", [1, 2, 3, 4, 96])  # floats
def test_feature_rows_need_16_bytes(offset):
    env = ut.Env(preset("fleet5", n_envs=2).replace(n_particles=64, d_model=0))
    env.est_set_weights(synth.mlp_params(seed=7, bias_scale=0.1))
    weights = env.est_get_weights()
    n = 40
    X = torch.randn(n * 96 + 96, device="cuda")[offset:offset + n * 96].view(n, 96)
    Y = torch.randn(n, 2, device="cuda")
    grad, out = torch.zeros(156930, device="cuda"), torch.zeros(n, 2, device="cuda")
    cfg = _abi.EstTrainConfig(1, n, 1e-3, 1, 0.9, 0.999, 1e-8, 0, 0.0)
    rcs = (ut.lib.est_forward(env.h, X.data_ptr(), out.data_ptr(), n),
           ut.lib.est_loss_grad(env.h, X.data_ptr(), Y.data_ptr(), n, n, 0, 0, 0.0, grad.data_ptr(), None),
           ut.lib.est_loss_grad(env.h, X.data_ptr(), Y.data_ptr(), n, 16, 0, 0, 0.0, grad.data_ptr(), None),
           ut.lib.est_train(env.h, X.data_ptr(), Y.data_ptr(), n, ctypes.byref(cfg), None))
    torch.cuda.synchronize()
    if offset % 4:
        assert rcs == (1, 1, 1, 1)  # UT_ERR_INVALID
        assert not grad.any() and not out.any() and (env.est_get_weights() == weights).all()
    else:
        assert rcs == (0, 0, 0, 0)
        assert bool(grad.any()) and bool(out.any())
    env.close()
