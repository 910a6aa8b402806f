"""Estimator loss and gradient at the edges of its 128-row tiles and of the 24
splits of its weight gradients (splits with one tile, unequal splits, splits
left without rows), against the FP64 oracle; bounds as in
test_gpu_estimator."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from parity import EST_GRAD_FRAC, check_elementwise  # noqa: E402
from test_gpu_estimator import _env, _features  # noqa: E402


@pytest.mark.parametrize("n", [127, 128, 129, 24 * 128, 24 * 128 + 1, 53 * 128 - 5])
def test_batch_edges_match_oracle(n):
    env, _ = _env()
    params = synth.mlp_params(seed=8, bias_scale=0.1)
    env.est_set_weights(params)
    X = _features(n, 12)
    Y = (np.random.default_rng(13).standard_normal((n, 2)) * 0.2).astype(np.float32)
    loss, grad = env.est_loss_grad(torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda())
    ref_loss, ref_grad = oracle.mlp_loss_grad(params, X, Y)
    assert abs(loss - ref_loss) <= 2e-2 * ref_loss
    check_elementwise(grad.cpu().numpy().astype(np.float64), ref_grad, synth.mlp_shapes(), EST_GRAD_FRAC)
