"""The CUDA-core path's paired products (the last block's queries over n rows
launched with its keys and values over n T): widths that leave part of a column
tile, row counts on either side of the row tiles, and splits along the rows that
differ between the two; outputs and gradients against the FP64 oracle, FP32
tolerances as in test_gpu_ppo."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2505_08222_gb300 import ppo  # noqa: E402
from test_gpu_ppo import FP32_TOL, _close, _grad_close, _inputs  # noqa: E402


# (d, H, tokens, samples)
@pytest.mark.parametrize("d,H,T,n", [(32, 2, 17, 129), (96, 6, 3, 65), (128, 8, 17, 1), (128, 8, 4, 64),
                                     (64, 4, 2, 700), (32, 4, 9, 2)])
def test_paired_products_match_oracle(d, H, T, n):
    L, NS = 2, T - 1
    prm = synth.policy_params(synth.PolicyDims(d, L, H, 1), seed=91)
    net = ppo.Tfm(prm, d, L, H, 1, NS, n, True, tensor_cores=False)
    tok, ne, h, tok_d, ne_d, h_d = _inputs(n, NS, d, 92)
    ref, _ = oracle.tfm_forward(prm, d, L, H, 1, tok, ne, h)
    _close(net.forward(tok_d, ne_d, h_d).cpu().numpy(), ref, FP32_TOL["out_atol"], FP32_TOL["out_rtol"])
    ret = np.random.default_rng(93).standard_normal(n).astype(np.float32)
    net.value_grad(tok_d, ne_d, h_d, torch.from_numpy(ret).cuda())
    _, g, _ = oracle.tfm_loss_grad(prm, d, L, H, 1, oracle.CRITIC, tok, ne, h, returns=ret)
    _grad_close(net.grad.cpu().numpy(), g, synth.policy_shapes(synth.PolicyDims(d, L, H, 1)), tol=FP32_TOL["grad"])
