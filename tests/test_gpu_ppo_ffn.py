"""The fused feed-forward sub-block of the training transformer (d = 64, tensor
cores) at the edges of its 128-row tiles and with more tiles than resident
CTAs, actor and critic gradients against the FP64 oracle; tolerances of the
BF16 path as in test_gpu_ppo."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2505_08222_gb300 import ppo  # noqa: E402
from test_gpu_ppo import _close_tc, _grad_close, _inputs, _ppo_args, _tol  # noqa: E402


# samples of 3 tokens: whole tiles, one row over, one short, 307 tiles
@pytest.mark.parametrize("n", [128, 129, 127, 13100])
def test_fused_feed_forward_matches_oracle(n):
    d, L, H, NS, no = 64, 2, 4, 2, 7
    shapes = synth.policy_shapes(synth.PolicyDims(d, L, H, no))
    prm = synth.policy_params(synth.PolicyDims(d, L, H, no), seed=71)
    net = ppo.Tfm(prm, d, L, H, no, NS, n, True)
    tok, ne, h, tok_d, ne_d, h_d = _inputs(n, NS, d, 72)
    out = net.forward(tok_d, ne_d, h_d).cpu().numpy()
    ref, _ = oracle.tfm_forward(prm, d, L, H, no, tok, ne, h)
    _close_tc(out, ref, True)
    act, logp_old, adv = _ppo_args(prm, d, L, H, no, tok, ne, h, 73)
    net.actor_grad(tok_d, ne_d, h_d, *(torch.from_numpy(x).cuda() for x in (act, logp_old, adv)), clip_eps=0.2,
                   ent_coef=0.01)
    _, g, _ = oracle.tfm_loss_grad(prm, d, L, H, no, oracle.ACTOR, tok, ne, h, act, logp_old, adv, 0.2, 0.01)
    _grad_close(net.grad.cpu().numpy(), g, shapes, tol=_tol(True)["grad"])
