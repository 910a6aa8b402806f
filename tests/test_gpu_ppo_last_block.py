"""The training network's last block, of which the head reads the recurrent
token alone: outputs, next embeddings and both gradients against the FP64
oracle where its kernels change form or can go wrong — a single block (the
last one is also the first), 17 and 2 tokens, head widths 8, 16 and 32, one
sample, on both GEMM paths.  Tolerances: those of test_gpu_ppo (the same
arithmetic per stage)."""
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

CASES = {
    # (d, L, H, NS, n)
    "one_block": (64, 1, 4, 10, 41),
    "one_sample": (64, 2, 4, 10, 1),
    "t17_two_blocks": (32, 2, 2, 16, 19),
    "t17_heads8": (32, 1, 4, 16, 23),
    "t2_heads32": (64, 2, 2, 1, 130),
    "t16_heads32": (96, 1, 3, 15, 33),
}


@pytest.mark.parametrize("tc", [False, True])
@pytest.mark.parametrize("case", list(CASES))
def test_last_block_matches_oracle(case, tc):
    d, L, H, NS, n = CASES[case]
    no = 7
    shapes = synth.policy_shapes(synth.PolicyDims(d, L, H, no))
    prm = synth.policy_params(synth.PolicyDims(d, L, H, no), seed=61)
    net = ppo.Tfm(prm, d, L, H, no, NS, n, True, tensor_cores=tc)
    tok, ne, h, tok_d, ne_d, h_d = _inputs(n, NS, d, 62)
    h_out = torch.empty_like(h_d)
    out = net.forward(tok_d, ne_d, h_d, h_out=h_out).cpu().numpy()
    ref, ref_h = oracle.tfm_forward(prm, d, L, H, no, tok, ne, h)
    _close_tc(out, ref, tc)
    _close_tc(h_out.cpu().numpy(), ref_h, tc)
    act, logp_old, adv = _ppo_args(prm, d, L, H, no, tok, ne, h, 63)
    net.actor_grad(tok_d, ne_d, h_d, *(torch.from_numpy(x).cuda() for x in (act, logp_old, adv)), clip_eps=0.2,
                   ent_coef=0.01)
    _, g, _ = oracle.tfm_loss_grad(prm, d, L, H, no, oracle.ACTOR, tok, ne, h, act, logp_old, adv, 0.2, 0.01)
    _grad_close(net.grad.cpu().numpy(), g, shapes, tol=_tol(tc)["grad"])

    shapes = synth.policy_shapes(synth.PolicyDims(d, L, H, 1))
    prm = synth.policy_params(synth.PolicyDims(d, L, H, 1), seed=64)
    net = ppo.Tfm(prm, d, L, H, 1, NS, n, True, tensor_cores=tc)
    ret = np.random.default_rng(65).standard_normal(n).astype(np.float32)
    net.value_grad(tok_d, ne_d, h_d, torch.from_numpy(ret).cuda())
    _, g, _ = oracle.tfm_loss_grad(prm, d, L, H, 1, oracle.CRITIC, tok, ne, h, returns=ret)
    _grad_close(net.grad.cpu().numpy(), g, shapes, tol=_tol(tc)["grad"])
