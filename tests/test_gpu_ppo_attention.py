"""The tensor-core attention of the training transformer (heads 16 wide, up to
16 tokens) in a block that is not the last, at the edges of its 16-row tiles
and of the elements of P that a lane holds (121 of 11 tokens fit four per lane,
144 of 12 do not): actor and critic gradients of two-block networks against the
FP64 oracle.

Tolerance, of every tensor's norm: the operands of a product are rounded to
BF16, a relative error of at most 2^-9, 2^-9 / sqrt(3) in the mean square, of
each of the two, so 1.6e-3 of a product's terms.  A gradient passes at most the
8 products of two blocks' forward and the 16 of their backward, whose errors are
independent: 1.6e-3 sqrt(24) = 7.8e-3, doubled for what the chain amplifies."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2505_08222_gb300 import ppo  # noqa: E402
from test_gpu_ppo import _inputs, _ppo_args  # noqa: E402

TOL = 1.6e-2


def _norms_close(got, ref, shapes):
    o = 0
    for name, shape, _ in shapes:
        n = int(np.prod(shape))
        g, r = got[o:o + n], ref[o:o + n]
        e = np.linalg.norm(g - r) / np.linalg.norm(r)
        assert e <= TOL, (name, e)
        o += n
    assert o == len(ref)


# (tokens, d, samples); the last has more row tiles than CTAs are resident
@pytest.mark.parametrize("T,d,n", [(2, 64, 300), (11, 64, 200), (12, 64, 200), (12, 128, 100), (13, 64, 200),
                                   (15, 32, 200), (16, 64, 200), (16, 128, 100), (16, 64, 2600)])
def test_two_block_gradients_match_oracle(T, d, n):
    L, H, NS, no = 2, d // 16, T - 1, 7
    shapes = synth.policy_shapes(synth.PolicyDims(d, L, H, no))
    prm = synth.policy_params(synth.PolicyDims(d, L, H, no), seed=81)
    tok, ne, h, tok_d, ne_d, h_d = _inputs(n, NS, d, 82)
    act, logp_old, adv = _ppo_args(prm, d, L, H, no, tok, ne, h, 83)
    net = ppo.Tfm(prm, d, L, H, no, NS, n, True)
    net.actor_grad(tok_d, ne_d, h_d, *(torch.from_numpy(x).cuda() for x in (act, logp_old, adv)), clip_eps=0.2,
                   ent_coef=0.01)
    _, g, _ = oracle.tfm_loss_grad(prm, d, L, H, no, oracle.ACTOR, tok, ne, h, act, logp_old, adv, 0.2, 0.01)
    _norms_close(net.grad.cpu().numpy(), g, shapes)

    shapes = synth.policy_shapes(synth.PolicyDims(d, L, H, 1))
    prm = synth.policy_params(synth.PolicyDims(d, L, H, 1), seed=84)
    ret = np.random.default_rng(85).standard_normal(n).astype(np.float32)
    net = ppo.Tfm(prm, d, L, H, 1, NS, n, True)
    net.value_grad(tok_d, ne_d, h_d, torch.from_numpy(ret).cuda())
    _, g, _ = oracle.tfm_loss_grad(prm, d, L, H, 1, oracle.CRITIC, tok, ne, h, returns=ret)
    _norms_close(net.grad.cpu().numpy(), g, shapes)
