"""The captured collection belongs to its critic: another GEMM path of the same
critic, or another critic (at the same address or not), captures it again; each
time it equals the step-by-step calls bit for bit."""
import pytest
import torch

import synth
from synth import preset

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2505_08222_gb300 as ut  # noqa: E402
from paper_2505_08222_gb300 import ppo  # noqa: E402


def _trainer():
    p = preset("fleet5", n_envs=6).replace(n_particles=64)
    env = ut.Env(p)
    prm = synth.policy_params(synth.PolicyDims(p.d_model, p.n_layers, p.n_heads, p.n_actions), seed=2)
    env.set_policy(prm)
    return ppo.Trainer(env, prm, _critic_params(p, 3), ppo.PPOConfig(T=5))


def _critic_params(p, seed):
    return synth.policy_params(synth.PolicyDims(p.d_model, p.n_layers, p.n_heads, 1), seed=seed)


def _check(tr):
    tr.collect_eager(9)
    torch.cuda.synchronize()
    want = tr.val.clone(), tr.ch.clone()
    tr.val.fill_(-7)
    tr.collect(9)
    torch.cuda.synchronize()
    assert torch.equal(tr.val, want[0]) and torch.equal(tr.ch, want[1])
    return want[0]


def test_gemm_path_of_the_critic():
    tr = _trainer()
    a = _check(tr)
    tr.critic.set_gemm_path(False)
    b = _check(tr)
    tr.critic.set_gemm_path(True)
    assert not torch.equal(a, b) and torch.equal(_check(tr), a)


def test_another_critic():
    tr = _trainer()
    p, seen = tr.env.params, [_check(tr)]
    for seed in (4, 5, 6):  # (an allocator gives a freed handle's address again)
        tr.critic.close()
        tr.critic = ppo.Tfm(_critic_params(p, seed), p.d_model, p.n_layers, p.n_heads, 1, tr.NS,
                            max(tr.mb_critic, tr.E), False, stream=tr.env._stream)
        seen.append(_check(tr))
        assert not torch.equal(seen[-1], seen[-2])
