"""Graph rollouts and graph collections under a new seed: a handle that has run
one seed's graph gives what a fresh handle gives under the other seed (every
random draw is a function of the seed)."""
import numpy as np
import pytest
import torch

import synth
from synth import preset

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2505_08222_gb300 as ut  # noqa: E402
from paper_2505_08222_gb300 import ppo  # noqa: E402

NAMES = ("ax", "ay", "apsi", "tx", "ty", "px", "py", "estx", "esty")


def _env(agent):
    p = preset("fleet5", n_envs=6).replace(n_particles=64, **({} if agent else {"d_model": 0}))
    env = ut.Env(p)
    if agent:
        env.set_policy(synth.policy_params(synth.PolicyDims(p.d_model, p.n_layers, p.n_heads, p.n_actions), seed=2))
    return env


def _state(env):
    torch.cuda.synchronize()
    st = env.state()
    return {k: st[k].cpu().numpy().copy() for k in NAMES}


@pytest.mark.parametrize("agent", [False, True])
def test_rollout_under_another_seed(agent):
    env, fresh = _env(agent), _env(agent)
    env.reset(1)
    env.rollout(4)
    for e in (env, fresh):
        e.reset(2)
        e.rollout(4)
    a, b = _state(env), _state(fresh)
    for k in NAMES:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    env.reset(1)  # and back
    env.rollout(4)
    fresh.reset(1)
    for _ in range(4):
        fresh.step()
    a, b = _state(env), _state(fresh)
    for k in NAMES:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)


def test_collection_under_another_seed():
    def trainer():
        env = _env(True)
        p = env.params
        d = synth.PolicyDims(p.d_model, p.n_layers, p.n_heads, p.n_actions)
        c = synth.PolicyDims(p.d_model, p.n_layers, p.n_heads, 1)
        return ppo.Trainer(env, synth.policy_params(d, seed=2), synth.policy_params(c, seed=3), ppo.PPOConfig(T=5))
    tr, fresh = trainer(), trainer()
    tr.collect(1)
    tr.collect(2)
    fresh.collect(2)
    torch.cuda.synchronize()
    for k in ("tok", "h", "act", "logp", "rew", "done", "ctok", "val"):
        assert torch.equal(getattr(tr, k), getattr(fresh, k)), k
