"""The transformer agent's two-kernel form (large batches: the last block's Wo
and FFN and the head on the recurrent rows of 128 agents per tile) against the
one-kernel form, which a stream capture keeps: the same arithmetic per row, so
logits, actions and embeddings are equal bit for bit."""
import numpy as np
import pytest
import torch

import synth
from synth import preset

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2505_08222_gb300 as ut  # noqa: E402


def _env(d, L, **kw):
    p = preset("fleet5", n_envs=4).replace(n_particles=32, d_model=d, n_layers=L, n_heads=d // 16, **kw)
    env = ut.Env(p)
    env.set_policy(synth.policy_params(synth.PolicyDims(d, L, d // 16), seed=5))
    env.reset(9)
    return env


def _one_kernel(env, tok, ne, h, step):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        logits, act = env.policy_forward(tok, ne, h, step=step, sample=True)
    g.replay()
    torch.cuda.synchronize()
    return logits, act


# agents just past three waves of tiles, past one chunk of agents, 16- and
# 17-token layouts, one block
@pytest.mark.parametrize("d,L,slots,n", [(64, 2, 10, 10033), (64, 1, 16, 6400), (128, 3, 16, 3333), (128, 2, 15, 3700),
                                         (64, 1, 1, 77824 + 70), (128, 1, 16, 58368 + 13)])
def test_two_kernels_equal_one(d, L, slots, n):
    env = _env(d, L)
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    tok = (0.4 * torch.randn(n, slots, 8, generator=g, device="cuda")).bfloat16()
    ne = torch.randint(0, slots + 1, (n,), generator=g, device="cuda", dtype=torch.int32)
    h = torch.randn(n, d, generator=g, device="cuda").bfloat16()
    h1, h2 = h.clone(), h.clone()
    a = env.policy_forward(tok, ne, h1, step=3, sample=True)
    b = _one_kernel(env, tok, ne, h2, 3)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and torch.equal(h1, h2)
    assert not torch.equal(h1, h)


def test_env_step_with_two_kernels():
    """4200 x 5 agents: the step's own policy launch against the one-kernel
    forward of the same tokens and embeddings; the launch count names both."""
    env = _env(64, 2, n_envs=4200)
    n = env.NA
    out = env.step()
    tok, h = out["obs"].clone().view(torch.bfloat16), env.state()["h"].clone().view(torch.bfloat16)
    out = env.step()
    got = out["logits"].clone(), out["actions"].clone(), env.state()["h"].clone().view(torch.bfloat16)
    ref = _one_kernel(env, tok, torch.full((n,), 10, dtype=torch.int32, device="cuda"), h, 2)
    assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1]) and torch.equal(got[2], h)
    s = env.rollout(2)
    assert s["kernel_launches"] == 2 * 6 and s["device_status"] == 0
