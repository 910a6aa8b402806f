"""The persistent rollout's environment warp runs one step ahead of the
filters (NT < 1024) or in turn with them (NT = 1024): the lengths at which the
look-ahead starts and stops, one and several filters per environment, both
reward types, against the graph rollout bit for bit."""
import numpy as np
import pytest
import torch

from synth import preset

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2505_08222_gb300 as ut  # noqa: E402

KEYS = ("ax", "ay", "apsi", "tx", "ty", "px", "py", "pvx", "pvy", "lpx", "lpy", "lpage", "estx", "esty", "velx", "vely")


def _run(p, form, T):
    env = ut.Env(p)
    env.reset(11)
    env.set_rollout_form(form)
    view = env.step()  # views of the step's outputs: the last rollout step writes them
    stats = [env.rollout(T) for _ in range(3)]
    torch.cuda.synchronize()
    st = env.state()
    out = {k: st[k].cpu().numpy().copy() for k in KEYS if st.get(k) is not None}
    out.update({k: view[k].cpu().numpy().copy() for k in ("obs", "reward", "done", "err")})
    env.close()
    return out, stats


@pytest.mark.parametrize("n_envs", [6, 153])  # up to one environment per SM, and more
@pytest.mark.parametrize("T", [1, 2, 3])
@pytest.mark.parametrize("name,kw", [
    ("small", {"n_particles": 3000}),                                       # NT = 1024, one filter
    ("ragged", {"n_particles": 2100, "d_model": 0, "reward_type": 0}),      # NT = 1024, several filters
    ("small", {"n_particles": 32, "reward_type": 1}),                       # one filter warp beside the environment's
    ("ragged", {"n_particles": 200, "d_model": 0, "shared_filter": 1}),
])
def test_rollout_stages(name, kw, T, n_envs):
    p = preset(name, n_envs=n_envs).replace(**kw)
    g, gs = _run(p, 0, T)
    r, rs = _run(p, 1, T)
    assert g.keys() == r.keys()
    for k in g:
        np.testing.assert_array_equal(r[k], g[k], err_msg=k)
    for a, b in zip(gs, rs):
        for k in ("n_err", "crash_count", "agent_steps", "steps", "device_status"):
            assert a[k] == b[k], k
        assert a["device_status"] == 0
        # the same double sums in another order
        assert b["sum_sq_err"] == pytest.approx(a["sum_sq_err"], rel=1e-12)
        assert b["reward_sum"] == pytest.approx(a["reward_sum"], rel=1e-12, abs=1e-9)
