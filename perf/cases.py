"""What a user of this framework has it do, as measurable cases.

Every case goes through the package's public entry points (``Env``, ``Tfm``):
environment steps of the tracking fleets with host-given actions or with the
transformer agent acting, whole rollouts, the agent's forward, the gradient
steps of the TransfMAPPO update and of the learned estimator.  Sizes are those
of the framework's five workloads (64 x 1 x 1 with 1000 particles; 4096 x 5 x 5
with 2048; ragged 1..8 x 1..8 with 1024; the learned-estimator fleet; 8 x 8
with 512 particles) and of the minibatches their training takes; ``draw``
spreads over the ranges between and around them.
"""
import math

import numpy as np
import torch

import paper_2505_08222_gb300 as ut
from paper_2505_08222_gb300 import ppo

STEP0 = 36          # global step of the injected states
HORIZON = 200       # steps after which the caller starts a new episode
N_ACTION_SETS = 8   # action batches that a host controller cycles through
EST_PARAMS = ((96, 256), (256, 256), (256, 256), (256, 2))


def listed():
    return [
        # one env_step of the smallest workload: what a host control loop waits for
        {"name": "step_small", "kind": "step", "envs": 64, "agents": 1, "targets": 1, "particles": 1000},
        # the same fleet's whole 200-step episode as one call (random actions)
        {"name": "rollout_small", "kind": "rollout", "envs": 64, "agents": 1, "targets": 1, "particles": 1000,
         "steps": 200},
        # the flagship step: the transformer agent acts, every agent filters every target
        {"name": "step_fleet5", "kind": "step", "envs": 4096, "agents": 5, "targets": 5, "particles": 2048, "d": 64,
         "layers": 2},
        # ragged fleets, 1..8 agents and targets per env, actions from outside
        {"name": "step_ragged", "kind": "step", "envs": 16384, "agents": 8, "targets": 8, "ragged": True,
         "particles": 1024},
        # many small filters: the 8 x 8 fleet
        {"name": "step_large", "kind": "step", "envs": 16384, "agents": 8, "targets": 8, "particles": 512},
        # the learned estimator in place of the filter
        {"name": "step_learned", "kind": "step", "envs": 4096, "agents": 5, "targets": 5, "particles": 64,
         "tracker": 1},
        # one vehicle team asks its agent for actions (serving, latency)
        {"name": "policy_team", "kind": "policy", "agents": 5, "slots": 10, "d": 64, "layers": 2},
        # the 8 x 8 fleet's agents, three layers of 128
        {"name": "policy_large", "kind": "policy", "agents": 131072, "slots": 16, "d": 128, "layers": 3},
        # actor minibatch of the PPO update (32 steps x 20480 agents in 4 minibatches)
        {"name": "actor_fleet5", "kind": "actor", "batch": 163840, "slots": 10, "d": 64, "layers": 2},
        # critic minibatch of the same update (true-state tokens, FP32)
        {"name": "critic_fleet5", "kind": "critic", "batch": 32768, "slots": 10, "d": 64, "layers": 2},
        # actor minibatch of the 8 x 8 fleet's network
        {"name": "actor_large", "kind": "actor", "batch": 16384, "slots": 16, "d": 128, "layers": 3},
        # one batch of the estimator's training
        {"name": "estimator_batch", "kind": "estimator", "batch": 16384},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "rollout", "policy", "actor", "critic", "estimator"])
    if kind == "step":
        a, t, p = rng.randint(1, 8), rng.randint(1, 8), _log(rng, 64, 4096)
        if rng.random() < 0.5:
            p = max(4, p // 4 * 4)
        most = (1 << 28) // (a * t * p)
        c = {"kind": kind, "envs": _log(rng, 16, max(16, min(16384, most))), "agents": a, "targets": t, "particles": p}
        option = rng.choice(["", "", "ragged", "agent", "learned", "shared", "ess"])
        if option == "ragged":
            c["ragged"] = True
        elif option == "agent":
            c.update(d=64, layers=rng.randint(1, 3))
        elif option == "learned":
            c.update(tracker=rng.randint(1, 3), particles=64)
        elif option == "shared":
            c["shared"] = True
        elif option == "ess":
            c["ess"] = rng.randint(4, 12)
        return c
    if kind == "rollout":
        return {"kind": kind, "envs": _log(rng, 8, 256), "agents": rng.randint(1, 2), "targets": rng.randint(1, 2),
                "particles": _log(rng, 64, 2048), "steps": _log(rng, 20, 200)}
    if kind == "policy":
        d = rng.choice([64, 128])
        return {"kind": kind, "agents": _log(rng, 1, 131072 if d == 64 else 65536), "slots": rng.randint(2, 16), "d": d,
                "layers": rng.randint(1, 3)}
    if kind in ("actor", "critic"):
        d = rng.choice([64, 64, 128])
        return {"kind": kind, "batch": _log(rng, 64, 65536 if d == 64 else 8192), "slots": rng.randint(2, 16), "d": d,
                "layers": rng.randint(1, 3)}
    return {"kind": kind, "batch": _log(rng, 128, 65536)}


# ------------------------------------------------------------------- the fleets
class Fleet:
    """Constants of one environment batch (the fields Env reads)."""

    def __init__(self, case):
        small = case["agents"] == 1 and case["targets"] == 1 and "d" not in case
        ts = (0.3, 0.3) if small else (0.5, 1.5)
        self.__dict__.update(
            n_envs=case["envs"], max_agents=case["agents"], max_targets=case["targets"],
            n_particles=case["particles"], horizon=HORIZON, agents_per_env=None, targets_per_env=None, dt=30.0,
            agent_speed=1.0, heading_noise=0.0 if small else 0.02, action_mode=0 if small else 1, n_rudder=5,
            n_actions=3 if small else 7, turn_angle=math.pi / 6, rudder_max=0.24, rudder_gain=1.45 / 0.24,
            target_model=0 if small else 1, target_speed_min=ts[0], target_speed_max=ts[1],
            target_drift_sigma=math.radians(10.0), target_depth_max=0.0, range_sigma=1.0, det_radius=1500.0,
            comm_radius=1500.0, comm_drop=0.0, pf_accel_sigma=0.1, pf_vcap=1.2 * ts[1], reward_type=0 if small else 1,
            eps_min=10.0, eps_max=50.0, follow_dmin=100.0, d_safe=10.0, spawn_min=50.0, spawn_radius=100.0,
            spawn_tries=64, feature_scale=1000.0, est_scale=100.0, id_env0=0, id_agent0=0, id_target0=0, id_filter0=0,
            d_model=case.get("d", 0), n_layers=case.get("layers", 0), n_heads=case.get("d", 0) // 16,
            shared_filter=int(case.get("shared", False)), id_pair0=0, pf_ess_num=case.get("ess", 0))
        if case.get("ragged"):  # one fleet composition per size, whatever the episode's seed
            r = np.random.default_rng(case["envs"])
            self.agents_per_env = r.integers(1, case["agents"] + 1, case["envs"]).astype(np.int32)
            self.targets_per_env = r.integers(1, case["targets"] + 1, case["envs"]).astype(np.int32)

    def counts(self):
        n = self.n_envs
        a, t = self.agents_per_env, self.targets_per_env
        return (np.full(n, self.max_agents, np.int32) if a is None else a,
                np.full(n, self.max_targets, np.int32) if t is None else t)

    def maps(self):
        """Agent and target of each filter, the filters of all envs one after the other."""
        a, t = (x.astype(np.int64) for x in self.counts())
        a0, t0 = np.cumsum(a) - a, np.cumsum(t) - t
        n = t if self.shared_filter else a * t
        env = np.repeat(np.arange(self.n_envs), n)
        j = np.arange(n.sum()) - np.repeat(np.cumsum(n) - n, n)
        agent = a0[env] + (0 if self.shared_filter else j // t[env])
        return env, agent, t0[env] + (j if self.shared_filter else j % t[env]), a, a0


def _rand(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g, (lambda *s: torch.randn(*s, generator=g, device="cuda")), \
        (lambda *s: torch.rand(*s, generator=g, device="cuda"))


def _fleet_state(p, seed):
    """An episode some steps old: everything in hearing range, each filter's
    cloud around its target, between a few and some tens of metres wide."""
    _, randn, rand = _rand(seed)
    env, agent, target, a, _ = p.maps()
    na, nt, nf, P = int(a.sum()), int(p.counts()[1].sum()), len(env), p.n_particles
    it = torch.from_numpy(target).cuda()
    st = {"ax": 600 * rand(na) - 300, "ay": 600 * rand(na) - 300, "apsi": 2 * math.pi * rand(na) - math.pi,
          "tx": 600 * rand(nt) - 300, "ty": 600 * rand(nt) - 300, "tz": torch.zeros(nt, device="cuda"),
          "tpsi": 2 * math.pi * rand(nt) - math.pi,
          "tspeed": p.target_speed_min + (p.target_speed_max - p.target_speed_min) * rand(nt)}
    width = 5 * torch.exp(2 * rand(nf))
    for k in ("x", "y"):
        off = width * 0.5 * randn(nf)
        st["est" + k] = st["t" + k][it] + off
        st["prev_est" + k] = st["est" + k] + 10 * randn(nf)
        st["vel" + k] = 5 * randn(nf)
        cloud = randn(nf, P).mul_(width[:, None]).add_(st["est" + k][:, None])
        st["p" + k] = cloud.view(-1)
        st["pv" + k] = (0.4 * p.pf_vcap * randn(nf * P)).clamp_(-p.pf_vcap, p.pf_vcap)
    acts = torch.randint(0, p.n_actions, (N_ACTION_SETS, na), generator=_rand(seed + 1)[0], device="cuda",
                         dtype=torch.int32)
    return st, acts


def _ring(p, seed, st):
    """16 pings per filter from the last steps, oldest first (qx, qy, r, step)."""
    _, randn, _ = _rand(seed + 2)
    _, agent, target, _, _ = p.maps()
    ia, it = torch.from_numpy(agent).cuda(), torch.from_numpy(target).cuda()
    n = len(agent)
    qx, qy = st["ax"][ia][:, None] + 150 * randn(n, 16), st["ay"][ia][:, None] + 150 * randn(n, 16)
    r = torch.hypot(qx - st["tx"][it][:, None], qy - st["ty"][it][:, None]) + 20 * randn(n, 16)
    g = (STEP0 - torch.arange(15, -1, -1, device="cuda") // max(1, p.max_agents)).float().expand(n, 16)
    return torch.stack([qx, qy, r, g], 2).contiguous()


def _params(shapes, seed, head_scale=1.0):
    """Usual initial weights, flat: matrices N(0, 1 / fan in), gains 1, biases small."""
    r = np.random.default_rng(seed)
    out = []
    for name, s in shapes:
        v = r.standard_normal(s)
        if len(s) == 2:
            v *= (head_scale if name == "Wh" else 1.0) / math.sqrt(s[1])
        else:
            v = 0.05 * v + (1.0 if "g" in name else 0.0)
        out.append(v.astype(np.float32).ravel())
    return np.concatenate(out)


def _agent_shapes(d, layers, n_out):
    s = [("We", (d, 8)), ("be", (d,))]
    for _ in range(layers):
        s += [("g1", (d,)), ("c1", (d,)), ("Wqkv", (3 * d, d)), ("bqkv", (3 * d,)), ("Wo", (d, d)), ("bo", (d,)),
              ("g2", (d,)), ("c2", (d,)), ("W1", (4 * d, d)), ("b1", (4 * d,)), ("W2", (d, 4 * d)), ("b2", (d,))]
    return s + [("gf", (d,)), ("cf", (d,)), ("Wh", (n_out, d)), ("bh", (n_out,))]


def _mlp_shapes():
    return [x for k, (i, o) in enumerate(EST_PARAMS) for x in (("Wh" if k == 3 else "W", (o, i)), ("b", (o,)))]


def _tokens(n, slots, seed, critic):
    """Entity tokens as the environment writes them, and their counts (full
    fleets mostly, some smaller)."""
    g, randn, rand = _rand(seed)
    tok = torch.zeros(n, slots, 8, device="cuda")
    tok[..., :3] = 0.3 * randn(n, slots, 3)
    if critic:
        psi = 2 * math.pi * rand(n, slots)
        tok[..., 3], tok[..., 4], tok[..., 5], tok[..., 6] = psi.cos(), psi.sin(), psi.cos(), psi.sin()
        tok[..., 7] = (rand(n, slots) < 0.5).float()
    else:
        tok.scatter_(2, torch.randint(3, 6, (n, slots, 1), generator=g, device="cuda"), 1.0)
        tok[..., 6] = (rand(n, slots) < 0.1).float()
        tok[..., 7] = tok[..., 6] / 16
    ne = torch.full((n,), slots, dtype=torch.int32, device="cuda")
    few = torch.randint(1, slots + 1, (n,), generator=g, device="cuda", dtype=torch.int32)
    ne = torch.where(rand(n) < 0.25, few, ne)
    tok *= (torch.arange(slots, device="cuda")[None, :, None] < ne[:, None, None])
    return tok if critic else tok.bfloat16(), ne


def _net_inputs(case, seed):
    """Weights, tokens, counts, recurrent embeddings and the loss's inputs."""
    critic = case["kind"] == "critic"
    n = case.get("batch", case.get("agents"))
    n_out = 1 if critic else 7
    # a policy head of small weights, as PPO starts with: near-uniform actions
    prm = _params(_agent_shapes(case["d"], case["layers"], n_out), seed + 5, 0.05 if case["kind"] == "actor" else 1.0)
    tok, ne = _tokens(n, case["slots"], seed + 6, critic)
    g, randn, _ = _rand(seed + 7)
    h = 0.7 * randn(n, case["d"])
    more = {"actions": torch.randint(0, n_out, (n,), generator=g, device="cuda", dtype=torch.int32),
            "logp_old": -math.log(n_out) + 0.1 * randn(n), "adv": randn(n), "returns": 3 * randn(n)}
    return prm, tok, ne, h, more


# ----------------------------------------------------------------- prepare, run
def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "t": 0, "seed": seed}
    if kind in ("step", "rollout"):
        p = Fleet(case)
        env = s["env"] = ut.Env(p, ring="tracker" in case)
        env.reset(seed)
        if case.get("d"):
            env.set_policy(_params(_agent_shapes(p.d_model, p.n_layers, p.n_actions), seed + 5))
            s["acts"] = [None]
        elif kind == "step":
            st, acts = _fleet_state(p, seed)
            if "tracker" in case:
                env.est_set_weights(_params(_mlp_shapes(), seed + 5, 0.1))
                env.est_set_mode(case["tracker"])
                st["ring"] = _ring(p, seed, st)
                st["ring_head"] = torch.zeros(env.F, dtype=torch.int32, device="cuda")
                st["ring_count"] = torch.full((env.F,), 16, dtype=torch.int32, device="cuda")
                for k in ("px", "py", "pvx", "pvy"):
                    del st[k]
            env.set_state(STEP0, 0, **st)
            s["acts"] = list(acts)
        else:
            env.set_rollout_form(1)  # the form that env.autotune keeps for fleets like these
            s["steps"] = case["steps"]
        v = env.state()
        s["state"] = {k: v[k] for k in ("ax", "ay", "apsi", "tx", "ty", "tpsi", "estx", "esty", "px", "py", "pvx",
                                        "pvy")}
        if "tracker" in case:
            s["state"] = {k: v[k] for k in ("ax", "ay", "tx", "ty", "velx", "vely", "prev_estx", "prev_esty")}
        for t in s["state"].values():
            t.owner = env  # the views borrow the handle's buffers: it lives as long as they do
        return s
    if kind == "estimator":
        _, randn, rand = _rand(seed)
        s["env"] = ut.Env(Fleet({"envs": 1, "agents": 1, "targets": 1, "particles": 64}))
        s["env"].reset(0)
        s["env"].est_set_weights(_params(_mlp_shapes(), seed + 5))
        s["X"], s["Y"] = _features(case["batch"], seed)
        return s
    prm, tok, ne, h, more = _net_inputs(case, seed)
    if kind == "policy":
        p = Fleet({"envs": 1, "agents": 2, "targets": 2, "particles": 64, "d": case["d"], "layers": case["layers"]})
        s["env"] = ut.Env(p)
        s["env"].reset(0)
        s["env"].set_policy(prm)
        s["h0"] = h.bfloat16()
        s["h"] = s["h0"].clone()
        s.update(tok=tok, ne=ne)
        return s
    s["tfm"] = ppo.Tfm(prm, case["d"], case["layers"], case["d"] // 16, 1 if kind == "critic" else 7, case["slots"],
                       case["batch"], kind == "actor")
    s.update(tok=tok, ne=ne, h=h, **more)
    return s


def _features(n, seed):
    """Recorded estimator rows: 16 pings, newest first, then the estimate's motion."""
    _, randn, rand = _rand(seed)
    X = torch.zeros(n, 96, device="cuda")
    ping = X[:, :80].view(n, 16, 5)
    ping[..., :2] = 1.5 * randn(n, 16, 2)
    ping[..., 2] = 0.3 * randn(n, 16)
    ping[..., 3] = torch.arange(16, device="cuda") // 5 / 16.0
    ping[..., 4] = 1.0
    X[:, 80:84] = 0.2 * randn(n, 4)
    return X, 0.4 * randn(n, 2)


def run(s):
    kind = s["kind"]
    if kind == "step":
        env = s["env"]
        if s["t"] == HORIZON:  # the episode is over: the caller starts the next one
            s["t"] = 0
            env.reset(s["seed"])
        out = env.step(s["acts"][s["t"] % len(s["acts"])])
        s["t"] += 1
        got = {k: out[k] for k in ("reward", "done", "estx", "esty", "err", "actions")}
        got["obs"] = out["obs"].view(torch.bfloat16)
        if out["logits"] is not None:
            got["logits"] = out["logits"]
        return got, s["state"]
    if kind == "rollout":
        s["env"].reset(s["seed"])
        st = s["env"].rollout(s["steps"])
        return [st[k] for k in ("sum_sq_err", "n_err", "rmse", "reward_sum", "crash_count", "agent_steps",
                                "steps")], s["state"]
    if kind == "policy":
        if s["t"] % HORIZON == 0:  # a new episode's recurrent embedding
            s["h"].copy_(s["h0"])
        s["t"] += 1
        logits, act = s["env"].policy_forward(s["tok"], s["ne"], s["h"], step=s["t"], sample=True)
        return logits, act, s["h"]
    if kind == "estimator":
        return s["env"].est_loss_grad(s["X"], s["Y"], huber=1.0)
    if kind == "actor":
        s["tfm"].actor_grad(s["tok"], s["ne"], s["h"], s["actions"], s["logp_old"], s["adv"], clip_eps=0.2,
                            ent_coef=0.01, stats=False)
    else:
        s["tfm"].value_grad(s["tok"], s["ne"], s["h"], s["returns"], stats=False)
    return s["tfm"].grad


# ------------------------------------------------------------------------- work
def work(case):
    kind = case["kind"]
    if kind in ("step", "rollout"):
        a, t, P = case["agents"], case["targets"], case["particles"]
        if case.get("ragged"):
            a, t = (a + 1) / 2, (t + 1) / 2
        na, nf = case["envs"] * a, case["envs"] * t * (1 if case.get("shared") else a)
        # per agent 24 B of state in and out and its tokens, per filter its estimate
        small = na * (24 + 16 * (case["agents"] + case["targets"])) + case["envs"] * t * 32 + nf * 12
        if kind == "rollout":
            return {"bytes": small + 16 * nf * P, "flops": case["steps"] * nf * P * (40 + 8 * a)}
        if "tracker" in case:
            return {"bytes": small + nf * 328, "flops": nf * 2 * (96 * 256 + 2 * 256 * 256 + 512)}
        w = {"bytes": small + (40 if case.get("ess") else 32) * nf * P, "flops": nf * P * (40 + 8 * a)}
        if case.get("d"):
            w["flops"] += na * _net_flops(case["agents"] + case["targets"], case["d"], case["layers"], 7)
            w["bytes"] += na * (4 * case["d"] + 28)
        return w
    if kind == "estimator":
        n = case["batch"]
        return {"bytes": n * 98 * 4 + 2 * 156930 * 4, "flops": n * 6 * (96 * 256 + 2 * 256 * 256 + 512)}
    d, T, n_out = case["d"], case["slots"], 1 if kind == "critic" else 7
    n = case.get("batch", case.get("agents"))
    prm = sum(int(np.prod(x)) for _, x in _agent_shapes(d, case["layers"], n_out))
    f = n * _net_flops(T, d, case["layers"], n_out)
    if kind == "policy":
        return {"bytes": n * (16 * T + 4 + 4 * d + 32) + 2 * prm, "flops": f}
    return {"bytes": n * ((32 if kind == "critic" else 16) * T + 4 + 4 * d + 12) + 8 * prm, "flops": 3 * f}


def _net_flops(slots, d, layers, n_out):
    """One sample's forward: every token through all blocks but the last, of
    which the output needs the keys and values of all tokens and the rest for
    the recurrent token alone."""
    T = 1 + slots
    full = T * 24 * d * d + 4 * T * T * d
    return (layers - 1) * full + T * 4 * d * d + 20 * d * d + 4 * T * d + 16 * slots * d + 2 * n_out * d


# ------------------------------------------------------- the same in 64 bits
def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors, key = seed."""
    m = 0xFFFFFFFF

    def mul(a, b):  # 32 x 32 -> (high, low)
        lo = (b & 0xFFFF) * a
        hi = (b >> 16) * a + (lo >> 16)
        return hi >> 16, ((hi & 0xFFFF) << 16) | (lo & 0xFFFF)

    k0, k1 = seed & m, (seed >> 32) & m
    for _ in range(10):
        ha, la = mul(0xD2511F53, c0)
        hb, lb = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = hb ^ c1 ^ k0, lb, ha ^ c3 ^ k1, la
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return c0, c1, c2, c3


def _normals(va, vb):
    rad = torch.sqrt(-2 * torch.log(((va >> 8) + 1).double() * 2.0 ** -24))
    ang = 2 * math.pi * (vb >> 8).double() * 2.0 ** -24
    return rad * ang.cos(), rad * ang.sin()


def _draw(ids, second, g, tag, seed):
    z = torch.zeros_like(ids)
    return _philox(ids, z + second, z + g, z + tag, seed)


def _exact_step(case, seed):
    """One step from the injected state: the move, the pings, and every
    filter's (or the estimator's) new estimate.  The resampled particles are a
    discontinuous function of the weights and have no value here."""
    p = Fleet(case)
    st, acts = _fleet_state(p, seed)
    env, agent, target, a, a0 = p.maps()
    dev = torch.device("cuda")
    g = STEP0 + 1
    x = {k: v.double() for k, v in st.items() if not k.startswith("p") or k.startswith("prev")}
    ids = torch.arange(len(st["ax"]), device=dev)
    angles = torch.tensor([(j - 1) * p.turn_angle for j in range(3)] if p.action_mode == 0 else
                          [p.rudder_gain * (-p.rudder_max + 2 * p.rudder_max * j / 6) for j in range(7)],
                          dtype=torch.float64, device=dev)
    r = _draw(ids, 0, g, 7, seed)
    psi = x["apsi"] + angles[acts[0].long()] + p.heading_noise * _normals(r[0], r[1])[0]
    psi = psi - 2 * math.pi * torch.floor((psi + math.pi) / (2 * math.pi))
    ax, ay = x["ax"] + p.dt * psi.cos(), x["ay"] + p.dt * psi.sin()
    ids = torch.arange(len(st["tx"]), device=dev)
    r = _draw(ids, 0, g, 8, seed)
    if p.target_model == 0:
        tpsi = 2 * math.pi * (r[0] >> 8).double() * 2.0 ** -24
    else:
        tpsi = x["tpsi"] + p.target_drift_sigma * _normals(r[0], r[1])[0]
    tpsi = tpsi - 2 * math.pi * torch.floor((tpsi + math.pi) / (2 * math.pi))
    tx, ty = x["tx"] + p.dt * x["tspeed"] * tpsi.cos(), x["ty"] + p.dt * x["tspeed"] * tpsi.sin()

    # every agent hears every target of its env and passes its range on:
    # sender b's ping of target k is pair (b, k) of the env
    nf, A = len(env), p.max_agents
    t_cnt = p.counts()[1].astype(np.int64)
    pair0 = np.cumsum(a * t_cnt) - a * t_cnt
    k = target - (np.cumsum(t_cnt) - t_cnt)[env]
    b = np.arange(A)[None, :]
    on = torch.from_numpy(b < a[env][:, None]).to(dev)
    snd = torch.from_numpy(np.minimum(a0[env][:, None] + b, len(st["ax"]) - 1)).to(dev)
    pair = torch.from_numpy(pair0[env][:, None] + b * t_cnt[env][:, None] + k[:, None]).to(dev)
    it = torch.from_numpy(target).to(dev)
    r = _draw(pair, 0, g, 9, seed)
    qx, qy = ax[snd], ay[snd]
    rng = torch.hypot(qx - tx[it][:, None], qy - ty[it][:, None]) + p.range_sigma * _normals(r[0], r[1])[0]

    move = {"ax": ax, "ay": ay, "tx": tx, "ty": ty}
    none = dict.fromkeys(("reward", "done", "actions", "obs"))
    if "tracker" in case:
        return _exact_learned(case, seed, p, st, x, on, qx, qy, rng, tx[it], ty[it], none, move)
    ex, ey = (torch.empty(nf, dtype=torch.float64, device=dev) for _ in "xy")
    P = p.n_particles
    block = max(1, (1 << 25) // P)
    odd = torch.arange(P, device=dev) % 2 == 1
    for f0 in range(0, nf, block):
        f = torch.arange(f0, min(nf, f0 + block), device=dev)
        half = torch.arange((P + 1) // 2, device=dev)[None, :].expand(len(f), -1)
        r = _draw(f[:, None].expand_as(half), half, g, 11, seed)
        n = [v.repeat_interleave(2, 1)[:, :P] for v in (*_normals(r[0], r[1]), *_normals(r[2], r[3]))]
        sl = slice(f0 * P, (f0 + len(f)) * P)
        vx, vy = (st[c][sl].view(-1, P).double() + p.pf_accel_sigma * torch.where(odd, n[i + 2], n[i])
                  for i, c in enumerate(("pvx", "pvy")))
        cap = torch.clamp(p.pf_vcap / torch.hypot(vx, vy), max=1.0)
        X = st["px"][sl].view(-1, P).double() + p.dt * vx * cap
        Y = st["py"][sl].view(-1, P).double() + p.dt * vy * cap
        ll = torch.zeros_like(X)
        for m in range(A):
            d = torch.hypot(X - qx[f, m][:, None], Y - qy[f, m][:, None]) - rng[f, m][:, None]
            ll -= torch.where(on[f, m][:, None], d * d, 0.0) / (2 * p.range_sigma ** 2)
        w = torch.exp(ll - ll.amax(1, keepdim=True))
        ex[f], ey[f] = (w * X).sum(1) / w.sum(1), (w * Y).sum(1) / w.sum(1)
    err = torch.hypot(ex - tx[it], ey - ty[it])
    return ({**none, "estx": ex, "esty": ey, "err": err},
            {**dict.fromkeys(("px", "py", "pvx", "pvy")), **move, "apsi": psi, "tpsi": tpsi, "estx": ex, "esty": ey})


def _exact_learned(case, seed, p, st, x, on, qx, qy, rng, tx, ty, none, move):
    g, L = STEP0 + 1, p.est_scale
    new = torch.stack([qx, qy, rng, torch.full_like(qx, g)], 2)
    ring = torch.cat([_ring(p, seed, st).double(), new], 1).flip(1)[:, :16]  # newest first
    e1x, e1y, e2x, e2y = (x[k] for k in ("estx", "esty", "prev_estx", "prev_esty"))
    vx, vy = 0.85 * x["velx"] + 0.15 * (e1x - e2x), 0.85 * x["vely"] + 0.15 * (e1y - e2y)
    dx, dy = ring[..., 0] - e1x[:, None], ring[..., 1] - e1y[:, None]
    f = torch.zeros(len(e1x), 96, dtype=torch.float64, device="cuda")
    f[:, :80] = torch.stack([dx / L, dy / L, (ring[..., 2] - torch.hypot(dx, dy)) / L, (g - ring[..., 3]) / 16,
                             torch.ones_like(dx)], 2).flatten(1)
    f[:, 80], f[:, 81], f[:, 82], f[:, 83] = (e1x - e2x) / L, (e1y - e2y) / L, vx / L, vy / L
    out = _mlp(torch.from_numpy(_params(_mlp_shapes(), seed + 5, 0.1)).cuda().double(), f).clamp(-3, 3)
    ex, ey = e1x + L * out[:, 0], e1y + L * out[:, 1]
    return ({**none, "estx": ex, "esty": ey, "err": torch.hypot(ex - tx, ey - ty)},
            {**move, "velx": vx, "vely": vy, "prev_estx": e1x, "prev_esty": e1y})


def _split(prm, shapes):
    out, at = [], 0
    for _, s in shapes:
        n = int(np.prod(s))
        out.append(prm[at:at + n].view(s))
        at += n
    return out


def _mlp(prm, x):
    w = _split(prm, _mlp_shapes())
    for k in range(3):
        x = torch.nn.functional.gelu(x @ w[2 * k].T + w[2 * k + 1])
    return x @ w[6].T + w[7]


def _agent(prm, d, layers, n_out, tok, ne, h):
    """The transformer of the agents and the critic: head output and the
    recurrent token after the last block."""
    w = iter(_split(prm, _agent_shapes(d, layers, n_out)))
    F = torch.nn.functional
    We, be = next(w), next(w)
    n, S, _ = tok.shape
    H = d // 16
    x = torch.cat([h[:, None], tok @ We.T + be], 1)
    off = (torch.arange(S + 1, device=tok.device)[None] > ne[:, None])[:, None, None]
    for _ in range(layers):
        g1, c1, Wqkv, bqkv, Wo, bo, g2, c2, W1, b1, W2, b2 = (next(w) for _ in range(12))
        q, k, v = (t.view(n, S + 1, H, 16).transpose(1, 2) for t in
                   (F.layer_norm(x, (d,), g1, c1) @ Wqkv.T + bqkv).split(d, -1))
        att = (q @ k.transpose(2, 3) / 4).masked_fill(off, -math.inf).softmax(-1) @ v
        x = x + att.transpose(1, 2).reshape(n, S + 1, d) @ Wo.T + bo
        x = x + F.gelu(F.layer_norm(x, (d,), g2, c2) @ W1.T + b1) @ W2.T + b2
    gf, cf, Wh, bh = (next(w) for _ in range(4))
    return F.layer_norm(x[:, 0], (d,), gf, cf) @ Wh.T + bh, x[:, 0]


def _exact_net(case, seed):
    prm, tok, ne, h, more = _net_inputs(case, seed)
    d, L, kind = case["d"], case["layers"], case["kind"]
    n_out = 1 if kind == "critic" else 7
    w = torch.from_numpy(prm).cuda().double().requires_grad_(kind != "policy")
    n, total = len(ne), None
    outs = []
    for i in range(0, n, 4096):
        sl = slice(i, i + 4096)
        h_in = h[sl].bfloat16() if kind == "policy" else h[sl]
        z, hn = _agent(w, d, L, n_out, tok[sl].double(), ne[sl], h_in.double())
        if kind == "policy":
            outs.append((z, hn))
            continue
        if kind == "critic":
            loss = ((z[:, 0] - more["returns"][sl].double()) ** 2).sum() / n
        else:
            lp = z.log_softmax(-1)
            ratio = (lp.gather(1, more["actions"][sl].long()[:, None])[:, 0] - more["logp_old"][sl].double()).exp()
            adv = more["adv"][sl].double()
            gain = torch.minimum(ratio * adv, ratio.clamp(0.8, 1.2) * adv)
            loss = -(gain + 0.01 * -(lp.exp() * lp).sum(-1)).sum() / n
        (grad,) = torch.autograd.grad(loss, w)
        total = grad if total is None else total + grad
    if kind == "policy":
        return torch.cat([o[0] for o in outs]), None, torch.cat([o[1] for o in outs])
    return total


def exact(case, seed):
    kind = case["kind"]
    if kind == "rollout" or (kind == "step" and case.get("d")):
        return None  # many steps, or steps whose actions come from the agent: one step and the agent are cases of their own
    if kind == "step":
        return _exact_step(case, seed)
    if kind == "estimator":
        X, Y = _features(case["batch"], seed)
        w = torch.from_numpy(_params(_mlp_shapes(), seed + 5)).cuda().double().requires_grad_()
        loss = torch.nn.functional.huber_loss(_mlp(w, X.double()), Y.double(), reduction="sum") / case["batch"]
        (grad,) = torch.autograd.grad(loss, w)
        return float(loss.detach()), grad
    return _exact_net(case, seed)
