"""The measured cases: what a user of this library has it do, through the public binding (auvenv.Env, Learner, ReplayBuffer).

A training program collects trajectories (env_rollout, env_step), turns them into advantages (env_observe, env_value,
env_gae), updates the networks (ppo_update, or ppo_grads and ppo_apply when gradients are averaged between ranks), or
differentiates through the simulator (env_shac_window), or feeds an off-policy learner (rbuf_insert, rbuf_sample).  Each
kind below is one of these calls; the listed sizes are the repository's workload presets and its benchmark's, the paper's
4,096 envs, and ragged sizes around them.

`exact` restates every path in 64-bit torch from the definitions in include/auvenv.h.  Tolerances are about four times the
distance between the library's results and that restatement, where the distance is rounding (32-bit sums, tf32 or bf16
operands) carried through the closed loop; inputs of one seed give the same bits on every run.
"""
import math

import numpy as np
import torch

from paper_2512_13359_gb300 import auvenv
from paper_2512_13359_gb300 import workloads as W

M32 = 0xFFFFFFFF
GAMMA, LAM = 0.99, 0.95


# ---- the cases ------------------------------------------------------------------------------------------------------------
def listed():
    return [
        # A host loop that steps the envs one control step a call (evaluation, a deployed controller): latency and launches.
        dict(name="step_256", kind="step", model="fossen", mlp="bf16", hidden=256, heads=16, value=False, n=256, steps=1, substeps=4, dr=1, full=False),
        # The smallest preset: 64 envs x 200 steps, exact fp32 networks of width 64, rewards and dones.
        dict(name="rollout_tiny_64", kind="rollout", model="fossen", mlp="fp32", hidden=64, heads=8, value=False, n=64, steps=200, substeps=1, dr=0, full=False),
        # The fp32 preset as its mlp="fp32" default runs it (exact 32-bit networks), the paper's env count.
        dict(name="rollout_fp32_4096", kind="rollout", model="fossen", mlp="fp32", hidden=256, heads=8, value=False, n=4096, steps=100, substeps=4, dr=0, full=False),
        # The domain-randomised preset with tf32 networks: 16,384 envs, rewards and dones.
        dict(name="rollout_dr_16384", kind="rollout", model="fossen", mlp="tf32", hidden=256, heads=8, value=False, n=16384, steps=128, substeps=4, dr=1, full=False),
        # The paper's own environment at its largest setting, 4,096 envs: a 50-step segment with full trajectory and values
        # (over a whole episode its closed loop grows bf16 rounding to a fifth of the observations).
        dict(name="rollout_paper_4096", kind="rollout", model="paper", mlp="bf16", hidden=256, heads=12, value=True, n=4096, steps=50, substeps=4, dr=1, full=True),
        # The benchmark's collection pass: 65,536 envs x 128 steps, bf16 networks, full trajectory and values.
        dict(name="rollout_ppo_65536", kind="rollout", model="fossen", mlp="bf16", hidden=256, heads=16, value=True, n=65536, steps=128, substeps=4, dr=1, full=True),
        # Advantages of a ragged batch: bootstrap value of the current observation, then GAE over the trajectory.
        dict(name="advantages_50007", kind="advantages", model="fossen", mlp="bf16", hidden=256, heads=16, value=True, n=50007, steps=100, substeps=4, dr=1, full=True),
        # One PPO epoch in the learner's fast mode: 32 gradient steps of 65,536 samples.
        dict(name="update_bf16_65536", kind="update", model="fossen", precision="bf16", hidden=256, n=65536, steps=32, batch=65536),
        # One data-parallel gradient step (gradient out, then Adam) of the paper model's networks, tf32, ragged minibatch.
        dict(name="grads_tf32_30011", kind="grads", model="paper", precision="tf32", hidden=256, n=4096, steps=64, batch=30011),
        # SHAC's actor gradient at the benchmark's size, tf32 products.
        dict(name="shac_tf32_65536", kind="shac", model="fossen", precision="tf32", hidden=256, n=65536, steps=32, substeps=4, dr=1, critic=True),
        # The same of the paper's environment at its env count in exact fp32.
        dict(name="shac_fp32_paper_4096", kind="shac", model="paper", precision="fp32", hidden=256, n=4096, steps=32, substeps=4, dr=1, critic=True),
        # Off-policy storage: a rollout into a wrapping ring of 2^22 transitions, then one 65,536-sample draw.
        dict(name="replay_65536", kind="replay", model="fossen", n=65536, steps=16, capacity=1 << 22, batch=65536),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("step", "rollout", "rollout", "rollout", "advantages", "update", "grads", "shac", "shac", "replay"))
    model = rng.choice(("fossen", "fossen", "paper"))
    act = 8 if model == "fossen" else 6
    if kind in ("step", "rollout"):
        mlp = rng.choice(("fp32", "tf32", "bf16", "bf16") if model == "fossen" else ("fp32", "bf16", "bf16"))
        hidden = rng.choice((64, 256)) if mlp == "fp32" else 256
        c = dict(kind=kind, model=model, mlp=mlp, hidden=hidden, heads=2 * act if mlp == "bf16" else rng.choice((act, 2 * act)),
                 value=mlp != "tf32" and rng.random() < 0.5, substeps=rng.choice((1, 2, 4)), dr=rng.choice((0, 1)), full=rng.random() < 0.6)
        if kind == "step":
            c.update(n=_log(rng, 1, 8192), steps=1, full=False, value=False)
        else:
            c.update(n=_log(rng, 30, 4096 if mlp == "fp32" else 65536), steps=_log(rng, 8, 50 if model == "paper" else 100 if mlp == "fp32" else 128))
            c["full"] = c["full"] or c["value"]
        return c
    if kind == "advantages":
        return dict(kind=kind, model=model, mlp="bf16", hidden=256, heads=2 * act, value=True, n=_log(rng, 100, 65536), steps=_log(rng, 5, 250),
                    substeps=4, dr=1, full=True)
    if kind in ("update", "grads"):
        precision = rng.choice(("bf16", "bf16", "tf32", "fp32"))
        n, steps = _log(rng, 512, 32768), _log(rng, 16, 64)
        rows = n * steps
        batch = min(max(_log(rng, 512, 65536), rows // 64), rows // 4) if kind == "update" else min(_log(rng, 512, 65536), rows)
        return dict(kind=kind, model=model, precision=precision, hidden=rng.choice((64, 256, 256)), n=n, steps=steps, batch=batch)
    if kind == "shac":
        return dict(kind=kind, model=model, precision=rng.choice(("tf32", "fp32")), hidden=rng.choice((64, 256)), n=_log(rng, 64, 32768),
                    steps=_log(rng, 4, 32), substeps=rng.choice((1, 2, 4)), dr=rng.choice((0, 1)), critic=rng.random() < 0.7)
    n, steps = _log(rng, 64, 65536), _log(rng, 4, 32)
    return dict(kind=kind, model=model, n=n, steps=steps, capacity=max(n * steps, _log(rng, 1 << 16, 1 << 22)), batch=_log(rng, 64, 65536))


# ---- inputs ---------------------------------------------------------------------------------------------------------------
def _workload(c, seed):
    base = "ppo_65536" if c["model"] == "fossen" else "paper_4096"
    return W.workload(base, n_envs=c["n"], steps=c["steps"], substeps=c.get("substeps", 4), hidden=c.get("hidden", 256),
                      mlp=c.get("mlp", "fp32"), policy_out=c.get("heads", 2 * _act(c)), has_value=int(c.get("value", False)),
                      dr_enable=c.get("dr", 1), current_range=0.3 if c.get("dr", 1) else 0.0, seed=seed, weight_seed=seed)


def _obs(c):
    return W.OBS_DIM if c["model"] == "fossen" else W.PAPER_OBS_DIM


def _act(c):
    return W.ACT_DIM if c["model"] == "fossen" else W.PAPER_ACT_DIM


def _cuda(a):
    return torch.from_numpy(a).cuda()


def _trajectory(c, seed):
    """A trajectory as a rollout leaves it: observations of a spread of states, actions and log-densities of the current
    policy, advantages that partly follow the action noise (a policy with something to learn), returns near the values."""
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    T, N, D, A = c["steps"], c["n"], _obs(c), _act(c)
    rand = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    obs = rand(T, D, N)
    obs[:, :3] *= 0.8
    obs[:, 3:] *= 0.5
    out = dict(obs=obs)
    if c["kind"] in ("update", "grads"):
        pw = W.mlp_weights(seed, D, c["hidden"], 2 * A, 0, 0.05)
        vw = W.mlp_weights(seed, D, c["hidden"], 1, 1, 0.05)
        act, logp, adv, ret = torch.empty(T, A, N, device="cuda"), *(torch.empty(T, N, device="cuda") for _ in range(3))
        for t in range(T):
            y = _mlp(_cuda(pw), obs[t].T, c["hidden"], 2 * A)
            ls = y[:, A:].clamp(-5.0, 2.0)
            eps = rand(N, A)
            act[t] = (y[:, :A] + ls.exp() * eps).T
            logp[t] = (-0.5 * eps * eps - ls - 0.5 * math.log(2 * math.pi)).sum(1)
            adv[t] = eps.sum(1) + 0.5 * rand(N)
            ret[t] = _mlp(_cuda(vw), obs[t].T, c["hidden"], 1)[:, 0] + obs[t, 0] + 0.5 * rand(N)
        out.update(act=act, logp=logp, adv=adv, ret=ret, pw=pw, vw=vw)
        return out
    out.update(act=rand(T, A, N), rew=-rand(T, N).abs(), value=-10.0 + rand(T, N),
               done=(torch.rand((T, N), generator=g, device="cuda") < 0.004).to(torch.uint8), last_obs=rand(D, N))
    return out


def _hp(c):
    return dict(clip_eps=0.2, vf_coef=0.5, ent_coef=0.01, max_grad_norm=0.5, lr=3e-4, adam_beta1=0.9, adam_beta2=0.999, adam_eps=1e-8,
                logstd_min=-5.0, logstd_max=2.0)


def prepare(case, seed):
    c = case
    s = dict(c=c)
    kind = c["kind"]
    if kind in ("step", "rollout", "advantages", "shac"):
        w = _workload(c, seed)
        env = s["env"] = auvenv.Env(w)
        if kind != "shac":
            env.set_weights(W.policy_weights(w), W.value_weights(w) if w["has_value"] else None)
        env.reset()
    if kind == "step":
        s["out"] = [torch.empty(_obs(c), c["n"], device="cuda"), torch.empty(c["n"], device="cuda"), torch.empty(c["n"], dtype=torch.uint8, device="cuda")]
    elif kind == "rollout":
        keys = ("obs", "act", "logp", "rew", "done") if c["full"] else ("rew", "done")
        s["traj"] = env.alloc_traj(c["steps"], keys + (("value",) if c["value"] else ()))
    elif kind == "advantages":
        s.update(_trajectory(c, seed))
        s.update(last=torch.empty(1, c["n"], device="cuda"), o=torch.empty(1, _obs(c), c["n"], device="cuda"),
                 adv=torch.empty_like(s["rew"]), ret=torch.empty_like(s["rew"]))
    elif kind in ("update", "grads"):
        tr = _trajectory(c, seed)
        lrn = s["learner"] = auvenv.Learner(_obs(c), _act(c), c["hidden"], c["batch"], precision=c["precision"], seed=seed, **_hp(c))
        lrn.set_weights(tr.pop("pw"), tr.pop("vw"))
        s.update(traj=tr, pol=torch.empty(lrn.n_policy, device="cuda"), val=torch.empty(lrn.n_value, device="cuda"),
                 stats=torch.zeros(8, device="cuda"), grad=torch.empty(lrn.n_policy + lrn.n_value, device="cuda"), j=0)
    elif kind == "shac":
        n, T = c["n"], c["steps"]
        s.update(pw=_cuda(W.mlp_weights(seed, _obs(c), c["hidden"], 2 * _act(c), 0, 0.05)), vw=_cuda(W.mlp_weights(seed, _obs(c), c["hidden"], 1, 1, 0.1)),
                 coef=torch.tensor([GAMMA ** t / (n * T) for t in range(T)], dtype=torch.float32, device="cuda"), J=torch.empty(n, device="cuda"),
                 obs=torch.empty(T, _obs(c), n, device="cuda"), rew=torch.empty(T, n, device="cuda"), done=torch.empty(T, n, dtype=torch.uint8, device="cuda"))
        s["grad"] = torch.empty_like(s["pw"])
    else:
        s.update(traj=_trajectory(c, seed), rb=auvenv.ReplayBuffer(_obs(c), _act(c), c["capacity"]), seed=seed, draw=0)
    return s


# ---- one pass -------------------------------------------------------------------------------------------------------------
def run(s):
    c, kind = s["c"], s["c"]["kind"]
    if kind == "step":
        s["env"].step(*s["out"])
        return s["out"] + [s["env"].state]
    if kind == "rollout":
        s["env"].rollout(c["steps"], s["traj"])
        return dict(s["traj"], state=s["env"].state)
    if kind == "advantages":
        env = s["env"]
        env.observe(s["o"])
        env.value(s["o"], s["last"])
        env.gae(s["rew"], s["done"], s["value"], s["last"], GAMMA, LAM, s["adv"], s["ret"])
        return dict(last=s["last"], adv=s["adv"], ret=s["ret"])
    if kind == "update":
        s["learner"].update(s["traj"], 1, _minibatches(c), s["stats"])
        s["learner"].export_weights(s["pol"], s["val"])
        return dict(policy=s["pol"], value=s["val"], stats=s["stats"])
    if kind == "grads":
        s["learner"].grads(s["traj"], 0, s["j"] % _minibatches(c), s["grad"], s["stats"])
        s["learner"].apply(s["grad"], s["stats"])
        s["learner"].export_weights(s["pol"], s["val"])
        s["j"] += 1
        return dict(policy=s["pol"], value=s["val"], stats=s["stats"], grad=s["grad"])
    if kind == "shac":
        s["env"].shac_window(s["pw"], s["vw"] if c["critic"] else None, s["coef"], GAMMA ** c["steps"] / c["n"], s["grad"], s["J"], s["rew"], s["done"],
                             s["obs"], precision=c["precision"])
        return dict(grad=s["grad"], J=s["J"], rew=s["rew"], done=s["done"], obs=s["obs"], state=s["env"].state[:13])
    t = s["traj"]
    s["rb"].insert(t["obs"], t["act"], t["rew"], t["done"], t["last_obs"])
    s["draw"] += 1
    return s["rb"].sample(c["batch"], s["seed"], s["draw"], with_idx=True)


def _minibatches(c):
    return c["n"] * c["steps"] // c["batch"]


# ---- what a pass cannot do without ------------------------------------------------------------------------------------------
def _net_flops(c, out):
    H = c["hidden"]
    return 2 * (_obs(c) * H + H * H + H * out)


def work(case):
    c, kind, n, T = case, case["kind"], case["n"], case["steps"]
    D, A = _obs(c), _act(c)
    state = 4 * n * (38 if c["model"] == "fossen" else 71)
    sub = 378 if c["model"] == "fossen" else 245
    if kind in ("step", "rollout"):
        step = _net_flops(c, c["heads"]) + (_net_flops(c, 1) if c["value"] else 0) + 450 + sub * c["substeps"]
        row = 5 + (4 * (D + A + 1) if c["full"] else 0) + (4 if c["value"] else 0) + (4 * D if kind == "step" else 0)
        return {"bytes": n * T * row + 2 * state, "flops": n * T * step}
    if kind == "advantages":
        return {"bytes": n * T * 17 + state + 4 * n * (D + 1), "flops": n * (_net_flops(c, 1) + 6 * T)}
    if kind in ("update", "grads"):
        steps = _minibatches(c) if kind == "update" else 1
        net = 3 * (_net_flops(c, 2 * A) + _net_flops(c, 1)) - 2 * 2 * D * c["hidden"]
        return {"bytes": steps * c["batch"] * 4 * (D + A + 3), "flops": steps * c["batch"] * net}
    if kind == "shac":
        step = 3 * _net_flops(c, 2 * A) + 3 * (450 + sub * c["substeps"])
        return {"bytes": n * T * (5 + 4 * D) + 2 * state, "flops": n * T * step + (2 * n * _net_flops(c, 1) if c["critic"] else 0)}
    return {"bytes": n * T * 4 * (D + A + 2) + n * T * 4 * (2 * D + A + 2) + 2 * c["batch"] * 4 * (2 * D + A + 2), "flops": 0}


def tolerance(case):
    kind = case["kind"]
    if kind == "replay":
        return "exact"   # copies and counter-based draws
    p = case.get("precision") or case.get("mlp")
    if p == "fp32":      # 32-bit sums, through up to 200 steps of closed loop or 64 Adam steps
        return {"rel": 1e-5, "max": 4e-3}
    if kind in ("step", "rollout"):   # rounding of the networks' operands, carried through the closed loop
        return {"rel": 3e-2, "max": 0.9}
    if kind == "advantages":          # the bootstrap value's bf16 network
        return {"rel": 1.6e-2, "max": 0.3}
    if kind == "shac":                # tf32 products; the gradient is a sum of terms that mostly cancel
        return {"rel": 3e-2, "max": 0.9}
    return {"rel": {"tf32": 4e-3, "bf16": 3e-2}[p], "max": {"tf32": 0.1, "bf16": 0.9}[p]}


# ---- the same in 64 bits ----------------------------------------------------------------------------------------------------
def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 over int64 tensors holding 32-bit words."""
    def mul(a, b):
        hi, lo = a * (b >> 16), a * (b & 0xFFFF)
        lo = ((hi & 0xFFFF) << 16) + lo
        return ((hi >> 16) + (lo >> 32)) & M32, lo & M32
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c0, c1, c2, c3


def _uniforms(ids, seed, index, stream, blocks):
    z = torch.zeros_like(ids)
    x = [w for b in range(blocks) for w in _philox(z + (index & M32), z + (index >> 32), z + stream, z + b, ids, z + seed)]
    return torch.stack([(2 * (v >> 9) + 1).double() * 2.0 ** -24 for v in x])


def _normals(ids, seed, t):
    u = _uniforms(ids, seed, t, 0, 2)
    r, ph = torch.sqrt(-2 * torch.log(u[0::2])), 2 * math.pi * u[1::2]
    return torch.stack([r * torch.cos(ph), r * torch.sin(ph)], 1).reshape(8, -1)


def _mlp(flat, x, H, out):
    """tanh MLP on rows x [n][in] with the flat [W1 | b1 | W2 | b2 | W3 | b3] weights."""
    D, o, p = x.shape[1], 0, []
    for shape in ((H, D), (H,), (H, H), (H,), (out, H), (out,)):
        p.append(flat[o:o + math.prod(shape)].reshape(shape))
        o += math.prod(shape)
    h = torch.tanh(torch.addmm(p[1], x, p[0].T))
    return torch.addmm(p[5], torch.tanh(torch.addmm(p[3], h, p[2].T)), p[4].T)


def _cross(a, b):
    return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]])


def _qmul(a, b):
    av, bv = a[1:], b[1:]
    return torch.cat([(a[0] * b[0] - (av * bv).sum(0))[None], a[0] * bv + b[0] * av + _cross(av, bv)])


def _rot(q):
    w, x, y, z = q
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]).reshape(3, 3, -1)


def _euler(roll, pitch, yaw):
    def axis(k, a):
        q = torch.zeros(4, a.numel(), dtype=torch.float64, device=a.device)
        q[0], q[1 + k] = torch.cos(a / 2), torch.sin(a / 2)
        return q
    return _qmul(axis(2, yaw), _qmul(axis(1, pitch), axis(0, roll)))


class _Sim:
    """The envs of one workload, [rows][n] float64 tensors; the step is differentiable."""

    def __init__(self, w, ids):
        self.w, self.ids, self.paper = w, ids, W.is_paper(w)
        self.ep, self.f = 0, (lambda v: torch.tensor(np.asarray(v, np.float64), device="cuda").reshape(-1, 1))
        if self.paper:
            m, inertia = w["mass"], np.asarray(w["inertia"], np.float64)
            b = np.sqrt(6.0 * (inertia.sum() - 2.0 * inertia) / m)
            rho, mu, d = w["fluid_density"], w["fluid_viscosity"], b.mean()
            self.kf = self.f(0.5 * rho * np.roll(b, -1) * np.roll(b, 1))
            self.kt = self.f(rho / 64.0 * b * (np.roll(b, -1) ** 4 + np.roll(b, 1) ** 4))
            self.cf, self.ct = 3 * math.pi * mu * d, math.pi * mu * d ** 3
        self.reset()

    def reset(self):
        w, sym = self.w, lambda u, r: (2 * u - 1) * r
        u = _uniforms(self.ids, w["seed"], self.ep, 1, 5)
        n = self.ids.numel()
        if self.paper:
            self.qd = _euler(*sym(u[3:6], w["goal_att_range"]))
            self.q = _euler(*sym(u[10:13], w["init_att_range"]))
            self.pd, self.p = sym(u[0:3], w["goal_pos_range"]), sym(u[7:10], w["init_pos_range"])
            self.g = w["g_eff"] + (sym(u[6], w["dr_gravity_range"]) if w["dr_enable"] else torch.zeros_like(u[6]))
            self.hist = [torch.zeros(6, n, dtype=torch.float64, device="cuda") for _ in range(w["mavg_len"])]
        else:
            self.p, self.pd, self.Vc = sym(u[0:3], w["init_pos_range"]), sym(u[6:9], w["goal_pos_range"]), sym(u[10:13], w["current_range"])
            self.q = _euler(*sym(u[3:6], w["init_att_range"]))
            self.qd = _euler(torch.zeros_like(u[0]), torch.zeros_like(u[0]), sym(u[9], w["goal_yaw_range"]))
            one, dr = torch.ones_like(u[0]), w["dr_enable"]
            lo, span = w["dr_scale_lo"], w["dr_scale_hi"] - w["dr_scale_lo"]
            self.sm, self.sa, self.sd = (u[13:16] * span + lo) if dr else (one, one, one)
            self.dB = sym(u[16], w["dr_buoy_range"]) if dr else 0 * one
            self.rb = sym(u[17:20], w["dr_cob_range"]) if dr else torch.zeros_like(u[0:3])
        self.nu = torch.zeros(6, n, dtype=torch.float64, device="cuda")
        self.nup, self.t_ep = self.nu, 0
        self.ep += 1

    def error_quat(self):
        return _qmul(torch.cat([self.qd[:1], -self.qd[1:]]), self.q)

    def observe(self):
        dp = torch.einsum("jin,jn->in", _rot(self.q), self.p - self.pd)
        qe = self.error_quat()
        if not self.paper:
            return torch.cat([dp, _rot(qe).transpose(0, 1).reshape(9, -1), self.nu])
        qe = qe * torch.where(qe[0] < 0, -1.0, 1.0)
        vn2 = (qe[1:] ** 2).sum(0)
        vn = torch.sqrt(torch.where(vn2 > 0, vn2, torch.ones_like(vn2)))
        th = torch.where(vn2 > 0, 2 * torch.atan2(vn, qe[0]) / vn, 2 / qe[0])
        return torch.cat([dp, th * qe[1:], self.nu])

    def substep(self, tau):
        w, h = self.w, self.w["dt"] / self.w["substeps"]
        R, v, om = _rot(self.q), self.nu[:3], self.nu[3:]
        inertia = self.f(w["inertia"])
        if self.paper:
            m = w["mass"]
            lin = (tau[:3] - self.kf * v.abs() * v - self.cf * v - m * self.g * R[2] - m * _cross(om, v)) / m
            rot = (tau[3:] - self.kt * om.abs() * om - self.ct * om - _cross(om, inertia * om)) / inertia
        else:
            A, dl, dq = self.f(w["added_mass"]), self.f(w["damp_lin"]), self.f(w["damp_quad"])
            grav = np.asarray(w["gravity"], np.float64)
            gn = float(np.linalg.norm(grav))
            Rt = R.transpose(0, 1)
            vc, kb = torch.einsum("ijn,jn->in", Rt, self.Vc), torch.einsum("ijn,jk->in", Rt, self.f(grav / gn))
            m, vr = self.sm * w["mass"], v - vc
            A1, A2 = self.sa * A[:3], self.sa * A[3:]
            nur = torch.cat([vr, om])
            damp = self.sd * (dl + dq * nur.abs()) * nur
            lin = tau[:3] - m * _cross(om, v) - _cross(om, A1 * vr) - damp[:3] - self.dB * kb - A1 * _cross(om, vc)
            rot = (tau[3:] - _cross(om, self.sm * inertia * om) - _cross(vr, A1 * vr) - _cross(om, A2 * om) - damp[3:]
                   - (m * gn + self.dB) * _cross(self.rb, kb))
            lin, rot = lin / (m + A1), rot / (self.sm * inertia + A2)
        self.nu = self.nu + h * torch.cat([lin, rot])
        self.p = self.p + h * torch.einsum("ijn,jn->in", R, self.nu[:3])
        half = 0.5 * h * self.nu[3:]
        a = torch.sqrt((half * half).sum(0))
        dq = torch.cat([torch.cos(a)[None], torch.where(a > 0, torch.sin(a) / a, torch.ones_like(a)) * half])
        q = _qmul(self.q, dq)
        self.q = q / torch.sqrt((q * q).sum(0))

    def step(self, act):
        """One control step with actions [A][n]: reward, and whether the episode ended."""
        w, ac = self.w, act.clamp(-1.0, 1.0)
        self.nup = self.nu
        tau = (torch.cat([w["f_max"] * ac[:3], w["tau_max"] * ac[3:]]) if self.paper
               else torch.tensor(w["alloc"] * w["thrust_max"], device="cuda") @ ac)
        for _ in range(w["substeps"]):
            self.substep(tau)
        if self.paper:
            o = self.observe()
            mean = sum(self.hist) / len(self.hist)
            r = (-w["w_pos"] * ((self.f(w["w_axes"]) * o[:3]) ** 2).sum(0) - w["w_att"] * (o[3:6] ** 2).sum(0) - w["w_act"] * (ac[3:] ** 2).sum(0)
                 - w["w_vel"] * (self.nu[3:] ** 2).sum(0) - w["w_mavg"] * ((ac - mean) ** 2).sum(0))
            self.hist[self.t_ep % len(self.hist)] = ac
        else:
            qe, d = self.error_quat(), self.p - self.pd
            theta = 2 * torch.atan2(torch.sqrt((qe[1:] ** 2).sum(0)), qe[0].abs())
            r = (-w["w_pos"] * torch.sqrt((d * d).sum(0)) - w["w_att"] * theta - w["w_act"] * (ac * ac).sum(0)
                 - w["w_vs"] * ((self.nu - self.nup) ** 2).sum(0))
        self.t_ep += 1
        done = self.t_ep == w["episode_len"]
        if done:
            self.reset()
        return r, done

    def rows(self):
        st = torch.cat([self.p, self.q, self.nu])
        if not self.paper:
            return torch.cat([st, self.nup])
        unused = torch.zeros(6 * (W.PAPER_HIST - len(self.hist)), st.shape[1], dtype=st.dtype, device="cuda")
        return torch.cat([st, *self.hist, unused])


def _sample(w, y, ids, t, A):
    eps = _normals(ids, w["seed"], t)[:A]
    ls = y[:, A:].T.clamp(w["logstd_min"], w["logstd_max"]) if y.shape[1] == 2 * A else torch.zeros_like(eps)
    return y[:, :A].T + torch.exp(ls) * eps, (-0.5 * eps * eps - ls - 0.5 * math.log(2 * math.pi)).sum(0)


def _exact_rollout(c, seed):
    w, T, A = _workload(c, seed), c["steps"], _act(c)
    ids = torch.arange(c["n"], device="cuda")
    sim = _Sim(w, ids)
    pw = _cuda(W.policy_weights(w)).double()
    vw = _cuda(W.value_weights(w)).double() if c["value"] else None
    keys = ("obs", "act", "logp", "rew", "done") if c["full"] or c["kind"] == "step" else ("rew", "done")
    out = {k: [] for k in keys + (("value",) if c["value"] else ())}
    for t in range(T):
        o = sim.observe()
        a, lp = _sample(w, _mlp(pw, o.T, w["hidden"], w["policy_out"]), ids, t, A)
        r, done = sim.step(a)
        row = dict(obs=o, act=a, logp=lp, rew=r, done=torch.full((c["n"],), int(done), dtype=torch.uint8, device="cuda"))
        if c["value"]:
            row["value"] = _mlp(vw, o.T, w["hidden"], 1)[:, 0]
        for k in out:
            out[k].append(row[k])
    out = {k: torch.stack(v) for k, v in out.items()}
    if c["kind"] == "step":
        return [out["obs"][0], out["rew"][0], out["done"][0], sim.rows()]
    return dict(out, state=sim.rows())


def _exact_advantages(c, seed):
    w, tr = _workload(c, seed), _trajectory(c, seed)
    sim = _Sim(w, torch.arange(c["n"], device="cuda"))
    last = _mlp(_cuda(W.value_weights(w)).double(), sim.observe().T, w["hidden"], 1)[:, 0]
    rew, v, live = tr["rew"].double(), tr["value"].double(), 1.0 - tr["done"].double()
    adv, a, nxt = torch.empty_like(rew), torch.zeros_like(last), last
    for t in range(c["steps"] - 1, -1, -1):
        a = rew[t] + GAMMA * live[t] * nxt - v[t] + GAMMA * LAM * live[t] * a
        adv[t], nxt = a, v[t]
    return dict(last=last[None], adv=adv, ret=adv + v)


def _permutation(seed, epoch, m, start, count):
    """Positions start .. start + count - 1 of the epoch's cycle-walked Feistel permutation of [0, m)."""
    bits = 2
    while (1 << bits) < m:
        bits += 2
    h, mask = bits // 2, (1 << (bits // 2)) - 1

    def feistel(x):
        left, right, z = x >> h, x & mask, torch.zeros_like(x)
        for j in range(4):
            f = _philox(right, z + j, z + epoch, z, z + seed, z)[0]
            left, right = right, left ^ (f & mask)
        return (left << h) | right
    x = feistel(torch.arange(start, start + count, device="cuda"))
    while bool((x >= m).any()):
        x = torch.where(x >= m, feistel(x), x)
    return x


def _exact_learner(c, seed):
    tr, hp = _trajectory(c, seed), _hp(c)
    T, N, A, B, H = c["steps"], c["n"], _act(c), c["batch"], c["hidden"]
    np_ = W.mlp_param_count(_obs(c), H, 2 * A)
    wt = torch.cat([_cuda(tr["pw"]), _cuda(tr["vw"])]).double().requires_grad_()
    m = v = torch.zeros_like(wt)
    steps = _minibatches(c) if c["kind"] == "update" else 1
    acc = torch.zeros(8, dtype=torch.float64, device="cuda")
    for k in range(steps):
        rows = _permutation(seed, 0, T * N, k * B, B)
        t, i = rows // N, rows % N
        x, a = tr["obs"][t, :, i].double(), tr["act"][t, :, i].double()
        lp0, adv, ret = (tr[q][t, i].double() for q in ("logp", "adv", "ret"))
        y, val = _mlp(wt[:np_], x, H, 2 * A), _mlp(wt[np_:], x, H, 1)[:, 0]
        ls = y[:, A:].clamp(hp["logstd_min"], hp["logstd_max"])
        lp = (-0.5 * ((a - y[:, :A]) / ls.exp()) ** 2 - ls - 0.5 * math.log(2 * math.pi)).sum(1)
        r, an = torch.exp(lp - lp0), (adv - adv.mean()) / (adv.std() + 1e-8)
        pg = torch.maximum(-an * r, -an * r.clamp(1 - hp["clip_eps"], 1 + hp["clip_eps"])).mean()
        vl, ent = 0.5 * ((val - ret) ** 2).mean(), (ls + 0.5 * (1 + math.log(2 * math.pi))).sum(1).mean()
        loss = pg + hp["vf_coef"] * vl - hp["ent_coef"] * ent
        g, = torch.autograd.grad(loss, wt)
        norm = g.norm()
        one = torch.ones_like(norm)
        acc = acc + torch.stack([pg, vl, ent, (lp0 - lp).mean(), ((r - 1).abs() > hp["clip_eps"]).double().mean(), norm, loss, one]).detach()
        gc = g * torch.clamp(hp["max_grad_norm"] / (norm + 1e-6), max=1.0)
        b1, b2 = hp["adam_beta1"], hp["adam_beta2"]
        m, v = b1 * m + (1 - b1) * gc, b2 * v + (1 - b2) * gc * gc
        new = wt - hp["lr"] * (m / (1 - b1 ** (k + 1))) / (torch.sqrt(v / (1 - b2 ** (k + 1))) + hp["adam_eps"])
        wt = new.detach().requires_grad_()
    stats = acc / steps
    stats[7] = steps
    out = dict(policy=wt.detach()[:np_], value=wt.detach()[np_:], stats=stats)
    return dict(out, grad=g) if c["kind"] == "grads" else out


def _exact_shac(c, seed):
    w, T, A, H = _workload(c, seed), c["steps"], _act(c), c["hidden"]
    pw = _cuda(W.mlp_weights(seed, _obs(c), H, 2 * A, 0, 0.05)).double().requires_grad_()
    vw = _cuda(W.mlp_weights(seed, _obs(c), H, 1, 1, 0.1)).double()
    parts, grad = [], torch.zeros_like(pw)
    for i0 in range(0, c["n"], 8192):   # groups of envs: the tape of 65,536 does not fit
        ids = torch.arange(i0, min(i0 + 8192, c["n"]), device="cuda")
        sim, J, rows = _Sim(w, ids), 0.0, []
        for t in range(T):
            o = sim.observe()
            a, _ = _sample(w, _mlp(pw, o.T, H, 2 * A), ids, t, A)
            r, done = sim.step(a)
            J = J + GAMMA ** t / (c["n"] * T) * r
            rows.append((o.detach(), r.detach(), torch.full(r.shape, int(done), dtype=torch.uint8, device="cuda")))
        if c["critic"]:
            J = J + GAMMA ** T / c["n"] * _mlp(vw, sim.observe().T, H, 1)[:, 0]
        g, = torch.autograd.grad(J.sum(), pw)
        grad = grad + g
        parts.append((J.detach(), *(torch.stack(x) for x in zip(*rows)), sim.rows()[:13].detach()))
    J, obs, rew, done, state = (torch.cat(x, -1) for x in zip(*parts))
    return dict(grad=grad.detach(), J=J, rew=rew, done=done, obs=obs, state=state)


def _exact_replay(c, seed):
    tr = _trajectory(c, seed)
    T, N, C, B = c["steps"], c["n"], c["capacity"], c["batch"]
    size = min(T * N, C)
    z = torch.zeros(B, dtype=torch.int64, device="cuda")
    word = _philox(z + torch.arange(B, device="cuda"), z + 0x52420000, z + 1, z, z + seed, z)[0]
    idx = (word * size) >> 32
    at = T * N - 1 - (T * N - 1 - idx) % C      # the last transition written to that slot
    t, i = at // N, at % N
    nxt = torch.cat([tr["obs"][1:], tr["last_obs"][None]])
    return dict(obs=tr["obs"][t, :, i], act=tr["act"][t, :, i], rew=tr["rew"][t, i], next_obs=nxt[t, :, i], done=tr["done"][t, i], idx=idx.to(torch.int32))


def exact(case, seed):
    kind = case["kind"]
    f = {"step": _exact_rollout, "rollout": _exact_rollout, "advantages": _exact_advantages, "update": _exact_learner, "grads": _exact_learner,
         "shac": _exact_shac, "replay": _exact_replay}[kind]
    return f(case, seed)
