"""The calls whose speed is measured: the steps of a training run and of a fleet
study, as a program that uses this library makes them, over the sizes of its
own workload presets.

Every kind goes through the public binding (``paper_2608_11226_gb300.pe``):

  iteration  rollout, GAE and PPO update of one small fp32 training iteration
  rollout    E envs x T steps under the policy network, then the value network
  replay     recorded actions replayed over the envs (no network)
  rule       the evaluation's baseline rule policies (no network)
  value      the value network on a batch of stored observations
  gae        generalised advantage estimation over a rollout buffer
  update     one PPO update (epochs x minibatches)
  fleet      window accounting of N composed fleets
  stagger    the greedy phase-staggered schedule

``exact`` restates each in 64 bits with plain torch, from the definitions in
the C header and not from the library's code.
"""
import math

import numpy as np
import torch

from paper_2608_11226_gb300 import pe
from paper_2608_11226_gb300 import workloads as W

GAMMA, LAMBDA = 0.99, 0.95
# networks by the preset that uses them
NETS = {"tiny": W.NetSpec(8, 64, 3, W.DTYPE_F32), "7b": W.NetSpec(16, 128, 5, W.DTYPE_F32),
        "72b": W.NetSpec(32, 256, 16, W.DTYPE_BF16), "stress": W.NetSpec(64, 512, 16, W.DTYPE_BF16)}
WINDOWS = (1, 60, 600)  # 0.5 s, 30 s and 5 min in half-second samples


def listed():
    return [
        # the Tiny preset whole: 64 envs x 128 steps, where launches and latency count
        dict(name="tiny_iteration", kind="iteration", preset="tiny", E=64, T=128, minibatch=2048, epochs=4),
        # one rollout of the 7B preset (its own envs and horizon), fp32 networks
        dict(name="rollout_7b", kind="rollout", preset="7b", E=4096, T=512),
        # the 72B preset's 65,536 envs on the bf16 networks, a slice of its 1,024 steps
        dict(name="rollout_72b", kind="rollout", preset="72b", E=65536, T=64),
        # the Stress preset's 262,144 envs, a slice of its 2,048 steps
        dict(name="rollout_stress", kind="rollout", preset="stress", E=262144, T=8),
        # recorded controllers replayed at the batch cadence, an odd number of envs
        dict(name="replay_cadence", kind="replay", preset="72b_cadence", E=10007, T=64),
        # GAE of the 7B rollout (narrow) and of the Stress rollout (the widest and longest)
        dict(name="gae_7b", kind="gae", E=4096, T=512),
        dict(name="gae_stress", kind="gae", E=262144, T=2048),
        # PPO updates at each preset's minibatch, over a slice of its rollout
        dict(name="update_7b", kind="update", preset="7b", n=131072, minibatch=8192, epochs=4),
        dict(name="update_72b", kind="update", preset="72b", n=524288, minibatch=65536, epochs=4),
        dict(name="update_stress", kind="update", preset="stress", n=262144, minibatch=65536, epochs=4),
        # a tenth of the fleet study's million compositions over its whole period
        dict(name="fleet_windows", kind="fleet", N=100000, L=380000, nw=3),
        # the phase-staggered schedule with every offset of the period as a candidate
        dict(name="fleet_stagger", kind="stagger", L=60000, stride=1, w=60),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["iteration", "rollout", "rollout", "replay", "rule", "value", "gae", "update", "update",
                       "fleet", "stagger"])
    if kind == "iteration":
        T = _log(rng, 32, 256)
        E = _log(rng, 16, 512)
        return dict(kind=kind, preset="tiny", E=E, T=T, minibatch=_log(rng, 256, max(512, E * T // 2)), epochs=rng.randint(1, 4))
    if kind == "rollout":
        preset = rng.choice(["tiny", "7b", "72b", "stress"])
        E = _log(rng, *{"tiny": (16, 4096), "7b": (256, 8192), "72b": (256, 65536), "stress": (256, 262144)}[preset])
        most = {"tiny": 256, "7b": 512, "72b": 64, "stress": 16}[preset]
        return dict(kind=kind, preset=preset, E=E, T=_log(rng, 4, most))
    if kind == "replay":
        return dict(kind=kind, preset=rng.choice(["7b", "72b", "72b_cadence", "stress"]), E=_log(rng, 100, 65536),
                    T=_log(rng, 8, 64))
    if kind == "rule":
        return dict(kind=kind, preset=rng.choice(["7b", "72b"]), rule=rng.choice(["random", "threshold", "hysteresis"]),
                    E=_log(rng, 100, 65536), T=_log(rng, 8, 256))
    if kind == "value":
        return dict(kind=kind, preset=rng.choice(["tiny", "7b", "72b", "stress"]), n=_log(rng, 64, 1 << 20))
    if kind == "gae":
        T = _log(rng, 64, 2048)
        return dict(kind=kind, E=_log(rng, 64, 262144), T=T)
    if kind == "update":
        preset = rng.choice(["7b", "72b", "stress"])
        mb = _log(rng, *{"7b": (512, 16384), "72b": (4096, 65536), "stress": (4096, 65536)}[preset])
        return dict(kind=kind, preset=preset, n=int(mb * rng.uniform(1.0, 4.0)), minibatch=mb, epochs=rng.randint(1, 4))
    if kind == "fleet":
        L = _log(rng, 4000, 380000)
        return dict(kind=kind, N=_log(rng, 200, min(100000, 20000000000 // L)), L=L, nw=rng.randint(1, 3))
    L = _log(rng, 3000, 60000)
    return dict(kind=kind, L=L, stride=rng.choice([1, 1, 4, 10]), w=rng.choice([1, 60, 600]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _workload(preset, E, seed):
    if preset == "tiny":
        return W.make_tiny(n_envs=E, seed=seed)
    if preset == "7b":
        return W.make_7b(n_envs=E, seed=seed)
    if preset == "72b":
        return W.make_72b(n_envs=E, seed=seed)
    if preset == "72b_cadence":
        return W.make_72b_cadence(n_envs=E, seed=seed)
    return W.make_stress(n_envs=E, seed=seed)


def _params(net, seed):
    """A controller some way into training: the initial weights with biases
    and a policy head ten times its initial size (logits around 0.1)."""
    p = torch.from_numpy(W.init_params(net, seed=seed, bias_scale=0.05))
    o = net.hidden * net.obs_dim + net.hidden + net.hidden * net.hidden + net.hidden
    p[o:o + net.n_actions * net.hidden] *= 10.0
    return p.cuda()


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _observations(preset, net, n, g):
    """Observations as the envs give them: power over budget around one, the
    occupancy and phase features on their grids, unused features zero."""
    x = 1.0 + 0.08 * torch.randn(n, net.obs_dim, generator=g, device="cuda")
    u = torch.rand(n, 3, generator=g, device="cuda")
    if preset == "tiny":
        x[:, 5] = 1.0 - x[:, 4]
        x[:, 6] = (u[:, 0] < 0.25).float()
        x[:, 7] = torch.floor(u[:, 1] * 3) / 2
    elif preset == "7b":
        x[:, 9] = 1.0 - x[:, 8]
        x[:, 10] = (u[:, 0] < 0.2).float()
        x[:, 11] = torch.floor(u[:, 1] * 6) / 5
        x[:, 12] = torch.floor(u[:, 2] * 8) / 7
        x[:, 14] -= 1.0
        x[:, 15] = 0.0
    else:
        x[:, 3] = 1.0 - x[:, 2]
        x[:, 4] -= 1.0
        x[:, 5] = torch.floor(u[:, 0] * 16 + 1) / 16
        x[:, 6] = torch.floor(u[:, 1] * 16 + 1) / 16
        x[:, 7] = torch.floor(u[:, 2] * 4) / 40
        if net.obs_dim == 32:
            x[:, 28:] = 0.0
    return x if net.dtype == W.DTYPE_F32 else x.bfloat16()


def _update_inputs(case, seed):
    net = NETS[case["preset"]]
    g = _gen(seed)
    n = case["n"]
    params = _params(net, seed)
    obs = _observations(case["preset"], net, n, g)
    logp = torch.empty(n, device="cuda")
    act = torch.empty(n, dtype=torch.uint8, device="cuda")
    pol = _split(params.double(), net)[0]
    for a in range(0, n, 65536):  # the behaviour policy that sampled the actions
        z = _mlp(pol, obs[a:a + 65536].double(), net)
        lp = torch.log_softmax(z, -1)
        gum = -torch.log(-torch.log(torch.rand(z.shape, generator=g, device="cuda").clamp(1e-7, 1 - 1e-7)))
        i = (lp + gum).argmax(-1)
        act[a:a + 65536] = i.to(torch.uint8)
        logp[a:a + 65536] = lp.gather(-1, i[:, None])[:, 0].float()
    adv = 8.0 * torch.randn(n, generator=g, device="cuda")
    ret = 20.0 * torch.randn(n, generator=g, device="cuda") - 30.0
    return params, obs, act, logp, adv, ret


def _ppo(case):
    return W.PPOSpec(epochs=case["epochs"], minibatch=case["minibatch"],
                     ent_coef=0.01 if case.get("preset") in ("72b", "stress") else 0.0)


def _rule(case, budget):
    if case["rule"] == "random":
        return W.random_rule()
    return W.threshold_rule(budget) if case["rule"] == "threshold" else W.hysteresis_rule(budget)


def _fleet(case, seed):
    fl = W.make_fleet(n_compositions=1, length=case["L"], seed=seed, windows=WINDOWS[:case.get("nw", 3)])
    return torch.from_numpy(fl.traces).cuda(), torch.from_numpy(fl.job_of_gpu).cuda(), fl.n_jobs, fl.budget_q


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, it=0)
    if kind in ("iteration", "rollout", "replay", "rule"):
        wl = _workload(case["preset"], case["E"], seed)
        s["env"] = pe.Env(wl.env, torch.from_numpy(wl.trace), torch.from_numpy(wl.phase))
        s["net"] = wl.net
        T, E = case["T"], case["E"]
        if kind == "replay":
            s["actions"] = torch.randint(0, wl.env.n_actions, (T, E), generator=_gen(seed), device="cuda").to(torch.uint8)
            s["buf"] = pe.alloc_rule_rollout(wl.env, T)
            return s
        if kind == "rule":
            s["rule"] = _rule(case, wl.env.budget_q)
            s["buf"] = pe.alloc_rule_rollout(wl.env, T)
            return s
        s["params"] = _params(wl.net, seed)
        s["buf"] = pe.alloc_rollout(wl.env, wl.net, T)
        s["ws"] = pe.alloc_workspace(pe.rollout_workspace_bytes(s["env"], wl.net))
        if kind == "iteration":
            s["adv"], s["ret"] = (torch.empty(T, E, device="cuda") for _ in range(2))
            s["seed"], n = seed, T * E
    elif kind == "value":
        s["net"] = net = NETS[case["preset"]]
        s["params"] = _params(net, seed)
        s["obs"] = _observations(case["preset"], net, case["n"], _gen(seed))
        s["out"] = torch.empty(case["n"], device="cuda")
        s["ws"] = pe.alloc_workspace(pe.value_workspace_bytes(net))
    elif kind == "gae":
        T, E, g = case["T"], case["E"], _gen(seed)
        s["reward"] = torch.randn(T, E, generator=g, device="cuda").mul_(3.0).sub_(1.0)
        s["value"] = torch.randn(T, E, generator=g, device="cuda").mul_(10.0).sub_(30.0)
        s["done"] = torch.randint(0, 500, (T, E), generator=g, device="cuda", dtype=torch.int16).eq_(0).to(torch.uint8)
        s["last"] = torch.randn(E, generator=g, device="cuda").mul_(10.0).sub_(30.0)
        s["adv"], s["ret"] = (torch.empty(T, E, device="cuda") for _ in range(2))
    elif kind == "update":
        s["net"], s["seed"], n = NETS[case["preset"]], seed, case["n"]
        s["params"], s["obs"], s["act"], s["logp"], s["adv"], s["ret"] = _update_inputs(case, seed)
    elif kind == "fleet":
        s["traces"], s["job"], s["J"], s["budget"] = _fleet(case, seed)
        s["off"] = torch.randint(0, case["L"], (case["N"], s["J"]), generator=_gen(seed), device="cuda", dtype=torch.int32)
        s["counts"], s["peaks"] = (torch.empty(case["N"], case["nw"], dtype=torch.int32, device="cuda") for _ in range(2))
        s["ws"] = pe.alloc_workspace(pe.fleet_workspace_bytes(s["J"], case["L"], case["L"]))
    else:
        s["traces"], s["job"], s["J"], s["budget"] = _fleet(case, seed)
        s["off"], s["peaks"] = (torch.empty(s["J"], dtype=torch.int32, device="cuda") for _ in range(2))
        s["ws"] = pe.alloc_workspace(pe.fleet_stagger_workspace_bytes(s["J"], case["L"], case["L"], case["stride"]))
    if kind in ("iteration", "update"):
        s["ppo"] = _ppo(case)
        s["p"], s["m"], s["v"] = s["params"].clone(), torch.zeros_like(s["params"]), torch.zeros_like(s["params"])
        s["stats"] = torch.empty(8, device="cuda")
        s["pws"] = pe.alloc_workspace(pe.ppo_workspace_bytes(s["net"], s["ppo"], n))
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _update(s, obs, act, logp, adv, ret, iteration):
    # every pass is the first update of a run: the weights start anew and so do Adam's moments
    s["p"].copy_(s["params"])
    s["m"].zero_()
    s["v"].zero_()
    pe.ppo_update(s["net"], s["ppo"], s["p"], s["m"], s["v"], 0, obs, act, logp, adv, ret, s["stats"], s["pws"],
                  seed=s["seed"], iteration=iteration)
    return dict(params=s["p"], adam_m=s["m"], adam_v=s["v"], stats=s["stats"])


def _tensors(buf):
    return {k: v for k, v in buf.items() if v is not None}


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("iteration", "rollout", "replay", "rule"):
        s["it"] += 1  # the envs go on where the last pass left them, as in a training run
    if kind == "rollout":
        pe.rollout(s["env"], s["net"], s["params"], case["T"], s["it"], s["buf"], workspace=s["ws"])
        return s["buf"]
    if kind == "iteration":
        b = s["buf"]
        pe.rollout(s["env"], s["net"], s["params"], case["T"], s["it"], b, workspace=s["ws"])
        pe.gae(b["reward"], b["value"], b["done"], b["last_value"], GAMMA, LAMBDA, s["adv"], s["ret"])
        u = _update(s, b["obs"], b["act"], b["logp"], s["adv"], s["ret"], s["it"])
        return dict(b, adv=s["adv"], ret=s["ret"], **u)
    if kind == "replay":
        pe.rollout_replay(s["env"], s["actions"], case["T"], s["it"], s["buf"])
        return _tensors(s["buf"])
    if kind == "rule":
        pe.rollout_rule(s["env"], s["rule"], case["T"], s["it"], s["buf"])
        return _tensors(s["buf"])
    if kind == "value":
        pe.value(s["net"], s["params"], s["obs"], s["out"], workspace=s["ws"])
        return s["out"]
    if kind == "gae":
        pe.gae(s["reward"], s["value"], s["done"], s["last"], GAMMA, LAMBDA, s["adv"], s["ret"])
        return dict(adv=s["adv"], ret=s["ret"])
    if kind == "update":
        return _update(s, s["obs"], s["act"], s["logp"], s["adv"], s["ret"], 1)
    if kind == "fleet":
        pe.fleet_windows(s["traces"], s["job"], s["J"], s["off"], case["L"], WINDOWS[:case["nw"]], s["budget"],
                         s["counts"], s["peaks"], s["ws"])
        return dict(counts=s["counts"], peaks=s["peaks"])
    pe.fleet_stagger(s["traces"], s["job"], s["J"], case["L"], case["w"], case["stride"], s["off"], s["peaks"], s["ws"])
    return dict(offsets=s["off"], peaks=s["peaks"])


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _net_flops(net, out):
    return 2 * (net.obs_dim * net.hidden + net.hidden * net.hidden + net.hidden * out)


def _rollout_work(case, network=True):
    E, T = case["E"], case["T"]
    # act, reward, done, power per step; counters per env
    b = E * T * (1 + 4 + 1 + 4) + E * (8 + 4 + 4 + 8 + 8)
    if not network:
        return dict(bytes=b, flops=E * T * 40)
    net = NETS[case["preset"]]
    es = 4 if net.dtype == W.DTYPE_F32 else 2
    b += E * (T + 1) * (net.obs_dim * es + 4) + E * T * 4
    return dict(bytes=b, flops=E * T * _net_flops(net, net.n_actions) + E * (T + 1) * _net_flops(net, 1))


def _update_work(net, n, epochs):
    fwd = _net_flops(net, net.n_actions) + _net_flops(net, 1)
    first = 2 * 2 * net.obs_dim * net.hidden  # no gradient with respect to the observations
    es = 4 if net.dtype == W.DTYPE_F32 else 2
    P = W.param_count(net.obs_dim, net.hidden, net.n_actions)
    return dict(bytes=n * (net.obs_dim * es + 13) + 2 * 3 * 4 * P, flops=epochs * n * (3 * fwd - first))


def work(case):
    kind = case["kind"]
    if kind in ("replay", "rule"):
        r = 33 if case["preset"] == "72b_cadence" else 1  # samples a step consumes, on average
        w = _rollout_work(case, network=False)
        return dict(bytes=w["bytes"], flops=w["flops"] * r)
    if kind == "rollout":
        return _rollout_work(case)
    if kind == "iteration":
        a, n = _rollout_work(case), case["E"] * case["T"]
        u = _update_work(NETS["tiny"], n, case["epochs"])
        return dict(bytes=a["bytes"] + u["bytes"] + 17 * n, flops=a["flops"] + u["flops"])
    if kind == "value":
        net = NETS[case["preset"]]
        es = 4 if net.dtype == W.DTYPE_F32 else 2
        return dict(bytes=case["n"] * (net.obs_dim * es + 4), flops=case["n"] * _net_flops(net, 1))
    if kind == "gae":
        n = case["E"] * case["T"]
        return dict(bytes=17 * n + 4 * case["E"], flops=8 * n)
    if kind == "update":
        return _update_work(NETS[case["preset"]], case["n"], case["epochs"])
    if kind == "fleet":
        # integer operations: one add per job and sample; a difference, a test and a maximum per window
        N, L = case["N"], case["L"]
        return dict(bytes=16 * L * 4 + N * (8 * 4 + case["nw"] * 8), flops=N * L * (8 + 3 * case["nw"]))
    # an add and a maximum per job, candidate and sample
    L = case["L"]
    return dict(bytes=16 * L * 4 + 64, flops=2 * 8 * ((L + case["stride"] - 1) // case["stride"]) * L)


def tolerance(case):
    """About four times what the start's code shows against exact(), or where
    rounding points are shared (bf16 networks) against another order of sums."""
    kind = case["kind"]
    if kind in ("replay", "rule"):
        # counts, powers and flags are whole numbers; the fp32 rewards and sums of a step or an env (1.5e-7)
        return {"rel": 1e-6, "max": 1e-5, "differ": 0.0}
    if kind in ("fleet", "stagger"):
        return "exact"
    if kind == "gae":
        return {"rel": 1e-6, "max": 4e-5}  # 1e-7 to 5e-7
    if kind == "value":
        return {"rel": 2e-6, "max": 1e-4} if NETS[case["preset"]].dtype == W.DTYPE_F32 else {"rel": 5e-3, "max": 0.1}
    if kind in ("rollout", "iteration"):
        # the fp32 outputs are 1e-6 off and the bf16 ones 1e-3, but an action next to a boundary of its
        # cumulative probability may fall on the other side, and its env then takes another way
        return {"rel": 1e-2, "max": 0.99, "differ": 2e-3}
    # an update: 2e-7 (fp32) and 2e-4 (bf16); Adam divides by the root of its second moment, so that the
    # rounding of the smallest gradients shows in single weights
    return {"rel": 2e-6, "max": 1e-2} if NETS[case["preset"]].dtype == W.DTYPE_F32 else {"rel": 1.5e-3, "max": 0.5}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _f32(x):
    """A scalar as the library receives it, in 32 bits."""
    return float(np.float32(x))


def _split(p, net):
    D, H, A = net.obs_dim, net.hidden, net.n_actions
    nets, o = [], 0
    for out in (A, 1):
        layers = []
        for rows, cols in ((H, D), (H, H), (out, H)):
            w = p[o:o + rows * cols].view(rows, cols)
            o += rows * cols
            layers.append((w, p[o:o + rows]))
            o += rows
        nets.append(layers)
    return nets


def _weight(w, net):
    """A bf16 network computes with its weights rounded to bf16 (the gradient passes to the master)."""
    return w if net.dtype == W.DTYPE_F32 else w + (w.float().bfloat16().double() - w).detach()


def _mlp(layers, x, net):
    for k, (w, b) in enumerate(layers):
        x = x @ _weight(w, net).T + b
        if k < 2:
            x = torch.tanh(x)
    return x


_M32 = 0xFFFFFFFF


def _mulhilo(m, c):
    t = m * (c & 0xFFFF)
    hi = (m * (c >> 16) + (t >> 16)) >> 16
    return hi & _M32, (t + ((m * (c >> 16)) << 16)) & _M32


def _philox(seed, c0, c1, c2, c3):
    """Philox4x32-10 of the counters (tensors of 32-bit values in int64) under the 64-bit key."""
    c = list(torch.broadcast_tensors(*[torch.as_tensor(x, device="cuda", dtype=torch.int64) for x in (c0, c1, c2, c3)]))
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
        h0, l0 = _mulhilo(0xD2511F53, c[0])
        h1, l1 = _mulhilo(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
    return c


class _Envs:
    """The environment from its definition, all envs at once: powers in whole 1/64 W, the rest in 64 bits."""

    def __init__(self, wl):
        s = self.s = wl.env
        self.E, self.C = s.n_envs, s.n_channels
        self.trace = torch.from_numpy(wl.trace).cuda().view(self.C, -1)
        self.phase = torch.from_numpy(wl.phase).cuda().long()
        if s.actuator_kind == W.ACT_INCDEC:
            sc = [[0.8 + 0.2 * l / s.g_max] * self.C for l in range(s.n_levels)]
        else:
            sc = s.level_scale
        self.scale = torch.tensor(sc, dtype=torch.float64).float().cuda()
        self.tokens = torch.tensor(s.level_tokens, dtype=torch.float32).double().cuda()
        self.ns = torch.tensor(s.level_samples or [1] * s.n_levels, device="cuda")
        self.e = torch.arange(self.E, device="cuda")
        for n in ("pos", "k", "level", "prev", "b", "til"):
            setattr(self, n, torch.zeros(self.E, dtype=torch.int64, device="cuda"))
        self.hist = torch.zeros(self.E, self.C, 60, dtype=torch.int32, device="cuda")  # newest last
        self.reset(torch.ones(self.E, dtype=torch.bool, device="cuda"), 0, 0, 2)

    def q(self, pos, level):
        """Actuated power of every channel at trace positions pos under levels, 1/64 W: [C, ...]."""
        x = self.trace[:, pos]
        on = (torch.tensor(self.s.scale_phase_mask, device="cuda") >> self.phase[pos]) & 1
        f = torch.where(on.bool(), self.scale[level].movedim(-1, 0), torch.ones((), device="cuda"))
        return torch.round(x * f * 64.0).to(torch.int32)

    def reset(self, who, t, it, purpose):
        i = who.nonzero()[:, 0]
        if not i.numel():
            return
        s = self.s
        span = s.trace_len - s.episode_len * int(self.ns.max()) - 60 + 1
        w = _philox(s.seed, i, t, it, purpose)[0]
        o = 60 + ((w * span) >> 32)
        self.pos[i], self.k[i], self.til[i] = o, 0, 0
        self.level[i], self.prev[i], self.b[i] = s.level_init, s.level_init, s.b_init
        back = o[:, None] + torch.arange(-60, 0, device="cuda")
        self.hist[i] = self.q(back, torch.full_like(back, s.level_init)).movedim(0, 1)

    def obs(self):
        s, B, C, h = self.s, float(self.s.budget_q), self.C, self.hist
        Q = h.sum(1).double()
        s20, s60 = Q[:, -20:].sum(1), Q.sum(1)
        ph = self.phase[self.pos - 1].double()
        if s.obs_kind == W.OBS_TINY8:
            return torch.cat([Q[:, -5:] / B, ((B - Q[:, -1]) / B)[:, None], ph[:, None],
                              (self.level / (s.n_levels - 1))[:, None]], 1)
        slope = (Q[:, -1] - Q[:, -11]) / B
        if s.obs_kind == W.OBS_7B16:
            cols = [s60 / (60 * B), 1 - s60 / (60 * B), ph, (self.level - s.g_min).double() / (s.g_max - s.g_min),
                    (self.b - s.b_min).double() / (s.b_max - s.b_min), s20 / (20 * B), slope, torch.zeros_like(ph)]
            return torch.cat([Q[:, -8:] / B, torch.stack(cols, 1)], 1)
        d = self.ns[self.level] / 40.0 if s.level_samples else self.til / 40.0
        core = torch.stack([Q[:, -1] / B, s20 / (20 * B), s60 / (60 * B), 1 - s60 / (60 * B), slope,
                            (self.level + 1) / s.n_levels, (self.prev + 1) / s.n_levels, d.clamp(max=1.0)], 1).double()
        hd = h.double()
        means = [C * hd[:, :, -20:].sum(2) / (20 * B), C * hd.sum(2) / (60 * B)]
        if s.obs_kind == W.OBS_OCC32:
            return torch.cat([core, (C * hd[:, :, -4:] / B).flatten(1), means[1], torch.zeros_like(means[1])], 1)
        return torch.cat([core, (C * hd[:, :, -12:] / B).flatten(1), means[0], means[1]], 1)

    def step(self, a, lam, t, it):
        s, B = self.s, self.s.budget_q
        new = a
        if s.actuator_kind == W.ACT_INCDEC:
            new = (self.level - (a == 1).long() + (a == 2).long()).clamp(s.g_min, s.g_max)
            self.b = (self.b - (a == 3).long() + (a == 4).long()).clamp(s.b_min, s.b_max)
        self.til = torch.where(new != self.level, 0, self.til + 1)
        self.prev, self.level = self.level, new
        rate = self.tokens[new]
        top = float(self.tokens.max())
        if s.actuator_kind == W.ACT_INCDEC:
            rate, top = rate * self.b / s.b_init, float(self.tokens[s.g_min:s.g_max + 1].max()) * s.b_max / s.b_init
        ns = self.ns[new]
        z = torch.zeros(self.E, dtype=torch.float64, device="cuda")
        o = dict(q=torch.zeros_like(new), v1=torch.zeros_like(new), v60=torch.zeros_like(new), tokens=z.clone(),
                 excess=z.clone(), samples=ns)
        peak, fixed = z.clone(), z.clone()
        for i in range(int(ns.max())):
            on = i < ns
            q = self.q(torch.where(on, self.pos, 0), new).movedim(0, 1)
            self.hist = torch.where(on[:, None, None], torch.cat([self.hist[:, :, 1:], q[:, :, None]], 2), self.hist)
            Q, s60 = q.sum(1).long(), self.hist.sum((1, 2)).long()
            v1, v60 = on & (Q > B), on & (s60 > 60 * B)
            ex = torch.where(v60, (s60 - 60 * B) / 3840.0, 0.0).double()
            o["q"] += Q * on
            o["v1"] += v1
            o["v60"] += v60
            o["excess"] += 0.5 * ex
            o["tokens"] += torch.where(on & (self.phase[self.pos * on] == 0), rate, 0.0)
            peak = torch.maximum(peak, ex)
            viol = v1 if s.reward_window == 1 else v60
            fixed += torch.where(on, torch.where(viol, s.r_viol, s.r_ok) + s.bonus_coef * rate / top, 0.0)
            self.pos = self.pos + on
        o["reward"] = o["tokens"] / 1000.0 - lam * o["excess"] - 2.0 * lam * peak if s.reward_kind == W.REWARD_LAGRANGE else fixed
        self.k = self.k + 1
        done = self.k == s.episode_len
        o["done"] = done.to(torch.uint8)
        self.reset(done, t, it, 1)
        return o


def _rule_actions(env, rule, t, it):
    s, Q = env.s, env.hist.sum(1)
    inc = s.actuator_kind == W.ACT_INCDEC
    if rule.kind == W.RULE_RANDOM:
        return (_philox(s.seed, env.e, t, it, 0)[0] * s.n_actions) >> 32
    hold = torch.zeros_like(env.level) if inc else env.level
    lower = torch.ones_like(env.level) if inc else (env.level - 1).clamp(min=0)
    up = torch.full_like(env.level, 2) if inc else (env.level + 1).clamp(max=s.n_levels - 1)
    if rule.kind == W.RULE_THRESHOLD:
        q = Q[:, -1]
        return torch.where(q > rule.hi_q, lower, torch.where(q < rule.lo_q, up, hold))
    s60, s20 = Q.sum(1), Q[:, -20:].sum(1)
    climb = (s60 < 60 * rule.climb30_q) & (s20 < 20 * rule.climb10_q)
    return torch.where(s60 > 60 * rule.drop30_q, lower, torch.where(climb, up, hold))


def _exact_rollout(case, seed):
    kind, T, it, lam = case["kind"], case["T"], 1, 1.0
    wl = _workload(case["preset"], case["E"], seed)
    env, net = _Envs(wl), wl.net
    nets = None
    if kind in ("rollout", "iteration"):
        nets = _split(_params(net, seed).double(), net)
    elif kind == "replay":
        given = torch.randint(0, wl.env.n_actions, (T, case["E"]), generator=_gen(seed), device="cuda").to(torch.uint8)
    rows = {k: [] for k in ("obs", "act", "logp", "value", "reward", "done", "q")}
    tot = {k: 0 for k in ("v1", "v60", "tokens", "excess", "q", "samples")}

    def seen(x):  # a bf16 network reads rounded observations
        return x if net.dtype == W.DTYPE_F32 else x.float().bfloat16().double()

    for t in range(T):
        if nets:
            x = env.obs()
            z = _mlp(nets[0], seen(x), net)
            lp = torch.log_softmax(z, -1)
            cum = torch.exp(z - z.max(-1, keepdim=True).values).cumsum(-1)
            u = (_philox(wl.env.seed, env.e, t, it, 0)[0] >> 8) * 2.0 ** -24
            a = (u[:, None] * cum[:, -1:] >= cum).sum(-1).clamp(max=net.n_actions - 1)
            rows["obs"].append(x)
            rows["logp"].append(lp.gather(-1, a[:, None])[:, 0])
            rows["value"].append(_mlp(nets[1], seen(x), net)[:, 0])
        else:
            a = given[t].long() if kind == "replay" else _rule_actions(env, _rule(case, wl.env.budget_q), t, it)
        o = env.step(a, lam, t, it)
        rows["act"].append(a.to(torch.uint8))
        for k in ("reward", "done"):
            rows[k].append(o[k])
        rows["q"].append(o["q"].to(torch.int32))
        for k in tot:
            tot[k] = tot[k] + o[k]
    out = {k: torch.stack(v) for k, v in rows.items() if v}
    out.update(viol=torch.stack([tot["v1"], tot["v60"]], 1).to(torch.int32), tokens=tot["tokens"], excess=tot["excess"],
               energy_q=tot["q"], samples=tot["samples"])
    if nets:
        x = env.obs()
        out.update(obs_last=x, last_value=_mlp(nets[1], seen(x), net)[:, 0])
    return out


def _exact_gae(r, v, d, last):
    adv = torch.empty(r.shape, dtype=torch.float64, device="cuda")
    gamma, gl = _f32(GAMMA), _f32(GAMMA) * _f32(LAMBDA)
    a, nv = torch.zeros_like(last), last
    for t in range(r.shape[0] - 1, -1, -1):
        on, vt = 1.0 - d[t].double(), v[t].double()
        a = r[t].double() + gamma * nv * on - vt + gl * on * a
        adv[t], nv = a, vt
    return adv, adv + v.double()


def _permutation(n, seed, epoch, it):
    keys = [int(k) for k in _philox(seed, epoch, 0, it, 3)]
    bits = 2
    while (1 << bits) < n:
        bits += 1
    half = (bits + 1) // 2
    mask = (1 << half) - 1

    def once(x):
        l, r = x >> half, x & mask
        for k in keys:
            f = r ^ k
            for sh, m in ((16, 0x7FEB352D), (15, 0x846CA68B)):
                f = ((f ^ (f >> sh)) * m) & _M32
            l, r = r, l ^ ((f ^ (f >> 16)) & mask)
        return (l << half) | r

    y = once(torch.arange(n, device="cuda"))
    while bool((y >= n).any()):
        y = torch.where(y >= n, once(y), y)
    return y


def _exact_update(case, net, params, obs, act, logp, adv, ret, seed, it):
    ppo, n = _ppo(case), act.numel()
    lr, clip, eps, b1, b2 = (_f32(x) for x in (ppo.lr, ppo.clip, ppo.eps, ppo.beta1, ppo.beta2))
    vf, ent_coef, top = _f32(ppo.vf_coef), _f32(ppo.ent_coef), _f32(ppo.max_grad_norm)
    p = params.double().clone().requires_grad_(True)
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    obs, act, logp, adv, ret = obs.reshape(n, -1), act.reshape(n).long(), logp.reshape(n), adv.reshape(n), ret.reshape(n)
    sums, norm, t = torch.zeros(6, dtype=torch.float64, device="cuda"), None, 0
    for ep in range(ppo.epochs):
        perm = _permutation(n, seed, ep, it)
        for a0 in range(0, n, ppo.minibatch):
            i = perm[a0:a0 + ppo.minibatch]
            x, M = obs[i].double(), i.numel()
            ad = adv[i].double()
            if M > 1:
                ad = (ad - ad.mean()) / (ad.std() + 1e-8)
            nets = _split(p, net)
            lp = torch.log_softmax(_mlp(nets[0], x, net), -1)
            val = _mlp(nets[1], x, net)[:, 0]
            logr = lp.gather(-1, act[i][:, None])[:, 0] - logp[i].double()
            rho = torch.exp(logr)
            pg = -torch.minimum(rho * ad, rho.clamp(1 - clip, 1 + clip) * ad).mean()
            vl = (ret[i].double() - val).square().mean()
            ent = -(torch.exp(lp) * lp).sum(-1).mean()
            loss = pg - ent_coef * ent + vf * vl
            (g,) = torch.autograd.grad(loss, p)
            with torch.no_grad():
                t += 1
                norm = g.norm()
                g = g * (top / (norm + 1e-6)).clamp(max=1.0)
                m = b1 * m + (1 - b1) * g
                v = b2 * v + (1 - b2) * g * g
                p -= lr * (m / (1 - b1 ** t)) / ((v / (1 - b2 ** t)).sqrt() + eps)
                kl, cf = ((rho - 1) - logr).mean(), ((rho - 1).abs() > clip).double().mean()
                sums += torch.stack([pg, vl, ent, kl, cf, loss])
    stats = torch.cat([sums / t, norm[None], torch.full((1,), float(t), dtype=torch.float64, device="cuda")])
    return dict(params=p.detach(), adam_m=m, adam_v=v, stats=stats)


def _job_power(traces, job, J):
    q = torch.round(traces * 64.0).to(torch.int32)
    return torch.stack([q[job == j].sum(0).to(torch.int32) for j in range(J)])


def _exact_fleet(case, seed):
    if case["N"] > 10000 or case["N"] * case["L"] > 4e9:
        return None  # whole numbers, compared bit for bit; over 20 seconds here
    traces, job, J, budget = _fleet(case, seed)
    L, N = case["L"], case["N"]
    off = torch.randint(0, L, (N, J), generator=_gen(seed), device="cuda", dtype=torch.int32)
    q = _job_power(traces, job, J)
    q2 = torch.cat([q, q], 1)
    counts, peaks = (torch.zeros(N, case["nw"], dtype=torch.int32, device="cuda") for _ in range(2))
    for n, o in enumerate(off.tolist()):
        P = sum(q2[j, o[j]:o[j] + L] for j in range(J))
        c = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), P.cumsum(0)])
        for k, w in enumerate(WINDOWS[:case["nw"]]):
            S = c[w:] - c[:-w]
            counts[n, k], peaks[n, k] = (S > budget * w).sum(), S.max()
    return dict(counts=counts, peaks=peaks)


def _exact_stagger(case, seed):
    traces, job, J, _ = _fleet(case, seed)
    L, w, stride = case["L"], case["w"], case["stride"]
    q = _job_power(traces, job, J)
    offs, pks = [], []
    rest = torch.zeros(L - w + 1, dtype=torch.int32, device="cuda")  # the placed jobs' window sums
    for j in range(J):
        c = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), torch.cat([q[j], q[j]]).cumsum(0)])
        S = (c[w:] - c[:-w]).to(torch.int32)
        cand = S.unfold(0, L - w + 1, stride)[:(L + stride - 1) // stride]
        peak = torch.cat([(rest + part).amax(1) for part in cand.split(2048)])
        best = int((peak == peak.min()).nonzero()[0])
        offs.append(best * stride)
        pks.append(int(peak[best]))
        rest = rest + cand[best]
    return dict(offsets=torch.tensor(offs, dtype=torch.int32), peaks=torch.tensor(pks, dtype=torch.int32))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("rollout", "replay", "rule", "iteration"):
        out = _exact_rollout(case, seed)
        if kind != "iteration":
            return out
        adv, ret = _exact_gae(out["reward"], out["value"], out["done"], out["last_value"])
        u = _exact_update(case, NETS["tiny"], _params(NETS["tiny"], seed), out["obs"], out["act"], out["logp"], adv, ret, seed, 1)
        return dict(out, adv=adv, ret=ret, **u)
    if kind == "value":
        net = NETS[case["preset"]]
        layers = _split(_params(net, seed).double(), net)[1]
        obs = _observations(case["preset"], net, case["n"], _gen(seed))
        return torch.cat([_mlp(layers, x.double(), net)[:, 0] for x in obs.split(65536)])
    if kind == "gae":
        s = prepare(case, seed)
        adv, ret = _exact_gae(s["reward"], s["value"], s["done"], s["last"].double())
        return dict(adv=adv, ret=ret)
    if kind == "update":
        return _exact_update(case, NETS[case["preset"]], *_update_inputs(case, seed), seed, 1)
    return _exact_fleet(case, seed) if kind == "fleet" else _exact_stagger(case, seed)
