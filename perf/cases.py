"""Performance cases: the calls a user of this library makes, over the sizes they come in.

A case is one call (or one training call) through the public entry points of
``paper_2311_13081_gb300``:

  dynamics  teacher-forced RK4 of a batch of bodies        qsim_dynamics_step
  step      one env step under the caller's own policy     qsim_step
  rollout   fused actor + env steps into the replay ring   qsim_rollout
  track     figure-eight tracking flights                  qsim_track
  recalc    reward recalculation of a filled ring          qsim_recalc_rewards
  update    TD3 updates of one learner from its ring       ac_update
  train     env steps + updates of one to 512 runs         ac_train, ac_plan_run
  vjp       loss and gradients of a simulated horizon      qsim_rollout_vjp, diff.rollout_loss

Inputs are synthetic and come from the seed alone: vehicles of the domain-randomised
distribution in mid-flight states, actors and critics with the sizes of freshly initialised
networks, Adam moments of a run in progress and replay rings of random transitions with
episodes of about 42 steps (what a random actor flies).  ``exact`` restates each call in
64-bit torch from the method (simulation, random streams, TD3), without the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2311_13081_gb300 as q
import workloads as W
from paper_2311_13081_gb300 import diff

DEV = "cuda"
F64 = torch.float64
NS = 17
HIDDENS = (32, 64, 128)
BATCHES = (128, 256, 512)
EPISODE_STEPS = 42  # mean episode length under a random actor
T_START, U_START = 100_000, 1_000  # counters of a run in progress


# ------------------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: a user's own policy steps a small env set, one call per step
        dict(name="step_own_policy", kind="step", n=1_000, layout=0, noise=True, slots=512, n_hist=16),
        # a batch of bodies integrated under given rotor speeds (model fitting, simulator use)
        dict(name="dynamics_million", kind="dynamics", n=1_000_000, steps=1, disturbed=True),
        # data collection with a few envs: what one training run or an evaluation does
        dict(name="rollout_small", kind="rollout", n=1_000, steps=128, hidden=64, noise=False, slots=128,
             n_hist=16),
        # the batched rollout workload: 65,536 randomised vehicles x 1,000 steps
        dict(name="rollout_65536", kind="rollout", n=65_536, steps=1_000, hidden=64, noise=False, slots=1_000,
             n_hist=16),
        # the widest actor
        dict(name="rollout_wide", kind="rollout", n=4_096, steps=64, hidden=128, noise=True, slots=64,
             n_hist=16),
        # evaluation of a controller: tracking flights of a fleet, an odd count
        dict(name="track_fleet", kind="track", n=20_001, steps=500, hidden=64, n_hist=16),
        # reward recalculation after a curriculum change
        dict(name="recalc_ring", kind="recalc", n=65_536, slots=64, layout=0),
        # one training run: updates between its env steps (critic, critic + actor)
        dict(name="update_single", kind="update", n=1, slots=10_000, hidden=64, batch=256, layout=0, noise=False,
             n_hist=16, updates=2),
        # many independent runs in one launch, mixed widths and batches (seeds, sweeps)
        dict(name="train_512_mixed", kind="train", runs=512, n=8, slots=2_048, hidden=0, batch=0, layout=0,
             noise=False, n_hist=16, steps=4, updates=1, plan=False),
        # privileged critics, 64 envs per run, a captured plan replayed
        dict(name="train_128_privileged", kind="train", runs=128, n=64, slots=4_096, hidden=64, batch=256, layout=1,
             noise=False, n_hist=16, steps=1, updates=16, plan=True),
        # policy gradient through the simulator (closed loop), buffers kept by the caller
        dict(name="vjp_closed_loop", kind="vjp", n=4_096, horizon=200, ckpt=20, closed=True, hidden=64,
             n_hist=16, autograd=False),
        # trajectory optimisation (open loop) through torch.autograd
        dict(name="vjp_open_loop", kind="vjp", n=4_096, horizon=200, ckpt=20, closed=False, hidden=64,
             n_hist=16, autograd=True),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("dynamics", "step", "rollout", "rollout", "track", "recalc", "update", "train", "train",
                       "vjp", "vjp"))
    n_hist = rng.choice((16, 16, 16, 8, 0))
    if kind == "dynamics":
        return dict(kind=kind, n=_log_int(rng, 1_000, 4_000_000), steps=rng.choice((1, 1, 10, 100)),
                    disturbed=rng.random() < 0.5)
    if kind == "step":
        return dict(kind=kind, n=_log_int(rng, 1, 65_536), layout=rng.randrange(4), noise=rng.random() < 0.5,
                    slots=_log_int(rng, 32, 512), n_hist=n_hist)
    if kind == "rollout":
        n = _log_int(rng, 64, 65_536)
        steps = _log_int(rng, 8, 1_000)
        hidden = rng.choice((64, 64, 64, 32, 128))
        if hidden != 64:
            steps = max(1, min(steps, 8_000_000 // n))
        return dict(kind=kind, n=n, steps=steps, hidden=hidden, noise=rng.random() < 0.3, slots=max(32, steps),
                    n_hist=n_hist)
    if kind == "track":
        return dict(kind=kind, n=_log_int(rng, 64, 65_536), steps=_log_int(rng, 50, 1_000), hidden=64,
                    n_hist=n_hist)
    if kind == "recalc":
        n = _log_int(rng, 8, 65_536)
        return dict(kind=kind, n=n, slots=_log_int(rng, 32, max(64, min(100_000, 8_000_000 // n))),
                    layout=rng.choice((0, 1)))
    # layouts whose critic reads the action history want one
    layout = rng.choice((0, 0, 1, 2, 3))
    hidden, batch = rng.choice(HIDDENS), rng.choice(BATCHES)
    if kind == "update":
        return dict(kind=kind, n=_log_int(rng, 1, 64), slots=_log_int(rng, 512, 10_000), hidden=hidden, batch=batch,
                    layout=layout, noise=rng.random() < 0.3, n_hist=n_hist, updates=2 * _log_int(rng, 1, 8))
    if kind == "train":
        runs = _log_int(rng, 1, 512)
        if rng.random() < 0.5:
            hidden, batch = 0, 0
        steps = _log_int(rng, 1, 8)
        n = _log_int(rng, 1, 64)
        updates = rng.choice((1, 1, 1, 2, 8)) if runs <= 128 else 1
        case = dict(kind=kind, runs=runs, n=n, slots=_log_int(rng, 256, 2_048), hidden=hidden, batch=batch,
                    layout=layout, noise=rng.random() < 0.3, n_hist=n_hist, steps=steps, updates=updates,
                    plan=rng.random() < 0.3)
        most = max(work(c)["flops"] for c in listed() if c["kind"] == kind)
        while work(case)["flops"] > most:
            key = "steps" if case["steps"] > 1 else "runs"
            case[key] = (case[key] + 1) // 2
        return case
    closed = rng.random() < 0.6
    return dict(kind="vjp", n=4 * _log_int(rng, 16, 1_024), horizon=_log_int(rng, 20, 200),
                ckpt=rng.choice((10, 20, 25)), closed=closed, hidden=rng.choice((64, 64, 32)), n_hist=n_hist,
                autograd=rng.random() < 0.5)


# ------------------------------------------------------------------------------ the inputs
def _gen(seed, *salt):
    g = torch.Generator(device=DEV)
    s = seed & 0x7FFFFFFF
    for x in salt:
        s = (s * 1_000_003 + int(x) + 12_345) & 0x7FFFFFFFFFFF
    g.manual_seed(s)
    return g


def _u(g, shape, lo, hi):
    return torch.rand(shape, generator=g, device=DEV) * (hi - lo) + lo


def _states(g, lead, n):
    """[*lead][17][n] mid-flight states: inside the box, tilted up to ~45 degrees."""
    s = torch.empty(*lead, NS, n, device=DEV)
    s[..., 0:3, :] = _u(g, (*lead, 3, n), -0.5, 0.5)
    quat = torch.randn((*lead, 4, n), generator=g, device=DEV) * 0.2
    quat[..., 0, :] = 1.0
    s[..., 3:7, :] = quat / quat.norm(dim=-2, keepdim=True)
    s[..., 7:13, :] = torch.randn((*lead, 6, n), generator=g, device=DEV)
    s[..., 13:17, :] = _u(g, (*lead, 4, n), 8_000.0, 21_000.0)
    return s


def _vehicles(g, n):
    """[8][n] parameters of the domain-randomised vehicle distribution."""
    v = W.VEHICLE
    p = torch.zeros(8, n, device=DEV)
    for i, (key, rel) in enumerate((("mass", 0.2), ("Jx", 0.2), ("Jy", 0.2), ("Jz", 0.2), ("kf", 0.1))):
        p[i] = v[key] * _u(g, (n,), 1.0 - rel, 1.0 + rel)
    p[5] = v["km"]
    p[6] = _u(g, (n,), 0.03, 0.15)
    return p


def _net(g, inp, hid, out, scale=1.0):
    """Flat parameters W1 b1 W2 b2 W3 b3, uniform in +-1/sqrt(fan-in)."""
    parts = []
    for rows, cols, fan, k in ((hid, inp, inp, 1.0), (hid, 1, inp, 1.0), (hid, hid, hid, 1.0), (hid, 1, hid, 1.0),
                               (out, hid, hid, scale), (out, 1, hid, scale)):
        b = k / math.sqrt(fan)
        parts.append(_u(g, (rows * cols,), -b, b))
    return torch.cat(parts)


def _hover_actor(g, inp, hid):
    """A random actor whose output stays near the hover action (tracking and the
    differentiable rollout start from such policies)."""
    p = _net(g, inp, hid, 4, scale=0.05)
    p[-4:] += math.atanh(W.hover_action())
    return p


def _sim(case, seed, run=0):
    """Simulation settings of a case as a plain dict (workloads' presets and overrides)."""
    d = W.config("c2")
    d.update(critic_layout=case.get("layout", 0), n_hist=case.get("n_hist", 16), learning_starts=0,
             seed=seed & 0x7FFFFFFF, run_id=run, reward=W.REWARD)
    if case.get("noise"):
        d.update(sig_p=0.002, sig_R=0.01, sig_v=0.01, sig_w=0.01, dist_f=0.0027, dist_tau=1.0e-6)
    return d


def _obs_dim(case):
    return 18 + 4 * case.get("n_hist", 16)


def _critic_in(case):
    da = _obs_dim(case)
    return {0: da + 4, 1: da + 10, 2: 28, 3: da}[case["layout"]] + 4


class _Handle:
    """A library handle, destroyed with its last reference."""

    def __init__(self, h, free):
        self.h, self.free = h, free

    def __del__(self):
        self.free(self.h)


class _View:
    """A device array of a handle; the tensor made of it keeps the handle alive."""

    def __init__(self, t, owner):
        self.__cuda_array_interface__ = t.__cuda_array_interface__
        self.owner = owner


def _kept(info, owner):
    return {k: torch.as_tensor(_View(v, owner), device=DEV) if isinstance(v, torch.Tensor) and v.is_contiguous() else v
            for k, v in info.items()}


class _Env:
    def __init__(self, d, n, slots):
        self.d = d
        self.h = q.qsim_create(q.make_config(d, n, slots, reward=W.REWARD, sigma_e=0.1), q.make_params(d))
        self.keep = _Handle(self.h, q.qsim_destroy)
        self.info = _kept(q.qsim_info_get(self.h), self.keep)


class _Learner:
    def __init__(self, hp, env, updates=1):
        self.a = q.ac_create(q.make_ac_config(hp, updates_per_step=updates), env.h)
        self.keep = _Handle(self.a, q.ac_destroy)
        self.info = _kept(q.ac_info_get(self.a), self.keep)


class _Plan:
    """A captured training launch; it goes before the runs and envs that it uses."""

    def __init__(self, runs, envs, steps):
        self.keep = [x.keep for x in runs + envs]
        self.p = q.ac_plan_create([r.a for r in runs], [e.h for e in envs], steps)

    def __del__(self):
        torch.cuda.synchronize()
        q.ac_plan_destroy(self.p)


def _live(g, case, d, ld):
    """Contents of an env set in mid-flight: states, parameters, disturbances, history and
    episode counters."""
    nh4 = 4 * case.get("n_hist", 16)
    hist = torch.zeros(64, ld, device=DEV)
    hist[:nh4] = (0.33 + 0.3 * torch.randn((nh4, ld), generator=g, device=DEV)).clamp(-1.0, 1.0)
    dist = torch.zeros(6, ld, device=DEV)
    if d["dist_f"]:
        dist[:3] = _u(g, (3, ld), -d["dist_f"], d["dist_f"])
        dist[3:] = _u(g, (3, ld), -d["dist_tau"], d["dist_tau"])
    step = torch.randint(16, EPISODE_STEPS, (ld,), generator=g, device=DEV, dtype=torch.int32)
    return dict(state=_states(g, (), ld), params=_vehicles(g, ld), dist=dist, hist=hist, ep_step=step)


def _ring(g, slots, ld, priv):
    """A full replay ring in time order: records [slots][F][ld] and side slots [slots][17][ld]."""
    rec = torch.empty(slots, 29 if priv else 23, ld, device=DEV)
    rec[:, :NS] = _states(g, (slots,), ld)
    rec[:, 17:21] = (0.33 + 0.3 * torch.randn((slots, 4, ld), generator=g, device=DEV)).clamp_(-1.0, 1.0)
    rec[:, 21] = 1.5 - torch.rand((slots, ld), generator=g, device=DEV)
    done = torch.rand((slots, ld), generator=g, device=DEV) < 1.0 / EPISODE_STEPS
    t = torch.arange(slots, device=DEV)[:, None].expand(slots, ld)
    # steps since the latest end before this record (envs start mid-episode)
    ended = torch.where(done, t + 1, torch.full_like(t, -20))
    start = torch.cat([torch.full((1, ld), -20, device=DEV, dtype=t.dtype), ended[:-1]]).cummax(0).values
    rec[:, 22] = (done.int() | ((t - start).int() << 8)).view(torch.float32)
    if priv:
        rec[:, 23:] = _u(g, (slots, 6, ld), -0.2, 0.2)
    side = torch.zeros(slots, NS, ld, device=DEV)
    side[:] = torch.where(done[:, None], rec[:, :NS] * 1.3, side)
    return rec, side


def _fill(g, case, env):
    """Puts an env set into the middle of training: live envs and a wrapped ring."""
    ld, slots = env.info["ld"], case["slots"]
    live = _live(g, case, env.d, ld)
    rec, side = _ring(g, slots, ld, env.d["critic_layout"] in (1, 2))
    head = int(torch.randint(0, slots, (1,), generator=g, device=DEV))
    for k, v in live.items():
        env.info[k].copy_(v)
    env.info["records"].copy_(rec.roll(head, 0))
    env.info["side"].copy_(side.roll(head, 0))
    q.qsim_set_counters(env.h, T_START, head, slots)


def _hyper(case, i):
    hp = dict(W.TD3)
    r = np.random.RandomState(1_000 + i)
    hp["hidden"] = case["hidden"] or int(r.choice(HIDDENS))
    hp["batch"] = case["batch"] or int(r.choice(BATCHES))
    return hp


def _networks(g, case, hp):
    """Weights, targets and Adam moments of a run in progress."""
    da, dc, h = _obs_dim(case), _critic_in(case), hp["hidden"]
    out = {}
    for name, inp, o, m in (("actor", da, 4, "a"), ("c1", dc, 1, "c1"), ("c2", dc, 1, "c2")):
        w = _net(g, inp, h, o)
        out[name] = w
        out[name + "_t"] = w + 0.01 * torch.randn(w.shape, generator=g, device=DEV)
        out["v_" + m] = (0.01 * _u(g, w.shape, 0.5, 1.5)) ** 2
        out["m_" + m] = 0.003 * torch.randn(w.shape, generator=g, device=DEV)
    return out


NETS = ("actor", "actor_t", "c1", "c1_t", "c2", "c2_t")
MOMENTS = ("m_a", "v_a", "m_c1", "v_c1", "m_c2", "v_c2")


def _learner_inputs(g, case, hp, learner):
    for k, v in _networks(g, case, hp).items():
        learner.info[k].copy_(v)
    q.ac_set_counters(learner.a, U_START // 2, U_START, U_START)


def _vjp_inputs(case, seed):
    g = _gen(seed, 7)
    n = case["n"]
    s0 = _states(g, (), n)
    s0[0:3] *= 0.4
    s0[7:13] *= 0.5
    x = (_hover_actor(g, _obs_dim(case), case["hidden"]) if case["closed"] else
         (W.hover_action() + 0.1 * torch.randn((case["horizon"], 4, n), generator=g, device=DEV)).clamp(-1, 1))
    return s0, _vehicles(g, n), x, _u(g, (n,), 0.5, 1.5)


WEIGHTS = (1.0, 0.5, 0.2, 0.05)  # of the differentiable rollout's loss


class _State:
    pass


def prepare(case, seed):
    st = _inputs(case, seed)
    st.outputs = _outputs(st)
    torch.cuda.synchronize()
    return st


def _inputs(case, seed):
    st = _State()
    st.case = case
    kind = case["kind"]
    if kind == "dynamics":
        n, ld = case["n"], (case["n"] + 3) // 4 * 4
        g = _gen(seed, 1)
        st.veh = q.make_params(W.VEHICLE)
        st.ld, st.s, st.p = ld, _states(g, (), ld), _vehicles(g, ld)
        st.rpm = _u(g, (4, ld), 5_000.0, 21_000.0)
        st.dist = None
        if case["disturbed"]:
            st.dist = torch.cat([_u(g, (3, ld), -0.0027, 0.0027), _u(g, (3, ld), -1e-6, 1e-6)])
        st.out = torch.empty_like(st.s)
        return st
    if kind == "vjp":
        st.s0, st.p, st.x, st.seed = _vjp_inputs(case, seed)
        st.veh = q.make_params(W.VEHICLE)
        if case["autograd"]:
            st.p.requires_grad_()
            st.x.requires_grad_()
            return st
        n = case["n"]
        st.desc = diff.make_desc(n, n, case["horizon"], case["ckpt"], int(case["closed"]), WEIGHTS,
                                 n_hist=case["n_hist"], hidden=case["hidden"])
        st.ws = torch.empty(q.qsim_vjp_workspace(st.desc) // 4 + 1, device=DEV)
        st.loss, st.gx, st.gp = torch.empty(n, device=DEV), torch.empty_like(st.x), torch.empty(4, n, device=DEV)
        return st
    if kind == "train":
        st.envs, st.runs = [], []
        for i in range(case["runs"]):
            hp = _hyper(case, i)
            env = _Env(_sim(case, seed, i), case["n"], case["slots"])
            run_ = _Learner(hp, env, case["updates"])
            _fill(_gen(seed, 2, i), case, env)
            _learner_inputs(_gen(seed, 3, i), case, hp, run_)
            st.envs.append(env)
            st.runs.append(run_)
        st.views = {k: [r.info[k] for r in st.runs] for k in NETS}
        st.views["state"] = [e.info["state"][:, : case["n"]] for e in st.envs]
        torch.cuda.synchronize()
        st.plan = _Plan(st.runs, st.envs, case["steps"]) if case["plan"] else None
        return st
    st.env = _Env(_sim(case, seed), case["n"], case.get("slots", 0))
    info = st.env.info
    g = _gen(seed, 2, 0)
    if kind in ("recalc", "update"):
        _fill(g, case, st.env)
    else:
        for k, v in _live(g, case, st.env.d, info["ld"]).items():
            info[k].copy_(v)
    if kind == "step":
        n, ld = case["n"], info["ld"]
        st.actions = (0.33 + 0.3 * torch.randn((4, ld), generator=g, device=DEV))
        st.obs_a = torch.zeros(info["obs_dim"], ld, device=DEV)
        st.obs_c = torch.zeros(info["critic_obs_dim"], ld, device=DEV)
        st.rew = torch.zeros(ld, device=DEV)
        st.term, st.trunc = (torch.zeros(ld, dtype=torch.uint8, device=DEV) for _ in range(2))
    elif kind == "rollout":
        st.actor = _net(_gen(seed, 3), _obs_dim(case), case["hidden"], 4)
    elif kind == "track":
        ld = info["ld"]
        st.actor = _hover_actor(_gen(seed, 3), _obs_dim(case), case["hidden"])
        st.period = torch.tensor([15.0, 5.5, 3.5], device=DEV).repeat(ld // 3 + 1)[:ld].contiguous()
        st.sq = torch.zeros(2, ld, dtype=F64, device=DEV)
        st.ok = torch.zeros(ld, dtype=torch.int32, device=DEV)
    elif kind == "update":
        hp = _hyper(case, 0)
        st.run = _Learner(hp, st.env)
        _learner_inputs(_gen(seed, 3, 0), case, hp, st.run)
    return st


# ------------------------------------------------------------------------------- the calls
def _outputs(st):
    """What a pass returns where it is the state's own buffers: views of the live envs."""
    case, kind = st.case, st.case["kind"]
    n = case["n"]
    if kind == "dynamics":
        return st.out[:, :n]
    if kind == "train":
        return None
    if kind == "vjp":
        return None if case["autograd"] else dict(loss=st.loss, g_x=st.gx, g_params=st.gp)
    i = st.env.info
    if kind == "step":
        return dict(obs_a=st.obs_a[:, :n], obs_c=st.obs_c[:, :n], reward=st.rew[:n], terminated=st.term[:n],
                    truncated=st.trunc[:n], state=i["state"][:, :n], hist=i["hist"][:, :n], ep_step=i["ep_step"][:n])
    if kind == "rollout":
        return dict(transitions=i["records"][:, :22, :n], flags=i["records"].view(torch.int32)[:, 22, :n],
                    state=i["state"][:, :n], hist=i["hist"][:, :n], ep_step=i["ep_step"][:n],
                    episodes=i["n_done"][:n], returns=i["ret_sum"][:n])
    if kind == "track":
        return dict(sq_err=st.sq[:, :n], steps_ok=st.ok[:n])
    if kind == "recalc":
        return i["records"][:, 21, :n]
    return {k: st.run.info[k] for k in NETS + MOMENTS + ("stats",)}


def run(st):
    case, kind = st.case, st.case["kind"]
    n = case["n"]
    if kind == "dynamics":
        q.qsim_dynamics_step(st.veh, st.p, st.dist, st.s, st.rpm, 0.01, 1, n, st.ld, case["steps"], st.out)
        return st.outputs
    if kind == "step":
        q.qsim_step(st.env.h, st.actions, st.obs_a, st.obs_c, st.rew, st.term, st.trunc)
        return st.outputs
    if kind == "rollout":
        q.qsim_rollout(st.env.h, st.actor, case["hidden"], case["steps"], 0.1)
        return st.outputs
    if kind == "track":
        q.qsim_track(st.env.h, st.actor, case["hidden"], case["steps"], st.period, st.sq, st.ok)
        return st.outputs
    if kind == "recalc":
        q.qsim_recalc_rewards(st.env.h)
        return st.outputs
    if kind == "update":
        q.ac_update(st.run.a, st.env.h, case["updates"])
        return st.outputs
    if kind == "train":
        # the runs' weights and env states (an update's Adam moments are what `update` returns)
        if st.plan is not None:
            q.ac_plan_run(st.plan.p, 1)
        else:
            q.ac_train([r.a for r in st.runs], [e.h for e in st.envs], case["steps"])
        return {k: torch.cat(v) for k, v in st.views.items()}
    # vjp
    if case["autograd"]:
        kw = dict(actor=st.x) if case["closed"] else dict(actions=st.x)
        loss = diff.rollout_loss(st.s0, st.p, st.veh, case["horizon"], case["ckpt"], WEIGHTS,
                                 n_hist=case["n_hist"], hidden=case["hidden"], **kw)
        gp, gx = torch.autograd.grad(loss, (st.p, st.x), st.seed)
        return dict(loss=loss.detach(), g_x=gx, g_params=gp[:4])
    acts, actor = (None, st.x) if case["closed"] else (st.x, None)
    g_acts, g_actor = (None, st.gx) if case["closed"] else (st.gx, None)
    q.qsim_rollout_vjp(st.desc, st.veh, st.s0, st.p, acts, actor, st.seed, st.loss, g_acts, g_actor, st.gp, None,
                       st.ws)
    return st.outputs


def _mlp_macs(inp, hid, out):
    return inp * hid + hid * hid + hid * out


def _update_flops(case, hp):
    """Multiply-adds x 2 of one TD3 update: target actor, twin target critics, critic
    regression (forward, input and weight gradients), every second update the actor's."""
    da, dc, h = _obs_dim(case), _critic_in(case), hp["hidden"]
    a, c = _mlp_macs(da, h, 4), _mlp_macs(dc, h, 1)
    macs = a + 2 * c + 2 * c + 4 * c + 0.5 * (a + 2 * c + 2 * a)
    return 2 * hp["batch"] * macs


def _update_bytes(case, hp):
    da, dc, h = _obs_dim(case), _critic_in(case), hp["hidden"]
    params = _mlp_macs(da, h, 4) + 2 * _mlp_macs(dc, h, 1)
    # a sample: state and next state, 17 actions, reward and flags; weights, targets and
    # both Adam moments read and written once
    return hp["batch"] * 4 * (2 * NS + 4 * (case.get("n_hist", 16) + 1) + 2) + 2 * 4 * 4 * params


RK4_FLOPS, STEP_FLOPS = 672, 60


def work(case):
    kind, n = case["kind"], case["n"]
    da = _obs_dim(case)
    if kind == "dynamics":
        return dict(bytes=4 * n * (NS + 7 + 4 + NS + (6 if case["disturbed"] else 0)),
                    flops=n * case["steps"] * RK4_FLOPS)
    fields = 29 if case.get("layout", 0) in (1, 2) else 23
    env_rw = 4 * (2 * NS + 7 + 6 + 8 * case.get("n_hist", 16) + 8)
    if kind == "step":
        return dict(bytes=n * (env_rw + 4 * (4 + fields + da + _critic_in(case) - 4) + 6),
                    flops=n * (RK4_FLOPS + STEP_FLOPS))
    step_flops = 2 * _mlp_macs(da, case.get("hidden") or 64, 4) + RK4_FLOPS + STEP_FLOPS
    if kind == "rollout":
        return dict(bytes=n * (case["steps"] * 4 * fields + env_rw), flops=n * case["steps"] * step_flops)
    if kind == "track":
        return dict(bytes=n * 4 * (7 + 6 + 1 + 5), flops=n * case["steps"] * step_flops)
    if kind == "recalc":
        return dict(bytes=n * case["slots"] * 4 * (NS + 4 + 1 + 1), flops=n * case["slots"] * 40)
    if kind == "update":
        hp = _hyper(case, 0)
        return dict(bytes=case["updates"] * _update_bytes(case, hp), flops=case["updates"] * _update_flops(case, hp))
    if kind == "train":
        b = f = 0.0
        for i in range(case["runs"]):
            hp = _hyper(case, i)
            b += case["steps"] * (n * (env_rw + 4 * fields) + case["updates"] * _update_bytes(case, hp))
            f += case["steps"] * (n * (2 * _mlp_macs(da, hp["hidden"], 4) + RK4_FLOPS + STEP_FLOPS)
                                  + case["updates"] * _update_flops(case, hp))
        return dict(bytes=b, flops=f)
    # reverse mode: about three times the forward step
    per = RK4_FLOPS + STEP_FLOPS + (2 * _mlp_macs(da, case["hidden"], 4) if case["closed"] else 0)
    size = 4 * (_mlp_macs(da, case["hidden"], 4) if case["closed"] else 8 * n * case["horizon"])
    return dict(bytes=4 * n * (NS + 7 + 1 + 5) + size, flops=3 * n * case["horizon"] * per)


# --------------------------------------------------------------- the same in 64 bits
# Plain torch in double precision, from the method's description: Philox4x32-10 streams,
# RK4 of the rigid body with first-order motors, observations, reward, reset, TD3.
M32 = 0xFFFFFFFF


def _f32(x):
    return float(np.float32(x))


def _philox(c0, c1, tag, sub, run, seed):
    """Four streams of 32-bit words (int64 tensors) at counters (c0, c1, tag, sub, run)."""
    c0 = torch.as_tensor(c0, device=DEV, dtype=torch.int64)
    c1 = torch.as_tensor(c1, device=DEV, dtype=torch.int64) & M32
    c0, c1 = torch.broadcast_tensors(c0, c1)
    c2 = torch.full_like(c0, (tag << 24) | sub)
    c3 = torch.full_like(c0, run)
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        hi0, lo0, hi1, lo1 = (p0 >> 32) & M32, p0 & M32, (p1 >> 32) & M32, p1 & M32
        c0, c1, c2, c3 = hi1 ^ c1 ^ k0, lo1, hi0 ^ c3 ^ k1, lo0
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c0, c1, c2, c3


def _u01(x):
    return ((x >> 9).to(F64) + 0.5) * 2.0 ** -23


def _normal(a, b):
    return torch.sqrt(-2.0 * torch.log(_u01(a))) * torch.cos(2.0 * math.pi * _u01(b))


class _Ref:
    """The simulation of one env set in double precision; fields as rows [.., n]."""

    def __init__(self, d, n, live=None):
        self.d, self.n = {k: (_f32(v) if isinstance(v, float) else v) for k, v in d.items()}, n
        self.e = torch.arange(n, device=DEV)
        v = W.VEHICLE
        self.rx = torch.tensor([_f32(x) for x in v["rotor_pos"][0::3]], device=DEV, dtype=F64)
        self.ry = torch.tensor([_f32(x) for x in v["rotor_pos"][1::3]], device=DEV, dtype=F64)
        self.dir = torch.tensor(v["rotor_dir"], device=DEV, dtype=F64)
        self.hi = _f32(v["rpm_max"])
        self.C = [_f32(x) for x in W.REWARD]
        if live is not None:
            self.s, self.p, self.f, self.hist = (live[k][:, :n].to(F64) for k in ("state", "params", "dist", "hist"))
            self.ep_step = live["ep_step"][:n].to(torch.int64)
            self.ep = torch.zeros(n, device=DEV, dtype=torch.int64)
            self.ep_ret, self.ret_sum = torch.zeros(n, device=DEV, dtype=F64), torch.zeros(n, device=DEV, dtype=F64)

    def draw(self, c0, c1, tag, sub=0):
        return _philox(c0, c1, tag, sub, self.d["run_id"], self.d["seed"])

    def deriv(self, s, u, p, f):
        qw, qx, qy, qz = s[3:7]
        w = s[10:13]
        thrust = p[4] * s[13:17] ** 2
        total = thrust.sum(0)
        tau = torch.stack([(self.ry[:, None] * thrust).sum(0), (-self.rx[:, None] * thrust).sum(0),
                           p[5] * (self.dir[:, None] * thrust).sum(0)]) + f[3:6]
        axis = torch.stack([2 * (qx * qz + qw * qy), 2 * (qy * qz - qw * qx), 1 - 2 * (qx * qx + qy * qy)])
        acc = (axis * total + f[0:3]) / p[0]
        acc = torch.cat([acc[:2], acc[2:3] - _f32(W.VEHICLE["g"])])
        dq = 0.5 * torch.stack([-qx * w[0] - qy * w[1] - qz * w[2], qw * w[0] + qy * w[2] - qz * w[1],
                                qw * w[1] - qx * w[2] + qz * w[0], qw * w[2] + qx * w[1] - qy * w[0]])
        J = p[1:4]
        dw = (tau - torch.linalg.cross(w, J * w, dim=0)) / J
        return torch.cat([s[7:10], dq, acc, dw, (u - s[13:17]) / p[6]])

    def rk4(self, s, u, p, f):
        h = _f32(self.d["dt"])
        u = u.clamp(0.0, self.hi)
        k1 = self.deriv(s, u, p, f)
        k2 = self.deriv(s + 0.5 * h * k1, u, p, f)
        k3 = self.deriv(s + 0.5 * h * k2, u, p, f)
        k4 = self.deriv(s + h * k3, u, p, f)
        s = s + h / 6.0 * (k1 + 2 * k2 + 2 * k3 + k4)
        quat = s[3:7] / s[3:7].norm(dim=0, keepdim=True)
        return torch.cat([s[:3], quat, s[7:]])

    @staticmethod
    def obs(s):
        w, x, y, z = s[3:7]
        R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                         2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                         2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)])
        return torch.cat([s[:3], R, s[7:13]])

    def noise(self, env, t):
        d = self.d
        sig = [d["sig_p"]] * 3 + [d["sig_R"]] * 9 + [d["sig_v"]] * 3 + [d["sig_w"]] * 3
        out = []
        for b in range(9):
            r = self.draw(env, t, 2, b)
            out += [sig[2 * b] * _normal(r[0], r[1]), sig[2 * b + 1] * _normal(r[2], r[3])]
        return torch.stack(out)

    def obs_actor(self, s, hist, env, t):
        o = self.obs(s)
        if self.d["sig_p"]:
            o = o + self.noise(env, t)
        return torch.cat([o, hist[: 4 * self.d["n_hist"]]])

    def rpm_norm(self, s):
        return 2.0 * s[13:17] / self.hi - 1.0

    def priv(self):
        d = self.d
        if d["critic_layout"] == 2:
            zero = torch.zeros_like(self.f)
            return torch.cat([self.f[:3] / d["dist_f"], self.f[3:] / d["dist_tau"]]) if d["dist_f"] else zero
        nom = [_f32(W.VEHICLE[k]) for k in ("mass", "Jx", "Jy", "Jz", "kf", "tm")]
        return torch.stack([self.p[i] / x - 1.0 for i, x in zip((0, 1, 2, 3, 4, 6), nom)])

    def obs_critic(self, s, hist, priv, oa):
        d = self.d
        if d["critic_layout"] == 3:
            return oa
        if d["critic_layout"] == 2:
            return torch.cat([self.obs(s), self.rpm_norm(s), priv])
        parts = [self.obs(s), hist[: 4 * d["n_hist"]], self.rpm_norm(s)]
        return torch.cat(parts + ([priv] if d["critic_layout"] == 1 else []))

    def reward(self, s, a, C=None):
        C = C or self.C
        return (-C[0] * (s[:3] ** 2).sum(0) - C[1] * (1 - s[3] ** 2) - C[2] * (s[7:10] ** 2).sum(0)
                - C[3] * (s[10:13] ** 2).sum(0) - C[4] * ((a - C[5]) ** 2).sum(0) + C[6])

    def start(self, env, ep):
        """State, parameters and disturbance that episode `ep` starts with."""
        d, v = self.d, {k: _f32(W.VEHICLE[k]) for k in ("mass", "Jx", "Jy", "Jz", "kf", "km")}
        U = torch.stack([_u01(x) for b in range(4) for x in self.draw(env, ep, 0, b)])
        sym = 2 * U - 1
        half = 0.5 * d["init_att"] * sym[3:6]
        (sr, sp, sy), (cr, cp, cy) = torch.sin(half), torch.cos(half)
        quat = torch.stack([cy * cp * cr + sy * sp * sr, cy * cp * sr - sy * sp * cr,
                            cy * sp * cr + sy * cp * sr, sy * cp * cr - cy * sp * sr])
        s = torch.cat([d["init_p"] * sym[:3], quat, d["init_v"] * sym[6:9], d["init_w"] * sym[9:12],
                       d["init_rpm_lo"] + (d["init_rpm_hi"] - d["init_rpm_lo"]) * U[12:16]])
        a, b = (torch.stack([_u01(x) for x in self.draw(env, ep, 1, k)]) for k in (0, 1))
        p = torch.stack([v["mass"] * (1 + d["dr_mass"] * (2 * a[0] - 1)), v["Jx"] * (1 + d["dr_J"] * (2 * a[1] - 1)),
                         v["Jy"] * (1 + d["dr_J"] * (2 * a[2] - 1)), v["Jz"] * (1 + d["dr_J"] * (2 * a[3] - 1)),
                         v["kf"] * (1 + d["dr_kf"] * (2 * b[0] - 1)), torch.full_like(a[0], v["km"]),
                         d["tm_lo"] + (d["tm_hi"] - d["tm_lo"]) * b[1], torch.zeros_like(a[0])])
        f = torch.zeros(6, len(env), device=DEV, dtype=F64)
        if d["dist_f"]:
            x, y = (torch.stack([2 * _u01(z) - 1 for z in self.draw(env, ep, 6, k)]) for k in (0, 1))
            f = torch.stack([d["dist_f"] * x[0], d["dist_f"] * x[1], d["dist_f"] * x[2], d["dist_tau"] * x[3],
                             d["dist_tau"] * y[0], d["dist_tau"] * y[1]])
        return s, p, f

    def step(self, a):
        """One env step with actions a [4][n]; returns the transition record's fields."""
        d = self.d
        s, priv = self.s, self.priv()
        s2 = self.rk4(s, (a + 1) * 0.5 * self.hi, self.p, self.f)
        r = self.reward(s2, a)
        term = (s2[:3].abs() > d["term_pos"]).any(0)
        after = self.ep_step + 1
        trunc = ~term & (after >= d["episode_len"])
        flags = term.long() | (trunc.long() << 1) | (self.ep_step << 8)
        done = term | trunc
        rec = dict(s=s, a=a, r=r, flags=flags, priv=priv, side=s2, done=done, term=term, trunc=trunc)
        nh = d["n_hist"]
        hist = torch.cat([a, self.hist[:-4]]) if nh else self.hist.clone()
        hist[4 * nh:] = self.hist[4 * nh:]
        self.ep_ret = self.ep_ret + r
        self.s, self.hist, self.ep_step = s2.clone(), hist, torch.where(done, torch.zeros_like(after), after)
        i = done.nonzero()[:, 0]
        if len(i):
            self.ret_sum = self.ret_sum + torch.where(done, self.ep_ret, torch.zeros_like(self.ep_ret))
            self.ep_ret = torch.where(done, torch.zeros_like(self.ep_ret), self.ep_ret)
            self.ep[i] += 1
            s0, p0, f0 = self.start(i, self.ep[i])
            self.p, self.f = self.p.clone(), self.f.clone()
            self.s[:, i], self.p[:, i], self.f[:, i], self.hist[:, i] = s0, p0, f0, 0.0
        return rec

    def explore(self, mu, t, sigma):
        r0, r1 = self.draw(self.e, t, 3, 0), self.draw(self.e, t, 3, 1)
        z = torch.stack([_normal(r0[0], r0[1]), _normal(r0[2], r0[3]), _normal(r1[0], r1[1]), _normal(r1[2], r1[3])])
        return (mu + _f32(sigma) * z).clamp(-1.0, 1.0)

    def act(self, actor, hidden, t, sigma):
        oa = self.obs_actor(self.s, self.hist, self.e, t)
        return self.explore(torch.tanh(_mlp(actor, oa.T, hidden, 4)).T, t, sigma)


def _mlp(w, x, hid, out):
    """Rows x [..][in] through in -> hid -> hid -> out (ReLU, ReLU, linear), flat weights."""
    inp, at = x.shape[-1], 0

    def take(*shape):
        nonlocal at
        m = math.prod(shape)
        at += m
        return w[at - m:at].reshape(shape)
    W1, b1, W2, b2, W3, b3 = take(hid, inp), take(hid), take(hid, hid), take(hid), take(out, hid), take(out)
    return torch.relu(torch.relu(x @ W1.T + b1) @ W2.T + b2) @ W3.T + b3


def _td3(ref, case, hp, net, ring, head, size, t_now, n_updates, u):
    """TD3 updates u, u+1, .. of the networks `net` (flat tensors, replaced in place)."""
    rec, side = ring
    d, cap, nh, n = ref.d, rec.shape[0], ref.d["n_hist"], ref.n
    B, H = hp["batch"], hp["hidden"]
    b1, b2, eps, lr = (_f32(hp[k]) for k in ("beta1", "beta2", "eps", "lr"))
    tau, gamma = _f32(hp["tau"]), _f32(hp["gamma"])
    j = torch.arange(B, device=DEV)
    ta, tc, stats = u // 2, u, [0.0, 0.0]

    def adam(name, m, g, t):
        net["m_" + m] = b1 * net["m_" + m] + (1 - b1) * g
        net["v_" + m] = b2 * net["v_" + m] + (1 - b2) * g * g
        net[name] = net[name] - lr * (net["m_" + m] / (1 - b1 ** t)) / (torch.sqrt(net["v_" + m] / (1 - b2 ** t)) + eps)

    for u in range(u, u + n_updates):
        lost = nh if size == cap else 0
        words = torch.stack(ref.draw(j >> 2, u, 4), -1)
        x = words.gather(1, (j & 3)[:, None])[:, 0]
        idx = (x * ((size - 1 - lost) * n)) >> 32
        k, env = idx // n, idx % n
        slot = (head - size + lost + k) % cap
        t_rec = t_now - size + lost + k
        row = rec[slot, :, env]
        fl = row[:, 22].contiguous().view(torch.int32).long()
        done, term, ep = (fl & 3) != 0, (fl & 1) != 0, fl >> 8
        nxt = torch.where(done[:, None], side[slot, :, env], rec[(slot + 1) % cap, :NS, env])
        s, s2, a, r = row[:, :NS].T.to(F64), nxt.T.to(F64), row[:, 17:21].T.to(F64), row[:, 21].to(F64)
        lags = [torch.where((ep >= i)[None], rec[(slot - i) % cap, 17:21, env].T.to(F64), torch.zeros_like(a))
                for i in range(1, nh + 1)]
        none = torch.zeros(0, B, device=DEV, dtype=F64)
        hist = torch.cat(lags) if lags else none
        hist2 = torch.cat(([a] + lags)[:nh]) if lags else none
        priv = row[:, 23:].T.to(F64) if rec.shape[1] > 23 else None
        oa, oa2 = ref.obs_actor(s, hist, env, t_rec), ref.obs_actor(s2, hist2, env, t_rec + 1)
        oc, oc2 = ref.obs_critic(s, hist, priv, oa).T, ref.obs_critic(s2, hist2, priv, oa2).T
        r0, r1 = ref.draw(j, u, 5, 0), ref.draw(j, u, 5, 1)
        z = torch.stack([_normal(r0[0], r0[1]), _normal(r0[2], r0[3]), _normal(r1[0], r1[1]), _normal(r1[2], r1[3])], 1)
        clip = _f32(hp["noise_clip"])
        a2 = (torch.tanh(_mlp(net["actor_t"], oa2.T, H, 4)) + (_f32(hp["sigma_t"]) * z).clamp(-clip, clip)).clamp(-1, 1)
        x2 = torch.cat([oc2, a2], 1)
        q2 = torch.minimum(_mlp(net["c1_t"], x2, H, 1), _mlp(net["c2_t"], x2, H, 1))[:, 0]
        y = r + torch.where(term, torch.zeros_like(q2), gamma * q2)
        xc = torch.cat([oc, a.T], 1)
        tc += 1
        loss = 0.0
        for name in ("c1", "c2"):
            w = net[name].detach().requires_grad_()
            lc = ((_mlp(w, xc, H, 1)[:, 0] - y) ** 2).mean()
            adam(name, name, torch.autograd.grad(lc, w)[0], tc)
            loss = loss + lc.detach()
        stats[0] = loss
        if u % hp["policy_delay"] == hp["policy_delay"] - 1:
            ta += 1
            w = net["actor"].detach().requires_grad_()
            la = -_mlp(net["c1"], torch.cat([oc, torch.tanh(_mlp(w, oa.T, H, 4))], 1), H, 1).mean()
            adam("actor", "a", torch.autograd.grad(la, w)[0], ta)
            stats[1] = la.detach()
            for name in ("actor", "c1", "c2"):
                net[name + "_t"] = tau * net[name] + (1 - tau) * net[name + "_t"]
    return stats


def _train_run(case, seed, i):
    """One run of a training case: its networks and final states."""
    hp, n, slots = _hyper(case, i), case["n"], case["slots"]
    ld = (n + 31) // 32 * 32
    d = _sim(case, seed, i)
    g = _gen(seed, 2, i)
    live = _live(g, case, d, ld)
    rec, side = _ring(g, slots, ld, d["critic_layout"] in (1, 2))
    head = int(torch.randint(0, slots, (1,), generator=g, device=DEV))
    rec, side = rec.roll(head, 0), side.roll(head, 0)
    net = {k: v.to(F64) for k, v in _networks(_gen(seed, 3, i), case, hp).items()}
    ref = _Ref(d, n, live)
    t, u = T_START, U_START
    if case["kind"] == "update":
        stats = _td3(ref, case, hp, net, (rec, side), head, slots, t, case["updates"], u)
        net["stats"] = torch.stack([*stats, torch.zeros_like(stats[0]), torch.zeros_like(stats[0])])
        return net
    for _ in range(case["steps"]):
        tr = ref.step(ref.act(net["actor"], hp["hidden"], t, 0.1))
        rec[head, :NS, :n], rec[head, 17:21, :n], rec[head, 21, :n] = tr["s"].float(), tr["a"].float(), tr["r"].float()
        rec[head, 22, :n] = tr["flags"].int().view(torch.float32)
        if rec.shape[1] > 23:
            rec[head, 23:, :n] = tr["priv"].float()
        side[head, :, :n] = torch.where(tr["done"], tr["side"].float(), side[head, :, :n])
        t, head = t + 1, (head + 1) % slots
        _td3(ref, case, hp, net, (rec, side), head, slots, t, case["updates"], u)
        u += case["updates"]
    return {**{k: net[k] for k in NETS}, "state": ref.s}


def _exact_vjp(case, seed):
    s0, p32, x32, w = _vjp_inputs(case, seed)
    d = W.config("c3")
    d.update(n_hist=case["n_hist"], seed=0, run_id=0)
    ref = _Ref(d, case["n"])
    wp, wq, wv, wa = (_f32(x) for x in WEIGHTS)
    p, x = p32.to(F64).requires_grad_(), x32.to(F64).requires_grad_()
    s, f = s0.to(F64), torch.zeros(6, case["n"], device=DEV, dtype=F64)
    hist = torch.zeros(64, case["n"], device=DEV, dtype=F64)
    loss = 0.0
    for t in range(case["horizon"]):
        if case["closed"]:
            oa = torch.cat([ref.obs(s), hist[: 4 * case["n_hist"]]])
            a = torch.tanh(_mlp(x, oa.T, case["hidden"], 4)).T
            hist = torch.cat([a, hist[:-4]])
        else:
            a = x[t]
        s = ref.rk4(s, (a + 1) * 0.5 * ref.hi, p, f)
        loss = (loss + wp * (s[:3] ** 2).sum(0) + wq * (1 - s[3] ** 2) + wv * (s[7:10] ** 2).sum(0)
                + wa * (a ** 2).sum(0))
    gp, gx = torch.autograd.grad(loss, (p, x), w.to(F64))
    return dict(loss=loss.detach(), g_x=gx, g_params=gp[:4])


def _exact_track(case, seed):
    d = _sim(case, seed)
    n = case["n"]
    ld = (n + 31) // 32 * 32
    ref = _Ref(d, n, _live(_gen(seed, 2, 0), case, d, ld))
    actor = _hover_actor(_gen(seed, 3), _obs_dim(case), case["hidden"]).to(F64)
    T = torch.tensor([15.0, 5.5, 3.5], device=DEV, dtype=F64).repeat(n // 3 + 1)[:n]
    dt, zero = _f32(d["dt"]), torch.zeros(n, device=DEV, dtype=F64)

    def target(k):
        th = 2 * math.pi * k * dt / T
        return (torch.stack([torch.cos(th), 0.5 * torch.sin(2 * th), zero]),
                2 * math.pi / T * torch.stack([-torch.sin(th), torch.cos(2 * th), zero]))

    p0, v0 = target(0)
    hover = torch.sqrt(ref.p[0] * _f32(W.VEHICLE["g"]) / (4 * ref.p[4])).clamp(0.0, ref.hi)
    s = torch.cat([p0, torch.stack([zero + 1, zero, zero, zero]), v0, torch.zeros(3, n, device=DEV, dtype=F64),
                   hover.expand(4, n)])
    hist = torch.zeros_like(ref.hist)
    alive, ok, sq = torch.ones(n, device=DEV, dtype=torch.bool), zero.long(), torch.zeros(2, n, device=DEV, dtype=F64)
    clip_p, clip_v = _f32(0.2), 1.0
    for k in range(case["steps"]):
        pr, vr = target(k)
        o = ref.obs(s)
        o = torch.cat([(o[:3] - pr).clamp(-clip_p, clip_p), o[3:12], (o[12:15] - vr).clamp(-clip_v, clip_v), o[15:]])
        a = torch.tanh(_mlp(actor, torch.cat([o, hist[: 4 * d["n_hist"]]]).T, case["hidden"], 4)).T.clamp(-1, 1)
        s2 = ref.rk4(s, (a + 1) * 0.5 * ref.hi, ref.p, ref.f)
        e = s2[:3] - target(k + 1)[0]
        alive = alive & ~(e.abs() > _f32(d["term_pos"])).any(0)
        sq = sq + torch.where(alive, torch.stack([(e ** 2).sum(0), (e[:2] ** 2).sum(0)]), torch.zeros_like(sq))
        ok = ok + alive
        s, hist = torch.where(alive, s2, s), torch.cat([a, hist[:-4]])
    return dict(sq_err=sq, steps_ok=None)


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind == "vjp":
        return _exact_vjp(case, seed)
    if kind == "dynamics":
        if n * case["steps"] > 20_000_000:
            return None
        ld = (n + 3) // 4 * 4
        g = _gen(seed, 1)
        s, p = _states(g, (), ld).to(F64), _vehicles(g, ld).to(F64)
        rpm, f = _u(g, (4, ld), 5_000.0, 21_000.0).to(F64), torch.zeros(6, ld, device=DEV, dtype=F64)
        if case["disturbed"]:
            f = torch.cat([_u(g, (3, ld), -0.0027, 0.0027), _u(g, (3, ld), -1e-6, 1e-6)]).to(F64)
        ref = _Ref(W.config("c2"), ld)
        for _ in range(case["steps"]):
            s = ref.rk4(s, rpm, p, f)
        return s[:, :n]
    if kind == "update":
        return _train_run(case, seed, 0)
    if kind == "train":
        if case["runs"] * case["steps"] * case["updates"] > 2_048:
            return None
        runs = [_train_run(case, seed, i) for i in range(case["runs"])]
        return {k: torch.cat([r[k] for r in runs]) for k in runs[0]}
    if kind == "track":
        return _exact_track(case, seed)
    d = _sim(case, seed)
    ld = (n + 31) // 32 * 32
    g = _gen(seed, 2, 0)
    live = _live(g, case, d, ld)
    ref = _Ref(d, n, live)
    if kind == "recalc":
        rec, side = _ring(g, case["slots"], ld, d["critic_layout"] in (1, 2))
        head = int(torch.randint(0, case["slots"], (1,), generator=g, device=DEV))
        out = torch.empty(case["slots"], n, device=DEV, dtype=F64)
        for t in range(case["slots"]):
            done = (rec[t, 22, :n].view(torch.int32) & 3) != 0
            nxt = rec[t + 1, :NS, :n] if t + 1 < case["slots"] else live["state"][:, :n]
            s2 = torch.where(done, side[t, :, :n], nxt).to(F64)
            out[t] = ref.reward(s2, rec[t, 17:21, :n].to(F64))
        return out.roll(head, 0)
    if kind == "step":
        a = (0.33 + 0.3 * torch.randn((4, ld), generator=g, device=DEV))[:, :n].to(F64).clamp(-1.0, 1.0)
        tr = ref.step(a)
        oa = ref.obs_actor(ref.s, ref.hist, ref.e, 1)
        return dict(obs_a=oa, obs_c=ref.obs_critic(ref.s, ref.hist, ref.priv(), oa), reward=tr["r"], terminated=None,
                    truncated=None, state=ref.s, hist=ref.hist, ep_step=None)
    # rollout.  Which step an episode ends at is a threshold on a rounded position, so over
    # enough episodes a 64-bit rollout takes another path than any 32-bit one: there is a
    # value to compare with only for a few thousand of them.
    if n * case["steps"] > 1 << 18:
        return None
    actor = _net(_gen(seed, 3), _obs_dim(case), case["hidden"], 4).to(F64)
    out = torch.zeros(case["slots"], 22, n, device=DEV, dtype=F64)
    for t in range(case["steps"]):
        tr = ref.step(ref.act(actor, case["hidden"], t, 0.1))
        out[t, :NS], out[t, 17:21], out[t, 21] = tr["s"], tr["a"], tr["r"]
    return dict(transitions=out, flags=None, state=ref.s, hist=ref.hist, ep_step=None, episodes=None,
                returns=ref.ret_sum)
