"""What the speed of this framework is measured on: the calls its users' programs make, through
the package's public entry points (``MarineEnv``, ``Sim``, ``adjoint.rollout``, ``NativeServer``),
over the sizes of the benchmark and of the tests and between them.

Kinds of case (the ``kind`` key) and what each stands for:

  env      one step of the Gym-style environment: a policy's throttles in, observation, reward
           and episode flags out, some envs finishing their episode and restarting inside the step
  control  a closed-loop controller that sets the throttles, advances a few sub-steps and reads the
           whole fleet's state back
  episode  a whole training episode: domain randomisation, reset, throttle schedule (buffered or
           procedural), the sub-steps with the launch shape the autotuner picks, state read-back
  rollout  an evaluation from given start states with a given schedule (nominal vehicles, or the
           full hydrodynamics with off-centre gravity)
  record   trajectory recording (system-identification data)
  adjoint  a differentiable rollout and its gradients with respect to the hydrodynamic
           coefficients, every throttle and the start state
  serve    a burst of rollout jobs of different sizes, horizons and vehicles through the native
           request loop, results collected

``exact`` evaluates the same vehicles in 64 bits with plain torch: Eq. 1 in matrix form, RK4 with
the attitude renormalised after each sub-step, and the documented counter-based draws.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2410_14117_gb300 import inputs as I
from paper_2410_14117_gb300.adjoint import rollout
from paper_2410_14117_gb300.autotune import Autotuner
from paper_2410_14117_gb300.env import TASKS, MarineEnv
from paper_2410_14117_gb300.serve import NativeServer, Request
from paper_2410_14117_gb300.sim import Sim

DT = float(np.float32(0.01))
LO, HI = float(np.float32(0.8)), float(np.float32(1.2))
CURRENT, NU0 = float(np.float32(0.2)), float(np.float32(0.3))
HOLD = 10  # sub-steps a throttle is held
RG_HALFWIDTH = float(np.float32(0.02))
COUPLING = 0.15

MAX_WORK = 262144 * 500  # env-sub-steps of the largest listed case


# ------------------------------------------------------------------------------- the cases

def listed():
    return [
        # a small training run's environment: station keeping, few vehicles, few sub-steps
        dict(name="env_station_1000", kind="env", n=1000, vehicle="rov", task="station",
             sub_steps=4, lookahead=1),
        # the usual size of a training run's environment
        dict(name="env_circle_4096", kind="env", n=4096, vehicle="heavy", task="circle",
             sub_steps=10, lookahead=4),
        # a large environment of mixed vehicles
        dict(name="env_helix_65536", kind="env", n=65536, vehicle="mixed", task="helix",
             sub_steps=10, lookahead=3),
        # a controller in the loop at every sub-step, an odd fleet
        dict(name="control_10007", kind="control", n=10007, vehicle="rov", k=1),
        # the small parity fleet: nominal vehicles, no current, default launch
        dict(name="rollout_1024", kind="rollout", n=1024, vehicle="rov", k=500, full=False),
        # the headline episode: the next episode's parameters drawn beside this one's steps
        dict(name="episode_65536", kind="episode", n=65536, vehicle="rov", k=1000, prefetch=True,
             procedural=False),
        # the largest fleet of the sweep, parameters drawn in line, procedural throttles
        dict(name="episode_1048576", kind="episode", n=1048576, vehicle="rov", k=100,
             prefetch=False, procedural=True),
        # a mixed fleet in uneven groups
        dict(name="episode_mixed_262144", kind="episode", n=262144, vehicle="mixed", k=500,
             prefetch=False, procedural=True),
        # off-centre gravity with full added-mass and damping matrices
        dict(name="hydro_16384", kind="rollout", n=16384, vehicle="rov", k=200, full=True),
        # trajectories of 8-thruster vehicles recorded after every sub-step
        dict(name="record_30000", kind="record", n=30000, vehicle="heavy", k=200),
        # gradients of a 200-sub-step rollout, checkpoints every 20
        dict(name="adjoint_4096", kind="adjoint", n=4096, vehicle="rov", k=200, c=20, full=False),
        # a burst of 12 rollout jobs of 64 to 32,768 vehicles
        dict(name="serve_12", kind="serve", jobs=12, n=32768, k=400, tick=100),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["env", "env", "control", "episode", "episode", "rollout", "record",
                       "adjoint", "serve"])
    vehicle = rng.choice(["rov", "rov", "heavy", "mixed"])
    if kind == "env":
        return dict(kind=kind, n=_log(rng, 256, 131072), vehicle=vehicle,
                    task=rng.choice(sorted(TASKS)), sub_steps=rng.randint(1, 20),
                    lookahead=rng.randint(1, 6))
    if kind == "control":
        return dict(kind=kind, n=_log(rng, 256, 262144), vehicle=vehicle, k=rng.choice([1, 1, 2, 5]))
    if kind == "episode":
        n = _log(rng, 1024, 1048576)
        return dict(kind=kind, n=n, vehicle=vehicle, k=min(_log(rng, 50, 1000), MAX_WORK // n),
                    prefetch=rng.random() < 0.5, procedural=rng.random() < 0.5)
    if kind == "rollout":
        n = _log(rng, 300, 131072)
        return dict(kind=kind, n=n, vehicle=vehicle, k=_log(rng, 20, 500), full=rng.random() < 0.6)
    if kind == "record":
        n = _log(rng, 300, 65536)
        return dict(kind=kind, n=n, vehicle=vehicle, k=min(_log(rng, 20, 400), 8000000 // n))
    if kind == "adjoint":
        n = _log(rng, 64, 8192)
        return dict(kind=kind, n=n, vehicle=vehicle, k=min(_log(rng, 20, 300), 4096 * 200 // n),
                    c=rng.choice([5, 10, 16, 20]), full=rng.random() < 0.35)
    return dict(kind=kind, jobs=rng.randint(3, 14), n=_log(rng, 512, 32768),
                k=_log(rng, 60, 500), tick=rng.choice([50, 100]))


# ------------------------------------------------------------------------------- inputs

def _gen(seed, salt=0):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 1000003 + salt)


def _types(case):
    n = case["n"]
    if case["vehicle"] == "mixed":  # groups of uneven size, 60 % of the first type
        return I.mixed_fleet(3, n, max_group=max(2, n // 8))
    return np.full(n, 0 if case["vehicle"] == "rov" else 1, dtype=np.int32)


def _n_thr(case):
    return 6 if case["vehicle"] == "rov" else 8


def _uniform(gen, shape, lo, hi):
    return torch.rand(shape, generator=gen, device="cuda") * (hi - lo) + lo


def _start_states(seed, n, types, spread, far=0.0):
    """States in the middle of a run: [n, 21] float32, p within `spread` m of the origin (a share
    `far` of the envs 5 m away), attitudes tilted up to some 60 degrees, any throttle state."""
    g = _gen(seed, 1)
    s = torch.zeros((n, 21), device="cuda")
    s[:, 0:3] = _uniform(g, (n, 3), -1, 1) * (spread / math.sqrt(3.0))
    if far:
        s[:, 0] += 5.0 * (torch.rand(n, generator=g, device="cuda") < far)
    e = torch.randn((n, 3), generator=g, device="cuda").clamp_(-2, 2) * 0.25
    q = torch.cat([torch.ones((n, 1), device="cuda"), e], dim=1)
    s[:, 3:7] = q / q.norm(dim=1, keepdim=True)
    s[:, 7:13] = 0.3 * torch.randn((n, 6), generator=g, device="cuda")
    thr = torch.tensor([6, 8], device="cuda")[torch.as_tensor(types, device="cuda").long()]
    s[:, 13:21] = _uniform(g, (n, 8), -1, 1) * (torch.arange(8, device="cuda") < thr[:, None])
    return s


def _schedule(seed, n_seg, n, w):
    return _uniform(_gen(seed, 2), (n_seg, n, w), -1, 1)


def _centres(case, seed, radius=2.0, spawn=0.5):
    """Reference centres and phases [n, 4] as MarineEnv draws them for this seed."""
    g = np.random.default_rng(seed)
    n = case["n"]
    phase = g.uniform(0.0, 2.0 * math.pi, n)
    c = np.zeros((n, 4))
    c[:, 3] = phase
    if case["task"] in ("circle", "helix"):
        c[:, 0], c[:, 1] = -radius * np.cos(phase), -radius * np.sin(phase)
    elif case["task"] == "lemniscate":
        den = 1.0 + np.sin(phase) ** 2
        c[:, 0] = -radius * np.cos(phase) / den
        c[:, 1] = -radius * np.sin(phase) * np.cos(phase) / den
    d = g.normal(size=(n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    c[:, :3] += d * (spawn * g.uniform(0.0, 1.0, (n, 1)) ** (1.0 / 3.0))
    return c


def _extension(seed, n):
    """Off-diagonal added mass and damping [n, 45] float32, 15 % coupling of the nominal diagonals
    (M_A above its diagonal, then D_l off its diagonal, row by row)."""
    g = _gen(seed, 3)
    p = I.fleet_vehicles()[0].params
    ma, dl = p[4:10], p[10:16]
    scale = [math.sqrt(ma[i] * ma[j]) for i in range(6) for j in range(i + 1, 6)]
    scale += [math.sqrt(dl[i] * dl[j]) for i in range(6) for j in range(6) if j != i]
    return _uniform(g, (n, 45), -1, 1) * torch.tensor(scale, dtype=torch.float32,
                                                      device="cuda") * COUPLING


def _jobs(case, seed):
    """Sizes log-uniform from 64, horizons and vehicles by the case; the seed keys the draws."""
    shape, keys = np.random.default_rng(42), np.random.default_rng(seed)
    out = []
    for i in range(case["jobs"]):
        n = int(round(math.exp(shape.uniform(math.log(64), math.log(case["n"])))))
        h = int(shape.integers(max(20, case["k"] // 8), case["k"] + 1))
        first = i == 0  # the largest of the burst
        out.append(dict(n_envs=case["n"] if first else n, horizon=case["k"] if first else h,
                        vehicle=int(shape.integers(0, 2)),
                        param_seed=int(keys.integers(1, 2**62)),
                        cmd_seed=int(keys.integers(1, 2**62))))
    return out


# A program keeps one tuner (it remembers what it picked) and one server.
_TUNER = None
_SERVERS = {}


def _server(tick):
    if tick not in _SERVERS:
        _SERVERS[tick] = NativeServer(I.fleet_vehicles(), budget_bytes=40e9,
                                      capacity_envs=16 * 32768, k=tick, record=True,
                                      keep_results=True)
    return _SERVERS[tick]


def _tune(sim, vehicles, general=False):
    global _TUNER
    if _TUNER is None:
        _TUNER = Autotuner(horizon=200, reps=2)
    _TUNER.tune(sim, vehicles, general)


# ------------------------------------------------------------------------------- prepare

def prepare(case, seed):
    kind = case["kind"]
    vs = I.fleet_vehicles()
    if kind == "serve":
        return dict(kind=kind, srv=_server(case["tick"]), jobs=_jobs(case, seed))
    n, types = case["n"], _types(case)
    if kind == "env":
        env = MarineEnv(n, task=case["task"], vehicle=types, sub_steps=case["sub_steps"],
                        seed=seed, nu0_sigma=NU0, lookahead=case["lookahead"])
        env.reset()
        env.sim.set_state(_start_states(seed, n, types, 1.0, far=0.02))
        acts = [_schedule(seed + 7 * i, 1, n, env.n_thr)[0] * 1.1 for i in range(2)]
        return dict(kind=kind, env=env, acts=acts, i=0)

    sim = Sim(n, types, vs)
    w = _n_thr(case)
    if w == 6:
        sim.set_action_width(6)
    st = dict(kind=kind, sim=sim, k=case["k"], seed=int(seed), i=0,
              out=torch.empty((n, 21), device="cuda"))
    n_seg = -(-case["k"] // HOLD)
    if kind == "control":
        sim.randomize(seed, LO, HI, CURRENT, NU0)
        sim.set_state(_start_states(seed, n, types, 1.0))
        st["acts"] = [_schedule(seed + 7 * i, 1, n, w) for i in range(2)]
    elif kind == "episode":
        _tune(sim, vs)
        if case["procedural"]:
            st["acts"] = None
        else:
            st["acts"] = _schedule(seed, n_seg, n, w)
        st["prefetch"] = case["prefetch"]
        if case["prefetch"]:
            sim.randomize_prefetch(seed, LO, HI, CURRENT)
    else:
        full = case.get("full", False)
        if kind != "rollout" or full:
            sim.randomize(seed, LO, HI, CURRENT, NU0, rg_halfwidth=RG_HALFWIDTH if full else 0.0)
        if full:
            sim.set_hydro_offdiag(_extension(seed, n))
            if kind == "rollout":
                _tune(sim, vs, general=True)
        st["s0"] = _start_states(seed, n, types, 1.0)
        st["acts"] = _schedule(seed, n_seg, n, w)
        if kind == "record":
            st["traj"] = torch.empty((case["k"], 13, n), device="cuda")
        if kind == "adjoint":
            st["c"] = case["c"]
            st["coef"] = sim.get_params()[:, 4:22].clone().requires_grad_(True)
            st["acts"].requires_grad_(True)
            st["s0"].requires_grad_(True)
            st["g"] = _loss_gradient(seed, case)
    return st


def _loss_gradient(seed, case):
    return torch.randn((case["k"], case["n"], 13), generator=_gen(seed, 4), device="cuda")


# ------------------------------------------------------------------------------- run

def run(st):
    kind = st["kind"]
    if kind == "env":
        st["i"] += 1
        return st["env"].step(st["acts"][(st["i"] - 1) % 2])
    if kind == "serve":
        reqs = [Request(arrival_s=0.0, hold=HOLD, **j) for j in st["jobs"]]
        done, _ = st["srv"].run(reqs, realtime=False)
        return [(r.final_state, r.traj) for r in reqs]
    sim, k = st["sim"], st["k"]
    if kind == "control":
        st["i"] += 1
        sim.set_actions_borrowed(st["acts"][(st["i"] - 1) % 2], 1)
        sim.step(k)
        return sim.get_state(st["out"])
    if kind == "episode":
        ep = st["seed"] + st["i"]
        st["i"] += 1
        sim.randomize(ep, LO, HI, CURRENT, NU0, wait=False)
        sim.reset()
        if st["acts"] is None:
            sim.set_procedural_actions(ep + 5678, HOLD)
        else:
            sim.set_actions_borrowed(st["acts"], HOLD)
        sim.step(k)
        if st["prefetch"]:
            sim.randomize_prefetch(ep + 1, LO, HI, CURRENT)
        return sim.get_state(st["out"])
    if kind == "adjoint":
        traj = rollout(sim, st["coef"], st["acts"], st["s0"], HOLD, k, st["c"])
        grads = torch.autograd.grad(traj, (st["coef"], st["acts"], st["s0"]), st["g"])
        return (traj.detach(),) + grads
    sim.set_state(st["s0"])
    sim.set_actions_borrowed(st["acts"], HOLD)
    if kind == "record":
        return sim.step_record(k, st["traj"]), sim.get_state(st["out"])
    sim.step(k)
    return sim.get_state(st["out"])


# ------------------------------------------------------------------------------- work

# Operations (an FMA is two) of one sub-step of one vehicle: four right-hand sides, the stage
# updates, the throttle lag and the renormalisation, for a diagonal mass matrix and for the full
# matrices (6 x 6 products for M^-1, M_A and D_l).
_FLOPS = {6: 1143, 8: 1223}
_FULL_FLOPS = 1300


def work(case):
    kind = case["kind"]
    if kind == "serve":
        b = f = 0.0
        for j in _jobs(case, 1):
            f += j["n_envs"] * j["horizon"] * _FLOPS[6]
            b += j["n_envs"] * 4 * (21 + 13 * j["horizon"])
        return {"bytes": b, "flops": f}
    n, w = case["n"], _n_thr(case)
    k = case["sub_steps"] if kind == "env" else case["k"]
    flops = n * k * (_FLOPS[w] + (_FULL_FLOPS if case.get("full") else 0))
    state, par = 4 * (13 + w), 4 * 34
    acts = 0 if case.get("procedural") else 4 * w * (1 if kind in ("env", "control") else -(-k // HOLD))
    b = par + acts
    if kind == "env":
        m = 1 if case["task"] == "station" else case["lookahead"]
        b += 2 * state + 24 + 4 * (6 * m + 6) + 4 + 1 + 4
    elif kind == "control":
        b += 2 * state + 4 * 21
    elif kind == "episode":
        b += 4 * 21
    else:
        b += 2 * 4 * 21 + (4 * 66 if case.get("full") else 0)
        if kind in ("record", "adjoint"):
            b += 4 * 13 * k
        if kind == "adjoint":
            b += 4 * 13 * k + 4 * (18 + 21) + acts
            flops *= 3  # the forward, and a transpose of about twice its operations
    return {"bytes": float(n * b), "flops": float(flops)}


def tolerance(case):
    """About four times the distance of the framework's results from `exact`, measured over the
    listed cases and drawn ones (32-bit state, rounded once a sub-step; the largest difference is
    that of a fast-turning vehicle among many)."""
    kind = case["kind"]
    if kind == "env":  # measured: rel 2.5e-7, max 2.7e-6
        return {"rel": 1e-6, "max": 1.2e-5, "differ": 1e-4}
    if kind == "control":  # 5.1e-8, 2.5e-7 for one sub-step
        return {"rel": 4e-7, "max": 3e-6}
    if kind == "adjoint":  # 4.1e-6 (the start state's gradient), 3.7e-5
        return {"rel": 1.6e-5, "max": 2e-4}
    return {"rel": 4e-6, "max": 4e-4}  # 1e-6, 1.1e-4


# ------------------------------------------------------------------------------- 64 bits
# Component-first arrays [components, n] in float64.

_M32 = 0xFFFFFFFF


def _mulhilo(m, c):
    hi = (m * (c >> 16) + ((m * (c & 0xFFFF)) >> 16)) >> 16
    return hi & _M32, (m * c) & _M32


def _philox(seed, gid, stream, block):
    """Philox4x32-10 words [4, n] (Salmon et al., SC 2011) of counter (gid lo, gid hi, stream,
    block) under key seed."""
    c = [gid & _M32, gid >> 32, torch.full_like(gid, stream), torch.full_like(gid, block)]
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for _ in range(10):
        h0, l0 = _mulhilo(0xD2511F53, c[0])
        h1, l1 = _mulhilo(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return torch.stack(c)


def _u01(x):
    return ((x >> 9).double() + 0.5) * 2.0 ** -23


def _normals(x):
    u = _u01(x)
    r = torch.sqrt(-2.0 * torch.log(u[0::2]))
    a = 2.0 * math.pi * u[1::2]
    return torch.stack([r * torch.cos(a), r * torch.sin(a)], dim=1).reshape(-1, x.shape[1])


def _gids(n):
    return torch.arange(n, dtype=torch.int64, device="cuda")


def _f32(x):
    return x.float().double()


def _nominal(types):
    tab = torch.tensor(np.stack([v.params for v in I.fleet_vehicles()]), device="cuda")
    return _f32(tab)[torch.as_tensor(types, device="cuda").long()].T.contiguous()


def _randomised(seed, types, rg_halfwidth=0.0):
    """Parameter records [35, n] as drawn by the domain randomisation, stored in 32 bits."""
    p = _nominal(types)
    g = _gids(p.shape[1])
    words = torch.cat([_philox(seed, g, 0, b) for b in range(7)])
    for j, idx in enumerate(I.RANDOMISED_INDICES):
        p[idx] *= LO + (HI - LO) * _u01(words[j])
    p[32:35] += CURRENT * _normals(_philox(seed, g, 1, 0))[:3]
    if rg_halfwidth:
        p[24:27] += rg_halfwidth * (2.0 * _u01(_philox(seed, g, 0, 7)[:3]) - 1.0)
    return _f32(p)


def _reset_nu(seed, n, episode):
    g = _gids(n)
    x = torch.cat([_philox(seed, g, 2, 2 * episode), _philox(seed, g, 2, 2 * episode + 1)])
    return NU0 * _normals(x[:6])


def _reset_state(seed, n, episode):
    s = torch.zeros((21, n), dtype=torch.float64, device="cuda")
    s[3] = 1.0
    s[7:13] = _reset_nu(seed, n, episode)
    return s


def _procedural(cmd_seed, types):
    thr = _thruster_mask(types)

    def at(seg):
        g = _gids(thr.shape[1])
        x = torch.cat([_philox(cmd_seed, g, 3, 2 * seg), _philox(cmd_seed, g, 3, 2 * seg + 1)])
        return (2.0 * _u01(x) - 1.0) * thr

    return at


def _buffered(acts, types):
    thr = _thruster_mask(types)

    def at(seg):
        a = acts[min(seg, acts.shape[0] - 1)].double().T
        c = torch.zeros_like(thr)
        return torch.cat([a, c[: 8 - a.shape[0]]]) * thr if a.shape[0] < 8 else a * thr

    return at


def _thruster_mask(types):
    nt = torch.tensor([6, 8], device="cuda")[torch.as_tensor(types, device="cuda").long()]
    return (torch.arange(8, device="cuda")[:, None] < nt).double()


def _cross(a, b):
    return torch.linalg.cross(a, b, dim=0)


def _turn(w, e, x):
    """R(q) x = x + 2 w e x x + 2 e x (e x x); with -w, R(q)^T x."""
    t = _cross(e, x)
    return x + 2.0 * w * t + 2.0 * _cross(e, t)


def _apply(A, x):
    return A * x if A.dim() == 2 else (A * x[None]).sum(1)


class _Vehicle:
    """Eq. 1 of a fleet in 64 bits; coef [18, n]: the diagonals of M_A, D_l and D_q."""

    def __init__(self, par, types, xh=None, coef=None):
        coef = par[4:22] if coef is None else coef
        self.ma, self.dl, self.dq = coef[0:6], coef[6:12], coef[12:18]
        self.m, self.ig = par[0], par[1:4]
        self.W, self.B, self.rg, self.rb = par[22], par[23], par[24:27], par[27:30]
        self.kT, self.itau, self.vc = par[30], 1.0 / par[31], par[32:35]
        n = par.shape[1]
        self.full = xh is not None
        if self.full:
            iu = torch.triu_indices(6, 6, 1, device="cuda")
            up = torch.zeros((6, 6, n), dtype=torch.float64, device="cuda")
            up[iu[0], iu[1]] = xh[:15]
            self.ma = torch.diag_embed(self.ma.T).permute(1, 2, 0) + up + up.transpose(0, 1)
            off = torch.zeros((6, 6, n), dtype=torch.float64, device="cuda")
            ij = [(i, j) for i in range(6) for j in range(6) if i != j]
            off[[i for i, _ in ij], [j for _, j in ij]] = xh[15:]
            self.dl = torch.diag_embed(self.dl.T).permute(1, 2, 0) + off
            eye = torch.eye(3, dtype=torch.float64, device="cuda")[:, :, None]
            rg = self.rg
            z = torch.zeros_like(rg[0])
            S = torch.stack([torch.stack([z, -rg[2], rg[1]]), torch.stack([rg[2], z, -rg[0]]),
                             torch.stack([-rg[1], rg[0], z])])
            Io = eye * self.ig[:, None] + self.m * (eye * (rg * rg).sum(0) - rg[:, None] * rg[None])
            rb = torch.cat([torch.cat([eye * self.m, -self.m * S], 1),
                            torch.cat([self.m * S, Io], 1)], 0)
            self.minv = torch.linalg.inv((rb + self.ma).permute(2, 0, 1)).permute(1, 2, 0)
        else:
            self.minv = 1.0 / (torch.cat([self.m.expand(3, n), self.ig]) + self.ma)
        vs = I.fleet_vehicles()
        d = torch.tensor(np.stack([v.d for v in vs]), dtype=torch.float32, device="cuda").double()
        r = torch.tensor(np.stack([v.r for v in vs]), dtype=torch.float32, device="cuda").double()
        self.alloc = torch.cat([d, torch.linalg.cross(r, d, dim=2)], dim=2).transpose(1, 2)
        t = torch.as_tensor(types, device="cuda").long()
        self.types = None if bool((t == t[0]).all()) else t
        self.type0 = int(t[0])

    def rhs(self, s, c):
        w4, e, v, w, nu, n = s[3], s[4:7], s[7:10], s[10:13], s[7:13], s[13:21]
        f = n * n.abs() * self.kT
        if self.types is None:
            tau = self.alloc[self.type0] @ f
        else:
            tau = torch.where(self.types == 0, self.alloc[0] @ f, self.alloc[1] @ f)
        vcb = _turn(-w4, e, self.vc)
        down = torch.zeros_like(e)
        down[2] = 1.0
        k = _turn(-w4, e, down)
        nur = torch.cat([v - vcb, w])
        Q = _apply(self.ma, nur)
        P1, P2 = self.m * v, self.ig * w
        if self.full:
            P1 = P1 + self.m * _cross(w, self.rg)
            P2 = P2 + self.m * (_cross(self.rg, v) - _cross(self.rg, _cross(self.rg, w)))
        cor = torch.cat([_cross(w, P1 + Q[:3]),
                         _cross(v, P1) + _cross(nur[:3], Q[:3]) + _cross(w, P2 + Q[3:])])
        g = torch.cat([(self.W - self.B) * k, _cross(self.W * self.rg - self.B * self.rb, k)])
        ca = torch.cat([_cross(w, vcb), torch.zeros_like(w)])
        damp = _apply(self.dl, nur) + self.dq * nur.abs() * nur
        nud = _apply(self.minv, tau - cor - damp + g - _apply(self.ma, ca))
        qd = torch.cat([-(e * w).sum(0, keepdim=True), w4 * w + _cross(e, w)]) * 0.5
        return torch.cat([_turn(w4, e, v), qd, nud, (c - n) * self.itau])

    def step(self, s, c, h=DT):
        k1 = self.rhs(s, c)
        k2 = self.rhs(s + 0.5 * h * k1, c)
        k3 = self.rhs(s + 0.5 * h * k2, c)
        k4 = self.rhs(s + h * k3, c)
        y = s + (h / 6.0) * (k1 + 2.0 * (k2 + k3) + k4)
        q = y[3:7]
        return torch.cat([y[:3], q / q.square().sum(0).sqrt(), y[7:]])

    def run(self, s, commands, hold, k, traj=None):
        for j in range(k):
            if j % hold == 0:
                c = commands(j // hold)
            s = self.step(s, c)
            if traj is not None:
                traj.append(s[:13])
        return s


def _reference(case, centres, t, radius=2.0, omega=0.3, vz=0.1):
    radius, omega, vz = (float(np.float32(x)) for x in (radius, omega, vz))
    s = omega * t + centres[3]
    sn, cs, z = torch.sin(s), torch.cos(s), torch.zeros_like(s)
    if case["task"] == "station":
        d = [z, z, z]
    elif case["task"] == "lemniscate":
        den = 1.0 + sn * sn
        d = [radius * cs / den, radius * sn * cs / den, z]
    else:
        d = [radius * cs, radius * sn, z + (vz * t if case["task"] == "helix" else 0.0)]
    return centres[:3] + torch.stack(d)


def _observe(case, centres, s, t):
    w, x, y, z = s[3], s[4], s[5], s[6]
    phi = torch.atan2(2 * (w * x + y * z), 1 - 2 * (x * x + y * y))
    theta = torch.asin((2 * (w * y - z * x)).clamp(-1, 1))
    psi = torch.atan2(2 * (w * z + x * y), 1 - 2 * (y * y + z * z))
    rows, m = [], 1 if case["task"] == "station" else case["lookahead"]
    for i in range(m):
        ti = t if case["task"] == "station" else t + 0.5 * (i + 1)
        rows += [s[:3] - _reference(case, centres, ti), torch.stack([phi, theta, psi])]
    return torch.cat(rows + [s[7:13]])


def _exact_env(case, seed):
    n, types = case["n"], _types(case)
    par = _randomised(seed, types)
    s = _start_states(seed, n, types, 1.0, far=0.02).double().T
    acts = (_schedule(seed, 1, n, 6 if int(np.max(types)) == 0 else 8) * 1.1).clamp(-1, 1)
    k = case["sub_steps"]
    s = _Vehicle(par, types).run(s, _buffered(acts, types), k, k)
    centres = torch.tensor(_centres(case, seed), dtype=torch.float32, device="cuda").double().T
    t = k * DT
    err = (s[:3] - _reference(case, centres, t)).square().sum(0).sqrt()
    done = err > 3.0
    obs = torch.where(done, _observe(case, centres, _reset_state(seed, n, 2), 0.0),
                      _observe(case, centres, s, t))
    return (obs.T, -err, None, {"episode_error": torch.where(done, err, torch.zeros_like(err))})


def exact(case, seed):
    kind = case["kind"]
    if kind == "env":
        return _exact_env(case, seed)
    if kind == "serve":
        out = []
        for j in _jobs(case, seed):
            n, types = j["n_envs"], np.full(j["n_envs"], j["vehicle"], dtype=np.int32)
            traj = []
            s = _Vehicle(_randomised(j["param_seed"], types), types).run(
                _reset_state(j["param_seed"], n, 0), _procedural(j["cmd_seed"], types), HOLD,
                j["horizon"], traj)
            out.append((s.T, torch.stack(traj)))
        return out
    n, types = case["n"], _types(case)
    w, k = _n_thr(case), case["k"]
    full = case.get("full", False)
    n_seg = -(-k // HOLD)
    if kind == "episode":
        par, s0 = _randomised(seed, types), _reset_state(seed, n, 0)
        cmd = (_procedural(seed + 5678, types) if case["procedural"]
               else _buffered(_schedule(seed, n_seg, n, w), types))
        return _Vehicle(par, types).run(s0, cmd, HOLD, k).T
    s0 = _start_states(seed, n, types, 1.0).double().T.contiguous()
    if kind == "control":
        cmd = _buffered(_schedule(seed, 1, n, w), types)
        return _Vehicle(_randomised(seed, types), types).run(s0, cmd, k, k).T
    par = (_randomised(seed, types, RG_HALFWIDTH if full else 0.0)
           if kind != "rollout" or full else _nominal(types))
    xh = _extension(seed, n).double().T.contiguous() if full else None
    acts = _schedule(seed, n_seg, n, w)
    if kind == "adjoint":
        coef = par[4:22].T.contiguous().requires_grad_(True)
        acts = acts.double().requires_grad_(True)
        s0 = s0.T.contiguous().requires_grad_(True)
        traj = []
        _Vehicle(par, types, xh, coef.T).run(s0.T, _buffered(acts, types), HOLD, k, traj)
        traj = torch.stack(traj).permute(0, 2, 1)
        grads = torch.autograd.grad(traj, (coef, acts, s0), _loss_gradient(seed, case).double())
        return (traj.detach(),) + grads
    veh, cmd = _Vehicle(par, types, xh), _buffered(acts, types)
    if kind == "record":
        traj = []
        s = veh.run(s0, cmd, HOLD, k, traj)
        return torch.stack(traj), s.T
    return veh.run(s0, cmd, HOLD, k).T
