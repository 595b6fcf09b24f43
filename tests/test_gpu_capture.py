"""A user's own CUDA graphs of the library's calls, replayed around parameter changes made outside
them: every replay must do what the same call made directly does then."""
import ctypes

import numpy as np
import pytest
import torch

from _helpers import TOL_STEP, oracle_geo, oracle_nominal, rel_err, vehicles
from oracle import oracle as O
from paper_2410_14117_gb300 import inputs as I
from paper_2410_14117_gb300._lib import MG_NSTATE, MG_NTRAJ, call
from paper_2410_14117_gb300.sim import Sim, _ptr

pytestmark = pytest.mark.gpu

N, T, C, HOLD = 300, 20, 8, 5


def _capture(stream, fn):
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
        fn()
    return g


def _advance(sim, how):
    """A function that advances sim and returns what it computes besides the state."""
    dev = dict(device="cuda", dtype=torch.float32)
    if how == "step":
        return lambda: sim.step(T)
    if how == "chunks":
        sim.set_launch(64, 7, False)
        return lambda: sim.step(T)
    if how == "queue":
        sim.set_schedule(True, True)
        return lambda: sim.step(T)
    if how == "noalloc":
        call("mg_step_noalloc", sim._h, 1)
        return lambda: (call("mg_step_noalloc", sim._h, T), None)[1]
    if how == "record":
        traj = torch.empty((T, MG_NTRAJ, N), **dev)
        return lambda: sim.step_record(T, traj)
    if how == "task":
        sim.set_task(1, torch.zeros((N, 4), **dev), lookahead=2)
        return lambda: sim.task_step(T)[0]
    if how == "env":
        sim.set_task(1, torch.zeros((N, 4), **dev), lookahead=2)
        out = (torch.empty((N, sim.obs_dim), **dev), torch.empty(N, **dev),
               torch.empty(N, device="cuda", dtype=torch.uint8), torch.empty(N, **dev))
        act = torch.tensor(I.commands(9, 1, N, sim.n_thr)[0], device="cuda")
        env = lambda: call("mg_env_step", sim._h, T, _ptr(act), *map(_ptr, out))  # noqa: E731
        env()  # the schedule's buffer is allocated by the first call

        def step():
            env()
            return out[0]
        return step
    traj, ckpt = torch.empty((T, MG_NTRAJ, N), **dev), torch.empty((-(-T // C), MG_NSTATE, N), **dev)
    step0 = ctypes.c_int64()
    g = torch.randn((T, MG_NTRAJ, N), generator=torch.Generator("cuda").manual_seed(3), **dev)
    dc, ds = torch.empty((N, 18), **dev), torch.empty((N, MG_NSTATE), **dev)
    da = torch.zeros((-(-T // HOLD), N, sim.act_w), **dev)

    def rollout():
        call("mg_rollout_forward", sim._h, T, C, _ptr(traj), _ptr(ckpt), ctypes.byref(step0))
        da.zero_()
        call("mg_rollout_backward", sim._h, T, C, _ptr(ckpt), _ptr(g), 0, _ptr(dc), _ptr(da),
             _ptr(ds))
        return torch.cat([dc.reshape(-1), da.reshape(-1), ds.reshape(-1), traj.reshape(-1)])
    rollout()
    return rollout


WAYS = ["step", "chunks", "queue", "noalloc", "record", "task", "env", "rollout"]


@pytest.mark.parametrize("kind", ["six", "mixed"])
@pytest.mark.parametrize("how", WAYS)
def test_captured_step_follows_buoyancy_off_the_axis(how, kind):
    """Captured while every r_b lies on the z axis (where the kernels of mirrored frames may leave
    the moments of G_x and G_y out); replayed with r_b off the axis, and on it again."""
    vs = vehicles()
    types = np.zeros(N, np.int32) if kind == "six" else I.mixed_fleet(4, N, max_group=60)
    nt = np.array([vs[t].n_thr for t in types])
    on = I.perturbed_params(5, oracle_nominal(vs)[types], N)
    off = on.copy()
    off[:, I.P_RB] = I.round_f32(np.random.default_rng(1).uniform(-0.02, 0.02, N))
    off[::3, I.P_RB + 1] = 0.015625
    states = I.random_states(6, N, nt)
    cmds = I.commands(7, -(-T // HOLD), N, nt)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        dev = lambda x: torch.tensor(x, dtype=torch.float32, device="cuda")  # noqa: E731
        acts, start = dev(cmds), dev(states)
        sims, fns = [], []
        for _ in range(2):
            sim = Sim(N, types, vs, stream=s)
            sim.set_launch(64, 50, False)
            sim.set_params(dev(on))
            sim.set_actions(acts, HOLD)
            fns.append(_advance(sim, how))
            sims.append(sim)
        for sim in sims:
            sim.set_actions(acts, HOLD)
        out = []
        g = _capture(s, lambda: out.append(fns[0]()))
        for params in (on, off, on):
            for sim in sims:
                sim.set_params(dev(params))
                sim.set_state(start)
                if how != "env":
                    sim.set_actions(acts, HOLD)
            g.replay()
            direct = fns[1]()
            torch.cuda.synchronize()
            assert torch.equal(sims[0].get_state(), sims[1].get_state())
            if direct is not None:
                assert torch.equal(out[0], direct)
            if how == "step":
                ref = O.rollout(params, oracle_geo(vs), types, states, cmds.astype(np.float64),
                                HOLD, T, h=0.01)
                got = sims[0].get_state().double().cpu().numpy()
                assert rel_err(got, ref).max() <= TOL_STEP * T
        for sim in sims:
            sim.close()


@pytest.mark.parametrize("also_step", [False, True])
def test_captured_draw_writes_the_parameters_in_use(also_step):
    """randomize(wait=False) and reset() in a user's graph; prefetched draws installed outside it
    before and after; each replay redraws what the next step reads."""
    vs = vehicles()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        a, b = (Sim(N, np.zeros(N, np.int32), vs, stream=s) for _ in range(2))
        for sim in (a, b):
            sim.randomize(1)
            sim.set_procedural_actions(7, HOLD)

        def draw(sim):
            sim.randomize(5, wait=False)
            sim.reset()
            if also_step:
                sim.step(3)
        g = _capture(s, lambda: draw(a))
        for ep in range(4):
            a.randomize_prefetch(50 + ep)
            for sim in (a, b):
                sim.randomize(50 + ep, wait=False)
                sim.reset()
                sim.step(11)
            assert torch.equal(a.get_params(), b.get_params()), ep
            assert torch.equal(a.get_state(), b.get_state()), ep
            if ep % 2:
                a.randomize_prefetch(70 + ep)  # drawn beside the replay, installed later
            g.replay()
            draw(b)
            for sim in (a, b):
                sim.step(9)
            assert torch.equal(a.get_params(), b.get_params()), ep
            assert torch.equal(a.get_state(), b.get_state()), ep
            if ep % 2:
                for sim in (a, b):
                    sim.randomize(70 + ep, wait=False)
                assert torch.equal(a.get_params(), b.get_params()), ep
        a.close()
        b.close()


def test_parameters_off_the_axis_stay_in_use_until_a_captured_draw_is_replayed():
    vs = vehicles()
    off = I.perturbed_params(5, oracle_nominal(vs)[np.zeros(N, int)], N)
    off[:, I.P_RB] = 0.015625
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        a, b = (Sim(N, np.zeros(N, np.int32), vs, stream=s) for _ in range(2))
        for sim in (a, b):
            sim.set_procedural_actions(7, HOLD)
            sim.set_params(torch.tensor(off, dtype=torch.float32, device="cuda"))
        g = _capture(s, lambda: a.randomize(5, wait=False))
        for sim in (a, b):
            sim.step(T)
        assert torch.equal(a.get_state(), b.get_state())
        g.replay()
        b.randomize(5, wait=False)
        for sim in (a, b):
            sim.step(T)
        assert torch.equal(a.get_state(), b.get_state())
        a.close()
        b.close()
