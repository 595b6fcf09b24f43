"""Thruster allocations of the diagonal-mass step (dense, vectored, mirrored frame) against the
FP64 oracle: vehicles on each side of every condition that picks one, one sub-step from random
states and a rollout, with the same bits from every kernel that steps them."""
import copy

import numpy as np
import pytest
import torch

from _helpers import TOL_ROLLOUT, TOL_STEP, oracle_nominal, rel_err, vehicles
from oracle import oracle as O
from paper_2410_14117_gb300 import inputs as I
from paper_2410_14117_gb300.adjoint import rollout
from test_gpu_parity import H, gpu_state, make_sim, oracle_types_geo

pytestmark = pytest.mark.gpu


def _swapped(v, i, j):  # the same vehicle, two thrusters numbered the other way round
    w = copy.deepcopy(v)
    w.r[[i, j]], w.d[[i, j]] = v.r[[j, i]], v.d[[j, i]]
    return w


def _moved(v, i, axis, by, what="r"):
    w = copy.deepcopy(v)
    getattr(w, what)[i, axis] += by
    return w


def _without(v, n):  # the vehicle's first n thrusters
    w = copy.deepcopy(v)
    w.n_thr = n
    w.r[n:], w.d[n:] = 0.0, 0.0
    return w


def _rb(v, x):  # centre of buoyancy off the z axis
    w = copy.deepcopy(v)
    w.params[I.P_RB] = x
    return w


ROV, HEAVY = vehicles()
FLEETS = {
    "six": ([ROV], 0), "eight": ([HEAVY], 0), "both": ([ROV, HEAVY], None),
    "literal frame": (vehicles("literal"), None),
    "swapped horizontals": ([_swapped(ROV, 0, 1), HEAVY], None),
    "swapped verticals": ([_swapped(HEAVY, 5, 6)], 0),
    "one arm longer": ([_moved(ROV, 4, 1, 0.05)], 0),
    "verticals ahead": ([_moved(_moved(ROV, 4, 0, 0.1), 5, 0, 0.1)], 0),
    "tilted horizontal": ([_moved(ROV, 2, 2, 0.3, "d")], 0),
    "four thrusters": ([_without(ROV, 4)], 0), "seven": ([_without(HEAVY, 7), ROV], None),
    "type off axis": ([_rb(ROV, 0.01), HEAVY], None),
    "record off axis": ([ROV, HEAVY], None),
}


@pytest.mark.parametrize("general", [False, True])  # True: off-centre gravity, full mass matrices
@pytest.mark.parametrize("name", FLEETS)
def test_allocation_matches_oracle_on_every_kernel(name, general):
    vs, only = FLEETS[name]
    n = 700
    types = np.full(n, 0, np.int32) if only == 0 else I.mixed_fleet(4, n, max_group=90)
    nt = np.array([vs[t].n_thr for t in types])
    params = I.perturbed_params(5, oracle_nominal(vs)[types], n)
    if name == "record off axis":
        params[n // 2, I.P_RB + 1] = 0.0078125
    if general:
        params[:, I.P_RG:I.P_RG + 3] = I.round_f32(
            np.random.default_rng(2).uniform(-0.02, 0.02, (n, 3)))
    states = I.random_states(6, n, nt)
    cmds = I.commands(7, 4, n, nt).astype(np.float64)
    t, geo = oracle_types_geo(types, vs)
    for k, tol in ((1, TOL_STEP), (40, TOL_ROLLOUT)):
        ref = O.rollout(params, geo, t, states, cmds, 10, k, h=H)
        out = []
        for queue, wide, spl in ((False, True, 50), (False, False, 7), (True, True, 9),
                                 (True, False, 50)):
            sim = make_sim(types, vs, epb=64, spl=spl, queue=queue, wide=wide)
            # the path follows the parameters: mirrored (if the types allow it) before this call
            sim.randomize(3, 0.8, 1.2, 0.2, 0.3)
            sim.set_params(torch.tensor(params, dtype=torch.float32, device="cuda"))
            sim.set_state(torch.tensor(states, dtype=torch.float32, device="cuda"))
            sim.set_actions(torch.tensor(cmds, dtype=torch.float32, device="cuda"), 10)
            sim.step(k)
            assert sim.sync() == 0
            out.append(gpu_state(sim))
            sim.close()
        assert rel_err(out[0], ref).max() <= tol
        for o in out[1:]:
            np.testing.assert_array_equal(o, out[0])


def test_recorded_and_rolled_out_states_equal_the_step():
    types = I.mixed_fleet(4, 500, max_group=90)
    got = []
    for record in (False, True):
        sim = make_sim(types, [ROV, HEAVY])
        sim.randomize(3, 0.8, 1.2, 0.2, 0.3)
        sim.reset()
        sim.set_procedural_actions(5, 10)
        sim.step_record(25) if record else sim.step(25)
        got.append(gpu_state(sim))
        sim.close()
    np.testing.assert_array_equal(got[0], got[1])


@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("which", [0, 1])
def test_adjoint_of_renumbered_thrusters(which, mode):
    """The same vehicles with thrusters 0 and 1 numbered the other way round: not a mirrored frame,
    so the dense transposes, whose gradients are the mirrored ones' with the actions permuted.
    Both sides sum the same terms in FP32 over 60 sub-steps: 1e-4 of each env's vector norm."""
    n, T, C = 97, 60, 16
    v = [ROV, HEAVY][which]
    perm = np.array([1, 0, 2, 3, 4, 5, 6, 7])
    types = np.zeros(n, np.int32)
    params = I.perturbed_params(5, oracle_nominal([v])[types], n)
    states = I.random_states(6, n, np.full(n, v.n_thr))
    cmds = I.commands(7, 6, n, v.n_thr)
    g = torch.randn((T, n, 13), generator=torch.Generator().manual_seed(3)).cuda()
    got = []
    for veh, p in ((v, np.arange(8)), (_swapped(v, 0, 1), perm)):
        sim = make_sim(types, [veh], queue=False)
        sim.set_adjoint_mode(mode)
        sim.set_params(torch.tensor(params, dtype=torch.float32, device="cuda"))
        coef = torch.tensor(params[:, 4:22], dtype=torch.float32, device="cuda", requires_grad=True)
        s = states.copy()
        s[:, 13:] = s[:, 13 + p]
        s = torch.tensor(s, dtype=torch.float32, device="cuda", requires_grad=True)
        a = torch.tensor(np.ascontiguousarray(cmds[:, :, p]), device="cuda", requires_grad=True)
        traj = rollout(sim, coef, a, s, 10, T, C)
        dc, da, ds = torch.autograd.grad(traj, (coef, a, s), g)
        ds = torch.cat([ds[:, :13], ds[:, 13 + p]], dim=1)
        got.append([x.double().cpu().numpy() for x in (dc, da[:, :, p].permute(1, 0, 2), ds)])
        sim.close()
    for x, y in zip(*got):
        x, y = x.reshape(n, -1), y.reshape(n, -1)
        err = np.linalg.norm(x - y, axis=1) / np.linalg.norm(y, axis=1)
        assert err.max() <= 1e-4


@pytest.mark.parametrize("kind", [0, 1, "mixed"])
@pytest.mark.parametrize("over", [0, 1])  # blocks past the static grid's register-budget line
def test_static_grid_register_budgets_give_the_same_bits(kind, over):
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    n = 32 * 12 * n_sm + over
    types = np.arange(n, dtype=np.int32) * 2 // n if kind == "mixed" else np.full(n, kind, np.int32)
    states = []
    for wide in (True, False):
        sim = make_sim(types, [ROV, HEAVY])
        sim.set_launch(32, 3, False)
        sim.set_schedule(False, wide)
        sim.randomize(7, 0.8, 1.2, 0.2, 0.3)
        sim.reset()
        sim.set_procedural_actions(11, 2)
        for k in (1, 5):
            sim.step(k)
        states.append(sim.get_state())
        sim.close()
    assert torch.equal(*states)


@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("how", ["static", "queue", "record", "task", "rollout"])
def test_lag_entries_past_the_thrusters_push_nothing(how, general):
    """A state whose throttle entries past a vehicle's thruster count are not zero moves as the same
    state with zeros there: those entries belong to no thruster."""
    n, k = 300, 12
    types = I.mixed_fleet(4, n, max_group=60)
    nt = np.array([(ROV, HEAVY)[t].n_thr for t in types])
    clean = torch.tensor(I.random_states(6, n, nt), dtype=torch.float32, device="cuda")
    dirty = clean.clone()
    dirty[torch.tensor(nt == 6, device="cuda"), 19:] = torch.tensor([0.75, -0.5], device="cuda")
    acts = torch.tensor(I.commands(7, 2, n, nt), device="cuda")
    got = []
    for start in (clean, dirty):
        sim = make_sim(types, [ROV, HEAVY], queue=how == "queue")
        sim.randomize(3, 0.8, 1.2, 0.2, 0.3, rg_halfwidth=0.02 if general else 0.0)
        sim.set_state(start)
        sim.set_actions(acts, 10)
        if how == "record":
            got.append([sim.step_record(k)])
        elif how == "task":
            sim.set_task(0, torch.zeros((n, 4), device="cuda"))
            got.append([sim.task_step(k)[0].clone()])
        elif how == "rollout":
            coef = sim.get_params()[:, 4:22].clone().requires_grad_(True)
            s = start.clone().requires_grad_(True)
            traj = rollout(sim, coef, acts, s, 10, k, 5)
            dc, ds = torch.autograd.grad(traj, (coef, s), torch.ones_like(traj))
            got.append([traj.detach(), dc, ds])
        else:
            sim.step(k)
            got.append([])
        got[-1].append(sim.get_state()[:, :19])
        sim.close()
    for x, y in zip(*got):
        assert torch.equal(x, y)
