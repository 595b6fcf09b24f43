"""The throttle lag's rounding error, against RK4 on n' = (c - n) / tau_m in 64 bits."""
import numpy as np
import pytest
import torch

from _helpers import vehicles
from paper_2410_14117_gb300 import inputs as I
from paper_2410_14117_gb300.sim import Sim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("which,steps,hold", [(0, 1, 1), (0, 20, 1), (1, 20, 1), (0, 200, 10)])
def test_lag_error_is_the_rounding_of_the_state(which, steps, hold, general):
    """Each sub-step rounds n once, a relative 3e-8 (2-norm) that the next ones damp by P = 1 + z +
    ... = 0.82 (tau_m = 0.05 s, h = 0.01 s): 3e-8 / sqrt(1 - P^2) = 5.3e-8.  The rounding of n - c
    and of the factor of it, 3e-8 each, is weighted by 1 - P = 0.18 and damped the same way: 1e-8
    each.  Together 5.5e-8; 8e-8 leaves half of that for the ranges of tau_m and c."""
    vs = vehicles()
    n, nt = 4096, vs[which].n_thr
    sim = Sim(n, np.full(n, which, np.int32), vs)
    sim.randomize(5, 0.8, 1.2, 0.2, 0.3, rg_halfwidth=0.02 if general else 0.0)
    tau = sim.get_params()[:, I.P_TAU].double().cpu().numpy()[:, None]
    states = I.random_states(6, n, np.full(n, nt)).astype(np.float32)
    cmds = I.commands(7, -(-steps // hold), n, nt)
    sim.set_state(torch.tensor(states, device="cuda"))
    sim.set_actions(torch.tensor(cmds, device="cuda"), hold)
    sim.step(steps)
    got = sim.get_state()[:, 13:13 + nt].double().cpu().numpy()
    sim.close()
    z = -float(np.float32(0.01)) / tau
    p = 1 + z * (1 + z / 2 * (1 + z / 3 * (1 + z / 4)))
    ref = states[:, 13:13 + nt].astype(np.float64)
    for k in range(steps):
        c = cmds[k // hold, :, :nt].astype(np.float64)
        ref = c + p * (ref - c)
    assert np.linalg.norm(got - ref) <= 8e-8 * np.linalg.norm(ref)
