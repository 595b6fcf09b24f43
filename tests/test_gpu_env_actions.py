"""The environment step's throttles, clamped inside its one launch: any 4-byte alignment of the
policy's buffer, both row widths, ragged fleets, and the schedule they leave behind."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2410_14117_gb300 import inputs as I
from paper_2410_14117_gb300._lib import call
from paper_2410_14117_gb300.sim import Sim

pytestmark = pytest.mark.gpu


def _sim(n, types, w):
    sim = Sim(n, types, I.fleet_vehicles())
    sim.set_launch(64, 20, True)
    sim.set_action_width(w)
    sim.randomize(3, 0.8, 1.2, 0.2, 0.3)
    sim.reset()
    sim.set_task(1, torch.zeros((n, 4), device="cuda"), lookahead=2, max_error=3.0,
                 episode_steps=15)
    return sim


@pytest.mark.parametrize("k", [1, 10, 20, 45])  # up to 20: one launch; 45: 40 sub-steps ahead of it
@pytest.mark.parametrize("n,w,kind", [(1, 6, 0), (33, 6, 0), (257, 8, 0), (700, 8, 1), (500, 8, 2)])
@pytest.mark.parametrize("off", [0, 1, 2])
def test_env_step_clamps_like_a_clamped_schedule(n, w, kind, off, k):
    types = I.mixed_fleet(8, n, max_group=90) if kind == 2 else np.full(n, kind, np.int32)
    a, b = _sim(n, types, w), _sim(n, types, w)
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    obs = torch.empty((n, a.obs_dim), device="cuda")
    rew, ep = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
    done = torch.empty(n, dtype=torch.uint8, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(5)
    buf = torch.empty(n * w + off, device="cuda")
    act = torch.zeros((1, n, w), device="cuda")
    for step in range(2):
        buf.copy_(torch.rand(n * w + off, generator=g, device="cuda") * 3 - 1.5)
        x = buf[off:]
        call("mg_env_step", a._h, k, p(x), p(obs), p(rew), p(done), p(ep))
        act[0] = x.view(n, w).clamp(-1, 1)
        b.set_actions_borrowed(act, 1 << 30)
        o2, e2, d2, ep2 = b.task_step(k)
        assert torch.equal(obs, o2) and torch.equal(rew, -e2)
        assert torch.equal(done, d2) and torch.equal(ep, ep2)
    a.step(7)  # the schedule the last step left
    b.step(7)
    assert torch.equal(a.get_state(), b.get_state())
    a.close()
    b.close()
