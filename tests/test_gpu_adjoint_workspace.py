"""The backward pass's workspace: none is needed to capture the default form, what a user's graph
uses outlives a larger one, and it can be given back."""
import ctypes

import numpy as np
import pytest
import torch

from _helpers import vehicles
from paper_2410_14117_gb300 import inputs as I
from paper_2410_14117_gb300._lib import MG_NSTATE, MG_NTRAJ, MGError, call
from paper_2410_14117_gb300.sim import Sim, _ptr

pytestmark = pytest.mark.gpu

T = 12


class _Case:
    """A sim with one recorded rollout and the buffers of its backward pass."""

    def __init__(self, n, general, stream=None):
        vs = vehicles()
        dev = dict(device="cuda", dtype=torch.float32)
        self.sim = sim = Sim(n, np.zeros(n, np.int32), vs, stream=stream)
        sim.randomize(5, rg_halfwidth=0.02 if general else 0.0)
        sim.reset()
        sim.set_actions(torch.tensor(I.commands(7, 2, n, 6), device="cuda"), 6)
        traj = torch.empty((T, MG_NTRAJ, n), **dev)
        self.ckpt = {c: torch.empty((-(-T // c), MG_NSTATE, n), **dev) for c in (3, 12)}
        step0 = ctypes.c_int64()
        start = sim.get_state()
        for c, ck in self.ckpt.items():
            sim.set_state(start)
            sim.set_actions(torch.tensor(I.commands(7, 2, n, 6), device="cuda"), 6)
            call("mg_rollout_forward", sim._h, T, c, _ptr(traj), _ptr(ck), ctypes.byref(step0))
        self.g = torch.randn((T, MG_NTRAJ, n), generator=torch.Generator("cuda").manual_seed(3),
                             **dev)
        self.out = [torch.empty((n, 18), **dev), torch.zeros((2, n, 8), **dev),
                    torch.empty((n, MG_NSTATE), **dev)]

    def backward(self, c):
        self.out[1].zero_()
        call("mg_rollout_backward", self.sim._h, T, c, _ptr(self.ckpt[c]), _ptr(self.g), 0,
             *map(_ptr, self.out))

    def result(self):
        torch.cuda.synchronize()
        return [x.clone() for x in self.out]


# fleets that the default runs with two warps per 32 envs, and with one thread per env
@pytest.mark.parametrize("n,general", [(97, False), (12000, False), (12000, True), (30000, True),
                                       (30000, False)])
def test_first_backward_can_be_captured(n, general):
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        case = _Case(n, general, s)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
            case.backward(3)
        g.replay()
        got = case.result()
        case.backward(3)
        assert all(torch.equal(x, y) for x, y in zip(got, case.result()))
        case.sim.close()


def test_two_warp_form_asked_for_needs_its_workspace_before_a_capture():
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        case = _Case(97, False, s)
        case.sim.set_adjoint_mode(2)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
            case.sim.step(1)
            with pytest.raises(MGError) as e:
                case.backward(3)
        assert e.value.code == "MG_ENOMEM"
        g.replay()  # the refused call left the capture as it was
        case.backward(3)
        case.sim.close()


def test_graph_keeps_its_workspace_when_a_larger_one_is_allocated():
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        case = _Case(4096, False, s)
        case.backward(3)
        want = case.result()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
            case.backward(3)
        case.backward(12)  # four times the records
        case.sim.set_adjoint_mode(1)
        free = torch.cuda.mem_get_info()[0]
        for _ in range(3):
            fill = torch.full((1 << 22,), -1.0, device="cuda")  # would land in freed memory
            g.replay()
            assert all(torch.equal(x, y) for x, y in zip(want, case.result()))
            del fill
        assert torch.cuda.mem_get_info()[0] <= free
        case.sim.close()


def test_workspace_is_given_back():
    case = _Case(16384, False)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    case.backward(12)
    want = case.result()
    held = before - torch.cuda.mem_get_info()[0]
    assert held >= 2 * 12 * 100 * 4 * 16384
    case.sim.set_adjoint_mode(1)
    assert before - torch.cuda.mem_get_info()[0] <= held - 2 * 12 * 100 * 4 * 16384
    case.sim.set_adjoint_mode(0)
    case.backward(12)
    assert all(torch.equal(x, y) for x, y in zip(want, case.result()))
    case.sim.close()


@pytest.mark.parametrize("general", [False, True])
def test_default_holds_a_workspace_only_while_every_block_is_resident(general):
    line = 32 * 4 * torch.cuda.get_device_properties(0).multi_processor_count
    for n, held in ((line, True), (line + 1, False)):
        case = _Case(n, general)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        case.backward(12)
        torch.cuda.synchronize()
        assert (before - torch.cuda.mem_get_info()[0] >= 2 * 12 * 100 * 4 * n) == held
        case.sim.close()
