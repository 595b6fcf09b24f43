"""The action cursor's rewind travels with the next step launch: every call that follows a schedule
change, in any order, and a user's own CUDA graph replayed around them, must see the cursor that an
immediate rewind gives."""
import numpy as np
import pytest
import torch

from paper_2410_14117_gb300 import inputs as I
from paper_2410_14117_gb300.sim import Sim

pytestmark = pytest.mark.gpu

N = 200


def _sim(stream=None, spl=50, queue=False):
    sim = Sim(N, np.zeros(N, np.int32), I.fleet_vehicles(), stream=stream)
    sim.set_launch(64, spl, False)
    sim.set_schedule(queue, True)
    sim.randomize(3, 0.8, 1.2, 0.2, 0.3)
    sim.reset()
    return sim


def _acts(seed):
    return torch.tensor(I.commands(seed, 12, N, 6), device="cuda")


# after the rewind: direct launch, two launches, recorded, split, task step, queue
AFTER = ["direct", "chunks", "record", "split", "task", "noalloc"]


def _advance(sim, how):
    if how == "direct":
        sim.step(7)
    elif how == "chunks":
        sim.step(60)
    elif how == "record":
        sim.step_record(7)
    elif how == "split":
        sim.step_split(1, torch.zeros((6, N), device="cuda"))
    elif how == "task":
        sim.set_task(0, torch.zeros((N, 4), device="cuda"))
        sim.task_step(7)
    else:
        from paper_2410_14117_gb300._lib import call
        call("mg_step_noalloc", sim._h, 7)


@pytest.mark.parametrize("how", AFTER)
@pytest.mark.parametrize("queue", [False, True])
def test_rewind_reaches_every_kind_of_step(how, queue):
    """Schedule, some sub-steps, the schedule again (a rewind), then `how` and a direct step: as
    on a fresh sim from the same state whose cursor never moved."""
    a, fresh = _sim(queue=queue), _sim(queue=queue)
    acts = _acts(1)
    a.set_actions(acts, 5)
    a.step(13)
    fresh.set_state(a.get_state())
    a.set_actions(acts, 5)
    fresh.set_actions(acts, 5)
    for sim in (a, fresh):
        _advance(sim, how)
        sim.step(9)
    assert torch.equal(a.get_state(), fresh.get_state())
    a.close()
    fresh.close()


@pytest.mark.parametrize("schedule_inside", [False, True])
@pytest.mark.parametrize("step_before_replay", [False, True])
@pytest.mark.parametrize("k", [5, 60])  # one launch; two
def test_captured_steps_replay_around_rewinds(k, schedule_inside, step_before_replay):
    """A graph of step(k) (with or without the schedule call inside) replayed between schedule
    changes, against the same calls made directly."""
    s = torch.cuda.Stream()
    acts, other = _acts(1), _acts(2)
    with torch.cuda.stream(s):
        a, b = _sim(s), _sim(s)
        b_step = lambda: ([b.set_procedural_actions(7, 5)] if schedule_inside else None,  # noqa: E731
                          b.step(k))
        for sim in (a, b):
            sim.set_actions(acts, 5)
            sim.step(4)
            sim.set_actions(acts, 5)  # a rewind is pending here
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
            if schedule_inside:
                a.set_procedural_actions(7, 5)
            a.step(k)
        if step_before_replay and not schedule_inside:
            a.step(3)
            b.step(3)
        for _ in range(3):
            g.replay()
            b_step()
        if not schedule_inside:
            for x in (other, acts):
                a.set_actions(x, 5)  # copied into the buffer the graph reads
                b.set_actions(x, 5)
                for _ in range(2):
                    g.replay()
                    b_step()
            a.step(2)
            b.step(2)
        torch.cuda.synchronize()
        assert torch.equal(a.get_state(), b.get_state())
        a.close()
        b.close()


def test_exchanged_parameters_around_a_captured_step():
    """Prefetched draws installed before and after step(5) is captured into a user's graph, whose
    replays must see each installed draw; an unmatched draw in between; graph-cached long steps."""
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        a, b = _sim(s), _sim(s)
        for sim in (a, b):
            sim.set_launch(64, 20, True)  # step(45) replays a cached graph
            sim.set_procedural_actions(7, 5)
        g = None
        for ep in range(6):
            for sim in (a, b):
                if ep != 3:
                    if sim is a:
                        sim.randomize_prefetch(50 + ep)
                    sim.randomize(50 + ep, nu0_sigma=0.3, wait=False)
                else:  # a draw for another seed stays in the buffer
                    if sim is a:
                        sim.randomize_prefetch(99)
                    sim.randomize(7, nu0_sigma=0.3)
                sim.reset()
                sim.step(45)
            if ep == 2:
                torch.cuda.synchronize()
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
                    a.step(5)
            if g is not None:
                g.replay()
                b.step(5)
            assert torch.equal(a.get_params(), b.get_params())
            assert torch.equal(a.get_state(), b.get_state()), ep
        a.close()
        b.close()
