"""The domain randomisation in two-float arithmetic against the FP64 oracle over its ranges, and the
parameter records through every alignment and ragged tail."""
import numpy as np
import pytest
import torch

from _helpers import TOL_STEP, f32, oracle_geo, oracle_nominal, rel_err, vehicles
from oracle import oracle as O
from paper_2410_14117_gb300 import inputs as I
from paper_2410_14117_gb300.sim import MGError, Sim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,lo,hi,sigma", [
    (1, 0.8, 1.2, 0.2), (127, 1.0, 1.0, 0.0), (129, 0.003, 7.5, 5.0), (20011, 0.8, 1.2, 0.2),
    (4096, 1e-3, 1e3, 1e-4)])
@pytest.mark.parametrize("background", [False, True])
def test_draws_are_the_fp64_values_rounded_once(n, lo, hi, sigma, background):
    vs = vehicles()
    types = I.mixed_fleet(3, n, max_group=max(1, n // 7))
    sim = Sim(n, types, vs)
    if background:
        sim.randomize_prefetch(77, lo, hi, sigma)
    sim.randomize(77, lo, hi, sigma, 0.3)
    got = sim.get_params().double().cpu().numpy()
    sim.close()
    ref = O.randomize(77, oracle_nominal(vs), types, f32(lo), f32(hi), f32(sigma))
    # half an FP32 ulp of the FP64 value; the two-float value is within 2^-35 of it before it is
    # rounded (2^-24 is half an ulp relative to the smallest mantissa)
    np.testing.assert_allclose(got, ref, rtol=2.0 ** -24 + 2.0 ** -34, atol=1e-30)


@pytest.mark.parametrize("lo,hi,sigma", [(0.8, 1.2, 0.2), (0.003, 7.5, 5.0), (1e-3, 1e3, 1e-4),
                                         (1.0, 1.0, 0.0)])
@pytest.mark.parametrize("background", [False, True])
@pytest.mark.parametrize("extreme", [False, True])
def test_draws_round_as_fp64_does(lo, hi, sigma, background, extreme):
    """Every stored value is the one FP64 arithmetic stores: a two-float value whose rounding its
    error leaves open is drawn again in FP64, and so is every value where a vehicle's are too small
    for two floats to hold."""
    vs = vehicles()
    n = 5003 if extreme else 100003
    if extreme:
        vs[0].params[I.P_DL:I.P_DL + 2] = 1e-33, 0.0
    types = I.mixed_fleet(3, n, max_group=9000)
    sim = Sim(n, types, vs)
    if background:
        sim.randomize_prefetch(78, lo, hi, sigma)
    sim.randomize(78, lo, hi, sigma, 0.3)
    got = sim.get_params().cpu().numpy()
    sim.close()
    ref = O.randomize(78, oracle_nominal(vs), types, f32(lo), f32(hi), f32(sigma))
    np.testing.assert_array_equal(got, ref.astype(np.float32))


@pytest.mark.parametrize("n", [1, 33, 128, 257, 1000])
@pytest.mark.parametrize("off", [0, 1, 2])
def test_records_round_trip_any_alignment(n, off):
    vs = vehicles()
    sim = Sim(n, np.zeros(n, np.int32), vs)
    p = np.ascontiguousarray(I.perturbed_params(5, oracle_nominal(vs)[np.zeros(n, int)], n))
    buf = torch.zeros(n * I.NPARAM + off + 1, device="cuda")
    rec = buf[off:off + n * I.NPARAM].view(n, I.NPARAM)
    rec.copy_(torch.tensor(p, dtype=torch.float32))
    sim.set_params(rec)
    out = torch.full_like(buf, -1.0)
    sim.get_params(out[off:off + n * I.NPARAM].view(n, I.NPARAM))
    assert torch.equal(out[off:off + n * I.NPARAM], buf[off:off + n * I.NPARAM])
    assert (out[:off] == -1).all() and out[-1] == -1
    sim.close()


def test_not_spd_records_are_seen():
    vs = vehicles()
    n = 300
    p = np.ascontiguousarray(I.perturbed_params(5, oracle_nominal(vs)[np.zeros(n, int)], n))
    p[17, I.P_MA + 2] = -p[17, I.P_M]  # M_33 = 0
    sim = Sim(n, np.zeros(n, np.int32), vs)
    with pytest.raises(MGError) as e:
        sim.set_params(torch.tensor(p, dtype=torch.float32, device="cuda"))
    assert e.value.code == "MG_ENOTSPD"
    assert np.array_equal(sim.get_params().double().cpu().numpy(), p)
    sim.close()


@pytest.mark.parametrize("back", ["set_params", "randomize", "randomize async", "prefetch"])
@pytest.mark.parametrize("axis", [0, 1])
def test_off_axis_records_are_seen_and_forgotten(axis, back):
    """One env's r_b off the z axis: the step keeps its moments (the oracle's step); with r_b back on
    the axis, by every way there, the steps are those of a sim that never left it."""
    vs = vehicles()
    n = 300
    types = I.mixed_fleet(4, n, max_group=60)
    nt = np.array([vs[t].n_thr for t in types])
    on = I.perturbed_params(5, oracle_nominal(vs)[types], n)
    off = on.copy()
    off[n - 1, I.P_RB + axis] = 0.03125
    states, cmds = I.random_states(6, n, nt), I.commands(7, 1, n, nt)
    dev = lambda x: torch.tensor(x, dtype=torch.float32, device="cuda")  # noqa: E731

    def step(sim):
        sim.set_state(dev(states))
        sim.set_actions(dev(cmds), 10)
        sim.step(5)
        return sim.get_state()

    def on_axis(sim):
        if back == "set_params":
            sim.set_params(dev(on))
        else:
            if back == "prefetch":
                sim.randomize_prefetch(9)
            sim.randomize(9, wait=back != "randomize async")
    sim, fresh = Sim(n, types, vs), Sim(n, types, vs)
    for params in (off, off):
        sim.set_params(dev(params))
        ref = O.rollout(params, oracle_geo(vs), types, states, cmds.astype(np.float64), 10, 5, h=0.01)
        assert rel_err(step(sim).double().cpu().numpy(), ref).max() <= 5 * TOL_STEP
        on_axis(sim)
        on_axis(fresh)
        assert torch.equal(step(sim), step(fresh))
        assert sim.kernel_info() == fresh.kernel_info()
    sim.close()
    fresh.close()
