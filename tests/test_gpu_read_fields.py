"""Reading phi, u and p: every value of every instance, in one piece and in several (a float handle converts as many rows at a
time as its next state's buffer holds), against the device's own copy of phi; a non-finite value anywhere is reported; and a
read leaves the run that follows as it is, although it uses the next state's buffer (the same bits as a run without)."""
import numpy as np
import pytest
import torch

from paper_1805_00007_gb300 import abi
from paper_1805_00007_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _setup(nx, ny, tau=1.0, **kw):
    p = wl.make_params(nx=nx, ny=ny, tau=tau, vel=wl.VEL_UNIFORM, ux0=0.03, uy0=-0.02, M=0.01, **kw)
    return p, wl.random_smooth_phi(nx, ny, seed=nx + ny)


@pytest.mark.parametrize("prec", ["f64", "f32", "f16s"])
@pytest.mark.parametrize("nx,ny", [(4, 4), (5, 260), (255, 3 * 64 + 1), (1030, 17)])
def test_phi_equals_the_device_copy(nx, ny, prec):
    p, phi0 = _setup(nx, ny)
    with abi.Simulation(p, phi0, prec=prec) as sim:
        sim.step(3)
        dev = torch.empty((ny, nx), dtype=torch.float64, device="cuda")
        if prec == "f64":
            abi.lb_ch_tape_phi(sim.h, dev.data_ptr())
            torch.cuda.synchronize()
        got = sim.phi()
        assert got.shape == (ny, nx) and np.isfinite(got).all()
        if prec == "f64":
            assert np.array_equal(got, dev.cpu().numpy())
        assert abs(got.sum() - sim.observe(abi.LBCH_OBS_MASS)) <= 1e-12 * np.abs(got).sum()
        assert got.max() == sim.observe(abi.LBCH_OBS_MAX) and got.min() == sim.observe(abi.LBCH_OBS_MIN)


@pytest.mark.parametrize("prec", ["f64", "f32", "f16s"])
@pytest.mark.parametrize("tau,steps", [(1.0, 1), (1.0, 6), (0.8, 3)])
def test_reading_leaves_the_run_as_it_is(prec, tau, steps):
    setups = [_setup(nx, ny, tau) for nx, ny in ((37, 20), (64, 33), (5, 9))]
    ps, fs = [s[0] for s in setups], [s[1] for s in setups]
    with abi.Simulation(ps, fs, prec=prec) as a, abi.Simulation(ps, fs, prec=prec) as b:
        for _ in range(3):
            a.step(steps)
            b.step(steps)
            for i in range(3):
                a.phi(i)
            a.observe_all(abi.LBCH_OBS_MASS)
        for i in range(3):
            assert np.array_equal(a.phi(i), b.phi(i))


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_reading_the_coupled_fields_leaves_the_run_as_it_is(prec):
    p, phi0 = wl.rayleigh_taylor(nx=33, ny=50, Re=300.0)
    with abi.Simulation(p, phi0, prec=prec) as a, abi.Simulation(p, phi0, prec=prec) as b:
        for _ in range(3):
            a.step(5)
            b.step(5)
            a.velocity(), a.pressure(), a.phi()
        assert np.array_equal(a.phi(), b.phi()) and np.array_equal(a.pressure(), b.pressure())
        assert np.array_equal(a.velocity(), b.velocity())


@pytest.mark.parametrize("prec", ["f64", "f32", "f16s"])
def test_a_value_that_is_not_finite_is_reported(prec):
    p, phi0 = _setup(70, 65)
    phi0[64, 69] = 1e300 if prec == "f64" else 1e38  # its chemical potential overflows in the first step
    with abi.Simulation(p, phi0, prec=prec) as sim:
        sim.step(2)
        with pytest.raises(abi.LbchError) as err:
            sim.phi()
        assert err.value.status == abi.LBCH_ENONFINITE
