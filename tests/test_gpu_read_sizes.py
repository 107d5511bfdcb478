"""Reading phi on both sides of the sizes at which it is staged in pinned memory, copied in one piece and in several: every
value at its place, in every precision, against the device's own copy (in the tape's type, float for the float states), and
the same values from an ensemble's instances.  Values are compared exactly: both come from the same stored numbers."""
import numpy as np
import pytest
import torch

from paper_1805_00007_gb300 import abi
from paper_1805_00007_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SIZES = [(4, 4), (64, 128), (91, 91), (8192, 4), (5, 1639), (128, 256), (181, 182), (32768, 4), (1030, 17), (700, 301)]


def _setup(nx, ny):
    p = wl.make_params(nx=nx, ny=ny, vel=wl.VEL_UNIFORM, ux0=0.03, uy0=-0.02, M=0.01)
    return p, wl.random_smooth_phi(nx, ny, seed=nx + ny)


@pytest.mark.parametrize("prec", ["f64", "f32", "f16s"])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_every_value_at_its_place(nx, ny, prec):
    p, phi0 = _setup(nx, ny)
    with abi.Simulation(p, phi0, prec=prec) as sim:
        sim.step(3)
        dev = torch.empty((ny, nx), dtype=torch.float64 if prec == "f64" else torch.float32, device="cuda")
        abi.lb_ch_tape_phi(sim.h, dev.data_ptr())
        torch.cuda.synchronize()
        assert np.array_equal(sim.phi().astype(np.float64 if prec == "f64" else np.float32), dev.cpu().numpy())


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_instances_of_an_ensemble(prec):
    setups = [_setup(nx, ny) for nx, ny in ((4, 4), (91, 91), (181, 182), (64, 128))]
    with abi.Simulation([s[0] for s in setups], [s[1] for s in setups], prec=prec) as sim:
        sim.step(3)
        for i, s in enumerate(setups):
            with abi.Simulation(*s, prec=prec) as one:
                one.step(3)
                assert np.array_equal(sim.phi(i), one.phi())


@pytest.mark.parametrize("nx,ny", [(64, 128), (91, 91), (181, 182)])
def test_a_value_that_is_not_finite_is_reported(nx, ny):
    p, phi0 = _setup(nx, ny)
    phi0[ny - 1, nx - 1] = 1e38
    with abi.Simulation(p, phi0, prec="f32") as sim:
        sim.step(2)
        with pytest.raises(abi.LbchError) as err:
            sim.phi()
        assert err.value.status == abi.LBCH_ENONFINITE
