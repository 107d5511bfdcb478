"""The bounded wait of the tile kernel with the first copy withheld: asked for by name, and from a handle that
steps with the row sweep, which has no such wait and goes over to the tile kernel's first shape.  The wait runs out
after about a second, as the hook's description has it (limit: five; the two-step kernel waits twice)."""
import time

import pytest

from paper_1805_00007_gb300 import abi
from paper_1805_00007_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _withhold(sim):
    abi.lb_ch_test_hook(sim.h, abi.LBCH_HOOK_SKIP_FIRST_LOAD, 1)
    kernel = sim.kernel()
    t = time.monotonic()
    sim.step(2)
    with pytest.raises(abi.LbchError) as ei:
        sim.observe(abi.LBCH_OBS_MASS)
    assert ei.value.status == abi.LBCH_ETIMEOUT and time.monotonic() - t < 5.0
    return kernel["form"], kernel["shape"]


@pytest.mark.parametrize("prec,shape,tau,form", [("f32", 3, 1.0, "tile_tau1"), ("f64", 4, 0.8, "tile")])
def test_tile_kernel_by_name(prec, shape, tau, form):
    p, phi0, _ = wl.zalesak(n=64, tau=tau)
    with abi.Simulation(p, phi0, prec=prec) as sim:
        abi.lb_ch_test_hook(sim.h, abi.LBCH_HOOK_TILE_KERNEL, 1)
        abi.lb_ch_test_hook(sim.h, abi.LBCH_HOOK_TILE_SHAPE, shape)
        assert _withhold(sim) == (form, shape)


@pytest.mark.parametrize("prec,tau,form", [("f32", 1.0, "tile_tau1"), ("f64", 0.8, "tile")])
def test_from_the_row_sweep(prec, tau, form):
    p, phi0, _ = wl.zalesak(n=64, tau=tau)
    with abi.Simulation(p, phi0, prec=prec) as sim:
        abi.lb_ch_test_hook(sim.h, abi.LBCH_HOOK_TILE_KERNEL, 0)
        abi.lb_ch_test_hook(sim.h, abi.LBCH_HOOK_TILE_SHAPE, 2)
        assert sim.kernel()["form"].startswith("sweep") and sim.kernel()["shape"] == 2
        assert _withhold(sim) == (form, 0)


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_two_step_kernel(prec):
    p, phi0, _ = wl.zalesak(n=64)
    with abi.Simulation(p, phi0, prec=prec) as sim:
        abi.lb_ch_test_hook(sim.h, abi.LBCH_HOOK_TWO_STEP, 1)
        assert _withhold(sim)[0] == "pair_tau1"
