"""The kernel that steps a handle until it is tuned: the rule of choose_default from the device's number of SMs, on both
sides of every line, and each choice's bits against the row sweep's (every form gives the same bits at one precision; with
half storage at tau_g = 1 both are the sweep)."""
import numpy as np
import pytest
import torch

from paper_1805_00007_gb300 import abi
from paper_1805_00007_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _tiles(nx, ny, tx, ty):
    return -(-nx // tx) * -(-ny // ty)


def _expected(prec, tau, nx, ny, walls, sms):
    """(form, shape), the shape None for the row sweep."""
    t = lambda tx, ty: _tiles(nx, ny, tx, ty)
    tau1 = tau == 1.0
    sweep = ("sweep_tau1" if tau1 else "sweep", None)
    tile = "tile_tau1" if tau1 else "tile"
    if prec == "f64":
        if t(32, 16) > 12 * sms:
            return sweep
        if t(16, 8) <= sms:
            return tile, 1
        if t(32, 8) <= sms:
            return tile, 2
        return tile, (4 if -(-t(32, 14) // sms) * 149 <= -(-t(32, 16) // sms) * 167 else 3)
    if not tau1:
        if 2 * t(16, 8) <= 5 * sms:
            return tile, 2
        if t(32, 16) <= sms:
            return tile, 3
        if t(32, 8) <= 3 * sms:
            return tile, 1
        return sweep
    if prec == "f16s" or walls:
        return sweep
    if t(16, 8) <= sms:
        return "pair_tau1", 2
    if t(32, 8) <= sms:
        return "pair_tau1", 3
    if t(32, 14) <= 2 * sms:
        return "pair_tau1", 1
    if t(32, 16) <= 2 * sms:
        return "pair_tau1", 0
    if 2 * t(32, 14) <= 5 * sms:
        return "pair_tau1", 1
    return sweep


def _edges(prec, tau, walls, sms):
    """Square grids n x (n + 3): the last before and the first after every change of the choice."""
    n, last, out = 16, None, []
    while n <= 1100:
        now = _expected(prec, tau, n, n + 3, walls, sms)
        if last is not None and now != last:
            out += [n - 1, n]
        last, n = now, n + 1
    return out or [16, 300]


CASES = [(p, t, w) for p in ("f32", "f64", "f16s") for t in (1.0, 0.8) for w in (0, 1)]


@pytest.mark.parametrize("prec,tau,walls", CASES)
def test_default_kernel_is_the_one_of_the_rule_with_the_bits_of_the_row_sweep(prec, tau, walls):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    seen = set()
    for n in _edges(prec, tau, walls, sms):
        p = wl.make_params(nx=n, ny=n + 3, tau=tau, walls=walls, vel=wl.VEL_SHEAR if walls else wl.VEL_UNIFORM, shear=1e-3,
                           ux0=0.03, uy0=-0.02, M=0.02)
        phi0 = wl.random_smooth_phi(n, n + 3, seed=n)
        with abi.Simulation(p, phi0, prec=prec) as sim, abi.Simulation(p, phi0, prec=prec) as ref:
            k = sim.kernel()
            want = _expected(prec, tau, n, n + 3, walls, sms)
            assert k["form"] == want[0] and want[1] in (None, k["shape"])
            seen.add(want)
            abi.lb_ch_test_hook(ref.h, abi.LBCH_HOOK_TILE_KERNEL, 0)
            assert ref.kernel()["form"].startswith("sweep")
            sim.step(5)
            ref.step(5)
            assert np.array_equal(sim.phi(), ref.phi())
    if sms == 152:
        assert len(seen) == {("f32", 1.0, 0): 5, ("f32", 0.8, 0): 4, ("f32", 0.8, 1): 4, ("f16s", 0.8, 0): 4, ("f16s", 0.8, 1): 4,
                             ("f64", 1.0, 0): 5, ("f64", 1.0, 1): 5, ("f64", 0.8, 0): 5, ("f64", 0.8, 1): 5}.get((prec, tau, walls), 1)
