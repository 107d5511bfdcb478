"""The coupled step where its storage can go wrong: rows of one group of 32 nodes, of a full last group and of one or two
nodes in it, between walls and periodic, against the FP64 oracle (1e-12: some tens of steps of operations of relative
error 1e-16 on values of order one), and the form that leaves the populations of the Cahn-Hilliard lattice unread at
tau_g = 1 against the general one (the same bits: it leaves out products with zero)."""
import numpy as np
import pytest

import oracle
from paper_1805_00007_gb300 import abi
from paper_1805_00007_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _setup(nx, ny, walls, tau):
    p = wl.make_params(nx=nx, ny=ny, walls=walls, vel=wl.VEL_COUPLED, phiA=1.0, phiB=-1.0, rhoA=1.0, rhoB=0.4, sigma=0.01,
                       W=3.0, M=0.02, tau=tau, nu=0.05, gx=1e-5, gy=-2e-5)
    return p, np.clip(wl.random_smooth_phi(nx, ny, seed=11 + nx + ny, amp=1.6, mean=0.0), -1, 1)


def _fields(p, phi0, nsteps, prec, general=False):
    with abi.Simulation(p, phi0, prec=prec) as sim:
        if general:
            abi.lb_ch_test_hook(sim.h, abi.LBCH_HOOK_GENERAL_PATH, 1)
        sim.step(nsteps)
        return [sim.phi(), *sim.velocity(), sim.pressure()]


@pytest.mark.parametrize("walls", [0, 1])
@pytest.mark.parametrize("nx,ny", [(4, 4), (31, 8), (32, 9), (33, 7), (34, 16), (64, 17), (65, 5), (98, 24)])
def test_group_edges(nx, ny, walls):
    tau = 1.0 if nx % 2 else 0.8
    p, phi0 = _setup(nx, ny, walls, tau)
    ref = oracle.ns_simulate(p, phi0, 40)
    for a, b in zip(_fields(p, phi0, 40, "f64"), ref):
        assert np.max(np.abs(a - b)) <= 1e-12


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_tau_one_form_gives_the_bits_of_the_general_one(prec):
    p, phi0 = _setup(47, 29, 1, 1.0)
    for a, b in zip(_fields(p, phi0, 70, prec), _fields(p, phi0, 70, prec, general=True)):
        assert np.array_equal(a, b)
