"""The step kernels where their cuts can go wrong, against the FP64 oracle and against one another.

FP64 against the oracle: 1e-12 (values of order one, operations of relative error 1e-16, some ten steps).  Forms of the step
against each other: the same bits, which every form promises at the same precision.  Adjoint: 1e-10 of the gradient's
largest value (the reverse step multiplies FP64 errors by the same factors as the gradient itself)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1805_00007_gb300 import abi
from paper_1805_00007_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _setup(nx, ny, tau, walls=0, model=2):
    if walls:
        p = wl.make_params(nx=nx, ny=ny, tau=tau, walls=1, vel=wl.VEL_SHEAR, shear=2e-3, M=0.02, sigma=0.02, W=3.0, model=model)
    else:
        p = wl.make_params(nx=nx, ny=ny, tau=tau, vel=wl.VEL_UNIFORM, ux0=0.03, uy0=-0.02, M=0.02, model=model)
    return p, wl.random_smooth_phi(nx, ny, seed=3 * nx + ny)


def _run(setups, prec, steps, form=None, shape=0, read=None):
    with abi.Simulation([s[0] for s in setups], [s[1] for s in setups], prec=prec) as sim:
        if form is not None:
            abi.lb_ch_test_hook(sim.h, abi.LBCH_HOOK_TILE_KERNEL, form == "tile")
            if form == "pair":
                abi.lb_ch_test_hook(sim.h, abi.LBCH_HOOK_TWO_STEP, 1)
            abi.lb_ch_test_hook(sim.h, abi.LBCH_HOOK_TILE_SHAPE, shape)
        for n in steps:
            sim.step(n)
        return [sim.phi(i) for i in range(len(setups))]


# strips of 58 columns from column -1 on (56 from 0 on with the populations): one strip, one with a node of the next, the
# strip's full width and one more; nodes with two images in x (nx < 6); domains of one warp's rows and fewer
SIZES = [(4, 4), (5, 7), (6, 6), (55, 9), (56, 12), (57, 5), (58, 8), (59, 4), (112, 6), (113, 31), (115, 10), (116, 33), (117, 7)]


@pytest.mark.parametrize("walls", [0, 1])
@pytest.mark.parametrize("tau", [1.0, 0.8])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_row_sweep_at_the_edges_of_its_strips(nx, ny, tau, walls):
    setup = _setup(nx, ny, tau, walls)
    ref = oracle.simulate(*setup, 7)[0]
    for shape in range(4):
        got = _run([setup], "f64", (7,), "sweep", shape)[0]
        assert np.max(np.abs(got - ref)) <= 1e-12
    for prec in ("f32",) if tau == 1.0 else ("f32", "f16s"):
        tile = _run([setup], prec, (7,), "tile")[0]
        for shape in range(4):
            assert np.array_equal(_run([setup], prec, (7,), "sweep", shape)[0], tile)


@pytest.mark.parametrize("tau", [1.0, 0.8])
def test_row_sweep_of_a_ragged_ensemble(tau):
    setups = [_setup(nx, ny, tau, walls=k % 2) for k, (nx, ny) in enumerate(SIZES)]
    for prec in ("f64", "f32"):
        tile = _run(setups, prec, (5,), "tile")
        for a, b in zip(_run(setups, prec, (5,), "sweep"), tile):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("prec,shapes", [("f32", 4), ("f64", 4)])
@pytest.mark.parametrize("nx,ny", [(4, 4), (5, 9), (31, 14), (33, 15), (47, 29), (64, 17)])
def test_two_step_kernel_at_the_edges_of_its_tiles(nx, ny, prec, shapes):
    setup = _setup(nx, ny, 1.0)
    one = _run([setup], prec, (9,), "sweep")[0]
    for shape in range(shapes):
        assert np.array_equal(_run([setup], prec, (9,), "pair", shape)[0], one)


# grids on both sides of the lines at which the default kernel changes (152 SMs)
@pytest.mark.parametrize("prec,tau,n", [("f32", 1.0, 152), ("f32", 1.0, 200), ("f32", 1.0, 264), ("f32", 1.0, 376), ("f32", 1.0, 400),
                                        ("f32", 1.0, 424), ("f32", 0.8, 204), ("f32", 0.8, 226), ("f32", 0.8, 300),
                                        ("f16s", 0.8, 272), ("f64", 0.8, 136), ("f64", 1.0, 200), ("f64", 1.0, 272)])
def test_default_kernel_gives_the_bits_of_the_row_sweep(prec, tau, n):
    setup = _setup(n, n + 3, tau)
    assert np.array_equal(_run([setup], prec, (5,))[0], _run([setup], prec, (5,), "sweep")[0])


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("form", ["sweep", "tile", "pair"])
def test_time_factors_over_batches_of_the_table(prec, form):
    """The same run by one call of 1100 steps (batches of the table of time factors, and a rest) and by calls of one and of
    several steps, which form them otherwise."""
    p = wl.make_params(nx=20, ny=12, vel=wl.VEL_VORTEX, U0=0.04, Tper=700.0, M=0.01)
    phi0 = wl.circle_phi(20, 12, 10, 6, 3, 3.0)
    whole = _run([(p, phi0)], prec, (1100,), form)[0]
    parts = _run([(p, phi0)], prec, (1, 2, 3, 64, 65, 1, 513, 450, 1), form)[0]
    assert np.array_equal(whole, parts)


@pytest.mark.parametrize("tau", [1.0, 0.85])
@pytest.mark.parametrize("model", [1, 2])
@pytest.mark.parametrize("nx,ny", [(4, 4), (5, 7), (31, 17), (32, 8), (33, 9), (65, 24)])
def test_adjoint_at_the_edges_of_its_tiles(nx, ny, tau, model):
    from paper_1805_00007_gb300.autograd import evolve

    p, phi0 = _setup(nx, ny, tau, model=model)
    phiT = oracle.simulate(p, phi0, 6)[0]
    target = np.roll(phi0, (1, 2), (0, 1))
    d, s = oracle.adjoint(p, phi0, 6, phiT - target)
    x = torch.tensor(phi0, device="cuda", requires_grad=True)
    scale = torch.tensor(1.0, device="cuda", dtype=torch.float64, requires_grad=True)
    y = evolve(x, scale, p, 6, prec="f64")
    gx, gs = torch.autograd.grad(0.5 * torch.sum((y - torch.tensor(target, device="cuda")) ** 2), (x, scale))
    assert np.max(np.abs(gx.cpu().numpy() - d)) <= 1e-10 * np.max(np.abs(d))
    assert abs(float(gs) - s) <= 1e-10 * max(abs(s), np.max(np.abs(d)))
