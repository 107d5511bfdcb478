"""The reciprocal in the force: against the device's own, and its range over the densities a handle can be given.

Bounds.  node_rcp: a Newton-Raphson step from an approximation within 2^-23 (float) leaves (2^-23)^2, a third-order step from one
within 2^-20 (double) 2^-60, so before the last rounding either is within a hundredth of a unit in the last place, and the
result is the correctly rounded one or its neighbour: 1.  Units of sigma and rho: powers of two round nothing, so the same bits.
Densities that make the force negligible, against the FP64 oracle over ten steps: 1e-12 in double, 1e-5 in float, as
elsewhere."""
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_1805_00007_gb300 import _build, abi
from paper_1805_00007_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cstdio>
#include <cstring>
#include "lbch_kernels.cuh"
using namespace lbch;
__device__ unsigned long long worst[2];
__device__ unsigned long long mix(unsigned long long z)
{
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
    return z ^ (z >> 31);
}
__device__ unsigned long long apart(long long a, long long b) { return a > b ? a - b : b - a; }
// every exponent of a normal number with a normal reciprocal, both signs; mantissas 0, 1, all ones and spread ones
__global__ void check()
{
    const unsigned long long t = blockIdx.x * 256ULL + threadIdx.x, m = t < 3 ? (t == 0 ? 0 : t == 1 ? 1 : ~0ULL) : mix(t);
    for (unsigned e = 1; e < 253; e++) {
        const unsigned b = (unsigned)(m & 0x807fffffU) | e << 23;
        const float v = __uint_as_float(b);
        atomicMax(&worst[0], apart(__float_as_int(node_rcp(v)), __float_as_int(__frcp_rn(v))));
    }
    for (unsigned e = 1; e < 2045; e++) {
        const double v = __longlong_as_double((long long)((m & 0x800fffffffffffffULL) | (unsigned long long)e << 52));
        atomicMax(&worst[1], apart(__double_as_longlong(node_rcp(v)), __double_as_longlong(1.0 / v)));
    }
}
int main()
{
    unsigned long long w[2] = {99, 99};
    check<<<64, 256>>>();
    if (cudaMemcpyFromSymbol(w, worst, sizeof w) != cudaSuccess) return 1;
    printf("%llu %llu\n", w[0], w[1]);
    return 0;
}
"""


def test_reciprocal_against_the_devices_own(tmp_path):
    src, exe = tmp_path / "rcp.cu", tmp_path / "rcp"
    src.write_text(SOURCE)
    subprocess.run([_build.nvcc(), *_build.COMPILE_FLAGS, "-I", _build.CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120, env=os.environ).stdout
    assert all(int(k) <= 1 for k in out.split()) and len(out.split()) == 2


def _setup(unit=0, **kw):
    u = 2.0 ** unit
    p = dict(nx=45, ny=38, vel=wl.VEL_UNIFORM, ux0=0.03, uy0=-0.02, sigma=0.02, M=0.02, rhoA=1000.0, rhoB=1.0, W=3.0)
    p.update(kw)
    p = wl.make_params(**p)
    p.update(sigma=p["sigma"] * u, rhoA=p["rhoA"] * u, rhoB=p["rhoB"] * u, M=p["M"] / u)
    return p, wl.random_smooth_phi(p["nx"], p["ny"], seed=5)


def _run(setup, prec, form):
    with abi.Simulation(setup[0], setup[1], prec=prec) as sim:
        if form == "pair":
            abi.lb_ch_test_hook(sim.h, abi.LBCH_HOOK_TWO_STEP, 1)
        elif form:
            abi.lb_ch_test_hook(sim.h, abi.LBCH_HOOK_TILE_KERNEL, form == "tile")
        sim.step(7)
        return sim.phi()


@pytest.mark.parametrize("prec,unit", [("f32", -60), ("f32", 90), ("f32", 112), ("f16s", 112), ("f64", 400), ("f64", 1005)])
@pytest.mark.parametrize("tau,model,form", [(1.0, 2, "sweep"), (1.0, 1, "tile"), (1.0, 2, "pair"), (0.8, 2, "sweep"),
                                            (0.8, 1, "tile"), (0.8, 3, "sweep"), (1.3, 3, "tile")])
def test_the_unit_of_tension_and_density_leaves_the_bits(prec, unit, tau, model, form):
    if prec == "f16s" and form == "pair":
        form = None
    a, b = _run(_setup(0, tau=tau, model=model), prec, form), _run(_setup(unit, tau=tau, model=model), prec, form)
    assert np.isfinite(a).all() and np.array_equal(a, b)


@pytest.mark.parametrize("prec,rho", [("f32", 1e34), ("f32", 2e36), ("f32", 3e38), ("f32", 1e39), ("f64", 1e39), ("f64", 1e307)])
@pytest.mark.parametrize("tau", [1.0, 0.8])
def test_densities_that_leave_no_force(prec, rho, tau):
    p, phi0 = _setup(0, rhoA=rho, rhoB=0.5 * rho, tau=tau)
    ref = oracle.simulate(p, phi0, 10)[0]
    for form in ("sweep", "tile"):
        with abi.Simulation(p, phi0, prec=prec) as sim:
            abi.lb_ch_test_hook(sim.h, abi.LBCH_HOOK_TILE_KERNEL, form == "tile")
            sim.step(10)
            assert np.max(np.abs(sim.phi() - ref)) <= (1e-12 if prec == "f64" else 1e-5)
