"""States in other units than order one against the oracle: the kernels' parts in pairs of FP32 are used only
where the units leave them their precision, so a solve in SI units of a thin or a dense gas, on kilometres or
fractions of a micrometre, meets parity_util's bars like one in units of order one."""
import dataclasses

import numpy as np
import pytest

from parity_util import check, run_gpu, run_oracle
from paper_2001_01570_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def in_units(spec, W, rho, a, length):
    """The problem and its planes with density, velocity and length in the given multiples."""
    nv, V = (3 if spec.dim == 1 else 4), W * rho
    for g in range(0, W.shape[0], nv):
        V[g + 1:g + nv - 1] *= a
        V[g + nv - 1] *= a * a
    V[nv:] /= length
    box = {k: getattr(spec, k) * length for k in ("x0", "x1", "y0", "y1")}
    return dataclasses.replace(spec, inflow=(rho, a, 0.0, rho * a * a), **box), V


def compare(spec, W, nsteps):
    g, _, sg = run_gpu(spec, W, nsteps)
    o, _, so = run_oracle(spec, W, nsteps)
    assert sg == so == nsteps
    check(None, g, o, dx=spec.dx, dy=spec.dy)


@pytest.mark.parametrize("mu", [0.0, 0.01])
@pytest.mark.parametrize("rho,a,length", [(1.2, 340.0, 1e-3), (3e-12, 800.0, 1e4), (1e-9, 1e3, 1e9), (1e-15, 1e4, 1e10),
                                          (1e4, 1e6, 1e-7)])
def test_vortex_in_units(rho, a, length, mu):
    spec, W = wl.isentropic_vortex(48)
    spec, W = in_units(spec, np.ascontiguousarray(W), rho, a, length)
    compare(dataclasses.replace(spec, mu=mu * rho * a * length), W, 20)


@pytest.mark.parametrize("char", [0, 1])
@pytest.mark.parametrize("length", [1e-42, 1e42])
def test_time_steps_out_of_a_floats_range(length, char):
    """A shock's non-equilibrium part, weighted by exp(-dt / (2 tau)), in units of time of 1e-45 and 1e39."""
    spec, W = wl.shock_tube_1d(100)
    spec, W = in_units(dataclasses.replace(spec, recon_vars=char), np.ascontiguousarray(W), 1.0, 1.0, length)
    compare(spec, W, 10)
    spec, W = wl.shock_vortex(nx=48, ny=24, mach=1.5)
    inflow = spec.inflow
    spec, W = in_units(dataclasses.replace(spec, recon_vars=char), np.ascontiguousarray(W), 1.0, 1.0, length)
    compare(dataclasses.replace(spec, inflow=inflow), W, 3)
