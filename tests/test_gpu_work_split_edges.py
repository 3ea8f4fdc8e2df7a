"""The edges of the kernels' work split against the oracle: 1D grids around a flux CTA's 64 faces and an
update chunk's 128 cells, 2D grids around the flux kernel's 8x4 strips (whole strips, one cell more and less,
whose last faces are a tile row of their own), and grids on both sides of the size from which an update
thread takes two cells (4 warps of cells per FP64 unit: 77,824 on 152 SMs), in both kinds of reconstruction
variables.  Tolerance: parity_util's, as for every other size."""
import dataclasses

import numpy as np
import pytest

from parity_util import check, run_gpu, run_oracle
from paper_2001_01570_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("char", [0, 1])
@pytest.mark.parametrize("n", [63, 64, 65, 127, 128, 129])
def test_1d_sizes(n, char):
    spec, W = wl.density_wave_1d(n, eps=0.2, cfl=0.3)
    spec = dataclasses.replace(spec, recon_vars=char)
    g, _, sg = run_gpu(spec, W, 3)
    o, _, so = run_oracle(spec, W, 3)
    assert sg == so == 3
    check(None, g, o, dx=spec.dx)


@pytest.mark.parametrize("char", [0, 1])
@pytest.mark.parametrize("nx,ny", [(16, 8), (15, 8), (17, 8), (16, 7), (16, 9), (33, 13)])
def test_2d_sizes(nx, ny, char):
    spec, W = wl.shock_vortex(nx=nx, ny=ny, mach=1.2)
    spec = dataclasses.replace(spec, recon_vars=char)
    g, _, sg = run_gpu(spec, W, 2)
    o, _, so = run_oracle(spec, W, 2)
    assert sg == so == 2
    check(None, g, o, dx=spec.dx, dy=spec.dy)


@pytest.mark.parametrize("nx,ny", [(304, 256), (304, 257)])
def test_cells_per_update_thread(nx, ny):
    spec, W = wl.shock_vortex(nx=nx, ny=ny, mach=1.2)
    g, _, sg = run_gpu(spec, W, 2)
    o, _, so = run_oracle(spec, W, 2)
    assert sg == so == 2
    check(None, g, o, dx=spec.dx, dy=spec.dy)
    assert np.isfinite(g).all()
