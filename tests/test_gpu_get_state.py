"""cgks_get_state into device planes, from sizes on both sides of the one from which 2D planes are copied, after an
odd and an even number of steps (the state is in either buffer): the planes of the host call."""
import numpy as np
import pytest

from paper_2001_01570_gb300 import cgks, workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(8, 8), (256, 256), (256, 257), (400, 300)])
@pytest.mark.parametrize("steps", [1, 2])
def test_device_planes_are_the_host_planes(nx, ny, steps):
    spec, W = wl.shock_vortex(nx=nx, ny=ny, mach=1.2)
    s = cgks.Solver(cgks.problem_from_spec(spec))
    s.set_state(W)
    s.step(steps)
    host, t, n = s.get_state()
    out = torch.empty(W.shape, dtype=torch.float64, device="cuda")
    assert cgks.cgks_get_state(s.handle, out) == (t, n) and n == steps
    assert np.array_equal(out.cpu().numpy(), host)
    s.close()
