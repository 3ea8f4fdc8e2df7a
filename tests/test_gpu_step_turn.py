"""No step asked of a state without a usable time step (an infinite speed of sound): no error; the first step
is refused and the state stays."""
import numpy as np
import pytest

from paper_2001_01570_gb300 import cgks, workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_no_steps_of_a_state_without_a_time_step():
    W = np.zeros((12, 8, 8))
    W[0], W[3] = 1e-160, 1e160
    spec = wl.ProblemSpec(dim=2, nx=8, ny=8, x0=0.0, x1=1.0)
    prob = cgks.problem_from_spec(spec)
    s = cgks.Solver(prob)
    s.set_state(W)
    s.step(0)
    assert s.get_state()[2] == 0
    d = torch.tensor(W, device="cuda")
    assert cgks.cgks_step_noalloc(prob, d, 0, t=0.5) == 0.5
    with pytest.raises(cgks.CgksError):
        s.step(1)
    out = np.empty_like(W)
    with pytest.raises(cgks.CgksError):
        cgks.cgks_get_state(s.handle, out)
    assert np.array_equal(out, W)
    s.close()
