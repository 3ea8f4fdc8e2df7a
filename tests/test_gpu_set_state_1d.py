"""cgks_set_state of 1D grids from device planes, on both sides of the size from which several CTAs do it: the
planes come back, a solve from them agrees with the oracle, and setting a large grid takes a small part of a step."""
import time

import numpy as np
import pytest

from parity_util import check, run_gpu, run_oracle
from paper_2001_01570_gb300 import cgks, workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [255, 256, 257, 511, 512, 513, 1025])
def test_sizes(n):
    spec, W = wl.density_wave_1d(n, eps=0.2, cfl=0.3)
    s = cgks.Solver(cgks.problem_from_spec(spec))
    d = torch.tensor(np.ascontiguousarray(W), device="cuda")
    out = torch.empty_like(d)
    cgks.cgks_set_state(s.handle, d, t=0.25)
    t, steps = cgks.cgks_get_state(s.handle, out)
    assert torch.equal(out, d) and t == 0.25 and steps == 0
    s.close()
    g, _, _ = run_gpu(spec, W, 2)
    o, _, _ = run_oracle(spec, W, 2)
    check(None, g, o, dx=spec.dx)


def test_a_large_grid_is_set_in_a_fraction_of_a_step():
    spec, W = wl.density_wave_1d(1 << 18, eps=0.2, cfl=0.3)
    s = cgks.Solver(cgks.problem_from_spec(spec))
    d = torch.tensor(np.ascontiguousarray(W), device="cuda")

    def best(f):
        f()
        ts = []
        for _ in range(5):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            f()
            torch.cuda.synchronize()
            ts.append(time.perf_counter() - t0)
        return min(ts)

    # 150 bytes and some 30 FP64 instructions a cell against some 1,000 of a step
    assert best(lambda: cgks.cgks_set_state(s.handle, d)) < 0.5 * best(lambda: cgks.cgks_step(s.handle, 1))
    s.close()
