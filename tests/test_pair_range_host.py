"""The choices between pairs of FP32 and FP64 in the flux kernel's arithmetic, run on the host over units of
density, velocity and length from 2^-120 to 2^120: the same segments through the kernels' functions with the
pairs and in FP64 alone (tests/pair_range_check.cpp).

Bound: a Gauss point's three states are within 2^-51 of their scale of the FP64 ones (tests/test_split_host.py) and
enter the fluxes and time derivatives with factors of order one; what is computed in pairs after them is kept
below the last bit of what it is added to.  2^-48 of the results' scale leaves 8 of those units; a pair that
lost its low words is off by 2^-24 of a correction, one that lost its range by all of it."""
import os
import subprocess

import numpy as np
import pytest
from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2001_01570_gb300", "csrc")
BOUND = 2.0 ** -48


def build(tmp, source, *defs):
    exe = str(tmp / ("check" + "".join(defs)))
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-std=c++20", "-w", "-Wno-unknown-pragmas", *defs, "-I", cuda,
                    "-I", CSRC, "-o", exe, os.path.join(ROOT, "tests", source)], check=True)
    return exe


@pytest.fixture(scope="module")
def points(tmp_path_factory):
    tmp = tmp_path_factory.mktemp("range")
    runs = [subprocess.run([build(tmp, "pair_range_check.cpp", *d)], check=True, capture_output=True).stdout
            for d in ((), ("-DCGKS_SPLIT_CHECK=1",))]
    a, b = (np.frombuffer(r).reshape(9, 8, 14, -1, 2, 5, 4) for r in runs)   # density, velocity, length, points
    assert np.array_equal(a[..., 1, :, :], b[..., 1, :, :])
    return np.abs(a[..., 0, :, :] - b[..., 0, :, :]) / a[..., 1, :, :]


@pytest.mark.parametrize("k,what", [(0, "flux"), (1, "F_t"), (2, "W(dt/2)"), (3, "W(dt)"), (4, "W_tt")])
def test_pairs_are_used_only_where_they_are_as_exact(points, k, what):
    worst = points[..., k, :].max(axis=(3, 4))
    assert np.all(worst <= BOUND), [(tuple(map(int, i)), float(np.log2(worst[tuple(i)]))) for i in np.argwhere(worst > BOUND)[:8]]


@pytest.mark.parametrize("k", range(5))
def test_pairs_are_used_in_units_of_order_one(points, k):
    """Density and velocity 1, cells of 2^-7: points differ from the FP64 ones in some last bits."""
    assert (points[5, 2, 5, :, k] > 0).any()


def test_numbers_out_of_a_floats_range(tmp_path):
    """ff_from_any keeps 47 bits from 2^-74 to 2^128 and errors below 2^-97 beneath; from 2^128 on, and for NaN,
    it and f_lead give no finite number, so that no bound on a result admits it."""
    src = tmp_path / "c.cpp"
    src.write_text('''
#include <cmath>
#include <cstdio>
#include <initializer_list>
#include <limits>
#include "cgks_split.cuh"
using namespace cgks;
int main()
{
    double rel = 0, low = 0; int bad = 0;
    for (int e = -400; e <= 400; ++e)
        for (int m = 0; m < 64; ++m)
            for (int sgn = -1; sgn <= 1; sgn += 2) {
                const double x = sgn * std::ldexp(1.0 + (m * 2654435761u % 1000003) / 1000003.0, e);
                const ff p = ff_from_any(x);
                const float f = f_lead(x);
                if (e >= 128) { bad += std::isfinite(p.h) + std::isfinite(f); continue; }
                const double err = std::fabs((double)p.h + (double)p.l - x), el = std::fabs((double)f - x);
                if (e >= -74) rel = std::fmax(rel, err / std::fabs(x));
                else low = std::fmax(low, err);
                if (e >= -126) bad += !(el < std::ldexp(std::fabs(x), -20));
                else bad += !(std::fabs((double)f) < std::ldexp(1.0, -126));
            }
    for (double x : {std::numeric_limits<double>::infinity(), -std::numeric_limits<double>::infinity(), (double)NAN})
        bad += std::isfinite(ff_from_any(x).h) + std::isfinite(f_lead(x));
    printf("%.17g %.17g %d\\n", rel, low, bad);
}
''')
    exe = str(tmp_path / "c")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, "-o", exe, str(src)], check=True)
    rel, low, bad = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert float(rel) <= 2.0 ** -47 and float(low) < 2.0 ** -97 and int(bad) == 0


def test_shear_is_measured_against_its_own_scale(tmp_path):
    """Characteristic variables, a shear layer in gases whose speed of sound is 1 to 2^-12 of the unit of
    velocity: the WENO-Z values' bound of tests/test_split_host.py (2^-51 of the scale, here rho, rho c and rho c^2)
    once for the field and once for the basis it goes through."""
    a, b = (np.frombuffer(subprocess.run([build(tmp_path, "char_scale_check.cpp", *d)], check=True, capture_output=True).stdout)
            .reshape(13, -1, 2, 2, 4) for d in ((), ("-DCGKS_SPLIT_CHECK=1",)))
    worst = (np.abs(a[:, :, 0] - b[:, :, 0]) / a[:, :, 1]).max(axis=(1, 2))
    assert (worst[0, 2] > 0) and np.all(worst <= 2.0 ** -50), np.log2(np.maximum(worst, 2.0 ** -60)).round(1)


def test_each_choice_is_its_bound(tmp_path):
    """Every function that chooses between the pairs and FP64, on data on both sides of its bound (1 % around it
    left out), against the bound worked out in FP64; slopes, second derivatives and rows that are infinite, NaN or
    out of a float's range are refused (tests/pair_choice_check.cpp)."""
    out = subprocess.run([build(tmp_path, "pair_choice_check.cpp")], check=True, capture_output=True, text=True).stdout
    rows = [(a[0], *map(int, a[1:])) for a in (ln.split() for ln in out.splitlines())]
    assert len(rows) == 9
    for name, yes, no, bad in rows:
        assert yes > 1000 and no > 1000 and bad == 0, (name, yes, no, bad)
