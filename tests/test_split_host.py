"""The split (pairs of FP32) arithmetic of the record and flux kernels, run on the host against
long double evaluations of the same rows and beside the FP64 formulas it stands in for (Sec. 3.3).

Bounds: a value is one FP64 rounding of the result and one of the first difference it is built from,
2^-53 (|value| + |difference|) <= 2^-52 of the row's scale (1.5), plus the pairs' part: about thirty
pair operations of 2^-47 each on third differences of at most 2^-7 of the scale, 2^-49 of the scale at
the very worst; errors that add up at random stay far below.  So the largest error may not exceed
2^-51, and neither the largest nor the rms error the FP64 formulas' own by more than a quarter of the
last place of the scale (2^-54)."""
import os
import subprocess

import pytest
from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2001_01570_gb300", "csrc")


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("split") / "split_check")
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-std=c++20", "-w", "-Wno-unknown-pragmas", "-I", cuda, "-I", CSRC,
                    "-o", exe, os.path.join(ROOT, "tests", "split_check.cpp")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    return [(a[0], int(a[1]), int(a[2]), int(a[3]), *map(float, a[4:])) for a in (ln.split() for ln in out.splitlines())]


def test_pairs_hold_47_bits(lines):
    (_, _, _, _, worst, exact, back, zero), = [ln for ln in lines if ln[0] == "pairs"]
    assert worst <= 2.0 ** -47 and exact == 0.0 and back == 0.0 and zero == 0.0


@pytest.mark.parametrize("what", ["weno8_value", "weno8_slope", "weno6_value", "weno6_slope"])
@pytest.mark.parametrize("base", ["1", "0"])   # 0: a momentum around zero, measured against the scale 1
def test_split_rows_are_as_exact_as_fp64(lines, what, base):
    rows = [ln for ln in lines if ln[0] == f"{what}_base{base}"]
    assert len(rows) == 6 and rows[-1][2] == rows[-1][3]        # every smooth row takes the split path
    for _, lev, taken, total, mx, mx64, rms, rms64 in rows:
        assert taken > 0
        assert mx <= 2.0 ** -51, (what, lev, mx)
        assert mx <= mx64 + 2.0 ** -54 and rms <= rms64 + 2.0 ** -54, (what, lev, mx, mx64, rms, rms64)


@pytest.mark.parametrize("what", ["tang_value", "tang_slope"])
def test_split_values_along_a_face_are_as_exact_as_fp64(lines, what):
    """The same bounds: third differences of at most 2^-6 of the scale times the Gauss points' 0.14,
    slope corrections of at most 2^-11."""
    rows = [ln for ln in lines if ln[0] == what]
    assert len(rows) == 5 and rows[-1][2] == rows[-1][3]
    for _, lev, taken, total, mx, mx64, rms, rms64 in rows:
        assert taken > 0 and mx <= 2.0 ** -51, (what, lev, mx)
        assert mx <= mx64 + 2.0 ** -54 and rms <= rms64 + 2.0 ** -54, (what, lev, mx, mx64, rms, rms64)


@pytest.mark.parametrize("what", ["slope_moments", "euler_second"])
def test_split_moments_and_time_derivatives_hold_41_bits_of_their_terms(lines, what):
    """Up to 140 pair operations of 2^-47 each on terms no larger than the size they are measured
    against: 2^-40 at the very worst; random signs leave far less.  The kernel takes them only where
    their weight is below 2^-7 of the quantity they are added to."""
    (_, _, n, total, mx, mx64, rms, _), = [ln for ln in lines if ln[0] == what]
    assert n == total and mx <= 2.0 ** -41 and rms <= 2.0 ** -46
    assert mx64 <= 2.0 ** -49
