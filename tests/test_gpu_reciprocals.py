"""The reciprocal and the reciprocal square root of the kernels' state variables (RegK::rcp3, RegK::rsq: a hardware
approximation, e below 2^-19 off, and one third-order step).

rcp3: y + y (e + e^2) with e = 1 - x y exact in one FMA: the rounding of the last FMA, 2^-53 of the result, and e^3 <
2^-57.  rsq: the same last rounding, and half of the 2^-53 that x y is rounded by on the way to e = 1 - x y^2."""
import pytest

from paper_2001_01570_gb300 import diag

pytestmark = pytest.mark.gpu


def test_relative_errors():
    rcp3, rsq = diag.rcp3_rsq_maxrel(1 << 22)
    assert 0.0 < rcp3 <= 2.0 ** -53 + 2.0 ** -57
    assert 0.0 < rsq <= 1.5 * 2.0 ** -53 + 2.0 ** -57
