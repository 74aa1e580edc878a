"""The FP64 inversion divides by a small integer through its correctly rounded
reciprocal and one residual (csrc/fcs_tasks.cu: inversion64).  The quotient has
to be the IEEE one, as the definition's division gives it: checked against it
in exact rational arithmetic for the fused operations."""
from fractions import Fraction

import numpy as np
import pytest


def _fma(a, b, c):  # rounded once (float() of a fraction rounds to nearest even)
    return float(Fraction(a) * Fraction(b) + Fraction(c))


@pytest.mark.parametrize("k0", [1, 17, 33, 49])
def test_quotients(k0):
    rng = np.random.default_rng(k0)
    for k in range(k0, k0 + 16):
        r = 1.0 / k
        # random significands, all-ones and sparse ones, and products near multiples of k
        n = np.concatenate([rng.uniform(1.0, 2.0, 150) * 2.0 ** rng.integers(-400, 4, 150),
                            np.nextafter(2.0 ** rng.integers(-30, 4, 20), 0.0), 2.0 ** rng.integers(-30, 4, 10),
                            np.nextafter(k * rng.uniform(0.0, 1.0, 20), rng.choice([0.0, 9.0], 20))])
        for x in map(float, n):
            q0 = x * r
            assert _fma(_fma(-q0, float(k), x), r, q0) == x / k, (k, x)
