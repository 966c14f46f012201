"""The fixed-point sums with the exponent that the FP64 element kernel gives them: one
per element and variable, so the two lines of a sum may lie below it, by up to 2 bits
(kSpareBits in csrc/cr_local64.cuh; elements with lines further down take FP64).

Bound: that of tests/test_fixed_point.py with the element's largest product in the place
of the lines', less its 2^-57 for the final shift, which rounds here (2^-58).  And down
to 1 bit below, no further from the exact sums on average than the FMA chain.
"""
from fractions import Fraction

import numpy as np
import pytest

import oracle
from tests import test_fixed_point as tfp


@pytest.fixture(scope="module")
def two_lines(tmp_path_factory):
    plain, tfp.SRC = tfp.SRC, tfp.SRC.replace("FixAcc acc{0, 0};", "FixAcc acc = fix_zero();")
    try:
        assert "fix_zero" in tfp.SRC
        return tfp.two_lines.__wrapped__(tmp_path_factory) if hasattr(tfp.two_lines, "__wrapped__") else None
    finally:
        tfp.SRC = plain


LINES = {
    "smooth": lambda r, xi: 1.0 + 0.01 * r.standard_normal(xi.size),
    "rough": lambda r, xi: r.standard_normal(xi.size),
    "through 0": lambda r, xi: r.uniform(0.3, 1.0) * (xi - r.uniform(0.0, 1.0)),
    "steep": lambda r, xi: np.exp(3.0 * r.standard_normal(xi.size)) * r.choice([-1.0, 1.0], xi.size),
}


@pytest.mark.parametrize("N", [1, 2, 3, 4])
@pytest.mark.parametrize("kind", sorted(LINES))
@pytest.mark.parametrize("bits", [0, 1, 2])
def test_lines_below_the_exponent(two_lines, N, kind, bits):
    rng = np.random.default_rng(N)
    n, (xi, _, _, _, D) = N + 1, oracle.tables(N)
    amax = Fraction(float(np.abs(D).max()))
    err_fix = err_fma = 0.0
    for it in range(60):
        x, y = LINES[kind](rng, xi), LINES[kind](rng, xi)
        top = amax * 2 ** bits * Fraction(float(max(np.abs(x).max(), np.abs(y).max())))
        for p in range(n):
            got = two_lines(D[p], x, D[p], y, D, D, -bits)
            c, want = 0.0, Fraction(0)
            for a, b in list(zip(D[p], x)) + list(zip(D[p], y)):       # one FMA at a time, exactly rounded
                t = Fraction(float(a)) * Fraction(float(b))
                want += t
                c = float(t + Fraction(c))
            e = abs(Fraction(got) - want)
            assert e <= top * Fraction(10 * n + 1, 2 ** 57) + abs(want) / 2 ** 53, (it, p, float(e))
            err_fix += float(e) ** 2
            err_fma += float(abs(Fraction(c) - want)) ** 2
    if bits <= 1:
        assert err_fix <= err_fma
