"""The state import's rounding of positions, checked on the CPU (no GPU needed).

The contract is q = rint((x - lo) / dq). The kernel multiplies by the rounded reciprocal of
dq and divides only within 2^-19 of a half or near the range's ends; IEEE doubles behave the
same here, so the rule is restated with numpy and compared with the division for random
coordinates, for representable ones and for the neighbours of every kind of half."""
import numpy as np
import pytest

LIM = 2147483000.0


def fast(d, dq):
    s = d * (1.0 / dq)
    exact = ~(np.abs(s - np.rint(s)) < 0.5 - 2.0 ** -19) | ~(np.abs(s) < 2147481600.0)
    s = np.where(exact, d / dq, s)
    inside = (s > -LIM) & (s < LIM)
    return np.where(inside, np.rint(np.where(inside, s, 0.0)), 0.0), inside, exact


@pytest.mark.parametrize("cell, bits", [(2.6 / 40, 22), (2.6 / 159, 21), (1.0 / 153, 22), (0.3, 17), (7.7e-5, 22)])
def test_reciprocal_rounding_equals_the_division(cell, bits):
    rng = np.random.default_rng(bits)
    dq = cell / 2 ** bits
    q = rng.integers(-2 ** 31 + 1000, 2 ** 31 - 1000, 200_000).astype(np.float64)
    halves = (q + 0.5) * dq
    d = np.concatenate([rng.uniform(-LIM, LIM, 400_000) * dq, q * dq, halves, np.nextafter(halves, np.inf),
                        np.nextafter(halves, -np.inf), halves * (1.0 + 2.0 ** -51), halves * (1.0 - 2.0 ** -51),
                        np.array([LIM * dq, np.nextafter(LIM * dq, 0.0), -LIM * dq, np.inf, -np.inf, np.nan, 0.0])])
    with np.errstate(invalid="ignore"):
        s = d / dq
        want_in = (s > -LIM) & (s < LIM)
        got, got_in, exact = fast(d, dq)
    np.testing.assert_array_equal(got_in, want_in)
    np.testing.assert_array_equal(got, np.where(want_in, np.rint(np.where(want_in, s, 0.0)), 0.0))
    assert exact[:600_000].mean() < 1e-3            # the division is rare on ordinary coordinates
