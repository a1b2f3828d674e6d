"""The bounds that csrc/boys_region.cuh states for its integer recurrence, for every order
0..32, on the model of tests/test_local_model.py (which asserts the range of every sum
T, 2^56 < T < 0.56 2^64, as it goes): 2^-53 relative before the cut to a double, derived
there.  The points are where it is nearest: just above powers of two, where X has
the fewest bits (from 32 on it holds the significand, and a sum keeps the product's
leading bits alone), just below x_1, where T is largest ((2x + e^{-x} / F_{l+1}) / 128
of 2^64, 0.556 at l = 31), and around x_0.
"""
import math

import pytest

from tests import test_local_model as M

POINTS = [M.X0, math.nextafter(M.X0, 0), M.X1, math.nextafter(M.X1, 0), 28.98, 2.8934195158947382, 6.69, 12.25146893730016,
          32.0, 32.375365956450544, 33.3757704437136, 64.25, 128.0014, 256.034, 515.015, 1044.0057104517814]


def _error(K, x):
    """The largest relative error of the model's values, as a power of two."""
    got, ref = M._model(K, x), M._algorithm1(K, x)
    worst = 0.0
    for l in range(K + 1):
        y, ex = got[l]
        v = y << (M.W + ex) if M.W + ex >= 0 else y >> -(M.W + ex)
        worst = max(worst, abs(v - ref[l]) / ref[l])
    return worst


@pytest.mark.parametrize("K", range(33))
def test_every_order(K):
    for x in POINTS:
        assert _error(K, x) <= 2.0 ** -53, (K, x)


@pytest.mark.parametrize("part", [0, 4, 8, 10])
def test_a_mistake_in_a_table_entry_shows(part):
    """A coefficient's last eight bits (16 in the fifth, which weighs 2^-8 at x = 3.3), the
    entry's exponent or e^{-x}'s, planted in the table: far outside the bound."""
    entry = M.TABLE[5][52]
    wrong = list(entry)
    wrong[part] += {0: 1 << 14, 4: 1 << 40, 8: 1, 10: 1 << 40}[part]
    M.TABLE[5][52] = type(entry)(wrong)
    try:
        assert _error(5, 3.3) > 2.0 ** -52
    finally:
        M.TABLE[5][52] = entry
    assert _error(5, 3.3) <= 2.0 ** -53
