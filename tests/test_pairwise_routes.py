"""boys_pairwise across its two ways to w(X) = sum_l c_l F_l(X) -- expansions
built by the call (X < 64, finite weights) and the evaluation order by
order -- and across the split of the j over a cluster of blocks.

Tolerance as in test_pairwise.py (5e-14 sum|c| sum|y| plus the rounding of the
sums); the expansions add at most 2^-54 sum|c_l|F_l of truncation and 2^-56 of X's
units, inside the rounding term.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2512_10059_gb300 as pb

pytestmark = pytest.mark.gpu


def _run(x, y, c):
    t = [torch.from_numpy(np.ascontiguousarray(v, dtype=np.float64)).to("cuda:0") for v in (x, y, c)]
    return pb.boys_pairwise(*t).cpu().numpy()


def _check(x, y, c):
    hi, lo = oracle.pairwise(x, y, c)
    s = np.abs(c).sum() * np.abs(y).sum()
    tol = 5e-14 * s + 2.0 ** -53 * (len(x) + len(c) + 1) * s + 1e-27
    assert np.max(np.abs((_run(x, y, c) - hi) - lo)) <= tol


@pytest.mark.parametrize("k", [0, 1, 23, 24, 25, 32])
@pytest.mark.parametrize("n", [1, 255, 257, 513, 1025])
def test_sizes_and_orders(n, k):
    rng = np.random.default_rng(1000 * k + n)
    _check(rng.uniform(0.0, 40.0, n), rng.standard_normal(n), rng.standard_normal(k + 1))


@pytest.mark.parametrize("k", [3, 24])
def test_interval_edges_and_the_end_of_the_table(k):
    """y one-hot pins single pairs: X on, just below and just above interval
    edges, at 64, and far beyond."""
    base = np.array([0.0, 1 / 16, 11.875, 11.9375, 28.9375, 29.0, 31.5, 63.9375, 64.0, 100.0, 1e6, 1e300])
    x = np.unique(np.concatenate([base, np.nextafter(base, 1e308), np.nextafter(base[1:], 0.0)]))
    c = np.random.default_rng(k).standard_normal(k + 1)
    for j in (0, 1, len(x) // 2):
        y = np.zeros(len(x))
        y[j] = 1.0
        hi, lo = oracle.pairwise(x, y, c)
        assert np.max(np.abs((_run(x, y, c) - hi) - lo)) <= (5e-14 + 2.0 ** -53 * (k + 3)) * np.abs(c).sum()


@pytest.mark.parametrize("l", [0, 12, 24, 32])
def test_small_values_keep_their_relative_accuracy(l):
    """One weight only: w = c_l F_l, down to 1e-22 at X = 63, where the table has the
    definition's values.  Truncation 2^-54, FP64 rounding of the expansion's leading
    coefficients 2^-53 each, an exponent's unit 2^-59 eight times, the rounding of the
    product by y: 2^-50 relative to the oracle."""
    x = np.array([22.5, 24.0, 27.0, 31.375])
    y = np.array([0.0, 0.0, 0.0, 1.0])
    c = np.zeros(l + 1)
    c[l] = -3.0
    hi, _ = oracle.pairwise(x, y, c)
    assert np.max(np.abs(_run(x, y, c) / hi - 1.0)) <= 2.0 ** -50


def test_invalid_arguments_and_weights():
    x = np.array([0.5, -1.0, 2.0, np.nan, np.inf, 70.0])
    y, c = np.ones(6), np.array([1.0, 0.5])
    z = _run(x, y, c)
    assert np.all(np.isnan(z))                      # every row meets the NaN
    x = np.array([0.5, -0.25, 2.0, np.inf, 70.0])   # only -0.25 - 0.25 < 0 is invalid
    z = _run(x, np.ones(5), c)
    assert np.isnan(z[1]) and np.all(np.isfinite(z[[0, 2, 3, 4]])) and z[3] == 0.0
    assert np.all(np.isnan(_run(np.array([1.0, 2.0]), np.ones(2), np.array([1.0, np.nan]))))
    assert np.all(_run(np.array([1.0, 2.0]), np.ones(2), np.zeros(3)) == 0.0)


@pytest.mark.parametrize("scale", [1e-250, 1e-30, 1e30, 1e200])
def test_weight_scales(scale):
    rng = np.random.default_rng(9)
    x, y, c = rng.uniform(0, 30, 300), rng.standard_normal(300), rng.standard_normal(13)
    a, b = _run(x, y, c), _run(x, y, c * scale)
    assert np.max(np.abs(b / scale - a)) <= 1e-15 * 300 * np.abs(c).sum()
