"""boys_pairwise where a block does without its table of expansions: few j, few rows,
pairs beyond the table (X >= 64) or formed with a negative argument, and weights
whose sum overflows.
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


def _pairs(x, j, c):
    """sum_l c_l F_l and sum_l |c_l| F_l at x_i + x_j."""
    f = np.stack(oracle.boys(x + x[j], len(c) - 1)).astype(np.longdouble).sum(0)
    return (f * c[:, None]).sum(0), (f * np.abs(c)[:, None]).sum(0)


@pytest.mark.parametrize("k", [0, 1, 12, 31, 32])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 7, 8, 9, 15, 16, 31, 33, 40, 47, 48, 49, 64, 65])
def test_short_batches(n, k):
    """All terms positive and in the table: 16 units of 2^-53 a pair and n for the sum."""
    rng = np.random.default_rng(100 * n + k)
    x, y, c = rng.uniform(0.0, 31.9, n), rng.uniform(0.5, 1.0, n), rng.uniform(0.5, 1.0, k + 1)
    hi, lo = oracle.pairwise(x, y, c)
    assert np.max(np.abs(((_run(x, y, c) - hi) - lo) / hi)) <= (n + 16) * 2.0 ** -53


@pytest.mark.parametrize("k", [0, 12, 32])
def test_expansions_of_single_pairs_have_the_tables_bits(k):
    rng = np.random.default_rng(k)
    x, c = rng.uniform(0.0, 31.9, 1200), rng.standard_normal(k + 1)
    for j in (0, 13, 23):
        y = np.zeros(1200)
        y[j] = 1.0
        assert np.array_equal(_run(x[:24], y[:24], c), _run(x, y, c)[:24])


@pytest.mark.parametrize("k", [0, 1, 12, 32])
@pytest.mark.parametrize("n", [6, 40, 600])
def test_pairs_beyond_the_table(n, k):
    """The closed form of region C.  Cuts of F_0 and of the sum 2 units of 2^-53 each, their
    product 1, the Horner sum's units below 1: 16 of sum |c_l| F_l; the asymptotic form
    itself is off by Gamma(l + 1/2, X) / (2 X^(l + 1/2)) < 1e-28 from X = 64 on."""
    rng = np.random.default_rng(n + k)
    x, c = rng.uniform(32.0, 2500.0, n), rng.standard_normal(k + 1)
    x[:2], c[0] = (32.0, 1e7), 1.0 + abs(c[0])
    for j in (0, 1, n - 1):
        y = np.zeros(n)
        y[j] = 1.0
        w, size = _pairs(x, j, c)
        assert np.all(np.abs(_run(x, y, c) - w) <= 2.0 ** -49 * size + 1e-28 * np.abs(c).sum())


@pytest.mark.parametrize("k", [0, 5, 12, 32])
@pytest.mark.parametrize("n", [8, 100, 700])
def test_negative_argument_with_a_larger_partner(n, k):
    """x_j = -20: the pairs with X >= 0 take the three-region evaluation order by order, in
    all its regions: 5e-14 an order and the rounding of the sum."""
    rng = np.random.default_rng(n + k)
    x, c = rng.uniform(20.0, 90.0, n), rng.standard_normal(k + 1)
    x[0], y = -20.0, np.zeros(n)
    y[0] = 1.0
    z = _run(x, y, c)
    f = np.stack(oracle.boys(x[1:] + x[0], k)).astype(np.longdouble).sum(0)
    assert np.isnan(z[0])
    assert np.max(np.abs(z[1:] - (f * c[:, None]).sum(0))) <= (5e-14 + 2.0 ** -53 * (k + 3)) * np.abs(c).sum()


@pytest.mark.parametrize("n", [5, 300])
def test_weights_whose_sum_overflows(n):
    rng = np.random.default_rng(n)
    x, c = rng.uniform(2.0, 60.0, n), np.full(3, 1e308)
    y = np.zeros(n)
    y[n // 2] = 1.0
    w, _ = _pairs(x, n // 2, np.ones(3))
    assert np.max(np.abs(_run(x, y, c) / 1e308 - w)) <= 3 * 5e-14 + 2.0 ** -50
