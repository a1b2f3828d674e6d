"""boys_pairwise where the sizes of y and of the weights offset each other: every
w_ij y_j is an ordinary number, however far from 1 its factors are.

All terms are positive, so the error is relative to z: per pair at most 16 units of
2^-53 (table, expansion and the product by y), the sum of n terms n more.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2512_10059_gb300 as pb

pytestmark = pytest.mark.gpu


def _check(x, y, c):
    t = [torch.from_numpy(np.ascontiguousarray(v, dtype=np.float64)).to("cuda:0") for v in (x, y, c)]
    z = pb.boys_pairwise(*t).cpu().numpy()
    hi, lo = oracle.pairwise(x, y, c)
    assert np.all(np.isfinite(hi)) and np.min(hi) > 1e-290
    assert np.max(np.abs(((z - hi) - lo) / hi)) <= (len(x) + 16) * 2.0 ** -53


@pytest.mark.parametrize("ys,cs", [(1.7e308, 1e-200), (1e300, 1e-308), (1e250, 1e-315), (1e-200, 1e200),
                                   (1e-300, 1e200), (1e-315, 1e270), (1e-10, 1.7e305)])
@pytest.mark.parametrize("k,n", [(0, 2), (12, 100), (32, 300)])
def test_offsetting_scales(ys, cs, k, n):
    rng = np.random.default_rng(k + n)
    # F_0 dominates the sums below X = 40
    _check(rng.uniform(0.0, 20.0, n), rng.uniform(0.25, 1.0, n) * ys, rng.uniform(0.25, 1.0, k + 1) * cs)


def test_small_y_against_a_high_order():
    """F_32 is about 1e-22 here: y times the scaled w would be far below the doubles."""
    x, c = np.linspace(25.0, 31.0, 64), np.zeros(33)
    c[32] = 1e280
    _check(x, np.full(64, 1e-305), c)
