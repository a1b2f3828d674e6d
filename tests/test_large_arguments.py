"""Arguments beyond the expansion tables (x > 2^28), down to where F_k leaves the normal
doubles: F_k = (sqrt(pi)/2) (2k-1)!!/2^k x^{-k-1/2}, formed to about 2^-55 an order
in 64-bit significands (2^-49 in all at order 32) and cut to a double, one unit of 2^-1074
below the normal range.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2512_10059_gb300 as pb

pytestmark = pytest.mark.gpu
X = np.array([m * 10.0 ** e for e in range(9, 300) for m in (1.0, 1.37, 4.2)])


def _close(got, hi):
    assert np.all(np.abs(got - hi) <= 2.0 ** -49 * np.abs(hi) + 2.0 ** -1074)


@pytest.mark.parametrize("k", [0, 1, 4, 5, 16, 32])
def test_gradual_underflow(k):
    hi, _ = oracle.boys(X, k)
    assert k == 0 or np.any((hi > 0) & (hi < 2.0 ** -1022))
    xt = torch.from_numpy(X).to("cuda:0")
    _close(pb.boys_eval(xt, k).cpu().numpy(), hi)
    if k < 32:  # one upstream gradient at a time gives -F_{l+1}
        hi, _ = oracle.boys(X, k + 1)
        for l in (0, k):
            g = torch.zeros((k + 1, X.size), dtype=torch.float64, device="cuda:0")
            g[l] = 1.0
            _close(-pb.boys_grad(xt, g, k).cpu().numpy(), hi[l + 1])


def test_ends_of_the_range():
    """The largest double, infinity and invalid arguments: as they were."""
    x = torch.tensor([1.7976931348623157e308, float("inf"), -1.0, float("nan"), -0.0], dtype=torch.float64, device="cuda:0")
    f = pb.boys_eval(x, 3).cpu().numpy()
    assert 0.0 < f[0, 0] < 1e-149 and np.all(f[1:, 0] == 0.0) and np.all(f[:, 1] == 0.0)
    assert np.all(np.isnan(f[:, 2:4])) and np.allclose(f[:, 4], [1, 1 / 3, 1 / 5, 1 / 7], rtol=1e-13)
