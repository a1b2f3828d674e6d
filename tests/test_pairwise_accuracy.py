"""Each pair of boys_pairwise on 36 <= X < 64, where the asymptotic form is exact and
what is left is rounding.

Derivation, in units of 2^-53 sum_l |c_l| F_l(X): the values of F_l at the interval's
edge are doubles (1); the partial sums of the leading coefficient, from the highest
order down, add sum_m (m + 1) |c_m| F_m (below 1.1 here, the orders fall off by at
least X / (l + 1/2)); the next coefficients, rounded likewise, weigh at most 1/16 (0.15 in
all); truncation of the expansion 0.5; units of the Horner sum 0.25; X in units of 2^-56
against the rounded x_i + x_j 0.5; the cut to a double 2.  5.5 in all; the bound is 8.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2512_10059_gb300 as pb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("positive", [True, False])
@pytest.mark.parametrize("k", [0, 4, 12, 32])
def test_pairs_in_the_asymptotic_range(k, positive):
    x = np.linspace(18.0, 31.999, 2000)
    xt = torch.from_numpy(x).to("cuda:0")
    for seed in range(3):
        c = np.random.default_rng(10 * k + seed).standard_normal(k + 1)
        c = np.abs(c) if positive else c
        ct = torch.from_numpy(c).to("cuda:0")
        for j in (0, 700, 1999):
            y = torch.zeros_like(xt)
            y[j] = 1.0
            w = pb.boys_pairwise(xt, y, ct).cpu().numpy()
            f = np.stack(oracle.boys(x + x[j], k)).astype(np.longdouble).sum(0)
            ref, size = (f * c[:, None]).sum(0), (f * np.abs(c)[:, None]).sum(0)
            assert np.max(np.abs((w - ref) / size)) <= 2.0 ** -50
