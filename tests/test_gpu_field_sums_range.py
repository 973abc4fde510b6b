"""GPU test of the weighted field sums at the upper end of the double range: the mean of values whose
plain sum overflows while every weighted term and the mean are finite, against math.fsum of the scaled
field (exact up to its final rounding; 2^-50 of the mean as for smaller fields)."""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(40, 24), (264, 200), (96, 64, 160)])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_mean_of_huge_values(n, sign):
    from paper_2506_02663_gb300 import amr
    X = np.abs(np.random.default_rng(n[0]).standard_normal(n)) + 0.5
    gh = amr.Hierarchy(len(n), n, [[((0,) * len(n), tuple(v - 1 for v in n))]])
    x = torch.from_numpy(gh.pack([[sign * np.ldexp(X, 1018)]])).cuda()
    m = amr.mean_zero(gh, x)
    exact = sign * math.fsum(X.ravel()) / X.size
    assert abs(math.ldexp(m, -1018) - exact) <= 2.0 ** -50 * abs(exact)
