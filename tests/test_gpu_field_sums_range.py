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


@pytest.mark.parametrize("n", [(64, 40), (264, 200), (96, 64, 160)])
def test_small_terms_between_cancelling_ones(n):
    """Values of size one that cancel in pairs, and as many of size 2^-60 between them: the sum keeps the
    small values' digits (a block has at most 2^12 terms here: bits down to 2^-114 of the largest
    value enter; the sum of the small ones and their count differ by less than 2^10)."""
    from paper_2506_02663_gb300 import amr
    rng = np.random.default_rng(n[0] + 1)
    f = np.ldexp(np.abs(rng.standard_normal(math.prod(n))) + 0.5, -60)
    big = rng.standard_normal(f.size // 4)
    at = rng.permutation(f.size)[:2 * big.size]
    f[at] = np.concatenate([big, -big])
    gh = amr.Hierarchy(len(n), n, [[((0,) * len(n), tuple(v - 1 for v in n))]])
    x = torch.from_numpy(gh.pack([[f.reshape(n)]])).cuda()
    exact = math.fsum(f) / f.size
    assert abs(amr.mean_zero(gh, x) - exact) <= 2.0 ** -50 * abs(exact)
