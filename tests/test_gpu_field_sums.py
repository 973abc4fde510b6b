"""GPU tests of the field sums in 128-bit fixed point (mean value of a composite field): against
math.fsum, which is exact up to its final rounding.  A sum of n doubles whose largest is M enters
with an error below n 2^-98 M (the frame keeps 100 bits below M, rows may come in a few frames),
and is then rounded a handful of times (sum, weight, division): 2^-50 of the mean."""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _mean(n, X):
    from paper_2506_02663_gb300 import amr
    gh = amr.Hierarchy(len(n), n, [[((0,) * len(n), tuple(v - 1 for v in n))]])
    x = torch.from_numpy(gh.pack([[X]])).cuda()
    return amr.mean_zero(gh, x), x


# rows shorter than a warp, of whole batches and with remainders; few and many rows per warp
@pytest.mark.parametrize("n", [(8, 8), (40, 24), (256, 32), (264, 200), (24, 16, 8), (96, 64, 160)])
@pytest.mark.parametrize("kind", ["normal", "cancelling", "wide", "growing", "negative", "tiny"])
def test_mean(n, kind):
    rng = np.random.default_rng(len(n) * 100 + n[0] + len(kind))
    X = rng.standard_normal(n)
    if kind == "cancelling":
        h = X.size // 2
        f = X.ravel()
        f[h:2 * h] = -f[:h][::-1]
        f[0] += 1e-12
    elif kind == "wide":
        X *= 2.0 ** rng.integers(-200, 200, n)
    elif kind == "growing":  # every batch of a row needs a new frame
        X *= 2.0 ** np.linspace(-300, 300, X.size).reshape(n)
    elif kind == "negative":
        X = -np.abs(X)
    elif kind == "tiny":
        X *= 1e-310
    m, _ = _mean(n, X)
    exact = math.fsum(X.ravel()) / X.size
    assert abs(m - exact) <= 2.0 ** -50 * abs(exact) + 2.0 ** -98 * float(np.abs(X).max()) + 1e-322  # w s may be subnormal


@pytest.mark.parametrize("bad", [math.nan, math.inf, -math.inf])
def test_non_finite(bad):
    X = np.random.default_rng(1).standard_normal((64, 40))
    X[13, 7] = bad
    assert math.isnan(_mean((64, 40), X)[0])
