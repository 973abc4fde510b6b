"""GPU test of the FP64 residual of a 2-D level where the field is small: a field of size 1e-8 with one
tall peak elsewhere.  Every cell's residual f - (alpha x + beta L x) has to be exact up to the rounding
of its own terms (16 units in the last place of their absolute sum: five additions per neighbour
sum, the combination, two products, two sums), whatever values stand far away."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n0", [(1024, 1024), (2048, 1024), (4096, 640)])
@pytest.mark.parametrize("ab", [(1.0, -1e-6), (0.0, 1.0)])
def test_small_values_keep_their_digits(n0, ab):
    from paper_2506_02663_gb300 import amr
    gh = amr.Hierarchy(2, n0, [[((0, 0), (n0[0] - 1, n0[1] - 1))]])
    op = amr.Operator(gh, *ab, [0, 1, 1, 0])
    rng = np.random.default_rng(6)
    X, F = 1e-8 * rng.standard_normal(n0), 1e-8 * rng.standard_normal(n0)
    X[300, 200] = 1.0
    x, f = (torch.from_numpy(gh.pack([[a]])).cuda() for a in (X, F))
    r = torch.zeros_like(f)
    op.residual(x, f, r)
    got = gh.unpack(r.cpu().numpy())[0][0]
    inv = n0[0] ** 2 / np.longdouble(12)

    def sums(a):
        def at(d, k):
            s = [slice(2, -2), slice(2, -2)]
            s[d] = slice(2 + k, n0[d] - 2 + k)
            return a[tuple(s)]
        return at(0, -1) + at(0, 1) + at(1, -1) + at(1, 1), at(0, -2) + at(0, 2) + at(1, -2) + at(1, 2), at(0, 0)

    s1, s2, c = sums(X.astype(np.longdouble))
    a1, a2, ac = sums(np.abs(X))
    alpha, beta = (np.longdouble(v) for v in ab)
    inner = (slice(2, -2), slice(2, -2))
    exact = F[inner] - (alpha * c + beta * inv * (16 * s1 - s2 - 60 * c))
    scale = np.abs(F[inner]) + abs(ab[0]) * ac + abs(ab[1]) * float(inv) * (16 * a1 + a2 + 60 * ac)
    err = np.abs((got[inner] - exact).astype(float))
    assert float((err / scale).max()) <= 16 * 2.0 ** -53
