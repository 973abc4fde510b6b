"""GPU test of the rounding of A x and f - A x on 3-D levels of any shape (FP64, Helmholtz with a small
beta, where alpha x carries the result).  L x is a sum of the cell and its neighbours of relative
error 8 u (three additions per neighbour sum, two combinations, the coefficient and its product;
u = 2^-53) of its terms' absolute sum, alpha x + beta L x is rounded once, f minus it once:
|error| <= u |A x| + u |f - A x| + 8 u |beta| / (12 h^2) (16 sum|x1| + sum|x2| + 90 |x|).  A sweep
x + w (f - A x) multiplies that by w and rounds once more."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n0", [(40, 36, 44), (72, 72, 72), (56, 48, 40), (144, 160, 144)])
def test_helmholtz_rounding(n0):
    from paper_2506_02663_gb300 import amr
    alpha, beta, u = 1.0, -1e-8, 2.0 ** -53
    gh = amr.Hierarchy(3, n0, [[((0, 0, 0), tuple(v - 1 for v in n0))]])
    op = amr.Operator(gh, alpha, beta, [0] * 6)
    rng = np.random.default_rng(8)
    X, F = rng.standard_normal(n0), rng.standard_normal(n0)
    x, f = (torch.from_numpy(gh.pack([[a]])).cuda() for a in (X, F))
    outs = [torch.zeros_like(f) for _ in range(3)]
    op.apply(x, outs[0])
    op.apply_transpose(x, outs[1])
    op.residual(x, f, outs[2])
    ones, zero = torch.ones_like(f), torch.zeros_like(f)
    op.smooth(0, 1, 2.0 / 3.0, zero, ones)  # from x = 0 with f = 1: the factor w itself
    w = float(gh.unpack(zero.cpu().numpy())[0][0][tuple(v // 2 for v in n0)])
    y = x.clone()
    op.smooth(0, 1, 2.0 / 3.0, y, f)
    ax, atx, res, swept = (gh.unpack(o.cpu().numpy())[0][0] for o in (*outs, y))

    def sums(a, m):
        def at(d, k):
            s = [slice(m, -m)] * 3
            s[d] = slice(m + k, n0[d] - m + k)
            return a[tuple(s)]
        return sum(at(d, k) for d in range(3) for k in (-1, 1)), sum(at(d, k) for d in range(3) for k in (-2, 2)), at(0, 0)

    for m, got, kind in ((2, ax, 0), (4, atx, 0), (2, res, 1), (2, swept, 2)):  # m: cells from the faces
        inner = (slice(m, -m),) * 3
        s1, s2, c = sums(X.astype(np.longdouble), m)
        a1, a2, ac = sums(np.abs(X), m)
        inv = np.longdouble(n0[0]) ** 2 / 12
        exact = np.longdouble(alpha) * c + np.longdouble(beta) * inv * (16 * s1 - s2 - 90 * c)
        bound = u * np.abs(exact) + 8 * u * abs(beta) * float(inv) * (16 * a1 + a2 + 90 * ac)
        if kind >= 1:
            exact = F[inner] - exact
            bound = bound + u * np.abs(exact)
        if kind == 2:
            exact = X[inner] + np.longdouble(w) * exact
            bound = w * bound + u * np.abs(exact)
        assert float((np.abs(got[inner] - exact) / bound).max()) <= 1.0, (m, kind)
