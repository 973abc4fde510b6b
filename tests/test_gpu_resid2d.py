"""GPU tests of the 2-D FP64 residual with exact fixed-point stencil sums (levels that are the
whole domain): against the plain FP64 kernel of the same operator (amr_set_fx_residual(0)).
The stencil sum is exact and every |x| is rounded once to 2^-56 of the frame, so with ghost
values of at most 50 times the interior's both differ from the exact residual by no more than
1e-13 of the operator's scale, and from one another by twice that."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture
def fx():
    from paper_2506_02663_gb300 import amr
    yield amr.set_fx_residual
    amr.set_fx_residual(1)


def _both(fx, op, x, f):
    out = []
    for on in (1, 0):
        fx(on)
        r = torch.zeros_like(f)
        op.residual(x, f, r)
        out.append(r)
    return out


# strips of 120 columns: whole, with a remainder, narrower than one; few chunks of rows and many
@pytest.mark.parametrize("n0", [(2048, 1024), (1536, 1408), (1920, 1152), (256, 8192), (8192, 256)])
@pytest.mark.parametrize("bc,ab", [([0, 1, 1, 0], (1.0, -1e-3)), ([1, 1, 1, 1], (0.0, 1.0)), ([1, 0, 0, 0], (1.0, -1e-6))])
def test_against_plain(fx, n0, bc, ab):
    from paper_2506_02663_gb300 import amr
    gh = amr.Hierarchy(2, n0, [[((0, 0), (n0[0] - 1, n0[1] - 1))]])
    op = amr.Operator(gh, *ab, bc)
    rng = np.random.default_rng(3)
    h = 1.0 / n0[0]
    for X in (rng.standard_normal(n0),
              np.sin(3 * (np.arange(n0[0]) + 0.5) / n0[0])[:, None] * np.cos(5 * (np.arange(n0[1]) + 0.5) / n0[1])[None, :],
              np.zeros(n0), np.full(n0, 1e-310)):
        x = torch.from_numpy(gh.pack([[X]])).cuda()
        f = torch.from_numpy(gh.pack([[rng.standard_normal(n0)]])).cuda()
        a, b = _both(fx, op, x, f)
        p = gh.patches[0]
        # alpha x + beta L x: the two-layer ghosts enter with up to 50 times the interior's size
        scale = float(f.abs().max()) + float(x.abs().max()) * (abs(ab[0]) + abs(ab[1]) * 128 / (12 * h * h) * 50)
        d = (gh.interior(a, p) - gh.interior(b, p)).abs().max()
        assert float(d) <= 2e-13 * scale, float(d) / scale
        if not X.any():
            assert torch.equal(a, b)


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_takes_the_plain_form(fx, bad):
    from paper_2506_02663_gb300 import amr
    n0 = (2048, 1024)
    gh = amr.Hierarchy(2, n0, [[((0, 0), (n0[0] - 1, n0[1] - 1))]])
    op = amr.Operator(gh, 1.0, -1e-3, [0, 1, 1, 0])
    rng = np.random.default_rng(4)
    X = rng.standard_normal(n0)
    X[7, 300] = bad
    x = torch.from_numpy(gh.pack([[X]])).cuda()
    f = torch.from_numpy(gh.pack([[rng.standard_normal(n0)]])).cuda()
    a, b = (t.cpu().numpy() for t in _both(fx, op, x, f))
    assert not np.isfinite(a).all()
    np.testing.assert_array_equal(np.isnan(a), np.isnan(b))
    np.testing.assert_array_equal(np.isinf(a), np.isinf(b))
    ok = np.isfinite(a)
    assert np.abs(a[ok] - b[ok]).max() <= 2e-13 * np.abs(b[ok]).max() * 50
