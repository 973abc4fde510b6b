"""GPU tests of the streamed 2-D legs at sizes that take them (from 768^2 cells below 1024^2, from 1.5
million cells above): one FP32 correction V-cycle of a mixed solve against the same V-cycle with one
launch per sweep (temporal_blocking = 0).  Both run the same linear program in FP32 with sums in
different orders: nine stencil passes and the transfers per level, each rounding at the FP32 unit
times the stencil's gain (at most about 90 next to a Dirichlet face), so the corrections agree to
2e-5 of their largest value."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _streams(lo, hi):
    n = [b - a + 1 for a, b in zip(lo, hi)]
    c = n[0] * n[1]
    return n[0] % 4 == 0 and n[1] % 2 == 0 and min(n) >= 16 and (768 * 768 <= c < 1024 * 1024 or c >= 1500000)


def _cycle(op, f, blk):
    from paper_2506_02663_gb300 import amr
    x = torch.zeros_like(f)
    op.solve(x, f, allow_not_converged=True,
             params=amr.default_params(rtol=1e-30, max_vcycles=1, precision=amr.MIXED, temporal_blocking=blk))
    return x


def _check(n0, boxes, bc, alpha, beta, seed):
    from paper_2506_02663_gb300 import amr
    gh = amr.Hierarchy(2, n0, boxes)
    op = amr.Operator(gh, alpha, beta, bc)
    rng = np.random.default_rng(seed)
    f = torch.from_numpy(gh.pack([[rng.standard_normal([hi[d] - lo[d] + 1 for d in range(2)]) for lo, hi in bl]
                                  for bl in boxes])).cuda()
    got, ref = _cycle(op, f, 1), _cycle(op, f, 0)
    scale = float(ref.abs().max())
    assert np.isfinite(scale) and scale > 0
    for p in gh.patches:
        d = (gh.interior(got, p) - gh.interior(ref, p)).abs().max()
        assert float(d) <= 2e-5 * scale, (p["level"], float(d), scale)


# one strip, a strip and a remainder, many; few chunks of rows and many; extents that end inside a
# strip; the smallest sizes of both ranges
@pytest.mark.parametrize("n0", [(128, 4608), (128, 6144), (192, 4096), (6144, 160), (4608, 128), (768, 768), (992, 608),
                                (608, 992), (928, 736), (1536, 1024), (1216, 1280), (2048, 1536)])
@pytest.mark.parametrize("bc,ab", [([0, 1, 1, 0], (1.0, -1e-3)), ([0, 0, 0, 0], (1.0, -1e-6)), ([1, 0, 0, 1], (0.0, 1.0))])
def test_single_level(n0, bc, ab):
    assert _streams((0, 0), (n0[0] - 1, n0[1] - 1))
    _check(n0, [[((0, 0), (n0[0] - 1, n0[1] - 1))]], bc, *ab, 11)


# boxes whose legs stream: inside the domain, touching faces (physical ghosts on some sides, zero
# coarse-fine ghosts on the others), and a level between two others (its second target)
@pytest.mark.parametrize("fine", [
    [[((264, 256), (1091, 1003))]],
    [[((0, 256), (799, 1055))]],
    [[((480, 480), (1279, 1279))]],
    [[((0, 0), (1279, 1199))]],
    [[((200, 200), (999, 999))], [((800, 780), (1611, 1579))]],
    [[((202, 200), (1001, 1003))], [((806, 780), (1617, 1579))]],
])
def test_refined_levels(fine):
    assert all(_streams(*b) for lev in fine for b in lev)
    _check((640, 640), [[((0, 0), (639, 639))]] + fine, [0, 1, 1, 0], 1.0, -1e-3, 13)
