"""GPU tests of the streamed 2-D legs (one warp per 128-column strip, four sweeps per pass): one
FP32 correction V-cycle of a mixed solve against the same V-cycle with one launch per sweep
(temporal_blocking = 0), on grids large enough to take them.  Both run the same linear program
in FP32 with sums in different orders: nine stencil passes and the transfers, each rounding at
the FP32 unit times the stencil's gain (at most about 90 next to a Dirichlet face), so the
corrections agree to 2e-5 of their largest value."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


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


# one strip, a strip and a remainder, many; a few chunks of rows and many; extents that end
# inside a strip; every face type
@pytest.mark.parametrize("n0", [(512, 512), (608, 448), (448, 608), (64, 4096), (4096, 64), (128, 2048), (2048, 320)])
@pytest.mark.parametrize("bc,ab", [([0, 1, 1, 0], (1.0, -1e-3)), ([1, 1, 1, 1], (0.0, 1.0)), ([0, 0, 0, 0], (1.0, -1e-6))])
def test_single_level(n0, bc, ab):
    _check(n0, [[((0, 0), (n0[0] - 1, n0[1] - 1))]], bc, *ab, 11)


# boxes whose legs stream: inside the domain, touching faces (physical ghosts on some sides, zero
# coarse-fine ghosts on the others), and a level between two others (its second target)
@pytest.mark.parametrize("fine", [
    [[((264, 256), (791, 803))]],
    [[((0, 256), (527, 803))]],
    [[((496, 484), (1023, 1023))]],
    [[((200, 200), (823, 827))], [((800, 780), (1327, 1311))]],
])
def test_refined_levels(fine):
    _check((512, 512), [[((0, 0), (511, 511))]] + fine, [0, 1, 1, 0], 1.0, -1e-3, 13)
