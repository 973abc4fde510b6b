"""GPU tests of the streamed 2-D legs on refined levels: one FP32 correction V-cycle of a mixed solve
against the same V-cycle with one launch per sweep (temporal_blocking = 0).  Both run the same
linear program in FP32 with sums in different orders: nine stencil passes and the transfers per
level, each rounding at the FP32 unit times the stencil's gain (at most about 90 next to a
Dirichlet face), so the corrections agree to 2e-5 of their largest value."""
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


# a box that starts on an odd coarse column: a lane's two coarse cells straddle an 8-byte boundary
@pytest.mark.parametrize("lo", [(202, 200), (206, 202)])
def test_odd_coarse_column(lo):
    box = (lo, (lo[0] + 999, lo[1] + 799))
    _check((640, 640), [[((0, 0), (639, 639))], [box]], [0, 1, 1, 0], 1.0, -1e-3, 17)
