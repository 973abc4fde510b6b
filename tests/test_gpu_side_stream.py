"""GPU tests of first calls on a side stream, which does not wait for the default stream that set-up
copies go to: the first gradient on a fresh hierarchy, and a migration, whose lists are uploaded inside
the call, against the same calls on the default stream (bit for bit)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

BOXES = [[((0, 0, 0), (31, 31, 31))], [((16, 16, 16), (47, 47, 47))]]
MOVED = [[((0, 0, 0), (31, 31, 31))], [((20, 12, 16), (51, 43, 47))]]


def _field(gh, seed):
    rng = np.random.default_rng(seed)
    return torch.from_numpy(gh.pack([[rng.standard_normal([b - a + 1 for a, b in zip(lo, hi)]) for lo, hi in bl]
                                     for bl in gh.boxes])).cuda()


def test_first_gradient():
    from paper_2506_02663_gb300 import amr
    out = []
    for side in (False, True):
        gh = amr.Hierarchy(3, (32, 32, 32), BOXES)
        x = _field(gh, 1)
        grads = [torch.zeros_like(x) for _ in range(3)]
        torch.cuda.synchronize()
        with torch.cuda.stream(torch.cuda.Stream() if side else torch.cuda.current_stream()):
            amr.gradient(gh, [0] * 6, x, grads)
        torch.cuda.synchronize()
        out.append([gh.interior(g, p).clone() for g in grads for p in gh.patches])
    assert all(torch.equal(a, b) for a, b in zip(*out))


def test_migration():
    from paper_2506_02663_gb300 import amr
    out = []
    for side in (False, True):
        old, new = amr.Hierarchy(3, (32, 32, 32), BOXES), amr.Hierarchy(3, (32, 32, 32), MOVED)
        x = _field(old, 2)
        y = torch.zeros(new.nelems, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        with torch.cuda.stream(torch.cuda.Stream() if side else torch.cuda.current_stream()):
            amr.migrate(old, x, new, y)
        torch.cuda.synchronize()
        out.append([new.interior(y, p).clone() for p in new.patches])
    assert all(torch.equal(a, b) for a, b in zip(*out))
