"""GPU test of the rounding of the interface ghosts' time derivative.  The four coarse fields differ
little (a large mean plus small changes), so the derivative's weights cancel.  Combining each coarse cell
over time and interpolating the result in space (here in numpy doubles) rounds the large values in
one sum only; the library's value and rate may not be further from extended precision than that
evaluation, up to 1.4 for another order of the folds and multiply-adds."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _window_weights():
    """1-D weights of the two halves of a cell over the averages of five cells (quartic)."""
    A = np.array([[((i + .5) ** (q + 1) - (i - .5) ** (q + 1)) / (q + 1) for q in range(5)] for i in range(-2, 3)])
    return [np.linalg.solve(A.T, [2 * (hi ** (q + 1) - lo ** (q + 1)) / (q + 1) for q in range(5)])
            for lo, hi in ((-.5, 0.), (0., .5))]


def _time_weights(eta, k):
    t = [(1 - i) * k for i in range(4)]  # coarse[i] at t_{-i}, eta counted from t_{-1}
    w = [np.prod([(eta - t[j]) / (t[i] - t[j]) for j in range(4) if j != i]) for i in range(4)]
    d = [sum(np.prod([(eta - t[j]) / (t[i] - t[j]) for j in range(4) if j not in (i, m)]) / (t[i] - t[m])
             for m in range(4) if m != i) for i in range(4)]
    return np.array(w), np.array(d)


def _refine(c, dt):
    """Children of every cell two or more away from the block's edges, axes in turn."""
    W = _window_weights()
    for ax in range(3):
        n = c.shape[ax] - 4
        halves = []
        for w in W:
            parts = [np.take(c, range(q, q + n), ax) * dt(w[q]) for q in range(5)]
            halves.append(sum(parts[1:], parts[0]))
        c = np.stack(halves, ax + 1).reshape(c.shape[:ax] + (2 * n,) + c.shape[ax + 1:])
    return c


def test_rate_of_slowly_changing_fields():
    from paper_2506_02663_gb300 import amr
    n, k = 32, 0.25
    lo, hi = 16, 47
    gh = amr.Hierarchy(3, (n,) * 3, [[((0,) * 3, (n - 1,) * 3)], [((lo,) * 3, (hi,) * 3)]])
    op = amr.Operator(gh, 1.0, -1e-3, [0] * 6)
    rng = np.random.default_rng(3)
    base = 1.0 + rng.random((n,) * 3)
    coarse = []
    for i in range(4):
        per = [[base + 1e-3 * rng.standard_normal((n,) * 3)], [np.zeros((hi - lo + 1,) * 3)]]
        c = torch.from_numpy(gh.pack(per)).cuda()
        coarse.append((c, per[0][0]))
    value, rate = torch.zeros_like(coarse[0][0]), torch.zeros_like(coarse[0][0])
    amr.cic_ghosts(gh, 1, [c for c, _ in coarse], k, 0.5 * k, value, rate)
    p = gh.patches[1]
    sl = slice((lo // 2 - 3), (hi + 1) // 2 + 3)  # the box's coarse cells and three more
    for got, w in zip((value, rate), _time_weights(0.5 * k, k)):
        flat = got.cpu().numpy()[p["offset"]:]
        m = hi - lo + 5
        pad = np.array([[flat[z * p["sz"] + y * p["sy"]:][:m] for y in range(m)] for z in range(m)]).transpose(2, 1, 0)
        ex = _refine(sum(np.longdouble(a) * x[sl, sl, sl].astype(np.longdouble) for a, (_, x) in zip(w, coarse)), np.longdouble)
        parts = [a * x[sl, sl, sl] for a, (_, x) in zip(w, coarse)]
        dbl = _refine(parts[0] + parts[1] + parts[2] + parts[3], float)
        e_got, e_dbl = [], []
        for d in range(3):
            for s in (slice(0, 2), slice(-2, None)):
                at = tuple(s if e == d else slice(2, -2) for e in range(3))
                assert float(np.abs(pad[at] - ex[at]).max()) <= 1e-12 * float(np.abs(ex).max()) + 1e-12
                e_got.append(((pad[at] - ex[at]) ** 2).mean())
                e_dbl.append(((dbl[at] - ex[at]) ** 2).mean())
        assert np.sqrt(np.mean(e_got)) <= 1.4 * np.sqrt(np.mean(e_dbl)), (np.sqrt(np.mean(e_got)), np.sqrt(np.mean(e_dbl)))
