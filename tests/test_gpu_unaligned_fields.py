"""GPU test of 2-D calls on fields that start at an odd element of a larger buffer (8-byte aligned only):
the whole-array passes (norm, FP32 copy, update) take their one-element form there, and every result
is that of the aligned fields, bit for bit (adjoint solves, which add atomically: to 1e-9)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _shifted(x):
    y = torch.zeros(x.numel() + 1, dtype=x.dtype, device=x.device)[1:]
    assert y.data_ptr() % 16 == 8
    y.copy_(x)
    return y


@pytest.mark.parametrize("n0,fine", [((40, 36), None), ((64, 64), [((32, 40), (87, 95))]), ((256, 200), [((128, 100), (383, 299))])])
def test_solves_and_residuals(n0, fine):
    from paper_2506_02663_gb300 import amr
    boxes = [[((0, 0), tuple(v - 1 for v in n0))]] + ([fine] if fine else [])
    gh = amr.Hierarchy(2, n0, boxes)
    rng = np.random.default_rng(9)
    f = torch.from_numpy(gh.pack([[rng.standard_normal([b - a + 1 for a, b in zip(lo, hi)]) for lo, hi in bl]
                                  for bl in boxes])).cuda()
    for alpha, beta, bc in ((1.0, -1e-4, [0] * 4), (0.0, 1.0, [1] * 4)):
        op = amr.Operator(gh, alpha, beta, bc)
        runs = []
        for move in (lambda t: t, _shifted):
            g, out, adj = move(f), [], []
            for prec in (0, 1):
                for graph in (0, 1):
                    x = move(torch.zeros_like(f))
                    st = op.solve(x, g, params=amr.default_params(rtol=1e-9, max_vcycles=100, precision=prec, use_graph=graph,
                                                                  cycles_per_refinement=1 + prec))
                    out += [x, torch.tensor([st["final_res"], st["vcycles"]])]
                y = move(torch.zeros_like(f))
                op.solve_transpose(y, g, params=amr.default_params(rtol=1e-9, max_vcycles=100, precision=prec))
                adj.append(y)
            r = move(torch.zeros_like(f))
            out += [torch.tensor(op.residual(out[0], g, r)), r]
            runs.append((out, adj))
        for a, b in zip(runs[0][1], runs[1][1]):
            assert float((a - b).abs().max()) <= 1e-9 * float(a.abs().max())
        for a, b in zip(runs[0][0], runs[1][0]):
            if a.numel() == gh.nelems:
                assert all(torch.equal(gh.interior(a, p), gh.interior(b, p)) for p in gh.patches)
            else:
                assert torch.equal(a, b)
