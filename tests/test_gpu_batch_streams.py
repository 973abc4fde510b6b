"""GPU tests of work-list batches whose descriptors change from call to call while the graph is kept:
other fields and other operators of the same sizes, on a side stream (which does not wait for the
default stream), against each problem's own captured solve (same kernels and cycles: 1e-13)."""
import pytest
import torch

pytestmark = pytest.mark.gpu

SIZES = (64, 96, 128, 384, 256, 64)


def _problems(seed, beta):
    from paper_2506_02663_gb300 import amr
    out = []
    g = torch.Generator(device="cuda").manual_seed(seed)
    for k, n in enumerate(SIZES):
        gh = amr.Hierarchy(2, (n, n), [[((0, 0), (n - 1, n - 1))]])
        f = torch.zeros(gh.nelems, dtype=torch.float64, device="cuda")
        blk = gh.interior(f, gh.patches[0])
        blk.copy_(torch.randn(blk.shape, dtype=torch.float64, device="cuda", generator=g))
        out.append((gh, amr.Operator(gh, 1.0, beta * (1 + k), [0] * 4), f))
    return out


@pytest.mark.parametrize("side", [True, False])
def test_alternating_fields_and_operators(side):
    from paper_2506_02663_gb300 import amr
    p = amr.default_params(rtol=1e-12, max_vcycles=100, precision=amr.MIXED, use_graph=1)
    sets = [_problems(1, -1e-4), _problems(2, -3e-4)]
    ref = []
    for probs in sets:
        ref.append([])
        for _, op, f in probs:
            x = torch.zeros_like(f)
            ref[-1].append((x, op.solve(x, f, params=p)["vcycles"]))
    other = [2 * f for _, _, f in sets[0]]  # the first set's operators, fields of their own
    torch.cuda.synchronize()
    st = torch.cuda.Stream() if side else torch.cuda.current_stream()
    with torch.cuda.stream(st):
        for _ in range(4):
            for probs, r in zip(sets, ref):
                xs = [torch.full_like(f, 3.0) for _, _, f in probs]
                stats, status = amr.batch_solve([q[1] for q in probs], xs, [q[2] for q in probs], params=p)
                assert all(s == 0 for s in status)
                for x, s, (y, vc) in zip(xs, stats, r):
                    assert s["vcycles"] == vc
                    assert float((x - y).abs().max()) <= 1e-13 * float(y.abs().max())
            xs = [torch.full_like(f, 3.0) for f in other]
            stats, status = amr.batch_solve([q[1] for q in sets[0]], xs, other, params=p)
            assert all(s == 0 for s in status)
            for x, s, (y, vc) in zip(xs, stats, ref[0]):  # twice the right-hand side: the same cycles, twice the solution
                assert s["vcycles"] == vc
                assert float((x - 2 * y).abs().max()) <= 2e-13 * float(y.abs().max())
    torch.cuda.synchronize()
