"""GPU test of stacked component batches (one replica of a 3-D hierarchy per problem): the replicas
run the kernels of the problems' own solves, coarse end included, so the V-cycle counts and every bit
of the solutions are those of the separate solves."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n0,fine", [((32, 32, 32), [((16, 20, 24), (39, 43, 47))]), ((40, 36, 44), [((20, 16, 24), (51, 47, 63))]),
                                     ((64, 64, 64), [((48, 48, 48), (79, 79, 79))]), ((48, 32, 40), None)])
def test_stacked_solves_equal_separate_ones(precision, n0, fine):
    from paper_2506_02663_gb300 import amr
    boxes = [[((0, 0, 0), tuple(v - 1 for v in n0))]] + ([fine] if fine else [])
    p = amr.default_params(rtol=1e-10, max_vcycles=100, precision=precision, use_graph=1)
    g = torch.Generator(device="cuda").manual_seed(n0[1])
    ghs, ops, fs, ref = [], [], [], []
    for _ in range(3):
        gh = amr.Hierarchy(3, n0, boxes)
        op = amr.Operator(gh, 1.0, -1e-4, [0] * 6)
        f = torch.zeros(gh.nelems, dtype=torch.float64, device="cuda")
        for q in gh.patches:
            blk = gh.interior(f, q)
            blk.copy_(torch.randn(blk.shape, dtype=torch.float64, device="cuda", generator=g))
        x = torch.zeros_like(f)
        ref.append((x, op.solve(x, f, params=p)["vcycles"]))
        ghs.append(gh)
        ops.append(op)
        fs.append(f)
    amr.set_stacked_batches(1)
    try:
        phis = [torch.zeros_like(f) for f in fs]
        stats, status = amr.batch_solve(ops, phis, fs, params=p)
    finally:
        amr.set_stacked_batches(0)
    assert all(s == 0 for s in status)
    for gh, x, s, (y, vc) in zip(ghs, phis, stats, ref):
        assert s["vcycles"] == vc
        for q in gh.patches:
            assert torch.equal(gh.interior(x, q), gh.interior(y, q)), q["level"]
