"""GPU tests of the work-list batch's choice between streamed and tiled legs: batches of a few large
problems (every depth in tiles), of several (the first depth streamed, the next in tiles) and of one
large problem among small ones, each problem against its own captured solve (the two forms of a leg run
the same operations per cell: 1e-13)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(512,), (384, 512, 768), (1024, 64), (1024, 1024), (2048,), (384,) * 14, (512, 96) * 8])
def test_batch_against_single_solves(sizes):
    from paper_2506_02663_gb300 import amr
    p = amr.default_params(rtol=1e-11, max_vcycles=100, precision=amr.MIXED, use_graph=1)
    g = torch.Generator(device="cuda").manual_seed(len(sizes))
    hs, ops, fs = [], [], []
    for k, n in enumerate(sizes):
        gh = amr.Hierarchy(2, (n, n), [[((0, 0), (n - 1, n - 1))]])
        f = torch.zeros(gh.nelems, dtype=torch.float64, device="cuda")
        blk = gh.interior(f, gh.patches[0])
        blk.copy_(torch.randn(blk.shape, dtype=torch.float64, device="cuda", generator=g))
        hs.append(gh)
        ops.append(amr.Operator(gh, 1.0, -1e-5 * (1 + k), [0] * 4))
        fs.append(f)
    xs = [torch.zeros_like(f) for f in fs]
    stats, status = amr.batch_solve(ops, xs, fs, params=p)
    assert all(s == 0 for s in status)
    for op, f, x, s in zip(ops, fs, xs, stats):
        y = torch.zeros_like(f)
        assert op.solve(y, f, params=p)["vcycles"] == s["vcycles"]
        assert float((x - y).abs().max()) <= 1e-13 * float(y.abs().max())
