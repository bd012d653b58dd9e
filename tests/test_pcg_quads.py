"""PCG vector kernels with three quads per thread (311 to 467 thousand quads), over solve lengths on either side of their
groups of two residuals."""
import pytest

from helpers import to_dev

from paper_1807_00467_gb300 import phantom

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("iters", [1, 2, 3, 12])
def test_three_quads_per_thread(iters):
    import torch
    from paper_1807_00467_gb300 import api
    m = (97, 97, 49)                              # 345 780 quads and a tail of three floats
    R = torch.zeros(tuple(k - 1 for k in m[::-1]), device="cuda")
    ctx = api.Context(R, R.clone(), (1.0, 1.0, 1.0), m, api.make_params(alpha=1.0, gamma=0.001), pcg_max=12)
    ctx.gn_linearize(torch.zeros((3, m[2], m[1], m[0]), device="cuda"))
    g = to_dev(phantom.smooth_grid_field(m, seed=8, amp=1.0))
    p, stats = ctx.gn_pcg_solve(g, iters)
    r = (-g - ctx.gn_matvec(p)).double()
    assert float(stats[0]) == float(iters)
    # Galerkin: r . p = 0 in exact arithmetic; FP32 vectors leave about 1e-6 of |r| |p|
    assert abs(float((r * p.double()).sum())) <= 1e-4 * float(r.norm() * p.double().norm())
    assert abs(float(r.norm()) - float(stats[2])) <= 1e-3 * float(stats[1])
    assert torch.equal(p, ctx.gn_pcg_solve(g, iters)[0])
