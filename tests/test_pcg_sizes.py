"""PCG vector kernels by vector length: one cluster (the fused launch, up to 16 blocks of 512 quads) and one quad per
thread beyond it, two and three quads, and the general partition; short solves against the FP64 oracle, with a solve
length that crosses a group of residuals."""
import numpy as np
import pytest

from helpers import gpu_context, oracle_problem, rel_l2, small_phantom, to_dev

from paper_1807_00467_gb300 import phantom

pytestmark = pytest.mark.gpu

CASES = [
    ((32, 32, 24), (9, 9, 7), 11),           # 425 quads: one block, a tail of one float
    ((64, 64, 56), (33, 17, 15), 10),        # 6311 quads: 13 blocks
    ((64, 64, 44), (33, 33, 12), 9),         # 9801 quads: 20 blocks, above a cluster
]


@pytest.mark.parametrize("n,m,iters", CASES)
def test_short_solves_against_oracle(n, m, iters):
    h = (1.0, 1.0, 1.5)
    ph = small_phantom(n, h, seed=31)
    u = phantom.motion_on_grid(ph, m, scale=0.5)
    ctx = gpu_context(ph, m, gamma=0.001)
    _, g = ctx.gn_linearize(to_dev(u))
    p, stats = ctx.gn_pcg_solve(g, iters)
    P = oracle_problem(ph, m, gamma=0.001)
    po, so = P.linearize(u).pcg(P.gradient(u)[1], iters)
    assert stats.cpu().numpy()[0] == so[0] == iters
    assert rel_l2(p.cpu().numpy(), po) <= 1e-4
    q, _ = ctx.gn_pcg_solve(g, iters)
    assert np.array_equal(p.cpu().numpy(), q.cpu().numpy())


@pytest.mark.parametrize("m", [(97, 65, 65), (129, 97, 65), (129, 129, 65)])   # one, two, three and more quads
def test_long_vectors_minimise_in_the_krylov_space(m):
    """Diagonal curvature-only system (flat images): the residual of the solve is orthogonal to its direction."""
    import torch
    from paper_1807_00467_gb300 import api
    n = tuple(k - 1 for k in m)
    R = torch.zeros(n[::-1], device="cuda")
    ctx = api.Context(R, R.clone(), (1.0, 1.0, 1.0), m, api.make_params(alpha=1.0, gamma=0.001), pcg_max=12)
    u = torch.zeros((3, m[2], m[1], m[0]), device="cuda")
    ctx.gn_linearize(u)
    g = to_dev(phantom.smooth_grid_field(m, seed=8, amp=1.0))
    p, stats = ctx.gn_pcg_solve(g, 12)
    r = (-g - ctx.gn_matvec(p)).double()
    assert float(stats[0]) == 12.0
    # Galerkin: r . p = 0 in exact arithmetic; FP32 vectors leave about 1e-6 of |r| |p|
    assert abs(float((r * p.double()).sum())) <= 1e-4 * float(r.norm() * p.double().norm())
    assert abs(float(r.norm()) - float(stats[2])) <= 1e-3 * float(stats[1])
