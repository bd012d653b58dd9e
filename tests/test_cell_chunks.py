"""Tile passes whose z chunks are one grid cell: objective, gradient and Gauss-Newton product against the FP64 oracle, at
the tolerances of test_gpu_parity.py."""
import pytest

from helpers import gpu_context, oracle_problem, rel, rel_l2, small_phantom, to_dev

from paper_1807_00467_gb300 import phantom

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [((48, 40, 16), (13, 11, 3)),       # two cells of eight planes, two chunks of one
                                 ((28, 16, 16), (8, 5, 3)),         # one tile in x-y
                                 ((40, 24, 24), (11, 7, 4))])       # three cells
def test_one_cell_per_chunk(n, m):
    ph = small_phantom(n, (1.0, 1.1, 1.6), seed=23)
    u, v = phantom.motion_on_grid(ph, m, scale=0.5), phantom.random_grid_field(m, seed=3)
    ctx, P = gpu_context(ph, m, gamma=0.001), oracle_problem(ph, m, gamma=0.001)
    terms, grad = ctx.gn_linearize(to_dev(u))
    ot, og, _ = P.gradient(u)
    assert rel(terms[4], ot[4]) <= 1e-6 and rel(ctx.ngf_objective(to_dev(u))[4], ot[4]) <= 1e-6
    assert rel_l2(grad.cpu().numpy(), og) <= 1e-5
    assert rel_l2(ctx.gn_matvec(to_dev(v)).cpu().numpy(), P.linearize(u).matvec(v)) <= 1e-5
