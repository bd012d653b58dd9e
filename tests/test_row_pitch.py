"""Volumes whose rows are not a multiple of four voxels (the stored linearisation is padded to that, so that the
TMA-fed products take them): linearisation by each pass, products, a short solve and the Jacobi diagonal in it, against
the FP64 oracle."""
import pytest

from helpers import gpu_context, oracle_problem, rel_l2, small_phantom, to_dev

from paper_1807_00467_gb300 import phantom
from paper_1807_00467_gb300._lib import RG_HOOK_PASS

pytestmark = pytest.mark.gpu

CASES = [
    ((70, 40, 24), (36, 21, 13), 1),     # rho (2, 2, 2): one column and a ragged one, by the column pass
    ((90, 36, 20), (46, 19, 6), 2),      # rho (2, 2, 4), by the tile pass
    ((182, 50, 13), (92, 26, 14), 0),    # rho (2, 2, 1), a plane count that is no whole number of ring cycles
    ((38, 24, 20), (20, 13, 11), 0),     # narrower than a column: the tile product
    ((22, 20, 12), (12, 11, 7), 0),      # narrower than its box: plain loads
]


@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("n,m,pass_", CASES)
def test_padded_rows_against_oracle(n, m, pass_, half):
    h = (1.0, 1.2, 1.6)
    ph = small_phantom(n, h, seed=51)
    u = phantom.motion_on_grid(ph, m, scale=0.5)
    ctx = gpu_context(ph, m, gamma=0.001, half=half)
    ctx.debug_hook(RG_HOOK_PASS, pass_)
    P = oracle_problem(ph, m, gamma=0.001, half=half)
    _, g = ctx.gn_linearize(to_dev(u))
    og, lin = P.gradient(u)[1], P.linearize(u)
    assert rel_l2(g.cpu().numpy(), og) <= 1e-5
    v = phantom.random_grid_field(m, seed=9)
    assert rel_l2(ctx.gn_matvec(to_dev(v)).cpu().numpy(), lin.matvec(v)) <= 1e-5
    p, _ = ctx.gn_pcg_solve(g, 5)
    assert rel_l2(p.cpu().numpy(), lin.pcg(og, 5)[0]) <= 1e-4
