"""Objective pass in 62 x 18 columns dealt plane by plane to the SMs (csrc/ngf_gobj.cu): extents at the edges of its
columns, cell ratios in every phase of a column's origin, few planes and many, against the FP64 oracle and the tile
pass; exactly zero for identical images."""
import pytest

from helpers import gpu_context, oracle_problem, rel, small_phantom, to_dev

from paper_1807_00467_gb300 import phantom
from paper_1807_00467_gb300._lib import RG_HOOK_PASS

pytestmark = pytest.mark.gpu

CASES = [
    ((64, 20, 4), (17, 6, 2)),        # one column, two planes of D, fewer pieces than SMs
    ((126, 38, 12), (64, 39, 13)),    # interior 124 x 36: exactly two columns each way; rho (2, 1, 1)
    ((128, 40, 24), (17, 11, 4)),     # two voxels more; rho (8, 4, 8)
    ((192, 56, 44), (49, 8, 23)),     # four columns in x, rho (4, 8, 2)
    ((250, 76, 66), (126, 39, 34)),   # odd multiples, rho (2, 2, 2)
]


@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("n,m", CASES)
def test_objective_against_oracle_and_tile_pass(n, m, half):
    h = (1.0, 1.1, 1.7)
    ph = small_phantom(n, h, seed=41)
    u = phantom.motion_on_grid(ph, m, scale=0.6)
    ctx = gpu_context(ph, m, half=half)
    ctx.debug_hook(RG_HOOK_PASS, 1)
    J = ctx.ngf_objective(to_dev(u))
    assert rel(J[0], oracle_problem(ph, m, half=half).objective(u)[0][0]) <= 1e-6
    ctx.debug_hook(RG_HOOK_PASS, 2)
    assert rel(J[0], ctx.ngf_objective(to_dev(u))[0]) <= 1e-7
    ctx.debug_hook(RG_HOOK_PASS, 1)
    far = to_dev(u) + 1000.0          # every sample beyond the volume: all clamped
    a = ctx.ngf_objective(far)
    ctx.debug_hook(RG_HOOK_PASS, 2)
    assert rel(a[0], ctx.ngf_objective(far)[0]) <= 1e-7
    same = gpu_context(phantom.Phantom(R=ph.R, T=ph.R, n=ph.n, h=ph.h, amps=ph.amps, centres=ph.centres), m, half=half)
    same.debug_hook(RG_HOOK_PASS, 1)
    assert float(same.ngf_objective(to_dev(u) * 0.0)[0]) == 0.0
