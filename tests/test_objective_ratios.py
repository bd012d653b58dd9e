"""Objective pass in columns (csrc/ngf_gobj.cu) with one voxel per cell along z, and along y and z: every plane starts a
cell, so the node ring is refilled in each step.  The bits tell it from the tile pass, so neither case is the tile pass
compared with itself."""
import pytest

from helpers import gpu_context, oracle_problem, rel, small_phantom, to_dev

from paper_1807_00467_gb300 import phantom
from paper_1807_00467_gb300._lib import RG_HOOK_PASS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("n,m", [((128, 40, 12), (65, 21, 13)),      # cells of 2 x 2 x 1 voxels: 33 x 11 staged nodes
                                 ((128, 38, 23), (33, 39, 24)),      # 4 x 1 x 1: 18 x 21
                                 ((64, 20, 4), (17, 6, 5))])         # 4 x 4 x 1, two planes of D
def test_objective_against_oracle_and_tile_pass(n, m, half):
    ph = small_phantom(n, (1.0, 1.1, 1.7), seed=47)
    ctx, P = gpu_context(ph, m, half=half), oracle_problem(ph, m, half=half)
    same_bits = []
    for scale in (0.2, 0.4, 0.6, 0.8):
        u = phantom.motion_on_grid(ph, m, scale=scale)
        ctx.debug_hook(RG_HOOK_PASS, 1)
        J = float(ctx.ngf_objective(to_dev(u))[0])
        assert rel(J, P.objective(u)[0][0]) <= 1e-6
        ctx.debug_hook(RG_HOOK_PASS, 2)
        tile = float(ctx.ngf_objective(to_dev(u))[0])
        assert rel(J, tile) <= 1e-7
        same_bits.append(J == tile)
    assert not all(same_bits)


def test_thin_slab_takes_columns():
    """A slab of few planes with a column per SM: the pass chosen by size is the column pass (its bits)."""
    import torch
    from paper_1807_00467_gb300 import api
    n, m = (512, 512, 8), (129, 129, 5)
    g = torch.Generator(device="cuda").manual_seed(3)
    R, T = (200.0 * torch.rand(n[::-1], generator=g, device="cuda") for _ in range(2))
    ctx = api.Context(R, T, (1.0, 1.0, 2.0), m, api.make_params(), pcg_max=1)
    u = to_dev(phantom.random_grid_field(m, seed=9))
    J = {}
    for hook in (0, 1, 2):
        ctx.debug_hook(RG_HOOK_PASS, hook)
        J[hook] = float(ctx.ngf_objective(u)[0])
    assert J[0] == J[1] and rel(J[1], J[2]) <= 1e-7 and J[1] != J[2]
