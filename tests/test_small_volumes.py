"""Volumes with few x-y tiles, whose tile passes split z into short chunks (down to one grid cell, with a ragged
last one): objective, gradient and Gauss-Newton product against the FP64 oracle, at the tolerances of
test_gpu_parity.py."""
import numpy as np
import pytest

from helpers import gpu_context, oracle_problem, rel, rel_l2, small_phantom, to_dev

from paper_1807_00467_gb300 import phantom

pytestmark = pytest.mark.gpu

CASES = [
    ((64, 64, 48), (1.0, 1.0, 2.5), (17, 17, 13)),     # chunks of one cell of four planes
    ((32, 24, 20), (1.0, 1.0, 2.0), (17, 13, 21)),     # one-plane cells: chunks of one plane
    ((48, 40, 56), (1.1, 0.9, 1.5), (13, 11, 8)),      # eight-plane cells
    ((60, 36, 46), (1.0, 1.0, 2.0), (31, 19, 24)),     # two-plane cells, ragged last chunk
]


@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("n,h,m", CASES)
def test_short_chunks_against_oracle(n, h, m, half):
    ph = small_phantom(n, h, seed=21)
    u = phantom.motion_on_grid(ph, m, scale=0.5)
    v = phantom.random_grid_field(m, seed=3)
    ctx = gpu_context(ph, m, gamma=0.001, half=half)
    P = oracle_problem(ph, m, gamma=0.001, half=half)
    terms, grad = ctx.gn_linearize(to_dev(u))
    ot, og, _ = P.gradient(u)
    assert rel(terms[4], ot[4]) <= 1e-6
    assert rel(ctx.ngf_objective(to_dev(u))[4], ot[4]) <= 1e-6
    assert rel_l2(grad.cpu().numpy(), og) <= 1e-5
    assert rel_l2(ctx.gn_matvec(to_dev(v)).cpu().numpy(), P.linearize(u).matvec(v)) <= 1e-5
    assert np.isfinite(grad.cpu().numpy()).all()
