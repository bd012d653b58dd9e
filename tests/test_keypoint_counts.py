"""Keypoint node sums for every number of keypoints per warp, spread (a few per cell, summed by one lane) and crowded
(summed by the warp): positions and targets are chosen so that every product and sum is exact in FP32."""
import numpy as np
import pytest

import oracle
from helpers import rel_l2, small_phantom, to_dev

from paper_1807_00467_gb300 import api, phantom

pytestmark = pytest.mark.gpu

N, M = (128, 128, 64), (33, 33, 17)


@pytest.mark.parametrize("nk", [1, 33, 1537, 3072, 3073, 6200, 12500, 24600, 50001])      # 1, 1, 1, 1, 4, 8, 16, 32, 32 per warp
def test_node_sums_are_exact(nk):
    import torch
    rng = np.random.default_rng(nk)
    x = rng.integers(0, 4 * (np.array(N) - 1), (nk, 3))
    crowd = rng.random(nk) < 0.1
    x[crowd, :2] = x[crowd, :2] % 64 + 128                 # some of them in 4 x 4 columns of cells,
    x[: min(nk, 150)] = x[: min(nk, 150)] % 16 + 160       # and 150 in one cell
    kx = (x / 4.0).astype(np.float32)
    ky = kx + rng.integers(-3, 4, (nk, 3)).astype(np.float32)
    R = torch.zeros(N[::-1], device="cuda")
    ctx = api.Context(R, R, (1.0, 1.0, 1.0), M, api.make_params(delta=1.0), nk_max=nk, pcg_max=1)
    ctx.set_keypoints(to_dev(kx), to_dev(ky))
    u = np.zeros((3, M[2], M[1], M[0]), np.float32)
    v = np.ones_like(u)
    P = oracle.Problem(np.zeros(N[::-1], np.float32), np.zeros(N[::-1], np.float32), (1.0, 1.0, 1.0), M, delta=1.0,
                       kx=kx.astype(np.float64), ky=ky.astype(np.float64))
    want, wantv = P.keypoints(u)[1], P.keypoints(u, v)[1]
    assert np.array_equal(ctx.regularizer_apply(api.RG_KP, to_dev(u))[1].cpu().numpy().astype(np.float64), want)
    assert np.array_equal(ctx.regularizer_apply(api.RG_KP, to_dev(u), to_dev(v))[1].cpu().numpy().astype(np.float64), wantv)


@pytest.mark.parametrize("nk", [3500, 13000, 30000])      # 4, 16 and 32 per warp
def test_preconditioner_of_many_keypoints(nk):
    """The keypoints' share of the Jacobi diagonal, dominant at delta = 5, through the first PCG step."""
    ph = small_phantom((64, 64, 32), (1.0, 1.0, 2.0), seed=29)
    m, rng = (17, 17, 9), np.random.default_rng(nk)
    kx = rng.uniform(0.0, 1.0, (nk, 3)) * (np.array(ph.n) * np.array(ph.h))
    kx[: nk // 8] = 20.0 + rng.uniform(0.0, 4.0, (nk // 8, 3))
    kx = kx.astype(np.float32)
    ky = (kx + rng.normal(0.0, 2.0, kx.shape)).astype(np.float32)
    import torch
    ctx = api.Context(torch.from_numpy(ph.R).cuda(), torch.from_numpy(ph.T).cuda(), ph.h, m,
                      api.make_params(delta=5.0), nk_max=nk)
    ctx.set_keypoints(to_dev(kx), to_dev(ky))
    P = oracle.Problem(ph.R, ph.T, ph.h, m, alpha=1.0, delta=5.0, kx=kx.astype(np.float64), ky=ky.astype(np.float64))
    u = phantom.motion_on_grid(ph, m, scale=0.5)
    _, g = ctx.gn_linearize(to_dev(u))
    p, _ = ctx.gn_pcg_solve(g, 1)
    po, _ = P.linearize(u).pcg(g.cpu().numpy().astype(np.float64), 1)
    assert rel_l2(p.cpu().numpy(), po) <= 1e-5      # as in test_gpu_parity.py
