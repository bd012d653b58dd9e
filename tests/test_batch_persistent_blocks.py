"""The persistent batched PCG runs several volume-change cell blocks one after the other on one shared scratch: with
the volume-change term on and enough cells for every group of threads to take four blocks in a row, repeated solves
keep the bits of the level graph's launches."""
import pytest

from paper_1807_00467_gb300 import batch, phantom

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gamma", [1.0, 0.0])
def test_repeated_solves_keep_the_bits(gamma):
    import torch
    from paper_1807_00467_gb300 import api
    ph = phantom.make_phantom((128, 96, 32), (1.2, 1.2, 2.5), seed=9, motion="small", n_vessels=12)
    R, T = torch.from_numpy(ph.R).cuda(), torch.from_numpy(ph.T).cuda()
    # 64 x 48 x 32 cells of two voxels along x and y, one plane each: 8 x 12 x 8 = 768 blocks of 8 x 4 x 4 cells,
    # and 136 ragged ones of the small volume
    pairs = batch.crop_pairs(R, T, ph.h, [(128, 96, 32), (72, 40, 24)])
    pairs = [(a, b, h, (a.shape[2] // 2 + 1, a.shape[1] // 2 + 1, a.shape[0] + 1)) for a, b, h, _ in pairs]
    params = api.make_params(eta=10.0, alpha=1.0, gamma=gamma)
    sched = dict(levels=1, gn_iters=1, pcg_iters=12)
    want = batch.register_batch_graph(pairs, params, **sched)[0]
    assert all(float(u.abs().max()) > 0.01 for u in want)
    for _ in range(20):
        got = batch.register_batch_graph(pairs, params, persistent=True, **sched)[0]
        assert all(torch.equal(a, b) for a, b in zip(want, got))
