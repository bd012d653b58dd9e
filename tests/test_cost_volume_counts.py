"""Cost volume by number of keypoints: the kernel of few keypoints (two z labels per CTA) and that of many (seven) give
the same bits, whichever a count takes; keypoints at the edges of the volume among them."""
import numpy as np
import pytest

from oracle import discrete as Dq

pytestmark = pytest.mark.gpu


def test_counts_give_the_same_rows():
    import torch
    from paper_1807_00467_gb300 import discrete
    rng = np.random.default_rng(4)
    shape = (40, 52, 44)
    F, M = (rng.normal(0.0, 200.0, shape).astype(np.float32) for _ in range(2))
    ff, fm = (discrete.features(torch.from_numpy(a).cuda()) for a in (F, M))
    kps = np.stack([rng.integers(0, k, 330) for k in shape[::-1]], axis=1).astype(np.int32)
    kps[:3] = [[0, 0, 0], [43, 51, 39], [22, 26, 20]]
    dev = torch.from_numpy(kps).cuda()
    D = discrete.cost_volume(ff, fm, dev)
    for nk in (1, 3, 100, 303, 304, 329):        # ten waves of five CTAs on 152 SMs from 304 on
        assert torch.equal(discrete.cost_volume(ff, fm, dev[:nk]), D[:nk])
    want = Dq.cost_volume(Dq.ngf_features(F, 10.0), Dq.ngf_features(M, 10.0), kps[:3])
    assert np.abs(D[:3].cpu().numpy() - want).max() <= 2e-6
