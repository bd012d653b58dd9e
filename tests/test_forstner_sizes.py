"""Foerstner detector (Sec. II-C1) at the edges of its blocks: rows shorter and
longer than a 256-voxel block, single voxels per axis, voxel counts that end
inside a word and a chunk, plateaus, non-finite image values."""
import numpy as np
import pytest

from oracle import discrete as Dq

pytestmark = pytest.mark.gpu


def _selected(resp, mask):
    """Keypoints of a response by the definition: positive, not exceeded in the
    window of offsets -3..2, linear index order."""
    n3, n2, n1 = resp.shape
    out = []
    for z, y, x in np.argwhere((resp > 0) & (mask != 0)):
        w = resp[max(0, z - 3):z + 3, max(0, y - 3):y + 3, max(0, x - 3):x + 3]
        if not (w > resp[z, y, x]).any():
            out.append((x, y, z))
    return np.array(out, dtype=np.int32).reshape(-1, 3)


@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 3, 5), (9, 1, 300), (7, 260, 1), (12, 17, 33), (4, 5, 517), (24, 32, 64)])
@pytest.mark.parametrize("masked", [False, True])
def test_response_and_keypoints(shape, masked):
    """Response against the oracle within 1e-12 of its maximum (FP64 on both
    sides, ~100 roundings per value on sums that the determinant subtracts: the
    bound the larger parity test uses); keypoints exactly those of the returned
    response."""
    import torch
    from paper_1807_00467_gb300 import discrete
    g = np.random.default_rng(sum(shape))
    img = (g.integers(-1000, 200, shape)).astype(np.float32)
    mask = (g.random(shape) < 0.6).astype(np.uint8) if masked else None
    k, resp = discrete.forstner(torch.as_tensor(img).cuda(), None if mask is None else torch.as_tensor(mask).cuda(),
                                response=True)
    resp = resp.cpu().numpy()
    Ro = Dq.forstner_response(img)
    assert np.abs(resp - Ro).max() <= 1e-12 * np.abs(Ro).max()
    np.testing.assert_array_equal(k.cpu().numpy(), _selected(resp, np.ones(shape, np.uint8) if mask is None else mask))


def test_plateaus_and_non_finite_values():
    """A periodic image (equal responses in every period: ties are all kept),
    and an image with infinities and NaN (their voxels' responses are not
    positive numbers or not exceeded; the rest as defined)."""
    import torch
    from paper_1807_00467_gb300 import discrete
    z, y, x = np.meshgrid(np.arange(16), np.arange(24), np.arange(48), indexing="ij")
    img = (100.0 * ((x // 2 + y // 2 + z // 2) % 2) + 30.0 * (x % 4)).astype(np.float32)
    bad = img.copy()
    bad[5, 6, 7], bad[8, 20, 40], bad[12, 3, 30] = np.inf, np.nan, -np.inf
    for im in (img, bad, np.full_like(img, 7.0)):
        k, resp = discrete.forstner(torch.as_tensor(im).cuda(), response=True)
        resp = resp.cpu().numpy()
        np.testing.assert_array_equal(k.cpu().numpy(), _selected(resp, np.ones(resp.shape, np.uint8)))
