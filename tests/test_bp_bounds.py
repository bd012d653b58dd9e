"""Where the min-convolution of the belief propagation may stop early: unary costs with NaN (a NaN never is a minimum,
so messages carry numbers wherever one is to be had) and a negative coupling, against every candidate in FP64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

S = 33
TOL_E = 1e-5     # of the largest energy, as in test_bp_trees.py


def _message(h, lam):
    out = h.reshape(S, S, S)
    for ax in range(3):
        v = np.moveaxis(out, ax, -1)
        i = np.arange(S)
        cost = lam * (2.0 * (i[:, None] - i[None, :])) ** 2
        out = np.moveaxis(np.fmin.reduce(v[..., None, :] + cost, axis=-1), -1, ax)
    return out.reshape(-1)


def _cases():
    rng = np.random.default_rng(3)
    flat = np.ones((3, S ** 3), np.float32)
    one, plane, line, noisy = flat.copy(), flat.copy(), flat.copy(), (flat + rng.random(flat.shape)).astype(np.float32)
    one[0, 17321] = np.nan
    plane.reshape(3, S, S, S)[1, 4] = np.nan                       # whole lines along x and y
    line.reshape(3, S, S, S)[2, 20, :, 7:30] = np.nan              # holes in rows
    noisy.reshape(-1)[rng.integers(0, noisy.size, 5000)] = np.nan
    inf = flat.copy()
    inf.reshape(3, S, S, S)[0, :16] = np.inf
    return {"one": (one, 0.2), "plane": (plane, 0.2), "line": (line, 0.2), "noisy": (noisy, 0.02), "inf": (inf, 0.2),
            "all": (np.full_like(flat, np.nan), 0.2), "negative": (flat, -6e-8), "negative_noisy": (noisy, -0.01)}


@pytest.mark.parametrize("name", list(_cases()))
def test_marginals_of_a_chain(name):
    import torch
    from paper_1807_00467_gb300 import discrete
    D, alpha = _cases()[name]
    kps = np.array([[0, 0, 0], [10, 0, 0], [20, 0, 0]], np.int32)      # edges of length 10
    edges, lam = np.array([[0, 1], [1, 2]], np.int32), np.float64(np.float32(alpha) / np.float32(10.0))
    D64 = D.astype(np.float64)
    m01, m21 = _message(D64[0], lam), _message(D64[2], lam)
    want = np.stack([D64[0] + _message(D64[1] + m21, lam), D64[1] + m01 + m21, D64[2] + _message(D64[1] + m01, lam)])
    dev = lambda a: torch.from_numpy(a).cuda()   # noqa: E731
    E = discrete.bp_marginals(dev(D), dev(kps), torch.zeros(3, device="cuda"), dev(edges), alpha=alpha).cpu().numpy()
    assert np.array_equal(np.isnan(E), np.isnan(want))
    finite = np.isfinite(want)
    assert np.array_equal(E[~finite & ~np.isnan(want)], want[~finite & ~np.isnan(want)])
    assert np.all(np.abs(E[finite] - want[finite]) <= TOL_E * np.abs(want[finite]).max(initial=1.0))
