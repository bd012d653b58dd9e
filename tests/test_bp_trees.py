"""Belief propagation on trees of every shape and coupling (kp_bp_marginals): chains, stars and random trees, from a
coupling of zero (every label distance counts) to one that ties neighbours to equal labels, against the FP64 oracle;
and a tree too large for the shared-memory sweeps, in closed form."""
import numpy as np
import pytest

from oracle import discrete as Dq

pytestmark = pytest.mark.gpu

TOL_E = 1e-5     # of the largest energy of a keypoint, as in test_discrete_gpu.py


def _dev(a, dtype=None):
    import torch
    t = torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")
    return t if dtype is None else t.to(dtype)


def _edges(kind, n, rng):
    if kind == "chain":
        e = [(i, i + 1) for i in range(n - 1)]
    elif kind == "star":
        e = [(n // 2, i) for i in range(n) if i != n // 2]
    else:
        e = [(int(rng.integers(0, i)), i) for i in range(1, n)]
    return np.array(sorted((min(a, b), max(a, b)) for a, b in e), dtype=np.int32)


@pytest.mark.parametrize("kind", ["chain", "star", "random"])
@pytest.mark.parametrize("alpha,spread", [(0.0, 1.0), (0.2, 1.0), (0.02, 200.0), (50.0, 20.0)])
def test_marginals_on_tree(kind, alpha, spread):
    import torch
    from paper_1807_00467_gb300 import discrete
    rng = np.random.default_rng(5)
    n = 2 if alpha == 50.0 and kind == "chain" else 17
    kps = rng.integers(0, 60, size=(n, 3))
    kps[1] = kps[0]                                   # an edge of zero length: lambda = inf (or 0 * inf for alpha = 0)
    if alpha == 0.0:
        kps[1] += 1
    inten = np.full(n, -850.0, np.float32)
    D = (spread * rng.random((n, Dq.N_STEPS ** 3))).astype(np.float32)
    e = _edges(kind, n, rng)
    with np.errstate(divide="ignore"):
        W = Dq.edge_weights(kps, inten)
        Eo = Dq.bp_marginals(D.astype(np.float64), e, W, alpha)
    E = discrete.bp_marginals(_dev(D), _dev(kps).int(), _dev(inten), _dev(e), alpha=alpha)
    assert torch.equal(E, discrete.bp_marginals(_dev(D), _dev(kps).int(), _dev(inten), _dev(e), alpha=alpha))
    err = np.abs(E.cpu().numpy() - Eo).max(axis=1)
    assert np.all(err <= TOL_E * np.abs(Eo).max(axis=1))


@pytest.mark.parametrize("n", [13000, 13001])
def test_large_tree_closed_form(n):
    """Equal unary costs of 1: every marginal is the number of keypoints, exactly; the tree from kp_mst."""
    import torch
    from paper_1807_00467_gb300 import discrete
    rng = np.random.default_rng(2)
    kps = _dev(rng.integers(0, 400, size=(n, 3))).int()
    inten = _dev(rng.normal(0.0, 50.0, n).astype(np.float32))
    e = discrete.mst(kps, inten)
    E = discrete.bp_marginals(torch.ones((n, Dq.N_STEPS ** 3), device="cuda"), kps, inten, e)
    assert bool((E == float(n)).all())
