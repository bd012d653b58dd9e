"""Spanning tree for intensity scales of either sign: with a negative one an edge may weigh less than its length, or
less than nothing (such weights order by their bit patterns), so no vertex may be passed over for its distance."""
import numpy as np
import pytest

from oracle import discrete as Dq

pytestmark = pytest.mark.gpu


def _kruskal(W):
    n = W.shape[0]
    a, b = np.triu_indices(n, 1)
    key = (W[a, b].view(np.uint32).astype(np.uint64) << np.uint64(32)) | (a.astype(np.uint64) << np.uint64(16)) | b.astype(np.uint64)
    root = np.arange(n)

    def find(v):
        while root[v] != v:
            root[v] = root[root[v]]
            v = root[v]
        return v

    edges = []
    for k in np.argsort(key):
        x, y = find(a[k]), find(b[k])
        if x != y:
            root[x] = y
            edges.append((a[k], b[k]))
    return np.array(sorted(edges))


@pytest.mark.parametrize("sigma", [150.0, -150.0, -5.0])
def test_tree_against_kruskal(sigma):
    import torch
    from paper_1807_00467_gb300 import discrete
    rng = np.random.default_rng(11)
    n = 700                                          # several groups of 256 candidates per vertex
    kps = rng.permutation(60 ** 3)[:n]
    kps = np.stack([kps % 60, kps // 60 % 60, kps // 3600], axis=1).astype(np.int32)
    inten = rng.normal(0.0, 100.0, n).astype(np.float32)
    got = discrete.mst(torch.from_numpy(kps).cuda(), torch.from_numpy(inten).cuda(), sigma_i=sigma).cpu().numpy()
    assert np.array_equal(got, _kruskal(Dq.edge_weights(kps, inten, sigma)))
