"""Volume-change kernels (csrc/vcc.cu): the two-cells-per-thread form taken on large grids gives the bits of the
one-cell form on a corner of the same field; folds and NaN make the objective +inf in both."""
import pytest

from helpers import to_dev

from paper_1807_00467_gb300 import api, phantom

pytestmark = pytest.mark.gpu


def _ctx(m, gamma=1.0):
    import torch
    n = tuple(max(4, 2 * (k - 1)) for k in m)
    R = torch.zeros(n[::-1], device="cuda")
    return api.Context(R, R.clone(), (1.0, 1.2, 1.5), m, api.make_params(gamma=gamma), pcg_max=1)


@pytest.mark.parametrize("small", [(9, 5, 5), (17, 18, 11), (20, 35, 30)])
def test_forms_give_the_same_bits(small):
    """A node below the corner grid's last one per axis has all its cells in both grids (4 x 152 blocks of 8 x 4 x 4
    cells separate the forms; 90 x 71 x 40 nodes are 2160 ragged blocks)."""
    import torch
    m = (90, 71, 40)
    u, v = (to_dev(s * phantom.random_grid_field(m, seed=k)) for k, s in ((6, 0.1), (5, 1.0)))
    cut = lambda f, d=0: f[:, :small[2] - d, :small[1] - d, :small[0] - d].contiguous()   # noqa: E731
    big, few = _ctx(m), _ctx(small)
    for args in ((u,), (u, v)):
        whole = big.regularizer_apply(api.RG_VCC, *args)[1]
        part = few.regularizer_apply(api.RG_VCC, *(cut(x) for x in args))[1]
        assert torch.equal(cut(whole, 1), cut(part, 1))


@pytest.mark.parametrize("m", [(17, 18, 11), (90, 71, 40)])
def test_fold_and_nan_are_infinite(m):
    import torch
    ctx = _ctx(m)
    u = torch.zeros((3, m[2], m[1], m[0]), device="cuda")
    for bad in (float("nan"), 100.0):        # one displaced node: NaN bounds, or negative ones
        w = u.clone()
        w[0, m[2] - 1, m[1] - 1, 0] = bad
        assert bool(torch.isinf(ctx.ngf_objective(w)[4]))
    assert float(ctx.ngf_objective(u)[2]) == 0.0
