"""Folds whose bounds overflow to -inf: their weight is 0 in the gradient and the Gauss-Newton product, whatever their
other factors are, and the objective is +inf."""
import pytest

from paper_1807_00467_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [(9, 5, 5), (90, 71, 40)])      # one and two cells per thread
def test_overflowing_folds_have_no_weight(m):
    import torch
    n = tuple(2 * (a - 1) for a in m)
    R = torch.zeros(n[::-1], device="cuda")
    ctx = api.Context(R, R.clone(), (0.5, 0.5, 0.5), m, api.make_params(gamma=1.0), pcg_max=1)      # node spacing 1
    axes = torch.meshgrid(*(torch.arange(float(k), device="cuda") for k in m[::-1]), indexing="ij")
    u = torch.stack([s * a for s, a in zip((-1e14, 1e14, 1e14), axes[::-1])]).contiguous()           # d = -1e42
    v = torch.stack([1e12 * a for a in axes[::-1]]).contiguous()                                     # grad d . v = -inf
    assert float(ctx.ngf_objective(u)[4]) == float("inf")
    for out in (ctx.regularizer_apply(api.RG_VCC, u)[1], ctx.regularizer_apply(api.RG_VCC, u, v)[1]):
        assert torch.equal(out, torch.zeros_like(out))
