"""Reference images that start on an odd element of their buffer: the column-marching passes load voxels in pairs, so
objective, gradient and linearisation take the tile pass there, also where the size or the hook asks for columns."""
import pytest

from helpers import small_phantom, to_dev

from paper_1807_00467_gb300 import phantom
from paper_1807_00467_gb300._lib import RG_HOOK_PASS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("n,m,hook", [((64, 24, 8), (17, 7, 5), 1),            # columns by the hook
                                      ((192, 192, 64), (49, 49, 17), 0)])      # by size: 4 x 11 columns of 62 planes
def test_odd_start(n, m, hook, half):
    import torch
    from paper_1807_00467_gb300 import api
    h = (1.0, 1.1, 1.7)
    ph = small_phantom(n, h, seed=43)
    u, v = to_dev(phantom.motion_on_grid(ph, m, scale=0.5)), to_dev(phantom.random_grid_field(m, seed=4))
    R, T = (torch.from_numpy(x).cuda() for x in (ph.R, ph.T))
    if half:
        R, T = (R + 1024.0).half(), (T + 1024.0).half()

    def results(shift, pas):
        buf = torch.zeros(R.numel() + 2, dtype=R.dtype, device="cuda")
        view = buf[shift:shift + R.numel()].view(R.shape)
        view.copy_(R)
        assert view.data_ptr() % (2 * R.element_size()) == shift * R.element_size()
        ctx = api.Context(view, T, h, m, api.make_params(gamma=0.001))
        ctx.debug_hook(RG_HOOK_PASS, pas)
        terms, grad = ctx.gn_linearize(u)
        return (ctx.ngf_objective(u), terms, grad, ctx.gn_matvec(v)) + tuple(ctx.ngf_gradient(u))

    for a, b in zip(results(1, hook), results(0, 2)):
        assert torch.equal(a, b)
