"""Rounding of the volume-change energy: a uniform stretch has equal bounds, all exact, so every cell's compensated sum
of 64 equal energies errs the same way and nothing averages out."""
import numpy as np
import pytest

from paper_1807_00467_gb300 import api

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


@pytest.mark.parametrize("m", [(9, 5, 5), (90, 71, 40)])      # one and two cells per thread
@pytest.mark.parametrize("k", [203, 325, 318, -115])
def test_uniform_stretch(k, m):
    """psi(d) = dm q with dm = d - 1 (exact) and q = dm / d rounded twice; summed with compensation, each addend is
    rounded once (relative error 2^-24) and the sum adds terms of second order."""
    import torch
    n = tuple(2 * (a - 1) for a in m)
    R = torch.zeros(n[::-1], device="cuda")
    ctx = api.Context(R, R.clone(), (0.5, 0.5, 0.5), m, api.make_params(gamma=1.0), pcg_max=1)      # node spacing 1
    u = torch.zeros((3, m[2], m[1], m[0]), device="cuda")
    u[0] = torch.arange(m[0], device="cuda") * (k / 256.0)
    d = np.float32(1.0 + k / 256.0)
    dm = d - np.float32(1.0)
    q = dm * (np.float32(1.0) / d)
    want = 64.0 * np.float64(dm) * np.float64(q) * (m[0] - 1) * (m[1] - 1) * (m[2] - 1)
    assert abs(float(ctx.ngf_objective(u)[2]) / want - 1.0) <= 1.1 * U
