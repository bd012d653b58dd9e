"""Bounds whose reciprocals leave the normal range: a positive subnormal bound (finite energy, 1 / d < 2^128) and bounds
above 2^126 (psi' = 1 to rounding), in the one-cell and the two-cell form."""
import numpy as np
import pytest

from paper_1807_00467_gb300 import api

pytestmark = pytest.mark.gpu

U = 2.0 ** -24
SMALL, LARGE = (8, 6, 6), (90, 71, 40)      # one and two cells per thread


def _ctx(m, g):
    import torch
    n = tuple(2 * (a - 1) for a in m)
    R = torch.zeros(n[::-1], device="cuda")
    return api.Context(R, R.clone(), tuple(x / 2.0 for x in g), m, api.make_params(gamma=1.0), pcg_max=1)


def _cut(f):
    return f[:, :SMALL[2] - 1, :SMALL[1] - 1, :SMALL[0] - 1]


def _subnormal(m):
    """Three skew edges of one cell shortened to k^2 2^-46 of their length (k = 5, 3, 3), so that their bound is
    2025 x 2^-138, exactly; no other bound of the field is below 1e-26."""
    import torch
    a = np.array([5.0, 3.0, 3.0]) * 2.0 ** -23
    u = np.zeros((3, m[2], m[1], m[0]), np.float32)
    for c, (x, y, z) in enumerate([(2, 2, 2), (3, 2, 3), (2, 3, 2)]):
        u[c, z, y, x] = 0.5 - a[c]
        u[c, z + (c == 2), y + (c == 1), x + (c == 0)] = -0.5
    return tuple(1.0 / (1.0 + a)), torch.from_numpy(u).cuda()


@pytest.mark.parametrize("m", [SMALL, LARGE])
def test_subnormal_bound(m):
    g, u = _subnormal(m)
    V = float(_ctx(m, g).ngf_objective(u)[2])
    # psi = (d - 1)^2 / d = 1 / d: one rounding of the reciprocal, one of the sum
    assert abs(V / (g[0] * g[1] * g[2] * 2.0 ** 138 / 2025.0) - 1.0) <= 2.0 * U + 1e-10


def _huge(m):
    import torch
    s = 1.25 * 2.0 ** 42                          # d = (1 + s)^3 = 1.95 x 2^126
    axes = torch.meshgrid(*(torch.arange(float(k), device="cuda") for k in m[::-1]), indexing="ij")
    return (1.0, 1.0, 1.0), torch.stack([s * x for x in axes[::-1]]).contiguous()


def test_huge_bounds():
    """psi' = 1 - 1 / d^2 = 1: the gradient of a uniform stretch is that of sum d, and only the outer nodes have one."""
    import torch
    m = SMALL
    g, u = _huge(m)
    grad = _ctx(m, g).regularizer_apply(api.RG_VCC, u)[1].cpu().double()
    s2 = (1.0 + 1.25 * 2.0 ** 42) ** 2
    ends = [torch.tensor([-1.0] + [0.0] * (k - 2) + [1.0], dtype=torch.float64) for k in m[::-1]]
    ones = [torch.tensor([1.0] + [2.0] * (k - 2) + [1.0], dtype=torch.float64) for k in m[::-1]]
    # d d / d u_x at the ends of an x-edge: +-s^2 for each of the 16 bounds of the (up to four) cells around it
    for c, ax in enumerate((2, 1, 0)):
        f = [ends[a] if a == ax else ones[a] for a in range(3)]
        want = 16.0 * s2 * f[0][:, None, None] * f[1][None, :, None] * f[2][None, None, :]
        # 16 equal terms of three roundings each, added plainly (at most 16 partial sums), four cells per node
        assert float((grad[c] - want).abs().max()) <= 32 * U * 64.0 * s2


def test_forms_agree():
    import torch
    for field in (_subnormal, _huge):
        few, big = (_ctx(m, field(m)[0]).regularizer_apply(api.RG_VCC, field(m)[1])[1] for m in (SMALL, LARGE))
        a, b = _cut(few), _cut(big)
        assert torch.equal(torch.isnan(a), torch.isnan(b)) and torch.equal(torch.nan_to_num(a), torch.nan_to_num(b))
