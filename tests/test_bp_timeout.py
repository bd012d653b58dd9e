"""Bounded waits of the belief propagation: when a message never completes the call returns RG_ETIMEOUT, the GPU stays
usable and the next call gives the normal result."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 60])
def test_wait_runs_out(n):
    import torch
    from paper_1807_00467_gb300 import _lib, discrete
    rng = torch.Generator(device="cuda").manual_seed(n)
    D = torch.rand((n, discrete.LABELS), generator=rng, device="cuda")
    kps = torch.randint(0, 60, (n, 3), generator=rng, device="cuda").int()
    inten = torch.zeros(n, device="cuda")
    edges = torch.stack([torch.arange(n - 1), torch.arange(1, n)], dim=1).int().cuda()      # a chain
    want = discrete.bp_marginals(D, kps, inten, edges)
    ws, wp, wb = discrete._scratch(n, "cuda")
    out = torch.empty_like(D)
    args = (n, *(C.c_void_p(t.data_ptr()) for t in (D, kps, inten, edges)), 150.0, 0.2, C.c_void_p(out.data_ptr()),
            C.c_void_p(wp), wb, C.c_void_p(torch.cuda.current_stream().cuda_stream))
    L = _lib.load()
    assert L.kp_bp_marginals_timeout(*args, 1024) == _lib.RG_ETIMEOUT
    assert L.kp_bp_marginals_timeout(*args, 0) == _lib.RG_EINVAL
    assert L.kp_bp_marginals(*args) == _lib.RG_OK
    assert torch.equal(out, want) and torch.equal(discrete.bp_marginals(D, kps, inten, edges), want)
