"""The link force where device memory is short: its smaller forms give the same bits,
and a context gives its workspace back when another allocation needs the memory."""
import numpy as np
import pytest

from paper_2004_08146_gb300 import synth
from gpu_util import make_ctx, dev, torch_cuda

pytestmark = pytest.mark.gpu
DIMS = (16, 16, 16, 16)          # workspaces of 270, 90 and 45 MB
MB = 1 << 20


def _leave(torch, left):
    """All of the device's free memory but `left` bytes."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")


def test_force_in_little_memory():
    torch = torch_cuda()
    U = synth.gauge_field(DIMS, 0.4, 31)
    n = 12 * int(np.prod(DIMS))
    g, psi = dev(synth.complex_gaussian(2 * n, 32)), dev(synth.complex_gaussian(2 * n, 33))
    ctx = make_ctx(U, DIMS, -0.3, 1.5)
    F0 = torch.empty(U.size, dtype=torch.complex128, device="cuda")
    F = torch.empty_like(F0)
    E0, E = torch.empty_like(F0), torch.empty_like(F0)
    ctx.qcd_bilinear_force_sum(2, g, psi, 1, F0)
    ctx.qcd_eig_force(1, psi, E0)
    for left in (160 * MB, 80 * MB):
        ctx.qcd_set_gauge(U, DIMS, -0.3, 1.5)          # drops the workspace
        hog = _leave(torch, left)
        try:
            F.fill_(float("nan"))
            E.fill_(float("nan"))
            ctx.qcd_bilinear_force_sum(2, g, psi, 1, F)
            ctx.qcd_eig_force(1, psi, E)
            torch.cuda.synchronize()
        finally:
            del hog
            torch.cuda.empty_cache()
        assert torch.equal(F, F0) and torch.equal(E, E0), left
    # 270 of 600 MB are the force's; the hierarchy (2^4 aggregates: P 144, stencil 226,
    # vectors 96) needs 466
    V = dev(synth.spinor(DIMS, 34, nvec=8))
    hog = _leave(torch, 600 * MB)
    try:
        ctx.qcd_bilinear_force_sum(2, g, psi, 1, F)
        ctx.qcd_mg_update_from_eigvecs(V, 8)
    finally:
        del hog
        torch.cuda.empty_cache()
    assert torch.equal(F, F0)
    ctx.close()
    make_ctx(U, DIMS, -0.3, 1.5).close()               # no error of the refused allocations is left
