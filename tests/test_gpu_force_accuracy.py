"""The link gradient of a batch is no further from the exact one (extended precision)
than the fields' gradients of the oracle in FP64 added up: a single chain of products
over all fields was 1.25 to 1.4 times as far."""
import numpy as np
import pytest

import oracle.dirac
from extended import CLD, dirac, rel
from paper_2004_08146_gb300 import synth
from gpu_util import make_ctx, dev, host, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("csw", [0.0, 1.5])
@pytest.mark.parametrize("nvec", [1, 7, 8])
def test_batch_gradient_error(csw, nvec):
    torch = torch_cuda()
    dims = (4, 4, 4, 4)
    U = synth.gauge_field(dims, 0.5, 13)
    g, psi = synth.spinor(dims, 14, nvec=nvec), synth.spinor(dims, 15, nvec=nvec)
    ctx = make_ctx(U, dims, -0.85, csw)
    F = torch.empty(U.size, dtype=torch.complex128, device="cuda")
    ctx.qcd_bilinear_force_sum(nvec, dev(g), dev(psi), 1, F)
    got = host(F)
    ctx.close()
    grads = {}
    for mod, dt in ((dirac, CLD), (oracle.dirac, np.complex128)):
        op = mod.WilsonClover(U.astype(dt), -0.85, csw)
        f = sum(mod.bilinear_force(op, g[j].astype(dt), psi[j].astype(dt)) for j in range(nvec))
        grads[dt] = 1j * (f @ op.U)
    err = rel(got, grads[CLD]), rel(grads[np.complex128], grads[CLD])
    assert err[0] <= err[1], err
