"""The Arnoldi launches of the device-controlled GMRES at the edges of their
splits: fields of fewer entries than one CTA takes, one to seventeen right-hand
sides (of which some converge early), steps on both sides of 4, 8 and 16 basis
vectors and up to 64, FP64 and FP32; the true residual as the oracle measures it
is what the library promises."""
import numpy as np
import pytest

from oracle.dirac import WilsonClover
from paper_2004_08146_gb300 import synth
from gpu_util import make_ctx, dev, host, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,nrhs,steps", [((2, 2, 2, 2), 1, 5), ((2, 2, 2, 2), 17, 64), ((4, 2, 6, 2), 3, 33),
                                             ((4, 4, 4, 4), 5, 20)])
@pytest.mark.parametrize("prec", [0, 1])
def test_gmres_steps(dims, nrhs, steps, prec):
    from paper_2004_08146_gb300 import qcd
    torch = torch_cuda()
    U = synth.gauge_field(dims, 0.3, 81)
    op = WilsonClover(U, 0.4, 1.0)
    ctx = make_ctx(U, dims, 0.4, 1.0, use_mg=0, correction_form=qcd.QCD_OP_Q, precision=prec, inner_maxiter=steps)
    b = synth.spinor(dims, 82, nvec=nrhs).reshape(nrhs, -1)
    b[nrhs // 2] *= 1e-3
    taus = [0.05 * j for j in range(nrhs)]
    bd = [dev(b[j]) for j in range(nrhs)]
    xd = [torch.zeros_like(v) for v in bd]
    rc, info = ctx.qcd_shifted_solve_batched(bd, xd, taus, 1e-9)
    assert rc == qcd.QCD_OK
    for j in range(nrhs):
        x = host(xd[j]).reshape(dims + (4, 3))
        r = b[j].reshape(x.shape) - (op.Q(x) - taus[j] * x)
        assert np.linalg.norm(r) <= (1e-9 + 1e-13) * np.linalg.norm(b[j]), j
    ctx.close()
