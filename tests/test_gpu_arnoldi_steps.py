"""GMRES takes the steps that the oracle's takes and reaches the tolerance in one cycle:
wrong coefficients, a lost projection or a wrong rotation would cost steps or another
cycle.  One to seventeen right-hand sides, basis sizes past 4, 8 and 16, FP64 and FP32
(whose inner tolerance stays above its floor); one step of slack at the threshold."""
import numpy as np
import pytest

from oracle import mg
from oracle.dirac import WilsonClover
from paper_2004_08146_gb300 import synth
from gpu_util import make_ctx, dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 2), 1), ((4, 2, 6, 2), 3), ((4, 4, 4, 4), 5), ((2, 2, 2, 4), 17)])
@pytest.mark.parametrize("prec,tol", [(0, 1e-9), (1, 1e-4)])
def test_steps_of_one_cycle(dims, nrhs, prec, tol):
    from paper_2004_08146_gb300 import qcd
    torch = torch_cuda()
    U = synth.gauge_field(dims, 0.3, 81)
    op = WilsonClover(U, 0.8, 1.0)
    b = synth.spinor(dims, 82, nvec=nrhs)
    taus = [0.02 * j for j in range(nrhs)]
    steps = []
    for j in range(nrhs):
        A = lambda v, t=taus[j]: mg.fine_apply(op, v.reshape(dims + (4, 3)), t, 'g5').reshape(1, -1)
        steps.append(int(mg.gmres(A, op.g5(b[j]).reshape(1, -1), 0.5 * tol, 64)[1][0]))
    assert max(steps) < 64
    ctx = make_ctx(U, dims, 0.8, 1.0, use_mg=0, precision=prec, inner_maxiter=64)
    bs = [dev(b[j]) for j in range(nrhs)]
    rc, info = ctx.qcd_shifted_solve_batched(bs, [torch.zeros_like(v) for v in bs], taus, tol)
    ctx.close()
    assert rc == qcd.QCD_OK and info.residual <= tol
    assert info.refinements == 1 and abs(info.iterations - max(steps)) <= 1, (info.refinements, info.iterations, steps)
