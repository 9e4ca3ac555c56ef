"""The 2^4-block SAP kernel at the shapes where it can go wrong: right-hand-side
counts that leave warps of a CTA without work (1, 3, 5, 7), extent-4 lattices
(both outside neighbours of a block are the same block) and unequal extents,
one step and more steps than the staged vectors need, periodic time, and a
16-site block of another shape (the general kernel).  Fixed block-GMRES steps
against the oracle in both forms; FP64 to 1e-10 relative, FP32 to 1e-4 (the
bounds of the other block families).  A run stopped at the block tolerance
leaves zero right-hand sides at zero."""
import numpy as np
import pytest

from oracle.dirac import WilsonClover
from oracle import mg
from paper_2004_08146_gb300 import synth
from gpu_util import make_ctx, dev, host, relerr, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,block,nrhs,iters,antip", [
    ((4, 4, 4, 4), (2, 2, 2, 2), 1, 1, 1), ((4, 8, 4, 4), (2, 2, 2, 2), 3, 10, 1),
    ((4, 4, 4, 12), (2, 2, 2, 2), 5, 3, 0), ((8, 4, 4, 4), (2, 2, 2, 2), 7, 4, 1),
    ((8, 4, 4, 4), (4, 2, 2, 1), 5, 4, 1)])
@pytest.mark.parametrize("prec,tol", [(0, 1e-10), (1, 1e-4)])
def test_cube_solves_match_oracle(dims, block, nrhs, iters, antip, prec, tol):
    from paper_2004_08146_gb300 import qcd
    torch_cuda()
    U = synth.gauge_field(dims, 0.5, 75)
    op = WilsonClover(U, -0.3, 1.3, antiperiodic_t=bool(antip))
    ctx = make_ctx(U, dims, -0.3, 1.3, sap_block=block, sap_block_iters=iters, antiperiodic_t=antip)
    dt = np.complex128 if prec == 0 else np.complex64
    b, x0 = synth.spinor(dims, 76, nvec=nrhs), synth.spinor(dims, 77, nvec=nrhs)
    taus = [0.1 - 0.07 * j for j in range(nrhs)]
    sap = mg.SAP(dims, block, block_iters=iters, block_tol=0.0)
    for opc, form in ((qcd.QCD_OP_D, 'g5'), (qcd.QCD_OP_Q, 'Q')):
        xd = dev(x0, dt)
        ctx.qcd_sap(opc, prec, nrhs, dev(b, dt), xd, taus, 1, -1.0)
        got = host(xd).reshape((nrhs,) + dims + (4, 3))
        for j in range(nrhs):
            ref = sap.smooth(lambda v, t=taus[j]: mg.fine_apply(op, v, t, form), b[j], x0[j], 1)
            assert relerr(got[j], ref) < tol, (form, j)
    ctx.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_zero_right_hand_side_stays_zero(prec):
    from paper_2004_08146_gb300 import qcd
    torch = torch_cuda()
    dims = (4, 4, 4, 8)
    ctx = make_ctx(synth.gauge_field(dims, 0.5, 78), dims, -0.3, 1.3)
    dt = torch.complex128 if prec == 0 else torch.complex64
    b = torch.zeros((2, int(np.prod(dims)) * 12), dtype=dt, device="cuda")
    b[1] = 1.0
    x = torch.zeros_like(b)
    ctx.qcd_sap(qcd.QCD_OP_D, prec, 2, b, x, [0.1, -0.1], 2, 0.1)
    assert float(x[0].abs().max()) == 0.0 and bool(torch.isfinite(torch.view_as_real(x[1])).all())
    assert float(x[1].abs().max()) > 0.0
    ctx.close()
