"""The stencils at the edges of their launch shapes: site counts that leave
warps partly idle, extents of 2 and odd extents (both neighbours of a site
equal, blocks of sites that wrap), batches, both shifted forms, and both FP64
kernels -- eight lanes per site below 65,536 sites, one thread per site from
there on -- against the oracle (FP64 1e-13, FP32 2e-6 relative, the bounds of the
operator tests).  A field gives the same bits alone and in a batch."""
import numpy as np
import pytest

from oracle.dirac import WilsonClover
from paper_2004_08146_gb300 import synth
from gpu_util import make_ctx, dev, host, relerr, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,antip", [((2, 2, 2, 2), 1), ((3, 5, 2, 7), 1), ((5, 3, 3, 3), 0),
                                        ((16, 16, 16, 15), 1), ((16, 16, 16, 16), 1)])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_stencil_shapes_match_oracle(dims, antip, nrhs):
    from paper_2004_08146_gb300 import qcd
    torch = torch_cuda()
    U = synth.gauge_field(dims, 0.5, 91)
    op = WilsonClover(U, -0.3, 1.3, antiperiodic_t=bool(antip))
    ctx = make_ctx(U, dims, -0.3, 1.3, antiperiodic_t=antip)
    psi = synth.spinor(dims, 92, nvec=nrhs)
    taus = [0.2 - 0.3 * j for j in range(nrhs)]
    g5 = np.array([1.0, 1, -1, -1])[:, None]
    ref = {}
    for j in range(nrhs):
        Dp = op.D(psi[j])
        ref[0, j], ref[1, j] = Dp - taus[j] * g5 * psi[j], g5 * Dp - taus[j] * psi[j]
    for prec, dt, tol in ((0, np.complex128, 1e-13), (1, np.complex64, 2e-6)):
        for opc in (qcd.QCD_OP_D, qcd.QCD_OP_Q):
            x = dev(psi, dt)
            y = torch.empty_like(x)
            ctx.qcd_apply(opc, prec, nrhs, x, y, taus)
            got = host(y).reshape((nrhs,) + dims + (4, 3))
            for j in range(nrhs):
                assert relerr(got[j], ref[opc, j]) < tol, (prec, opc, j)
            one = torch.empty(x.numel() // nrhs, dtype=x.dtype, device="cuda")
            last = x[(nrhs - 1) * one.numel():]
            ctx.qcd_apply(opc, prec, 1, last, one, taus[-1:])
            assert np.array_equal(host(one).reshape(dims + (4, 3)), got[-1]), (prec, opc)
    ctx.close()


@pytest.mark.parametrize("dims,nrhs", [((8, 8, 8, 16), 25), ((3, 5, 2, 7), 2)])
@pytest.mark.parametrize("offset", [0, 2])
def test_fp32_batches_and_alignment(dims, nrhs, offset):
    """FP32 batches past the line where a thread takes two right-hand sides (an
    odd count leaves one alone), and fields aligned to 16 bytes only, whose
    results have the same bits as aligned ones."""
    from paper_2004_08146_gb300 import qcd
    torch = torch_cuda()
    U = synth.gauge_field(dims, 0.5, 93)
    op = WilsonClover(U, -0.3, 1.3)
    ctx = make_ctx(U, dims, -0.3, 1.3)
    psi = synth.spinor(dims, 94, nvec=nrhs)
    taus = [0.2 - 0.03 * j for j in range(nrhs)]
    x = dev(psi, np.complex64)
    xo = torch.empty(x.numel() + offset, dtype=x.dtype, device="cuda")[offset:].copy_(x)
    yo = torch.empty(x.numel() + offset, dtype=x.dtype, device="cuda")[offset:]
    y = torch.empty_like(x)
    ctx.qcd_apply(qcd.QCD_OP_Q, 1, nrhs, xo, yo, taus)
    ctx.qcd_apply(qcd.QCD_OP_Q, 1, nrhs, x, y, taus)
    got = host(yo).reshape((nrhs,) + dims + (4, 3))
    assert np.array_equal(got.reshape(-1), host(y))
    for j in (0, nrhs - 1):
        assert relerr(got[j], op.Q_shift(psi[j], taus[j])) < 2e-6, j
    ctx.close()
