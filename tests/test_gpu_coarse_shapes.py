"""The FP32 coarse stencil at the edges of its tiles: blocks that do not fill 16
rows or 8 columns, right-hand sides from one to past one pass over the blocks,
coarse extents 1 and 2 (a neighbour in both directions), against the FP64 stencil
on the same data.  A sum of 9 nc complex products rounded once per real product,
rms 2^-24 sqrt(18 nc) relative, plus the rounding of blocks and vectors; the
unaligned vectors of the general kernel meet the same bound."""
import numpy as np
import pytest

from paper_2004_08146_gb300 import synth
from gpu_util import make_ctx, dev, host, relerr, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,agg,nv", [((4, 4, 4, 4), (4, 4, 2, 2), 1), ((4, 4, 4, 4), (2, 2, 2, 2), 3),
                                         ((4, 4, 4, 6), (2, 2, 2, 2), 8), ((4, 4, 4, 4), (2, 2, 2, 2), 9),
                                         ((8, 4, 4, 4), (2, 2, 4, 4), 17), ((4, 4, 4, 4), (2, 2, 4, 4), 24),
                                         ((4, 4, 4, 4), (4, 2, 2, 4), 29), ((4, 4, 4, 4), (4, 4, 2, 2), 32)])
def test_coarse_stencil_tiles(dims, agg, nv):
    from paper_2004_08146_gb300 import qcd
    torch = torch_cuda()
    ctx = make_ctx(synth.gauge_field(dims, 0.5, 95), dims, -0.3, 1.3, sap_block=agg)
    ctx.qcd_mg_update_from_eigvecs(dev(synth.spinor(dims, 96, nvec=nv)), nv)
    nco = int(np.prod(dims)) // int(np.prod(agg)) * 2 * nv
    tol = 2.0 ** -24 * (np.sqrt(18 * 2 * nv) + 2)
    for nrhs in (1, 4, 5, 8, 11, 16, 17):
        x = synth.complex_gaussian((nrhs, nco), 155)
        taus = [0.01 * j - 0.1 for j in range(nrhs)]
        y64 = torch.empty(nrhs * nco, dtype=torch.complex128, device="cuda")
        for op in (qcd.QCD_OP_D, qcd.QCD_OP_Q):
            ctx.qcd_coarse_apply(op, 0, nrhs, dev(x), y64, taus)
            ref = host(y64).reshape(nrhs, nco)
            for offset in (0, 1):
                xin = torch.zeros(nrhs * nco + offset, dtype=torch.complex64, device="cuda")[offset:]
                xin.copy_(dev(x, np.complex64))
                y = torch.full((nrhs * nco,), np.nan, dtype=torch.complex64, device="cuda")
                ctx.qcd_coarse_apply(op, 1, nrhs, xin, y, taus)
                got = host(y).reshape(nrhs, nco)
                for j in range(nrhs):
                    assert relerr(got[j], ref[j]) < tol, (nrhs, op, offset, j)
    ctx.close()
