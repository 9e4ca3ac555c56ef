"""Every tile of the FP64 restriction (1 x 1, 2 x 1, 4 x 1 and 4 x 2, chosen by test
vectors and right-hand sides per CTA), both prolongations, and a last chunk that needs
fewer warps than the others, in FP32 too: against P applied with numpy (FP64 1e-13, FP32
2e-6 relative, the bounds of the other transfer tests)."""
import numpy as np
import pytest

from paper_2004_08146_gb300 import qcd, synth
from gpu_util import make_ctx, dev, host, relerr, torch_cuda
from test_gpu_transfer_shapes import _split

pytestmark = pytest.mark.gpu

DIMS, AGG = (8, 8, 8, 8), (2, 2, 2, 2)


@pytest.mark.parametrize("nv", [5, 13, 20, 32])
def test_transfer_tiles_of_full_lattices(nv):
    torch = torch_cuda()
    ctx = make_ctx(synth.gauge_field(DIMS, 0.5, 95), DIMS, -0.3, 1.3, sap_block=AGG, precision=qcd.QCD_FP64)
    ctx.qcd_mg_update_from_eigvecs(dev(synth.spinor(DIMS, 96, nvec=nv)), nv)
    P = ctx.qcd_mg_get_P().reshape(256, 2, nv, -1)
    n = 4096 * 12
    r = synth.spinor(DIMS, 97, nvec=18).reshape(18, n)
    xc = synth.complex_gaussian((18, 256, 2, nv), 98)
    down = np.einsum("scie,nsce->nsci", P.conj(), _split(r, DIMS, AGG))
    up = np.einsum("scie,nsci->nsce", P, xc)
    for prec, dt, tol in ((0, np.complex128, 1e-13), (1, np.complex64, 2e-6)):
        for nrhs in (1, 4, 7, 18):
            yc = torch.empty(nrhs * 512 * nv, dtype=torch.complex128 if prec == 0 else torch.complex64, device="cuda")
            x = torch.empty(nrhs * n, dtype=yc.dtype, device="cuda")
            ctx.qcd_mg_restrict(prec, nrhs, dev(r[:nrhs], dt), yc)
            ctx.qcd_mg_prolong(prec, nrhs, dev(xc[:nrhs], dt), x)
            got, gotx = host(yc).reshape(down[:nrhs].shape), _split(host(x).reshape(nrhs, n), DIMS, AGG)
            for j in range(nrhs):
                assert relerr(got[j], down[j]) < tol, (prec, nrhs, j)
                assert relerr(gotx[j], up[j]) < tol, (prec, nrhs, j)
    ctx.close()
