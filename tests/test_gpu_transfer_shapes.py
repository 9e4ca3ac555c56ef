"""Restriction and prolongation at the edges of their tiles: numbers of test
vectors and right-hand sides that do not fill a tile (nv 1, 5, 7, 30; 1 to 17
right-hand sides, past one pass over P), aggregates of 2 to 256 sites and of
unequal extents, FP64 and FP32, FP32 fields aligned to 8 bytes only, and
right-hand sides that a tile covers beyond the last.  Against P of the library
applied with numpy (FP64 1e-13, FP32 2e-6 relative)."""
import numpy as np
import pytest

from paper_2004_08146_gb300 import synth
from gpu_util import make_ctx, dev, host, relerr, torch_cuda

pytestmark = pytest.mark.gpu


def _split(f, dims, agg):
    """[n, coarse sites, chirality, local entries] of fields [n, V*12]."""
    n = f.shape[0]
    sh = [n]
    for d, a in zip(dims, agg):
        sh += [d // a, a]
    f = f.reshape(sh + [2, 6]).transpose(0, 1, 3, 5, 7, 9, 2, 4, 6, 8, 10)
    return f.reshape(n, -1, 2, int(np.prod(agg)) * 6)


@pytest.mark.parametrize("dims,agg,nv,nrhs", [
    ((4, 4, 2, 2), (2, 1, 1, 1), 1, 1), ((4, 4, 4, 4), (2, 2, 2, 2), 5, 3), ((4, 6, 4, 4), (4, 3, 1, 2), 7, 17),
    ((8, 4, 4, 4), (4, 4, 4, 4), 30, 9), ((4, 4, 4, 4), (2, 2, 2, 2), 8, 4), ((6, 2, 2, 3), (3, 2, 2, 3), 4, 2)])
@pytest.mark.parametrize("prec,offset", [(0, 0), (1, 0), (1, 1)])
def test_transfer_tiles(dims, agg, nv, nrhs, prec, offset):
    torch = torch_cuda()
    ctx = make_ctx(synth.gauge_field(dims, 0.5, 95), dims, -0.3, 1.3, sap_block=agg)
    ctx.qcd_mg_update_from_eigvecs(dev(synth.spinor(dims, 96, nvec=nv)), nv)
    nb = int(np.prod(dims)) // int(np.prod(agg))
    P = ctx.qcd_mg_get_P().reshape(nb, 2, nv, -1)
    n = int(np.prod(dims)) * 12
    r = synth.spinor(dims, 97, nvec=nrhs).reshape(nrhs, n)
    xc = synth.complex_gaussian((nrhs, nb, 2, nv), 98)
    dt, tol = (np.complex128, 1e-13) if prec == 0 else (np.complex64, 2e-6)
    rd = torch.empty(nrhs * n + offset, dtype=torch.complex128 if prec == 0 else torch.complex64, device="cuda")[offset:]
    rd.copy_(dev(r, dt))
    yc = torch.empty(xc.size, dtype=rd.dtype, device="cuda")
    ctx.qcd_mg_restrict(prec, nrhs, rd, yc)
    ref = np.einsum("scie,nsce->nsci", P.conj(), _split(r, dims, agg))
    got = host(yc).reshape(ref.shape)
    x = torch.empty(nrhs * n + offset, dtype=rd.dtype, device="cuda")[offset:]
    ctx.qcd_mg_prolong(prec, nrhs, dev(xc, dt), x)
    fine = np.einsum("scie,nsci->nsce", P, xc)
    gotx = _split(host(x).reshape(nrhs, n), dims, agg)
    for j in range(nrhs):
        assert relerr(got[j], ref[j]) < tol, j
        assert relerr(gotx[j], fine[j]) < tol, j
    ctx.close()
