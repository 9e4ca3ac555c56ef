"""Long sums of complex products are no further from the exact ones (extended
precision, on the data as the library holds it) than serial sums in the working
precision that round each product before it is added: the lanes of a warp along an
aggregate's entries, added at the end, for the restriction, the test vectors in
turn for the prolongation, the columns of the nine blocks for the coarse stencil; the
interpolation (Gram-Schmidt twice) to 5 % of numpy's in FP64.  Chains of fused multiply-adds through the running sum
round it twice per product and are 1.25 to 1.4 times as far."""
import numpy as np
import pytest

from extended import CLD, rel
from paper_2004_08146_gb300 import synth
from gpu_util import make_ctx, dev, host, torch_cuda
from test_gpu_transfer_shapes import _split

pytestmark = pytest.mark.gpu


def serial(terms, axis=0):
    """Sum along `axis` one after the other, in the precision of the terms."""
    terms = np.moveaxis(terms, axis, 0)
    s = terms[0].copy()
    for t in terms[1:]:
        s = s + t
    return s


def mg_context(dims, agg, nv, seed):
    torch_cuda()
    ctx = make_ctx(synth.gauge_field(dims, 0.5, seed), dims, -0.3, 1.3, sap_block=agg)
    ctx.qcd_mg_update_from_eigvecs(dev(synth.spinor(dims, seed + 1, nvec=nv)), nv)
    nb = int(np.prod(dims)) // int(np.prod(agg))
    return ctx, ctx.qcd_mg_get_P().reshape(nb, 2, nv, -1), nb


@pytest.mark.parametrize("prec,dt", [(0, np.complex128), (1, np.complex64)])
@pytest.mark.parametrize("dims,agg,nv,nrhs", [((8, 8, 4, 4), (4, 4, 4, 4), 20, 3), ((8, 4, 4, 4), (4, 4, 4, 4), 23, 9),
                                              ((8, 8, 8, 4), (4, 2, 4, 2), 12, 2)])
def test_transfer_error(dims, agg, nv, nrhs, prec, dt):
    torch = torch_cuda()
    ctx, P, nb = mg_context(dims, agg, nv, 95)
    P = P.astype(dt)
    n = int(np.prod(dims)) * 12
    r = synth.spinor(dims, 97, nvec=nrhs).reshape(nrhs, n).astype(dt)
    xc = synth.complex_gaussian((nrhs, nb, 2, nv), 98).astype(dt)
    yc = torch.empty(xc.size, dtype=torch.complex128 if prec == 0 else torch.complex64, device="cuda")
    x = torch.empty(r.size, dtype=yc.dtype, device="cuda")
    ctx.qcd_mg_restrict(prec, nrhs, dev(r), yc)
    ctx.qcd_mg_prolong(prec, nrhs, dev(xc), x)
    down, up = host(yc), _split(host(x).reshape(nrhs, n), dims, agg)
    ctx.close()
    rs = _split(r, dims, agg)
    terms = P.conj()[None] * rs[:, :, :, None]                       # [n, sites, chirality, i, entries]
    plain = serial(serial(terms.reshape(terms.shape[:-1] + (-1, 32)), -2), -1)
    exact = np.sum(P.astype(CLD).conj()[None] * rs.astype(CLD)[:, :, :, None], axis=-1)
    assert rel(down, exact) <= rel(plain, exact), (rel(down, exact), rel(plain, exact))
    terms = P[None] * xc[..., None]
    plain = serial(terms, 3)
    exact = np.sum(P.astype(CLD)[None] * xc.astype(CLD)[..., None], axis=3)
    assert rel(up, exact) <= rel(plain, exact), (rel(up, exact), rel(plain, exact))


@pytest.mark.parametrize("prec,dt,offset", [(0, np.complex128, 0), (1, np.complex64, 0), (1, np.complex64, 1)])
@pytest.mark.parametrize("nv,nrhs", [(20, 3), (7, 5)])
def test_coarse_stencil_error(nv, nrhs, prec, dt, offset):
    from paper_2004_08146_gb300 import qcd
    torch = torch_cuda()
    dims, agg = (8, 8, 8, 4), (4, 4, 4, 4)
    ctx = make_ctx(synth.gauge_field(dims, 0.5, 95), dims, -0.3, 1.3, sap_block=agg, precision=qcd.QCD_FP64)
    ctx.qcd_mg_update_from_eigvecs(dev(synth.spinor(dims, 96, nvec=nv)), nv)
    g, nc = (2, 2, 2, 1), 2 * nv
    A = np.asarray(ctx.qcd_mg_get_coarse()).reshape(8, 9, nc, nc).astype(dt)     # [site][direction][row][column]
    x = synth.complex_gaussian((nrhs, 8, nc), 98).astype(dt)
    xd = torch.empty(x.size + offset, dtype=torch.complex128 if prec == 0 else torch.complex64, device="cuda")[offset:]
    xd.copy_(dev(x))
    y = torch.empty_like(xd)
    ctx.qcd_coarse_apply(qcd.QCD_OP_D, prec, nrhs, xd, y, [0.0] * nrhs)
    got = host(y)
    ctx.close()
    nb = np.empty((8, 9), dtype=int)
    for s in range(8):
        for d in range(9):
            c = list(np.unravel_index(s, g))
            if d:
                c[(d - 1) % 4] = (c[(d - 1) % 4] + (1 if d <= 4 else -1)) % g[(d - 1) % 4]
            nb[s, d] = np.ravel_multi_index(c, g)
    xn = x[:, nb]                                                                # [n, site, direction, column]
    plain = serial((A[None] * xn[:, :, :, None]).transpose(0, 1, 3, 2, 4).reshape(nrhs, 8, nc, -1), -1)
    exact = np.sum(A.astype(CLD)[None] * xn.astype(CLD)[:, :, :, None], axis=(2, 4))
    assert rel(got, exact) <= rel(plain, exact), (rel(got, exact), rel(plain, exact))


@pytest.mark.parametrize("dims,agg,nv", [((8, 8, 4, 4), (4, 4, 4, 4), 20), ((4, 4, 4, 8), (2, 2, 2, 2), 12)])
def test_interpolation_error(dims, agg, nv):
    ctx, P, _ = mg_context(dims, agg, nv, 95)
    ctx.close()

    def schmidt(dt):
        q = list(_split(synth.spinor(dims, 96, nvec=nv).reshape(nv, -1), dims, agg).astype(dt))
        for _ in range(2):
            for i in range(nv):
                for j in range(i):
                    q[i] = q[i] - np.sum(q[j].conj() * q[i], axis=-1, keepdims=True) * q[j]
                q[i] = q[i] / np.sqrt(np.sum(np.abs(q[i]) ** 2, axis=-1, keepdims=True))
        return np.stack(q, axis=2)

    exact = schmidt(CLD)
    plain = rel(schmidt(np.complex128), exact)
    assert rel(P, exact) <= 1.05 * plain, (rel(P, exact), plain)
