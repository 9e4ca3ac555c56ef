"""The aggregation P on both sides of the line between vectors in shared and in
global memory (nv x sites of an aggregate = 512), one vector to more than the warps
of a CTA, entries that do not fill a warp: orthonormal columns per aggregate and
chirality, whose span holds the test vectors.  Gram-Schmidt applied twice leaves a
few rounding errors of 2^-53 per product: 1e-13."""
import numpy as np
import pytest

from paper_2004_08146_gb300 import synth
from gpu_util import make_ctx, dev, torch_cuda
from test_gpu_transfer_shapes import _split

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,agg,nv", [((4, 4, 2, 2), (2, 1, 1, 1), 1), ((6, 2, 2, 3), (3, 1, 1, 1), 7),
                                         ((4, 4, 4, 4), (2, 2, 2, 2), 8), ((4, 4, 4, 4), (2, 2, 2, 2), 32),
                                         ((4, 4, 4, 4), (4, 4, 4, 1), 11), ((8, 4, 4, 4), (4, 4, 4, 4), 9)])
def test_build_P(dims, agg, nv):
    torch_cuda()
    ctx = make_ctx(synth.gauge_field(dims, 0.5, 95), dims, -0.3, 1.3, sap_block=agg)
    v = synth.spinor(dims, 96, nvec=nv)
    ctx.qcd_mg_update_from_eigvecs(dev(v), nv)
    nb = int(np.prod(dims)) // int(np.prod(agg))
    P = ctx.qcd_mg_get_P().reshape(nb, 2, nv, -1)
    gram = np.einsum("scie,scje->scij", P.conj(), P)
    assert np.max(np.abs(gram - np.eye(nv))) < 1e-13
    r = _split(v.reshape(nv, -1), dims, agg)
    back = np.einsum("scie,nsci->nsce", P, np.einsum("scie,nsce->nsci", P.conj(), r))
    assert np.linalg.norm(back - r) < 1e-13 * np.linalg.norm(r)
    ctx.close()
