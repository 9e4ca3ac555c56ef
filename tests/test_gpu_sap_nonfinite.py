"""Block solves whose right-hand side is not finite: the solution of the block shows it
(it is not silently left as it was), the blocks that do not see it are untouched by it."""
import numpy as np
import pytest

from oracle import mg
from paper_2004_08146_gb300 import synth
from gpu_util import make_ctx, dev, host, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,half", [(0, 0), (1, 0), (1, 1)])
@pytest.mark.parametrize("tol", [-1.0, 0.1])
def test_infinite_right_hand_side_shows(prec, half, tol):
    from paper_2004_08146_gb300 import qcd
    torch_cuda()
    dims, block = (8, 4, 4, 4), (2, 2, 2, 2)
    dt = np.complex128 if prec == 0 else np.complex64
    blk = mg.Blocking(dims, block)
    b, x0 = synth.spinor(dims, 76).astype(dt).reshape(-1, 12), synth.spinor(dims, 77).astype(dt).reshape(-1, 12)
    ctx = make_ctx(synth.gauge_field(dims, 0.5, 75), dims, -0.3, 1.3, sap_block=block, sap_half=half)
    out = []
    for bad in (False, True):
        c = b.copy()
        if bad:
            c[blk.sites[0][3], 5] = np.inf
        xd = dev(x0, dt)
        ctx.qcd_sap(qcd.QCD_OP_D, prec, 1, dev(c), xd, [0.1], 1, tol)
        out.append(host(xd).reshape(-1, 12))
    ctx.close()
    assert not np.isfinite(out[1][blk.sites[0]]).any()
    same = np.nonzero(blk.colour == blk.colour[0])[0][1:]
    sites = blk.sites[same].reshape(-1)
    assert np.array_equal(out[0][sites], out[1][sites]) and np.isfinite(out[0]).all()
