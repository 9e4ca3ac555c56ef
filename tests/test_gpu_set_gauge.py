"""Loading a gauge field from device memory, and again on a lattice the context
already holds: the same bits as a fresh context loaded from the host, a dropped
hierarchy, refused links, and a new lattice."""
import numpy as np
import pytest

from paper_2004_08146_gb300 import synth
from gpu_util import make_ctx, dev, host, torch_cuda

pytestmark = pytest.mark.gpu


def _apply(ctx, dims, prec):
    torch = torch_cuda()
    dt = np.complex128 if prec == 0 else np.complex64
    x = dev(synth.spinor(dims, 5, nvec=2), dt)
    y = torch.empty_like(x)
    ctx.qcd_apply(1, prec, 2, x, y, [0.1, -0.2])
    return host(y)


def test_set_gauge_device_and_again():
    from paper_2004_08146_gb300 import qcd
    torch_cuda()
    a, b = (4, 4, 4, 4), (2, 4, 6, 4)
    ctx = make_ctx(synth.gauge_field(a, 0.4, 1), a, -0.2, 1.0)
    ctx.qcd_mg_setup(4, (2, 2, 2, 2))
    for dims, seed, m0, csw in ((a, 2, -0.1, 1.5), (a, 3, -0.2, 0.0), (b, 4, -0.1, 1.0), (b, 5, -0.3, 1.0), (a, 6, 0.1, 1.0)):
        U = synth.gauge_field(dims, 0.4, seed)
        if seed % 2:
            ctx.qcd_set_gauge(U, dims, m0, csw)
        else:
            ctx.qcd_set_gauge_device(dev(U), dims, m0, csw)
        with pytest.raises(qcd.QcdError):   # the hierarchy went with the old field
            ctx.qcd_mg_get_P()
        fresh = make_ctx(U, dims, m0, csw)
        for prec in (0, 1):
            assert np.array_equal(_apply(ctx, dims, prec), _apply(fresh, dims, prec))
        fresh.close()
    with pytest.raises(ValueError):
        ctx.qcd_set_gauge_device(dev(U)[:-1], a, 0.1, 1.0)
    assert np.array_equal(_apply(ctx, a, 0), _apply(make_ctx(U, a, 0.1, 1.0), a, 0))   # still the last field
    with pytest.raises(qcd.QcdError):
        ctx.qcd_set_gauge_device(dev(1.1 * U), a, 0.1, 1.0)
    with pytest.raises(qcd.QcdError):
        _apply(ctx, a, 0)                                                              # no field is left
    ctx.qcd_set_gauge_device(dev(U), a, 0.1, 1.0)
    assert np.array_equal(_apply(ctx, a, 0), _apply(make_ctx(U, a, 0.1, 1.0), a, 0))
    ctx.close()


@pytest.mark.parametrize("dims", [(2, 2, 2, 3), (2, 3, 5, 2), (3, 4, 2, 7)])
@pytest.mark.parametrize("csw", [0.0, 1.7])
def test_clover_blocks(dims, csw):
    """The clover blocks on lattices that do not fill a CTA of the build, with
    neighbours that coincide (extent 2) and odd extents, through Q in FP64 (sums of
    about 60 products: 1e-14) and FP32 (2e-6) against the oracle."""
    from oracle.dirac import WilsonClover
    U = synth.gauge_field(dims, 0.6, 12)
    op = WilsonClover(U, -0.1, csw)
    ctx = make_ctx(U, dims, -0.1, csw)
    x = synth.spinor(dims, 5, nvec=2).reshape((2,) + dims + (4, 3))
    for prec, tol in ((0, 1e-14), (1, 2e-6)):
        got = _apply(ctx, dims, prec).reshape(x.shape)
        for j, tau in enumerate((0.1, -0.2)):
            ref = op.Q(x[j]) - tau * x[j]
            assert np.linalg.norm(got[j] - ref) < tol * np.linalg.norm(ref)
    ctx.close()
