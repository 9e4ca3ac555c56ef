"""qcd_set_gauge_device hands a raw device pointer to the library: tensors whose memory
is not the links on the device are refused before the call."""
import pytest
import torch

from paper_2004_08146_gb300 import qcd


@pytest.mark.parametrize("links", [
    torch.zeros(16, 4, 3, 3, dtype=torch.complex128),                     # host memory
    torch.zeros(16, 4, 3, 3, dtype=torch.complex128).conj(),
    torch.zeros(16, 4, 3, 3, dtype=torch.complex128, device="meta").conj()])
def test_refuses_what_is_not_device_links(links):
    ctx = qcd.Context.__new__(qcd.Context)                                # no GPU needed: refused before the call
    ctx.h = None
    with pytest.raises(ValueError):
        ctx.qcd_set_gauge_device(links, (2, 2, 2, 2), 0.0, 1.0)


@pytest.mark.gpu
def test_refuses_lazy_views_and_keeps_the_field():
    from gpu_util import dev, host, make_ctx, torch_cuda
    from paper_2004_08146_gb300 import synth
    torch_cuda()
    dims = (2, 2, 2, 4)
    U = synth.gauge_field(dims, 0.4, 3)
    ctx = make_ctx(U, dims, -0.1, 1.0)
    for view in (dev(U).conj(), dev(U)[:-1], torch.from_numpy(U.reshape(-1))):
        with pytest.raises(ValueError):
            ctx.qcd_set_gauge_device(view, dims, -0.1, 1.0)
    x = dev(synth.spinor(dims, 5))
    y = torch.empty_like(x)
    ctx.qcd_apply(1, 0, 1, x, y, [0.1])                                   # the field is still there
    assert bool(torch.isfinite(torch.view_as_real(y)).all()) and host(y).any()
    ctx.close()
