"""An infinite entry of a field reaches the same real and imaginary parts of the result
in both FP64 stencils (eight lanes per site, one thread per site) as in the FP32 one:
the real diagonal of the clover blocks does not mix the two parts of an entry."""
import numpy as np
import pytest

from paper_2004_08146_gb300 import synth
from gpu_util import make_ctx, dev, host, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (16, 16, 16, 16)])
@pytest.mark.parametrize("part", ["real", "imag"])
def test_infinite_entry(dims, part):
    torch = torch_cuda()
    ctx = make_ctx(synth.gauge_field(dims, 0.5, 91), dims, -0.3, 1.3)
    psi = synth.spinor(dims, 92).reshape(-1, 12)
    for k in range(12):
        getattr(psi, part)[37 + 18 * k, k] = np.inf
    for op in (0, 1):
        seen = []
        for prec, dt in ((0, np.complex128), (1, np.complex64)):
            x = dev(psi, dt)
            y = torch.empty_like(x)
            ctx.qcd_apply(op, prec, 1, x, y, [0.1])
            y = host(y)
            seen.append(np.stack([np.isfinite(y.real), np.isfinite(y.imag)]))
        assert not seen[1].all() and np.array_equal(seen[0], seen[1])
    ctx.close()
