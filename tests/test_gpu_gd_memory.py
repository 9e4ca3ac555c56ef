"""Device memory of an eigensolve on a tiny lattice (n = 192): basis, locked vectors
and pencil take less than 4 MB at the default sizes, so the context stays below 8."""
import pytest

from paper_2004_08146_gb300 import synth
from gpu_util import make_ctx, torch_cuda

pytestmark = pytest.mark.gpu


def test_eigensolve_workspace():
    from paper_2004_08146_gb300 import qcd
    torch = torch_cuda()
    dims = (2, 2, 2, 2)
    U = synth.gauge_field(dims, 0.3, 71)
    used = []
    for _ in range(2):                 # the first call loads the kernels
        ctx = make_ctx(U, dims, -0.1, 1.0, use_mg=0, correction_form=qcd.QCD_OP_Q)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        assert ctx.qcd_eigs(4, 1e-8)[0] == qcd.QCD_OK
        torch.cuda.synchronize()
        used.append(free - torch.cuda.mem_get_info()[0])
        ctx.close()
    assert used[1] < 8 << 20, used
