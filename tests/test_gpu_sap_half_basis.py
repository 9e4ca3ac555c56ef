"""The block solves with the FP16-stored basis follow modified Gram-Schmidt one vector
at a time: emulated in FP64 with the same FP16 roundings, they are nearer to that than
to projections on two vectors at a time, which FP16 leaves orthogonal to 3e-4 only."""
import numpy as np
import pytest

from oracle import mg
from oracle.dirac import WilsonClover
from paper_2004_08146_gb300 import synth
from gpu_util import make_ctx, dev, host, torch_cuda

pytestmark = pytest.mark.gpu


def _half(v):
    return v.real.astype(np.float16).astype(np.float64) + 1j * v.imag.astype(np.float16).astype(np.float64)


def _solve(M, r, steps, width):
    """GMRES correction, projecting on `width` basis vectors at a time."""
    beta = np.linalg.norm(r)
    V, H = [_half(r / beta)], np.zeros((steps + 1, steps), dtype=complex)
    for j in range(steps):
        w = M @ V[j]
        for i in range(0, j + 1, width):
            some = range(i, min(i + width, j + 1))
            for k in some:
                H[k, j] = np.vdot(V[k], w)
            w = w - sum(H[k, j] * V[k] for k in some)
        H[j + 1, j] = np.linalg.norm(w)
        V.append(_half(w / H[j + 1, j]))
    rhs = np.zeros(steps + 1, dtype=complex)
    rhs[0] = beta
    y = np.linalg.lstsq(H, rhs, rcond=None)[0]
    return sum(y[i] * V[i] for i in range(steps))


@pytest.mark.parametrize("steps", [6, 10])
def test_fp16_basis_projects_one_vector_at_a_time(steps):
    from paper_2004_08146_gb300 import qcd
    torch = torch_cuda()
    dims, tau = (4, 4, 4, 8), 0.1
    U = synth.gauge_field(dims, 0.5, 75)
    op = WilsonClover(U, -0.3, 1.3)
    sap = mg.SAP(dims, (2, 2, 2, 2))
    M = sap.block_matrices(lambda v: mg.fine_apply(op, v, tau, 'g5'), 0)
    sites = sap.blk.sites[sap.members[0]]
    b = synth.spinor(dims, 76).astype(np.complex64)
    ctx = make_ctx(U, dims, -0.3, 1.3, sap_block=(2, 2, 2, 2), sap_block_iters=steps, sap_half=1)
    x = torch.zeros(b.size, dtype=torch.complex64, device="cuda")
    ctx.qcd_sap(qcd.QCD_OP_D, qcd.QCD_FP32, 1, dev(b), x, [tau], 1, -1.0)
    got = host(x).reshape(-1, 12)[sites].reshape(len(sites), -1)
    ctx.close()
    rb = b.reshape(-1, 12)[sites].reshape(len(sites), -1).astype(np.complex128)
    dist = [np.linalg.norm(got - np.array([_solve(M[q], rb[q], steps, width) for q in range(len(sites))]))
            for width in (1, 2)]
    assert dist[0] < dist[1], dist
