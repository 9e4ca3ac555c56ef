"""The double-float Gram-Schmidt kernels of the Davidson basis at the edges of
their splits: vectors of fewer entries than one CTA reads, with remainders, and
basis plus locked sets from one vector to more than a CTA's share."""
import numpy as np
import pytest

from oracle.dirac import WilsonClover
from paper_2004_08146_gb300 import synth
from gpu_util import make_ctx, host, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,k", [((2, 2, 2, 2), 1), ((2, 2, 2, 2), 20), ((6, 2, 2, 2), 9), ((4, 2, 6, 2), 33),
                                    ((4, 4, 6, 2), 17)])
def test_gd_vectors(dims, k):
    """Each pair meets ||Q v - lambda v|| <= tol as the oracle measures it (plus
    FP64 roundoff of the measurement), so lambda lies within tol of an eigenvalue
    of the Hermitian Q; the vectors are orthonormal to far below the double-float
    2^-48 times the number of entries."""
    from paper_2004_08146_gb300 import qcd
    torch = torch_cuda()
    tol = 1e-8
    U = synth.gauge_field(dims, 0.3, 71)
    op = WilsonClover(U, -0.1, 1.0)
    ev = np.linalg.eigvalsh(op.dense('Q'))
    ctx = make_ctx(U, dims, -0.1, 1.0, use_mg=0, correction_form=qcd.QCD_OP_Q)
    V = torch.zeros(k * op.n, dtype=torch.complex128, device="cuda")
    rc, lam, info = ctx.qcd_eigs(k, tol, V)
    assert rc == qcd.QCD_OK and info.converged
    V = host(V).reshape(k, -1)
    for j in range(k):
        v = V[j].reshape(dims + (4, 3))
        assert np.linalg.norm(op.Q(v) - lam[j] * v) <= tol + 1e-13
        assert np.min(np.abs(ev - lam[j])) <= tol + 1e-13
    assert np.max(np.abs(V.conj() @ V.T - np.eye(k))) <= op.n * 2.0 ** -48
