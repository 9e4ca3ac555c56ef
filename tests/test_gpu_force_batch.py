"""The force kernels at the edges of their shapes: odd extents and extents of 2
(both neighbours of a site equal), one and several fields, with and without
the clover term, against the oracle element by element (1e-12 of the largest
entry, the bound of the other force tests); the summed call against the sum of
the single ones; and a lattice past the size to which all six planes are done
in one launch, where sum tr(X F) has to reproduce the directional derivative
(1e-12)."""
import numpy as np
import pytest

from oracle.dirac import WilsonClover
from paper_2004_08146_gb300 import synth
from gpu_util import make_ctx, dev, host, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,antip,csw,nvec", [((2, 2, 2, 2), True, 1.5, 1), ((3, 5, 2, 3), True, 1.5, 3),
                                                 ((4, 3, 3, 5), False, 1.1, 2), ((3, 2, 5, 2), True, 0.0, 2)])
@pytest.mark.parametrize("grad", [0, 1])
def test_summed_force_matches_oracle(dims, antip, csw, nvec, grad):
    torch = torch_cuda()
    from oracle.dirac import bilinear_force
    U = synth.gauge_field(dims, 0.5, 191)
    op = WilsonClover(U, -0.3, csw, antiperiodic_t=antip)
    ctx = make_ctx(U, dims, -0.3, csw, antiperiodic_t=int(antip))
    g, psi = synth.spinor(dims, 192, nvec=nvec), synth.spinor(dims, 193, nvec=nvec)
    nl = 36 * int(np.prod(dims))
    S = torch.full((nl,), float("nan"), dtype=torch.complex128, device="cuda")
    F = torch.full((nvec * nl,), float("nan"), dtype=torch.complex128, device="cuda")
    ctx.qcd_bilinear_force_sum(nvec, dev(g), dev(psi), grad, S)
    ctx.qcd_bilinear_force(nvec, dev(g), dev(psi), grad, F)
    ref = sum(bilinear_force(op, g[j], psi[j]) for j in range(nvec))
    ref = 1j * (ref @ U) if grad else ref
    got, one = host(S).reshape(ref.shape), host(F).reshape((nvec,) + ref.shape).sum(axis=0)
    assert np.max(np.abs(got - ref)) < 1e-12 * np.max(np.abs(ref))
    assert np.max(np.abs(one - ref)) < 1e-12 * np.max(np.abs(ref))
    ctx.close()


def test_force_one_plane_per_launch():
    torch = torch_cuda()
    dims = (32, 32, 18, 17)
    U = synth.gauge_field(dims, 0.4, 195)
    ctx = make_ctx(U, dims, -0.3, 1.5)
    v = dev(synth.spinor(dims, 196, nvec=1))
    F = torch.empty(36 * int(np.prod(dims)), dtype=torch.complex128, device="cuda")
    ctx.qcd_eig_force(1, v, F)
    X = synth.su3_directions(dims, 197, 1)[0]
    der = ctx.qcd_eig_derivative(X, 1, v)[0]
    con = np.einsum('iab,iba->', host(F).reshape(-1, 3, 3), X.reshape(-1, 3, 3)).real
    scale = np.linalg.norm(host(F)) * np.linalg.norm(X)
    assert abs(con - der) < 1e-12 * max(abs(der), scale * 1e-2), (con, der)
    ctx.close()
