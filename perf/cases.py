"""Performance cases of the library: the calls a program makes through the
``qcd`` binding (and ``autograd.apply_Q``), over the sizes they are made at.

``listed()`` names twelve of them, ``draw(rng)`` gives another of the same
ranges, ``prepare(case, seed)`` builds what a program holds before the call,
``run(state)`` is one pass, ``work(case)`` the bytes and operations it cannot
do without and ``exact(case, seed)`` its result in plain torch at 64 bits (the
operator, block and coarse solves and derivatives written out below from the
conventions stated in ``include/qcd.h``).

Links are U = exp(i eps H) with eps, c_sw and m0 of the 16 x 8^3 workload.
Block solves that stop at a tolerance are compared at 16 x 8^3; the large
smoother case takes a fixed number of steps, because among half a million
block solves some residual always lies within rounding of the threshold.  For
the same reason the FP16-stored block basis has no case of its own: a last-bit
change of an FP32 sum moves FP16 roundings.
"""
import math

import numpy as np
import torch

from paper_2004_08146_gb300 import autograd, qcd

EPS, CSW, M0 = 0.5, 1.5, -0.85
DEV = "cuda"
C128 = torch.complex128


def listed():
    return [
        # the operator at the smallest lattice of the tests: a call a program makes
        # inside its own solver on a tiny lattice, where the launch is the cost
        _case("apply_q_4x4c3", "apply", (4, 4, 4, 4), "f64", 1, form="Q"),
        # the FP64 operator of residuals and Rayleigh quotients at an ordinary size
        _case("apply_q_32x16c3", "apply", (32, 16, 16, 16), "f64", 1, form="Q"),
        # the FP32 operator of the inner solves on the largest lattice
        _case("apply_f32_64x32c3", "apply", (64, 32, 32, 32), "f32", 1, form="D"),
        # the same for a batch of 16 shifted systems (32 x 16^3 workload: 16 targets)
        _case("apply_f32_32x16c3_n16", "apply", (32, 16, 16, 16), "f32", 16, form="D"),
        # a training step through the operator: forward, and backward to spinors and links
        _case("autograd_16c4_n8", "autograd", (16, 16, 16, 16), "f64", 8),
        # the smoother as the 16 x 8^3 eigensolve calls it: 4 targets, stopped at 1e-1
        _case("sap_16x8c3_n4", "sap", (16, 8, 8, 8), "f32", 4, sweeps=4, block_tol=0.1),
        # the smoother where the chip is full: 16 targets, ten steps per block solve
        _case("sap_32x16c3_n16", "sap", (32, 16, 16, 16), "f32", 16, sweeps=2, block_tol=-1.0),
        # restriction of 16 residuals and prolongation of 16 corrections (32 x 16^3 workload)
        _case("transfer_32x16c3_n16", "transfer", (32, 16, 16, 16), "f32", 16, nv=20, agg=4),
        # the level-1 stencil of the three-level hierarchy for 16 systems: the blocks
        # (0.7 GB) are the bulk of the bytes
        _case("coarse_32c4_n16", "coarse", (32, 32, 32, 32), "f32", 16, nv=24, agg=4),
        # one preconditioner application of the 16 x 8^3 workload
        _case("cycle_16x8c3_n4", "cycle", (16, 8, 8, 8), "f32", 4, nv=8),
        # whole call: four shifted systems solved to 1e-12 from a given hierarchy
        _case("solve_16x8c3_n4", "solve", (16, 8, 8, 8), "f64", 4, nv=8),
        # whole call: setup and 24 eigenpairs (8 guard pairs) of a 16 x 8^3 field
        _case("eigs_16x8c3_k24", "eigs", (16, 8, 8, 8), "f64", 4, nv=8, k=24),
    ]


def _case(name, kind, dims, prec, nrhs, **more):
    c = {"kind": kind, "prec": prec, "nrhs": nrhs}
    if name:
        c = {"name": name, **c}
    c.update({"L%d" % mu: int(d) for mu, d in enumerate(dims)})
    c.update(more)
    return c


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _extents(rng, vmin, vmax, unit, most):
    """Four extents, multiples of `unit` (at least 2), with vmin <= volume <= vmax."""
    while True:
        d = tuple(max(2, unit * max(1, round(_loguniform(rng, max(2, unit), most) / unit))) for _ in range(4))
        if vmin <= d[0] * d[1] * d[2] * d[3] <= vmax:
            return d


def draw(rng):
    kind = rng.choice(["apply", "apply", "autograd", "sap", "sap", "transfer", "coarse", "cycle", "solve"])
    if kind == "apply":
        # any extents, odd ones among them
        target = _loguniform(rng, 64, 2 << 20)
        d = _extents(rng, target // 2, min(2 * target, 2 << 20), 1, 64)
        prec = rng.choice(["f64", "f32", "f32"])
        vol = d[0] * d[1] * d[2] * d[3]
        n = max(1, min(_loguniform(rng, 1, 24), (4 << 20) // vol))
        return _case("", kind, d, prec, n, form=rng.choice(["D", "Q"]))
    if kind == "autograd":
        d = _extents(rng, 64, 32768, 1, 16)
        return _case("", kind, d, "f64", rng.randint(1, 8))
    if kind == "sap":
        d = _extents(rng, 256, 65536, 4, 32)
        vol = d[0] * d[1] * d[2] * d[3]
        fixed = rng.random() < 0.5
        n = max(1, min(rng.randint(1, 16), ((1 << 20) if fixed else 65536) // vol))
        return _case("", kind, d, rng.choice(["f32", "f32", "f64"]), n, sweeps=rng.randint(1, 4),
                     block_tol=-1.0 if fixed else 0.1)
    if kind in ("transfer", "coarse"):
        agg = rng.choice([2, 4])
        d = _extents(rng, 256, 131072, agg, 32)
        return _case("", kind, d, rng.choice(["f32", "f32", "f64"]), rng.randint(1, 20), nv=rng.randint(2, 24), agg=agg)
    d = _extents(rng, 1024, 8192, 4, 16)
    return _case("", kind, d, "f32" if kind == "cycle" else "f64", rng.randint(1, 6), nv=rng.randint(4, 10))


def _dims(c):
    return tuple(int(c["L%d" % mu]) for mu in range(4))


# ---------------------------------------------------------------- inputs
def _links(dims, seed):
    """Seeded links exp(i EPS H), H traceless Hermitian with unit-variance Gaussian entries."""
    gen = torch.Generator(device=DEV).manual_seed(int(seed) * 2 + 1)
    G = torch.randn(dims + (4, 3, 3), dtype=C128, device=DEV, generator=gen) * math.sqrt(2.0)
    H = 0.5 * (G + G.mH)
    del G
    tr = torch.diagonal(H, dim1=-2, dim2=-1).sum(-1).real / 3.0
    X = (1j * EPS / 16.0) * (H - tr[..., None, None] * torch.eye(3, dtype=C128, device=DEV))
    del H
    E = torch.eye(3, dtype=C128, device=DEV).expand(X.shape)
    for k in range(10, 0, -1):                       # Taylor of exp(X) by Horner's rule
        E = torch.eye(3, dtype=C128, device=DEV) + _mm(X, E) / k
    for _ in range(4):
        E = _mm(E, E)
    r0 = E[..., 0, :]
    r0 = r0 / torch.linalg.vector_norm(r0, dim=-1, keepdim=True)
    r1 = E[..., 1, :] - (r0.conj() * E[..., 1, :]).sum(-1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
    r2 = torch.linalg.cross(r0, r1, dim=-1).conj()
    return torch.stack([r0, r1, r2], dim=-2).contiguous()


def _field(n, dims, seed, salt, dtype=C128):
    gen = torch.Generator(device=DEV).manual_seed(int(seed) * 16 + salt)
    return torch.randn((n,) + dims + (4, 3), dtype=dtype, device=DEV, generator=gen) * math.sqrt(2.0)


def _prec(c):
    return (qcd.QCD_FP64, C128) if c["prec"] == "f64" else (qcd.QCD_FP32, torch.complex64)


def _taus(n, width=0.2):
    """Distinct shifts on both sides of zero, as the targets of one outer iteration have."""
    return [width * (2.0 * j + 1.0 - n) / n + 0.01 for j in range(n)]


def _context(c, U, **params):
    ctx = qcd.Context(stream=torch.cuda.current_stream().cuda_stream, **params)
    ctx.qcd_set_gauge(U.cpu().numpy(), _dims(c), M0, CSW)
    return ctx


def _near_kernel(U, nv, seed):
    """Test vectors: random fields with the upper spectrum of D^H D damped."""
    D = Wilson(U)
    V = _field(nv, U.shape[:4], seed, 5)
    for _ in range(24):
        V = V - D(D(V) * D.g5) * D.g5 / 48.0
    return V


def prepare(case, seed):
    kind, dims, n = case["kind"], _dims(case), case["nrhs"]
    prec, dtype = _prec(case)
    U = _links(dims, seed)
    s = {"kind": kind, "n": n, "prec": prec, "dims": dims}
    if kind == "apply":
        s["ctx"] = _context(case, U)
        s["op"] = qcd.QCD_OP_Q if case["form"] == "Q" else qcd.QCD_OP_D
        s["taus"] = _taus(n)
        s["x"] = _field(n, dims, seed, 1, dtype)
        s["y"] = torch.empty_like(s["x"])
    elif kind == "autograd":
        s["ctx"] = qcd.Context(stream=torch.cuda.current_stream().cuda_stream)
        s["links"] = U.requires_grad_(True)
        s["x"] = _field(n, dims, seed, 1).requires_grad_(True)
        s["g"] = _field(n, dims, seed, 2)
    elif kind == "sap":
        s["ctx"] = _context(case, U)
        s["taus"] = _taus(n)
        s["b"] = _field(n, dims, seed, 1, dtype)
        s["x"] = torch.zeros_like(s["b"])
        s["sweeps"], s["tol"] = case["sweeps"], case["block_tol"]
    elif kind in ("transfer", "coarse"):
        nv, agg = case["nv"], case["agg"]
        s["ctx"] = _context(case, U, precision=qcd.QCD_FP64 if case["prec"] == "f64" else qcd.QCD_MIXED,
                            sap_block=(agg,) * 4)
        s["ctx"].qcd_mg_update_from_eigvecs(_field(nv, dims, seed, 5), nv)
        s["taus"] = _taus(n)
        vc = dims[0] * dims[1] * dims[2] * dims[3] // agg ** 4
        gen = torch.Generator(device=DEV).manual_seed(int(seed) * 16 + 3)
        s["xc"] = torch.randn((n, vc, 2 * nv), dtype=dtype, device=DEV, generator=gen) * math.sqrt(2.0)
        s["yc"] = torch.empty_like(s["xc"])
        if kind == "transfer":
            s["r"] = _field(n, dims, seed, 1, dtype)
            s["x"] = torch.empty_like(s["r"])
    elif kind in ("cycle", "solve"):
        s["ctx"] = _context(case, U, coarse_maxiter=12)
        s["ctx"].qcd_mg_update_from_eigvecs(_near_kernel(U, case["nv"], seed), case["nv"])
        s["taus"] = _taus(n, 0.02)
        s["b"] = _field(n, dims, seed, 1, dtype)
        s["x"] = torch.empty_like(s["b"])
    else:
        s["ctx"] = _context(case, U, coarse_maxiter=12, block=n, guard=8)
        s["nv"], s["k"] = case["nv"], case["k"]
    return s


def run(s):
    ctx, kind, n, prec = s["ctx"], s["kind"], s["n"], s["prec"]
    if kind == "apply":
        if n == 1 and prec == qcd.QCD_FP64 and s["op"] == qcd.QCD_OP_Q:
            ctx.qcd_apply_Q(s["x"], s["y"], s["taus"][0])
        else:
            ctx.qcd_apply(s["op"], prec, n, s["x"], s["y"], s["taus"])
        return s["y"]
    if kind == "autograd":
        y = autograd.apply_Q(ctx, s["x"], 0.05, links=s["links"], lattice=(s["dims"], M0, CSW))
        gx, gu = torch.autograd.grad(y, (s["x"], s["links"]), grad_outputs=s["g"])
        return y.detach(), gx, gu
    if kind == "sap":
        s["x"].zero_()
        ctx.qcd_sap(qcd.QCD_OP_D, prec, n, s["b"], s["x"], s["taus"], s["sweeps"], s["tol"])
        return s["x"]
    if kind == "transfer":
        ctx.qcd_mg_restrict(prec, n, s["r"], s["yc"])
        ctx.qcd_mg_prolong(prec, n, s["xc"], s["x"])
        return s["yc"], s["x"]
    if kind == "coarse":
        ctx.qcd_coarse_apply(qcd.QCD_OP_D, prec, n, s["xc"], s["yc"], s["taus"])
        return s["yc"]
    if kind == "cycle":
        ctx.qcd_mg_cycle(qcd.QCD_OP_D, prec, n, s["b"], s["x"], s["taus"])
        return s["x"]
    if kind == "solve":
        ctx.qcd_shifted_solve_batched(list(s["b"]), list(s["x"]), s["taus"], 1e-12)
        return s["x"]
    ctx.qcd_mg_setup(s["nv"], (2, 2, 2, 2))
    return ctx.qcd_eigs(s["k"], 1e-8)[1]


# ---------------------------------------------------------------- work
def _sap_work(vol, n, es, sweeps, steps):
    # per site: its residual, then per GMRES step four hops inside the block, the
    # clover term and Gram-Schmidt against the block basis
    flops = sweeps * vol * n * (1824.0 + steps * 1250.0 + 96.0 * steps * (steps + 2))
    return vol * (n * 48.0 + 144.0) * es, flops


def _cycle_work(vol, n, es, nv):
    nc, vc = 2 * nv, vol / 16
    b, f = _sap_work(vol, n, es, 4, 4)
    b += vol * 24.0 * nv * es + vc * 9.0 * nc * nc * 2 * es
    f += 2 * 96.0 * vol * nv * n + 12 * 8.0 * 9 * nc * nc * vc * n
    return b, f


def work(case):
    kind, n = case["kind"], case["nrhs"]
    es = 8.0 if case["prec"] == "f64" else 4.0
    d = _dims(case)
    vol = float(d[0] * d[1] * d[2] * d[3])
    if kind == "apply":
        b, f = vol * (48.0 * n + 144.0) * es, 1824.0 * vol * n
    elif kind == "autograd":
        # two applies per field; colour outer products per field; the four-link
        # products of the clover derivative once (they are linear in the outer products)
        b, f = vol * (96.0 * n + 216.0) * es, vol * (n * (2 * 1824.0 + 5760.0) + 46700.0)
    elif kind == "sap":
        b, f = _sap_work(vol, n, es, case["sweeps"], 10 if case["block_tol"] < 0 else 4)
    elif kind == "transfer":
        b = vol * es * (2 * 24.0 * case["nv"] + 2 * 24.0 * n)
        f = 2 * 96.0 * vol * case["nv"] * n
    elif kind == "coarse":
        nc, vc = 2.0 * case["nv"], vol / case["agg"] ** 4
        b, f = vc * (9 * nc * nc + 2 * n * nc) * 2 * es, 8.0 * 9 * nc * nc * vc * n
    elif kind == "cycle":
        b, f = _cycle_work(vol, n, es, case["nv"])
    else:
        # about 60 preconditioned FP32 iterations per system solved or pair found
        _, f1 = _cycle_work(vol, 1, 4.0, case["nv"])
        m = case["k"] if kind == "eigs" else n
        b, f = vol * (24.0 * m * 2 + 144.0) * 8.0, 60.0 * m * (f1 + 1824.0 * vol)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- 64-bit results
def _mm(a, b):
    """Products of batches of 3 x 3 matrices."""
    return sum(a[..., :, k, None] * b[..., None, k, :] for k in range(3))


def _spin_mono(v, perm, phase):
    """(M v)_r = phase[r] v[perm[r]] on the spin axis (-2) of extent 2."""
    return torch.stack([phase[r] * v[..., perm[r], :] for r in range(2)], dim=-2)


# gamma_mu = [[0, B], [B^H, 0]]: B_0 = -1, B_k = -i sigma_k; rows (column, phase)
_B = [((0, 1), (-1, -1)), ((1, 0), (-1j, -1j)), ((1, 0), (-1, 1)), ((0, 1), (-1j, 1j))]
_BH = [((0, 1), (-1, -1)), ((1, 0), (1j, 1j)), ((1, 0), (1, -1)), ((0, 1), (1j, -1j))]


def _dense(mono):
    M = np.zeros((2, 2), dtype=complex)
    for r in range(2):
        M[r, mono[0][r]] = mono[1][r]
    return M


class Wilson:
    """D of Eq. 2.5 with the clover term, antiperiodic in time, on fields
    [n, L0, L1, L2, L3, 4, 3]; `block` drops the hops that leave a block."""

    def __init__(self, U, block=None):
        self.U, self.dims = U, tuple(U.shape[:4])
        self.g5 = torch.tensor([1.0, 1, -1, -1], dtype=torch.float64, device=U.device)[:, None]
        self.block = block
        self.A = self._clover()

    def _clover(self):
        U = self.U
        u = [U[..., mu, :, :] for mu in range(4)]

        def sh(f, mu, k, nu=0, m=0):          # f(x + k mu + m nu)
            f = torch.roll(f, -k, dims=mu) if k else f
            return torch.roll(f, -m, dims=nu) if m else f

        A = [0.0, 0.0]
        for mu in range(4):
            for nu in range(mu + 1, 4):
                a, b = u[mu], u[nu]
                q = _mm(_mm(a, sh(b, mu, 1)), _mm(b, sh(a, nu, 1)).mH)
                q = q + _mm(_mm(b, sh(a, mu, -1, nu, 1).mH), _mm(sh(b, mu, -1).mH, sh(a, mu, -1)))
                q = q + _mm(_mm(sh(b, mu, -1, nu, -1), sh(a, mu, -1)).mH, _mm(sh(a, mu, -1, nu, -1), sh(b, nu, -1)))
                q = q + _mm(_mm(sh(b, nu, -1).mH, sh(a, nu, -1)), _mm(sh(b, mu, 1, nu, -1), a.mH))
                F = (q - q.mH) / 8.0
                for chi in range(2):
                    X, Y = (_B, _BH) if chi == 0 else (_BH, _B)
                    sig = 0.5j * (_dense(X[mu]) @ _dense(Y[nu]) - _dense(X[nu]) @ _dense(Y[mu]))
                    sig = torch.from_numpy(sig).to(U.device) * (0.5j * CSW)
                    A[chi] = A[chi] + sig[:, None, :, None] * F[..., None, :, None, :]
        one = torch.eye(6, dtype=C128, device=U.device) * (M0 + 4.0)
        return [a.reshape(self.dims + (6, 6)) + one for a in A]

    def _inside(self, f, mu, fwd):
        """f with the entries zeroed whose hop in direction mu leaves the block."""
        if self.block is None:
            return f
        x = torch.arange(self.dims[mu], device=f.device) % self.block
        keep = (x != self.block - 1) if fwd else (x != 0)
        shape = [1] * f.dim()
        shape[1 + mu] = -1
        return f * keep.to(torch.float64).reshape(shape)

    def __call__(self, psi):
        n = psi.shape[0]
        out = []
        for chi in range(2):
            v = psi[..., 2 * chi:2 * chi + 2, :].reshape((n,) + self.dims + (6,))
            w = sum(self.A[chi][..., :, k] * v[..., k, None] for k in range(6))
            out.append(w.reshape((n,) + self.dims + (2, 3)))
        up, dn = psi[..., :2, :], psi[..., 2:, :]
        for mu in range(4):
            bd = _spin_mono(dn, *_B[mu])
            sign = torch.ones(self.dims[mu], dtype=torch.float64, device=psi.device)
            if mu == 0:
                sign[-1] = -1.0                     # the hop between the last and the first slice
            shape = [1] * psi.dim()
            shape[1 + mu] = -1
            u = self.U[..., mu, :, :]
            h = torch.roll(up - bd, -1, dims=1 + mu) * sign.reshape(shape)
            o = sum(u[..., None, :, k] * h[..., k, None] for k in range(3))
            o = self._inside(o, mu, True) * -0.5
            h = up + bd
            p = sum(u[..., None, k, :].conj() * h[..., k, None] for k in range(3)) * sign.reshape(shape)
            p = self._inside(torch.roll(p, 1, dims=1 + mu), mu, False) * -0.5
            out[0] = out[0] + o + p
            out[1] = out[1] + _spin_mono(p - o, *_BH[mu])
        return torch.cat(out, dim=-2)

    def shifted(self, psi, taus, form="D"):
        t = torch.tensor(taus, dtype=torch.float64, device=psi.device).reshape((-1,) + (1,) * (psi.dim() - 1))
        if form == "D":
            return self(psi) - t * (self.g5 * psi)
        return self.g5 * self(psi) - t * psi


class Blocks:
    """Inner products and scalings block by block of extent `b`."""

    def __init__(self, dims, b):
        self.dims, self.b = dims, b
        self.shape = sum(([d // b, b] for d in dims), [])

    def split(self, f):                             # [n, grid..., b..., 4, 3]
        n = f.shape[0]
        return f.reshape([n] + self.shape + [4, 3]).permute(0, 1, 3, 5, 7, 2, 4, 6, 8, 9, 10)

    def join(self, f):
        return f.permute(0, 1, 5, 2, 6, 3, 7, 4, 8, 9, 10).reshape((f.shape[0],) + self.dims + (4, 3))

    def dot(self, a, b):
        return self.split(a.conj() * b).sum(dim=(5, 6, 7, 8, 9, 10))

    def scale(self, c, f):
        return self.join(self.split(f) * c[..., None, None, None, None, None, None])


def _gmres(apply, r, dot, scale, steps, tol):
    """`steps` GMRES steps from zero on every group of `dot` (stopped at tol times its norm): the correction."""
    def inv(x):
        return torch.where(x > 0, 1.0 / torch.where(x > 0, x, torch.ones_like(x)), torch.zeros_like(x))

    beta = dot(r, r).real.sqrt()
    v = [scale(inv(beta).to(C128), r)]
    g, cols, cs, sn = [beta.to(C128)], [], [], []
    kdim = torch.full(beta.shape, steps, device=r.device)
    done = beta <= 0
    for j in range(steps):
        w, h = apply(v[j]), []
        for i in range(j + 1):
            h.append(dot(v[i], w))
            w = w - scale(h[i], v[i])
        hn = dot(w, w).real.sqrt()
        v.append(scale(inv(hn).to(C128), w))
        for i in range(j):
            h[i], h[i + 1] = cs[i] * h[i] + sn[i] * h[i + 1], cs[i] * h[i + 1] - sn[i].conj() * h[i]
        rr = (h[j].abs() ** 2 + hn ** 2).sqrt()
        cs.append(h[j].abs() * inv(rr))
        sn.append(h[j] * inv(h[j].abs()) * hn * inv(rr))
        h[j] = cs[j] * h[j] + sn[j] * hn
        g.append(-sn[j].conj() * g[j])
        g[j] = cs[j] * g[j]
        cols.append(h)
        now = (~done) & (g[j + 1].abs() <= tol * beta)
        kdim = torch.where(now, torch.full_like(kdim, j + 1), kdim)
        done = done | now
        if bool(done.all()):
            break
    e = torch.zeros_like(r)
    y = {}
    for i in reversed(range(len(cols))):
        # columns past a group's own step count are left out, and its g ends there
        s = g[i]
        for k in range(i + 1, len(cols)):
            s = s - cols[k][i] * y[k]
        y[i] = torch.where((kdim > i) & (beta > 0), s / torch.where(cols[i][i] == 0, 1.0, cols[i][i]), 0.0)
        e = e + scale(y[i], v[i])
    return e


def _sap(U, b, x, taus, sweeps, tol, steps=10):
    full, inner, B = Wilson(U), Wilson(U, block=2), Blocks(tuple(U.shape[:4]), 2)
    grid = torch.meshgrid(*[torch.arange(d // 2, device=DEV) for d in U.shape[:4]], indexing="ij")
    colour = (grid[0] + grid[1] + grid[2] + grid[3]) % 2
    for _ in range(sweeps):
        for c in range(2):
            mask = (colour == c).to(C128)[None]
            r = B.scale(mask, b - full.shifted(x, taus))
            x = x + _gmres(lambda v: inner.shifted(v, taus), r, B.dot, B.scale, steps, tol)
    return x


class Aggregates:
    """P of the test vectors V [nv, ...] over aggregates of extent b: [sites, chirality, nv, entries]."""

    def __init__(self, V, b):
        self.dims, self.blocks, self.nv = tuple(V.shape[1:5]), Blocks(tuple(V.shape[1:5]), b), V.shape[0]
        q = list(self.local(V).unbind(0))           # each [sites, chirality, entries]
        for _ in range(2):
            for i in range(self.nv):
                for j in range(i):
                    q[i] = q[i] - (q[j].conj() * q[i]).sum(-1, keepdim=True) * q[j]
                q[i] = q[i] / torch.linalg.vector_norm(q[i], dim=-1, keepdim=True)
        self.P = torch.stack(q, dim=2)

    def local(self, f):                             # [n, sites, chirality, entries]
        n, b = f.shape[0], self.blocks.b
        s = self.blocks.split(f).reshape(n, -1, b ** 4, 2, 6)
        return s.permute(0, 1, 3, 2, 4).reshape(n, s.shape[1], 2, -1)

    def restrict(self, f):                          # [n, sites, 2 nv]
        return torch.stack([torch.einsum("scie,sce->sci", self.P.conj(), v) for v in self.local(f)]).flatten(2)

    def prolong(self, xc):
        n, b = xc.shape[0], self.blocks.b
        y = xc.reshape(n, -1, 2, self.nv)
        f = torch.stack([torch.einsum("scie,sci->sce", self.P, v) for v in y])
        f = f.reshape(n, -1, 2, b ** 4, 6).permute(0, 1, 3, 2, 4)
        grid = [d // b for d in self.dims]
        return self.blocks.join(f.reshape([n] + grid + [b] * 4 + [4, 3]))


def exact(case, seed):
    kind, dims, n = case["kind"], _dims(case), case["nrhs"]
    if kind == "eigs":
        return None
    _, dtype = _prec(case)
    U = _links(dims, seed)
    if kind == "apply":
        return Wilson(U).shifted(_field(n, dims, seed, 1, dtype).to(C128), _taus(n), case["form"])
    if kind == "autograd":
        U.requires_grad_(True)
        x = _field(n, dims, seed, 1).requires_grad_(True)
        y = Wilson(U).shifted(x, [0.05] * n, "Q")
        gx, gu = torch.autograd.grad(y, (x, U), grad_outputs=_field(n, dims, seed, 2))
        with torch.no_grad():                       # tangent to SU(3): i F U, F traceless Hermitian
            M = 1j * _mm(U, gu.mH)
            F = 0.5 * (M + M.mH)
            tr = torch.diagonal(F, dim1=-2, dim2=-1).sum(-1).real / 3.0
            F = F - tr[..., None, None] * torch.eye(3, dtype=C128, device=DEV)
            return y.detach(), gx, 1j * _mm(F, U)
    if kind == "sap":
        b = _field(n, dims, seed, 1, dtype).to(C128)
        return _sap(U, b, torch.zeros_like(b), _taus(n), case["sweeps"], case["block_tol"])
    if kind in ("transfer", "coarse"):
        P = Aggregates(_field(case["nv"], dims, seed, 5), case["agg"])
        gen = torch.Generator(device=DEV).manual_seed(int(seed) * 16 + 3)
        vc = dims[0] * dims[1] * dims[2] * dims[3] // case["agg"] ** 4
        xc = (torch.randn((n, vc, 2 * case["nv"]), dtype=dtype, device=DEV, generator=gen) * math.sqrt(2.0)).to(C128)
        if kind == "transfer":
            return P.restrict(_field(n, dims, seed, 1, dtype).to(C128)), P.prolong(xc)
        D, taus = Wilson(U), _taus(n)
        return torch.cat([P.restrict(D.shifted(P.prolong(xc[j:j + 1]), taus[j:j + 1])) for j in range(n)])
    taus = _taus(n, 0.02)
    b = _field(n, dims, seed, 1, dtype).to(C128)
    D = Wilson(U)
    if kind == "cycle":
        P = Aggregates(_near_kernel(U, case["nv"], seed), 2)
        xc = _gmres(lambda v: P.restrict(D.shifted(P.prolong(v), taus)), P.restrict(b),
                    lambda a, c: (a.conj() * c).sum(dim=(1, 2)), lambda c, f: c[:, None, None] * f, 12, 0.5)
        return _sap(U, b, P.prolong(xc), taus, 4, 0.1)
    # conjugate gradients on the normal equations (Q - tau is Hermitian)
    Q = lambda v: D.shifted(v, taus, "Q")  # noqa: E731
    x = torch.zeros_like(b)
    r = Q(b)
    p, rr = r, r.abs().square().sum(dim=(1, 2, 3, 4, 5, 6), keepdim=True)
    stop = rr * 1e-30
    for it in range(2500):
        q = Q(Q(p))
        a = rr / (p.conj() * q).real.sum(dim=(1, 2, 3, 4, 5, 6), keepdim=True).clamp_min(1e-300)
        x, r = x + a * p, r - a * q
        new = r.abs().square().sum(dim=(1, 2, 3, 4, 5, 6), keepdim=True)
        p, rr = r + (new / rr.clamp_min(1e-300)) * p, new
        if it % 50 == 49 and bool((rr <= stop).all()):
            break
    return x
