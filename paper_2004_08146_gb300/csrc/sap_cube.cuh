// SAP block solves on 2^4 blocks with the residual formed in the same launch
// (Eq. 2.10; included by mg.cu inside its anonymous namespace).
//
// One warp solves one block for one right-hand side: lane chi * 16 + l holds
// chirality half chi (spins 2 chi, 2 chi + 1) of block site l, so every block
// vector is 32 lanes x 6 complex, kept in shared memory as [6][32]: a lane's
// own entries and those of any neighbour lane are read without bank conflicts.
// In a 2^4 block each site has exactly one neighbour inside the block and one
// outside it per direction.  The inside link of every direction (daggered
// where the hop is backward, times -1/2) stays in registers for the whole solve
// (FP64: in shared memory); the clover block is read from shared memory once
// per step, which leaves the registers that two basis vectors at a time need.
// The residual b - op(tau) x is formed here from x of the block and of its
// 8-neighbourhood, whose blocks have the other colour and are not written by
// this launch; the separate residual pass computed it on both colours and went
// through memory.
// Arnoldi by modified Gram-Schmidt over pairs of basis vectors (one reduction
// of four values per pair instead of two of two; one by one with the FP16 basis, 1258
// against 1165 us per colour at ten steps, 578 against 564 stopped at 1e-1); every lane
// carries the plane rotations of
// the new column in registers while the projections run, and the triangular
// solve runs one row per lane, so no step waits for a serial lane.  The
// rotation of (a, b), b real, is (conj(c), s; -s, c) with c = a / r complex and
// s = b / r real, r = sqrt(|a|^2 + b^2): the diagonal of R and the rotated
// right-hand side g stay real, the residual is |g| and one reciprocal square
// root serves c, s and the triangular solve (no divisions).
// Bound: instruction issue and the latency of the reductions at 12 warps per SM
// (3 CTAs: registers and the FP32 basis of 10 vectors allow no more).  Measured
// on 32 x 16^3, 16 right-hand sides, ten steps: 1.19 ms per colour (65,536
// solves) with the residual, against 2.64 ms for the solves (site-major block
// vectors: 4- to 8-way bank conflicts, rotations by one lane) and 0.27 ms for
// the residual pass before; on 16 x 8^3, 4 right-hand sides, stopped at 1e-1:
// 19 us against 27 + 11 us.

// Shared memory of a CTA of rw warps: outside and inside links [mu][9][16] and
// the lanes' clover blocks ([16-byte piece][32]) once, then per warp the basis
// (iters vectors [6][32]; the same space first holds x of the block and its four outside neighbours per site, 5 vectors in
// the working precision), R (column-major, reciprocal diagonal), rotations
// (s, c) and g.
template <typename R> struct alignas(16) CubeRot { R s, cx, cy, unused; };
struct CubeLayout {
    size_t el, il, cl, warps, rm, rot, g, perwarp, total;
};
template <typename R, typename BT>
__host__ __device__ inline CubeLayout cube_layout(int iters, int rw) {
    auto up = [](size_t v) { return (v + 15) & ~size_t(15); };
    constexpr size_t lnk = (size_t)36 * 16 * sizeof(cplx<R>);
    const size_t stage = (size_t)5 * 192 * sizeof(cplx<R>);
    size_t basis = (size_t)iters * 192 * sizeof(BT);
    if (basis < stage) basis = stage;
    CubeLayout L;
    L.el = 0;
    L.cl = lnk;
    size_t o = lnk + (size_t)36 * 32 * sizeof(R);
    // FP32: the inside links are only staged here on their way to registers;
    // they share warp 0's basis behind the staged x when that is long enough
    if (sizeof(R) == 4 && basis >= stage + lnk) {
        L.warps = o;
        L.il = o + stage;
    } else {
        L.il = o;
        o += lnk;
        L.warps = o;
    }
    size_t w = up(basis);
    L.rm = w;  w = up(w + (size_t)iters * iters * sizeof(cplx<R>));
    L.rot = w; w = up(w + (size_t)iters * sizeof(CubeRot<R>));
    L.g = w;   w = up(w + (size_t)iters * sizeof(cplx<R>));
    L.perwarp = w;
    L.total = L.warps + (size_t)rw * w;
    return L;
}

// half a spinor (6 complex entries, 16-byte aligned)
__device__ __forceinline__ void load_half(const float2* p, float2 (&v)[6]) {
    const float4* q = reinterpret_cast<const float4*>(p);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float4 t = q[k];
        v[2 * k] = make_float2(t.x, t.y);
        v[2 * k + 1] = make_float2(t.z, t.w);
    }
}
__device__ __forceinline__ void load_half(const double2* p, double2 (&v)[6]) {
#pragma unroll
    for (int k = 0; k < 6; ++k) v[k] = p[k];
}
__device__ __forceinline__ void store_half(float2* p, const float2 (&v)[6]) {
    float4* q = reinterpret_cast<float4*>(p);
#pragma unroll
    for (int k = 0; k < 3; ++k) q[k] = make_float4(v[2 * k].x, v[2 * k].y, v[2 * k + 1].x, v[2 * k + 1].y);
}
__device__ __forceinline__ void store_half(double2* p, const double2 (&v)[6]) {
#pragma unroll
    for (int k = 0; k < 6; ++k) p[k] = v[k];
}
// the lane's 36 reals of the clover term, staged in 16-byte pieces [piece][32]
__device__ __forceinline__ void stage_clover(const float* p, float* sm, int lane) {
    const float4* q = reinterpret_cast<const float4*>(p);
    float4 t[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) t[k] = __ldg(q + k);
#pragma unroll
    for (int k = 0; k < 9; ++k) reinterpret_cast<float4*>(sm)[k * 32 + lane] = t[k];
}
__device__ __forceinline__ void stage_clover(const double* p, double* sm, int lane) {
    const double2* q = reinterpret_cast<const double2*>(p);
#pragma unroll
    for (int k = 0; k < 18; ++k) reinterpret_cast<double2*>(sm)[k * 32 + lane] = __ldg(q + k);
}
__device__ __forceinline__ void load_clover(const float* sm, int lane, float (&a)[36]) {
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const float4 t = reinterpret_cast<const float4*>(sm)[k * 32 + lane];
        a[4 * k] = t.x; a[4 * k + 1] = t.y; a[4 * k + 2] = t.z; a[4 * k + 3] = t.w;
    }
}
__device__ __forceinline__ void load_clover(const double* sm, int lane, double (&a)[36]) {
#pragma unroll
    for (int k = 0; k < 18; ++k) {
        const double2 t = reinterpret_cast<const double2*>(sm)[k * 32 + lane];
        a[2 * k] = t.x; a[2 * k + 1] = t.y;
    }
}
// y = off-diagonal part of the block times x (first products written, not
// added); the diagonal comes last, so that the small terms are summed first
template <typename R>
__device__ __forceinline__ void clover_half_off(const R (&a)[36], const cplx<R> (&x)[6], cplx<R> (&y)[6]) {
#pragma unroll
    for (int i = 0; i < 6; ++i) {
#pragma unroll
        for (int j = i + 1; j < 6; ++j) {
            const int o = herm_off(i, j);
            const cplx<R> aij = mk<R>(a[o], a[o + 1]);
            if (i == 0 && j == 1) y[0] = aij * x[1];
            else cmac(y[i], aij, x[j]);
            if (i == 0) y[j] = cmulc(aij, x[0]);
            else cmacc(y[j], aij, x[i]);
        }
    }
}

// Sum of a complex number over the warp: the two halves of the warp first
// split re and im between them (7 shuffles, the last two independent, where
// two butterflies would take 10).
template <typename R>
__device__ __forceinline__ cplx<R> warp_sum2(cplx<R> v, int lane) {
    const bool up = lane & 16;
    R k = (up ? v.y : v.x) + __shfl_xor_sync(0xffffffffu, up ? v.x : v.y, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
    return mk<R>(__shfl_sync(0xffffffffu, k, 0), __shfl_sync(0xffffffffu, k, 16));
}
// Two complex sums at once: 10 shuffles, six deep.
template <typename R>
__device__ __forceinline__ void warp_sum4(cplx<R>& a, cplx<R>& b, int lane) {
    const bool up = lane & 16, q = lane & 8;
    const R kx = (up ? b.x : a.x) + __shfl_xor_sync(0xffffffffu, up ? a.x : b.x, 16);
    const R ky = (up ? b.y : a.y) + __shfl_xor_sync(0xffffffffu, up ? a.y : b.y, 16);
    R k = (q ? ky : kx) + __shfl_xor_sync(0xffffffffu, q ? kx : ky, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
    a = mk<R>(__shfl_sync(0xffffffffu, k, 0), __shfl_sync(0xffffffffu, k, 8));
    b = mk<R>(__shfl_sync(0xffffffffu, k, 16), __shfl_sync(0xffffffffu, k, 24));
}

// Adds the hop of direction mu to this lane's half: v is a block vector
// [6][32], n the lane site it is read at, e the link as applied (times -1/2),
// pm = -1 for a forward hop and +1 for a backward one.  h_s (s = chi) =
// up_s + pm (B dn)_s; the partner lane (lane ^ 16) has the other s.  Phases
// i of B and B^H occur for mu = 1, 3 only and the column swap for mu = 1, 2
// only, so all but the signs are known at compile time.
template <typename R, int mu, typename V, typename E>
__device__ __forceinline__ void cube_hop(const V* v, int n, int chi, R pm, const E& e, cplx<R> (&acc)[6]) {
    constexpr bool swap = mu == 1 || mu == 2;
    constexpr bool imag = mu == 1 || mu == 3;
    // B = -1, -i sigma_1, -i sigma_2, -i sigma_3: sign of row chi
    const R cb = (mu == 0 || mu == 1) ? -pm : (chi ? pm : -pm);
    const int sp = swap ? 1 - chi : chi;
    cplx<R> h[3], os[3], ot[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const cplx<R> up = bload(v + (chi * 3 + a) * 32 + n);
        const cplx<R> dn = bload(v + (sp * 3 + a) * 32 + 16 + n);
        h[a] = imag ? mk<R>(up.x - cb * dn.y, up.y + cb * dn.x) : mk<R>(up.x + cb * dn.x, up.y + cb * dn.y);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        cplx<R> s = e(mu * 9 + a * 3) * h[0];
#pragma unroll
        for (int b = 1; b < 3; ++b) cmac(s, e(mu * 9 + a * 3 + b), h[b]);
        os[a] = s;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a)
        ot[a] = mk<R>(__shfl_xor_sync(0xffffffffu, os[a].x, 16), __shfl_xor_sync(0xffffffffu, os[a].y, 16));
    // chi = 0: acc_s += o_s; chi = 1: acc_s += pm (B^H o)_s
    const bool own0 = swap || chi == 0;   // row 0 takes this lane's o
    if (!imag) {
        const R d0 = chi ? (mu == 0 ? -pm : pm) : R(1);
        const R d1 = chi ? -pm : R(1);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const cplx<R> p0 = own0 ? os[a] : ot[a], p1 = own0 ? ot[a] : os[a];
            acc[a].x += d0 * p0.x;
            acc[a].y += d0 * p0.y;
            acc[3 + a].x += d1 * p1.x;
            acc[3 + a].y += d1 * p1.y;
        }
    } else {
        const R f0 = chi ? pm : R(1), f1 = chi ? (mu == 1 ? pm : -pm) : R(1);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const cplx<R> p0 = own0 ? os[a] : ot[a], p1 = own0 ? ot[a] : os[a];
            const cplx<R> q0 = chi ? mk<R>(-p0.y, p0.x) : p0, q1 = chi ? mk<R>(-p1.y, p1.x) : p1;
            acc[a].x += f0 * q0.x;
            acc[a].y += f0 * q0.y;
            acc[3 + a].x += f1 * q1.x;
            acc[3 + a].y += f1 * q1.y;
        }
    }
}

// diagonal and shift: D - t Gamma5, or Gamma5 D - t
template <typename R>
__device__ __forceinline__ void cube_diag(int op, R t, int chi, const R (&a)[36], const cplx<R> (&psi)[6],
                                          cplx<R> (&acc)[6]) {
    const R g5 = chi ? R(-1) : R(1);
    const R ts = op == QCD_OP_D ? -t * g5 : -t;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        acc[k].x = fma(a[k], psi[k].x, acc[k].x);
        acc[k].y = fma(a[k], psi[k].y, acc[k].y);
    }
    if (op != QCD_OP_D)
#pragma unroll
        for (int k = 0; k < 6; ++k) acc[k] = g5 * acc[k];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        acc[k].x = fma(ts, psi[k].x, acc[k].x);
        acc[k].y = fma(ts, psi[k].y, acc[k].y);
    }
}

// 1 / sqrt(v) to working accuracy (0 for v = 0 and for infinity): the hardware
// estimate with one Newton step in FP32
__device__ __forceinline__ float inv_sqrt(float v) {
    const float r = rsqrtf(v);
    return v > 0.f && r > 0.f ? r * fmaf(-0.5f * v * r, r, 1.5f) : 0.f;
}
__device__ __forceinline__ double inv_sqrt(double v) { return v > 0.0 ? rsqrt(v) : 0.0; }

template <typename R> __device__ __forceinline__ R cube_threshold(double tol, R beta) {
    // largest working-precision value not above tol * beta
    const double t = tol * (double)beta;
    if constexpr (sizeof(R) == 4) return __double2float_rd(t);
    else return t;
}

// FP32: three CTAs of 128 threads per SM, the most that shared memory allows for
// ten basis vectors, so up to 168 registers cost nothing.
template <typename R, typename BT>
__global__ void __launch_bounds__(128, sizeof(R) == 4 ? 3 : 1)
sap_cube_kernel(Geom g, Blocking B, const cplx<R>* __restrict__ U, const R* __restrict__ A,
                const int* __restrict__ blocks, int op, Shifts tau, const cplx<R>* __restrict__ b, cplx<R>* x,
                int iters, double tol, const int* __restrict__ act, int nrhs) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, rw = blockDim.x >> 5;
    const int chi = lane >> 4, l = lane & 15;
    const CubeLayout LY = cube_layout<R, BT>(iters, rw);
    unsigned char* wbase = smraw + LY.warps + (size_t)wid * LY.perwarp;
    cplx<R>* el = reinterpret_cast<cplx<R>*>(smraw + LY.el);   // [mu * 9 + k][16]
    cplx<R>* il = reinterpret_cast<cplx<R>*>(smraw + LY.il);
    R* sclov = reinterpret_cast<R*>(smraw + LY.cl);
    cplx<R>* xs = reinterpret_cast<cplx<R>*>(wbase);           // [5][6][32], before the basis
    BT* basis = reinterpret_cast<BT*>(wbase);                  // [iters][6][32]
    cplx<R>* Rm = reinterpret_cast<cplx<R>*>(wbase + LY.rm);   // column-major, ld = iters
    CubeRot<R>* rot = reinterpret_cast<CubeRot<R>*>(wbase + LY.rot);
    cplx<R>* gv = reinterpret_cast<cplx<R>*>(wbase + LY.g);

    int x0[4];
    block_coords(B, blocks[blockIdx.x], x0);
    int ms[4];   // site stride of direction mu
    ms[3] = 1;
    ms[2] = g.L[3];
    ms[1] = g.L[3] * g.L[2];
    ms[0] = g.L[3] * g.L[2] * g.L[1];
    int y0 = 0;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        x0[mu] *= 2;
        y0 += x0[mu] * ms[mu];
    }
    // site of lane site ll, and its neighbour outside the block in direction
    // mu (backward where o_mu = 0, forward where o_mu = 1)
    auto o_of = [](int ll, int mu) { return (ll >> (3 - mu)) & 1; };
    auto site_of = [&](int ll) {
        int s = y0;
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) s += o_of(ll, mu) * ms[mu];
        return s;
    };
    auto outside_of = [&](int ll, int mu, bool& wraps) {
        const int o = o_of(ll, mu);
        const int xm = x0[mu] + (o ? 2 : -1);
        wraps = xm < 0 || xm >= g.L[mu];
        const int xw = xm < 0 ? g.L[mu] - 1 : (xm >= g.L[mu] ? 0 : xm);
        return site_of(ll) + (xw - x0[mu] - o) * ms[mu];
    };
    // ---- stage the links, as applied, times -1/2: 64 inside, 64 outside
    for (int t = threadIdx.x; t < 128; t += blockDim.x) {
        const int ll = t & 15, mu = (t >> 4) & 3, out = t >> 6;
        int msm = ms[0];
        if (mu == 1) msm = ms[1];
        if (mu == 2) msm = ms[2];
        if (mu == 3) msm = ms[3];
        const int o = (ll >> (3 - mu)) & 1;
        const int ys = site_of(ll);
        const bool fw = out ? o == 1 : o == 0;
        R sc = R(-0.5);
        int src = ys;
        if (!fw) src = ys - msm;
        if (out) {
            int Lm = g.L[0], xm = x0[0];
            if (mu == 1) { Lm = g.L[1]; xm = x0[1]; }
            if (mu == 2) { Lm = g.L[2]; xm = x0[2]; }
            if (mu == 3) { Lm = g.L[3]; xm = x0[3]; }
            const bool wraps = fw ? xm + 2 >= Lm : xm == 0;
            if (!fw && wraps) src = ys + (Lm - 1) * msm;
            if (wraps && mu == 0 && g.antiperiodic) sc = R(0.5);
        }
        const cplx<R>* u = U + ((size_t)src * 4 + mu) * 9;
        cplx<R>* dst = (out ? el : il) + mu * 9 * 16 + ll;
        cplx<R> e[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) e[k] = sc * __ldg(u + k);
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int c = 0; c < 3; ++c) dst[(a * 3 + c) * 16] = fw ? e[a * 3 + c] : conj(e[c * 3 + a]);
    }
    const int j = blockIdx.y * rw + wid;
    const bool mine = j < nrhs && (act == nullptr || act[j]);
    const size_t fstride = (size_t)g.V * 12;
    const int y = site_of(l);
    cplx<R> psi[6], w[6];
    if (wid == rw - 1) stage_clover(A + (size_t)y * 72 + 36 * chi, sclov, lane);
    if (mine) {
        b += j * fstride;
        x += j * fstride;
        load_half(x + (size_t)y * 12 + 6 * chi, psi);
        load_half(b + (size_t)y * 12 + 6 * chi, w);
        cplx<R> v[4][6];
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
            bool wr;
            load_half(x + (size_t)outside_of(l, mu, wr) * 12 + 6 * chi, v[mu]);
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) xs[k * 32 + lane] = psi[k];
#pragma unroll
        for (int mu = 0; mu < 4; ++mu)
#pragma unroll
            for (int k = 0; k < 6; ++k) xs[((mu + 1) * 6 + k) * 32 + lane] = v[mu][k];
    }
    __syncthreads();
    cplx<R> lk[sizeof(R) == 4 ? 36 : 1];
    if constexpr (sizeof(R) == 4) {
        if (mine) {
#pragma unroll
            for (int k = 0; k < 36; ++k) lk[k] = il[k * 16 + l];
        }
        __syncthreads();   // warp 0's basis may now overwrite the staged inside links
    }
    if (!mine) return;
    auto inside = [&](int k) {
        if constexpr (sizeof(R) == 4) return lk[k];
        else return il[k * 16 + l];
    };
    auto outside = [&](int k) { return el[k * 16 + l]; };
    const R t = (R)tau.t[j];
    R pm[4];   // of the inside hop: forward (-1) where o_mu = 0
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) pm[mu] = o_of(l, mu) ? R(1) : R(-1);
    // ---- residual w = b - op(tau) x on the block
    {
        cplx<R> acc[6];
        R cl[36];
        load_clover(sclov, lane, cl);
        clover_half_off<R>(cl, psi, acc);
        cube_hop<R, 0>(xs, l ^ 8, chi, pm[0], inside, acc);
        cube_hop<R, 1>(xs, l ^ 4, chi, pm[1], inside, acc);
        cube_hop<R, 2>(xs, l ^ 2, chi, pm[2], inside, acc);
        cube_hop<R, 3>(xs, l ^ 1, chi, pm[3], inside, acc);
        cube_hop<R, 0>(xs + 192, l, chi, -pm[0], outside, acc);
        cube_hop<R, 1>(xs + 384, l, chi, -pm[1], outside, acc);
        cube_hop<R, 2>(xs + 576, l, chi, -pm[2], outside, acc);
        cube_hop<R, 3>(xs + 768, l, chi, -pm[3], outside, acc);
        cube_diag<R>(op, t, chi, cl, psi, acc);
#pragma unroll
        for (int k = 0; k < 6; ++k) w[k] -= acc[k];
    }
    R nn = 0;
#pragma unroll
    for (int k = 0; k < 6; ++k) nn += w[k].x * w[k].x + w[k].y * w[k].y;
    nn = warp_sum(nn);
    if (!(nn > R(0))) return;
    // an infinite norm: vectors of zeros where the entries are finite (no correction),
    // of NaN where they are not, so that x shows it
    const R ib = inv_sqrt(nn), beta = ib > R(0) ? nn * ib : R(1);
    const R thr = cube_threshold<R>(tol, beta);
    __syncwarp();   // x of the neighbours is read
    {
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            bstore(basis + k * 32 + lane, ib * w[k]);
            psi[k] = bround<BT>(ib * w[k]);
        }
    }
    R gc = beta;
    int kdim = 0;
    for (int jj = 0; jj < iters; ++jj) {
        __syncwarp();
        const BT* vj = basis + (size_t)jj * 192;
        R cl[36];
        load_clover(sclov, lane, cl);
        clover_half_off<R>(cl, psi, w);
        cube_hop<R, 0>(vj, l ^ 8, chi, pm[0], inside, w);
        cube_hop<R, 1>(vj, l ^ 4, chi, pm[1], inside, w);
        cube_hop<R, 2>(vj, l ^ 2, chi, pm[2], inside, w);
        cube_hop<R, 3>(vj, l ^ 1, chi, pm[3], inside, w);
        cube_diag<R>(op, t, chi, cl, psi, w);
        // modified Gram-Schmidt, two basis vectors at a time where they are
        // orthogonal to each other to the working precision; vectors rounded to FP16
        // are so to 3e-4 only and go one by one.  rc: entry of the new column under
        // rotation
        constexpr bool kPairs = sizeof(BT) == sizeof(cplx<R>);
        cplx<R> rc = czero<R>();
        auto rotate = [&](int i, cplx<R> h) {
            if (i == 0) {
                rc = h;
                return;
            }
            const CubeRot<R> q = rot[i - 1];
            const cplx<R> c = mk<R>(q.cx, q.cy);
            cplx<R> up = q.s * h, dn = (-q.s) * rc;
            cmacc(up, c, rc);
            cmac(dn, c, h);
            if (lane == 0) Rm[(size_t)jj * iters + i - 1] = up;
            rc = dn;
        };
        int i = 0;
        for (; kPairs && i < jj; i += 2) {
            const BT* vi = basis + (size_t)i * 192 + lane;
            cplx<R> a0[6], a1[6], h0 = czero<R>(), h1 = czero<R>();
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                a0[k] = bload(vi + k * 32);
                a1[k] = bload(vi + 192 + k * 32);
                cmacc(h0, a0[k], w[k]);
                cmacc(h1, a1[k], w[k]);
            }
            warp_sum4<R>(h0, h1, lane);
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                cmsub(w[k], h0, a0[k]);
                cmsub(w[k], h1, a1[k]);
            }
            rotate(i, h0);
            rotate(i + 1, h1);
        }
        for (; i <= jj; ++i) {
            const BT* vi = basis + (size_t)i * 192 + lane;
            cplx<R> a[6], h = czero<R>();
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                a[k] = bload(vi + k * 32);
                cmacc(h, a[k], w[k]);
            }
            h = warp_sum2<R>(h, lane);
#pragma unroll
            for (int k = 0; k < 6; ++k) cmsub(w[k], h, a[k]);
            rotate(i, h);
        }
        R hn2 = 0;
#pragma unroll
        for (int k = 0; k < 6; ++k) hn2 += w[k].x * w[k].x + w[k].y * w[k].y;
        hn2 = warp_sum(hn2);
        const R ih = inv_sqrt(hn2), hn = hn2 * ih;
        const R irr = inv_sqrt(rc.x * rc.x + rc.y * rc.y + hn2);
        const R sn = irr > R(0) ? hn * irr : R(1);
        const cplx<R> c = irr * rc;
        if (lane == 0) {
            Rm[(size_t)jj * iters + jj] = mk<R>(irr, R(0));
            rot[jj] = CubeRot<R>{sn, c.x, c.y, R(0)};
            gv[jj] = gc * conj(c);
        }
        gc = -sn * gc;
        kdim = jj + 1;
        if ((tol >= 0.0 && fabs(gc) <= thr) || kdim == iters) break;
        BT* vn = basis + (size_t)kdim * 192 + lane;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            bstore(vn + k * 32, ih * w[k]);
            psi[k] = bround<BT>(ih * w[k]);
        }
    }
    __syncwarp();
    // ---- triangular solve, row i on lane i (iters <= 32)
    cplx<R> yv = lane < kdim ? gv[lane] : czero<R>();
    for (int k = kdim - 1; k >= 0; --k) {
        const R id = Rm[(size_t)k * iters + k].x;   // 0 for a zero pivot: no contribution
        const cplx<R> yk = id * mk<R>(__shfl_sync(0xffffffffu, yv.x, k), __shfl_sync(0xffffffffu, yv.y, k));
        if (lane < k) cmsub(yv, Rm[(size_t)k * iters + lane], yk);
        else if (lane == k) yv = yk;
    }
    if (lane == 0) count_sap_work(16, kdim);
    load_half(x + (size_t)y * 12 + 6 * chi, psi);
    for (int i = 0; i < kdim; ++i) {
        const cplx<R> yi = mk<R>(__shfl_sync(0xffffffffu, yv.x, i), __shfl_sync(0xffffffffu, yv.y, i));
        const BT* vi = basis + (size_t)i * 192 + lane;
#pragma unroll
        for (int k = 0; k < 6; ++k) cmac(psi[k], yi, bload(vi + k * 32));
    }
    store_half(x + (size_t)y * 12 + 6 * chi, psi);
}
