// Device building blocks of the Wilson-clover operator (Eq. 2.5 plus the
// clover term): spinor loads/stores, SU(3) products, spin projection with
// the chiral-basis monomials of common.cuh and the packed clover apply.
#pragma once
#include "common.cuh"

namespace qcd {

template <typename R> struct Spinor { cplx<R> c[12]; };   // index = spin*3 + colour

template <typename R> __device__ __forceinline__ void load_spinor(const cplx<R>* __restrict__ p, Spinor<R>& s);
template <> __device__ __forceinline__ void load_spinor<double>(const double2* __restrict__ p, Spinor<double>& s) {
#pragma unroll
    for (int k = 0; k < 12; ++k) s.c[k] = __ldg(p + k);
}
template <> __device__ __forceinline__ void load_spinor<float>(const float2* __restrict__ p, Spinor<float>& s) {
    const float4* q = reinterpret_cast<const float4*>(p);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        float4 v = __ldg(q + k);
        s.c[2 * k] = make_float2(v.x, v.y);
        s.c[2 * k + 1] = make_float2(v.z, v.w);
    }
}
// 32 bytes per load and store (complex64, 32-byte aligned): a warp reading one
// 96-byte spinor per lane touches 24 lines with every load, so three loads of 32
// bytes cost the L1 pipe half of what six of 16 bytes do
__device__ __forceinline__ void load8(const float2* __restrict__ p, float2* v) {
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(v[0].x), "=f"(v[0].y), "=f"(v[1].x), "=f"(v[1].y), "=f"(v[2].x), "=f"(v[2].y), "=f"(v[3].x), "=f"(v[3].y)
        : "l"(p));
}
__device__ __forceinline__ void store8(float2* p, const float2* v) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0].x), "f"(v[0].y),
                 "f"(v[1].x), "f"(v[1].y), "f"(v[2].x), "f"(v[2].y), "f"(v[3].x), "f"(v[3].y)
                 : "memory");
}
template <bool W32> __device__ __forceinline__ void load_spinor_w(const float2* __restrict__ p, Spinor<float>& s) {
    if constexpr (W32) {
#pragma unroll
        for (int k = 0; k < 3; ++k) load8(p + 4 * k, s.c + 4 * k);
    } else {
        load_spinor<float>(p, s);
    }
}

template <typename R> __device__ __forceinline__ void store_spinor(cplx<R>* __restrict__ p, const Spinor<R>& s);
template <> __device__ __forceinline__ void store_spinor<double>(double2* __restrict__ p, const Spinor<double>& s) {
#pragma unroll
    for (int k = 0; k < 12; ++k) p[k] = s.c[k];
}
template <> __device__ __forceinline__ void store_spinor<float>(float2* __restrict__ p, const Spinor<float>& s) {
    float4* q = reinterpret_cast<float4*>(p);
#pragma unroll
    for (int k = 0; k < 6; ++k) q[k] = make_float4(s.c[2 * k].x, s.c[2 * k].y, s.c[2 * k + 1].x, s.c[2 * k + 1].y);
}

template <typename R> struct Link { cplx<R> e[9]; };
template <typename R> __device__ __forceinline__ void load_link(const cplx<R>* __restrict__ p, Link<R>& u) {
#pragma unroll
    for (int k = 0; k < 9; ++k) u.e[k] = __ldg(p + k);
}

// y = U h (dag = false) or U^H h (dag = true) on a 2-spinor h[2][3]
template <typename R, bool dag>
__device__ __forceinline__ void su3_mul_half(const Link<R>& u, const cplx<R> h[6], cplx<R> o[6]) {
#pragma unroll
    for (int s = 0; s < 2; ++s) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            cplx<R> acc = czero<R>();
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                if (b == 0) acc = dag ? cmulc(u.e[a], h[s * 3]) : u.e[a * 3] * h[s * 3];
                else if (dag) cmacc(acc, u.e[b * 3 + a], h[s * 3 + b]);
                else cmac(acc, u.e[a * 3 + b], h[s * 3 + b]);
            }
            o[s * 3 + a] = acc;
        }
    }
}

// Hop contribution of direction mu: psi is the neighbour spinor (with the
// boundary sign already folded into `sgn`), U the link (U_mu(x) forward,
// U_mu(x-mu) backward, used daggered).  Adds
//   forward : -1/2 (1 - gamma_mu) U psi   -> up += -1/2 U h,  dn += +1/2 B^H U h,  h = up - B dn
//   backward: -1/2 (1 + gamma_mu) U^H psi -> up += -1/2 U^H h, dn += -1/2 B^H U^H h, h = up + B dn
template <typename R, int mu, bool fwd>
__device__ __forceinline__ void hop_accumulate(const Spinor<R>& psi, const Link<R>& u, R sgn, Spinor<R>& acc) {
    constexpr SpinMono B = kB(mu);
    constexpr SpinMono BH = kBH(mu);
    cplx<R> h[6], o[6];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            cplx<R> bd = mul_ipow(psi.c[(2 + B.perm[s]) * 3 + a], B.ph[s]);
            h[s * 3 + a] = fwd ? (psi.c[s * 3 + a] - bd) : (psi.c[s * 3 + a] + bd);
        }
    }
    su3_mul_half<R, !fwd>(u, h, o);
    const R half = R(-0.5) * sgn;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            acc.c[s * 3 + a] += half * o[s * 3 + a];
            cplx<R> bo = mul_ipow(o[BH.perm[s] * 3 + a], BH.ph[s]);
            if (fwd) acc.c[(2 + s) * 3 + a] -= half * bo;
            else     acc.c[(2 + s) * 3 + a] += half * bo;
        }
    }
}

// The same hop with the direction chosen at run time (fwd: U_mu(x) and
// 1 - gamma_mu; otherwise U_mu(x-mu)^H and 1 + gamma_mu), so that lanes with
// neighbours on different sides share one instruction stream.
template <typename R, int mu>
__device__ __forceinline__ void hop_accumulate_dir(const Spinor<R>& psi, const Link<R>& u, R sgn, bool fwd,
                                                   Spinor<R>& acc) {
    constexpr SpinMono B = kB(mu);
    constexpr SpinMono BH = kBH(mu);
    const R pm = fwd ? R(-1) : R(1);
    cplx<R> h[6], o[6];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const cplx<R> bd = mul_ipow(psi.c[(2 + B.perm[s]) * 3 + a], B.ph[s]);
            h[s * 3 + a] = psi.c[s * 3 + a] + pm * bd;
        }
    }
    cplx<R> e[9];   // U or U^H
#pragma unroll
    for (int a = 0; a < 3; ++a) {
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const cplx<R> d = u.e[a * 3 + b], t = u.e[b * 3 + a];
            e[a * 3 + b] = fwd ? d : conj(t);
        }
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            cplx<R> accv = czero<R>();
#pragma unroll
            for (int b = 0; b < 3; ++b) cmac(accv, e[a * 3 + b], h[s * 3 + b]);
            o[s * 3 + a] = accv;
        }
    }
    const R half = R(-0.5) * sgn;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            acc.c[s * 3 + a] += half * o[s * 3 + a];
            const cplx<R> bo = mul_ipow(o[BH.perm[s] * 3 + a], BH.ph[s]);
            acc.c[(2 + s) * 3 + a] += (pm * half) * bo;
        }
    }
}

// y = (off-diagonal part of A) x for one packed Hermitian 6x6 block (diagonal
// reals, then the upper triangle as (re, im) pairs in herm_off order).  The
// diagonal term, the largest of a row, is added last (clover_diag), so that the
// partial sums before it are small and round less.
template <typename R>
__device__ __forceinline__ void herm_off_apply(const R* a, const cplx<R>* xs, cplx<R>* ys) {
#pragma unroll
    for (int i = 0; i < 6; ++i) {
#pragma unroll
        for (int j = i + 1; j < 6; ++j) {
            const int o = herm_off(i, j);
            const cplx<R> aij = mk<R>(a[o], a[o + 1]);
            if (i == 0 && j == 1) ys[0] = aij * xs[1];
            else cmac(ys[i], aij, xs[j]);
            if (i == 0) ys[j] = cmulc(aij, xs[0]);
            else cmacc(ys[j], aij, xs[i]);
        }
    }
}

// y = A x for the two packed blocks of a site
template <typename R>
__device__ __forceinline__ void clover_apply_regs(const R* a0, const Spinor<R>& x, Spinor<R>& y) {
#pragma unroll
    for (int chi = 0; chi < 2; ++chi) {
        herm_off_apply<R>(a0 + 36 * chi, x.c + 6 * chi, y.c + 6 * chi);
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            const R d = a0[36 * chi + i];
            cplx<R>& v = y.c[6 * chi + i];
            v.x = fma(d, x.c[6 * chi + i].x, v.x);
            v.y = fma(d, x.c[6 * chi + i].y, v.y);
        }
    }
}

template <typename R>
__device__ __forceinline__ void clover_apply(const R* __restrict__ A, const Spinor<R>& x, Spinor<R>& y) {
    // the 72 reals of the site in 16-byte loads (288 B in FP32, 576 B in FP64)
    R ar[72];
    if constexpr (sizeof(R) == 4) {
        const float4* q = reinterpret_cast<const float4*>(A);
#pragma unroll
        for (int k = 0; k < 18; ++k) {
            const float4 v = __ldg(q + k);
            ar[4 * k] = v.x; ar[4 * k + 1] = v.y; ar[4 * k + 2] = v.z; ar[4 * k + 3] = v.w;
        }
    } else {
        const double2* q = reinterpret_cast<const double2*>(A);
#pragma unroll
        for (int k = 0; k < 36; ++k) {
            const double2 v = __ldg(q + k);
            ar[2 * k] = v.x; ar[2 * k + 1] = v.y;
        }
    }
    clover_apply_regs<R>(ar, x, y);
}

// Same product with the packed blocks in shared memory.
template <typename R>
__device__ __forceinline__ void clover_apply_smem(const R* A, const Spinor<R>& x, Spinor<R>& y) {
    clover_apply_regs<R>(A, x, y);
}
// neighbour site and boundary sign
__device__ __forceinline__ int nb_fwd(const Geom& g, const int x[4], int s, int mu, int& sgn_neg) {
    int y[4] = {x[0], x[1], x[2], x[3]};
    y[mu] += 1;
    sgn_neg = 0;
    if (y[mu] == g.L[mu]) { y[mu] = 0; if (mu == 0 && g.antiperiodic) sgn_neg = 1; }
    return site_index(g, y);
}
__device__ __forceinline__ int nb_bwd(const Geom& g, const int x[4], int s, int mu, int& sgn_neg) {
    int y[4] = {x[0], x[1], x[2], x[3]};
    y[mu] -= 1;
    sgn_neg = 0;
    if (y[mu] < 0) { y[mu] = g.L[mu] - 1; if (mu == 0 && g.antiperiodic) sgn_neg = 1; }
    return site_index(g, y);
}

}  // namespace qcd
