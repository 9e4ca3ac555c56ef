// Fine-lattice operator kernels: clover construction (Sec. 4, Table 1 clover
// term; Sheikholeslami-Wohlert) and the Wilson-clover stencil of Eq. 2.5 in
// the shifted forms D - tau Gamma5 (Eq. 3.7) and Q - tau (Eq. 3.6).
#include <algorithm>
#include <cstring>

#include "internal.h"
#include "dirac.cuh"

namespace qcd {

// ------------------------------------------------------------------ SU(3) helpers
template <typename R> struct M3 { cplx<R> e[3][3]; };
__device__ __forceinline__ M3<double> m3_load(const double2* p) {
    M3<double> m;
    for (int a = 0; a < 3; ++a) for (int b = 0; b < 3; ++b) m.e[a][b] = p[a * 3 + b];
    return m;
}
// One element of x y.  kTwo: the terms with Re x and with Im x in sums of their own;
// seven operations per component round as little as the eight of products added up
// one by one, where six in one chain round 5 % more (rms), and a chain on top of a
// running sum twice as much (link gradient, 4^4: 2.07e-16 from the exact one against
// 2.22e-16 with single chains, the plaquettes 1.93 ms against 1.49 on 16^4).
template <bool kTwo>
__device__ __forceinline__ double2 m3_row(const M3<double>& x, const M3<double>& y, int a, int b) {
    const double2 u = x.e[a][0], v = y.e[0][b];
    if constexpr (!kTwo) {
        double2 s = u * v;
        cmac(s, x.e[a][1], y.e[1][b]);
        cmac(s, x.e[a][2], y.e[2][b]);
        return s;
    }
    double2 s = make_double2(u.x * v.x, u.x * v.y), t = make_double2(u.y * v.y, u.y * v.x);
#pragma unroll
    for (int c = 1; c < 3; ++c) {
        const double2 p = x.e[a][c], q = y.e[c][b];
        s.x = fma(p.x, q.x, s.x);
        s.y = fma(p.x, q.y, s.y);
        t.x = fma(p.y, q.y, t.x);
        t.y = fma(p.y, q.x, t.y);
    }
    return make_double2(s.x - t.x, s.y + t.y);
}
template <bool kTwo = true>
__device__ __forceinline__ M3<double> m3_mul(const M3<double>& x, const M3<double>& y) {
    M3<double> r;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) r.e[a][b] = m3_row<kTwo>(x, y, a, b);
    return r;
}
// z += x y
__device__ __forceinline__ void m3_mac(M3<double>& z, const M3<double>& x, const M3<double>& y) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) z.e[a][b] += m3_row<true>(x, y, a, b);
}
__device__ __forceinline__ M3<double> m3_dag(const M3<double>& x) {
    M3<double> r;
    for (int a = 0; a < 3; ++a) for (int b = 0; b < 3; ++b) r.e[a][b] = conj(x.e[b][a]);
    return r;
}

__device__ __forceinline__ int shifted(const Geom& g, const int x[4], int mu, int dmu, int nu, int dnu) {
    int y[4] = {x[0], x[1], x[2], x[3]};
    y[mu] = (y[mu] + dmu + g.L[mu]) % g.L[mu];
    y[nu] = (y[nu] + dnu + g.L[nu]) % g.L[nu];
    return site_index(g, y);
}

// sigma^chi_{mu nu} (2x2, chirality block chi) = (i/2)(B_mu B_nu^H - B_nu B_mu^H)
// for chi = 0 and (i/2)(B_mu^H B_nu - B_nu^H B_mu) for chi = 1.
__device__ void spin_block_dense(int mu, bool herm, double2 M[2][2]) {
    SpinMono m = herm ? kBH(mu) : kB(mu);
    for (int r = 0; r < 2; ++r) for (int c = 0; c < 2; ++c) M[r][c] = make_double2(0, 0);
    for (int r = 0; r < 2; ++r) M[r][m.perm[r]] = mul_ipow(make_double2(1, 0), m.ph[r]);
}
__device__ void sigma_block(int mu, int nu, int chi, double2 S[2][2]) {
    double2 A[2][2], Bh[2][2], Bn[2][2], Ah[2][2];
    // chi = 0: X_mu = B_mu, Y_nu = B_nu^H ; chi = 1: X_mu = B_mu^H, Y_nu = B_nu
    spin_block_dense(mu, chi == 1, A);
    spin_block_dense(nu, chi == 0, Bh);
    spin_block_dense(nu, chi == 1, Bn);
    spin_block_dense(mu, chi == 0, Ah);
    for (int r = 0; r < 2; ++r) for (int c = 0; c < 2; ++c) {
        double2 s = make_double2(0, 0);
        for (int k = 0; k < 2; ++k) s += A[r][k] * Bh[k][c] - Bn[r][k] * Ah[k][c];
        S[r][c] = mul_ipow(0.5 * s, 1);
    }
}

// The packed blocks A_chi = (m0 + 4) + C_chi with C = c_sw (i/2) sum_{mu<nu}
// sigma_{mu nu} (x) F_{mu nu}, F_{mu nu} = (Q_{mu nu} - Q_{mu nu}^H)/8 from the four
// plaquette leaves.  With the staples above and below the link (x, mu)
//   D = U_nu(x+mu) U_mu(x+nu)^H U_nu(x)^H - U_nu(x+mu-nu)^H U_mu(x-nu)^H U_nu(x-nu)
// the leaves pair up: Q - Q^H = [U_mu(x) D(x) + D(x-mu) U_mu(x-mu)] - h.c., so a plane
// takes four products per site for D and two more, where the leaves by themselves
// take twelve.  Bound by the FP64 pipe.  16^4: 1.46 ms with one thread per site and
// its 72 sums in local memory, 0.62 now; the error of F against 80-bit arithmetic is
// the same (3.0e-17 rms at eps 0.3).

// plane p = 0 .. 5: (0,1) (0,2) (0,3) (1,2) (1,3) (2,3)
__device__ __forceinline__ void plane_dirs(int p, int& mu, int& nu) {
    mu = p < 3 ? 0 : (p < 5 ? 1 : 2);
    nu = p < 3 ? p + 1 : (p < 5 ? p - 1 : 3);
}
// D of planes 2 k, 2 k + 1 lives in d[k], [site][2][9]
struct StapleBufs { double2* d[3]; };

__global__ void __launch_bounds__(128) clover_staples_kernel(const double2* __restrict__ U, Geom g, StapleBufs D) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x, p = blockIdx.y;
    if (s >= g.V) return;
    int mu, nu, x[4];
    plane_dirs(p, mu, nu);
    site_coords(g, s, x);
    auto L = [&](int site, int d) { return m3_load(U + ((size_t)site * 4 + d) * 9); };
    const int down = shifted(g, x, mu, 0, nu, -1);
    M3<double> up = m3_mul<false>(m3_mul<false>(L(shifted(g, x, mu, 1, nu, 0), nu), m3_dag(L(shifted(g, x, mu, 0, nu, 1), mu))),
                           m3_dag(L(s, nu)));
    const M3<double> dn = m3_mul<false>(m3_mul<false>(m3_dag(L(shifted(g, x, mu, 1, nu, -1), nu)), m3_dag(L(down, mu))), L(down, nu));
    double2* o = D.d[p >> 1] + ((size_t)s * 2 + (p & 1)) * 9;
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) o[3 * a + b] = up.e[a][b] - dn.e[a][b];
}

// Warp p of a CTA makes F of plane p for 32 sites (9 reals, anti-Hermitian: Im of the
// diagonal, then (0,1), (0,2), (1,2)); then the CTA writes their blocks.  Per
// chirality sigma_{0k} = +-sigma_k and sigma_{jk} = -eps_jkl sigma_l, so C = sum_k
// sigma_k (x) E_k with E_1 = +-F_01 - F_23, E_2 = +-F_02 + F_13, E_3 = +-F_03 - F_12.
__global__ void __launch_bounds__(192) clover_assemble_kernel(const double2* __restrict__ U, Geom g, StapleBufs D,
                                                              double m0, double csw, double* __restrict__ A64,
                                                              float* __restrict__ A32) {
    __shared__ double F[6][9][32];
    const int lane = threadIdx.x & 31, p = threadIdx.x >> 5, s0 = blockIdx.x * 32, s = s0 + lane;
    if (csw != 0.0 && s < g.V) {
        int mu, nu, x[4];
        plane_dirs(p, mu, nu);
        site_coords(g, s, x);
        const int sm = shifted(g, x, mu, -1, nu, 0);
        auto Dl = [&](int site) { return m3_load(D.d[p >> 1] + ((size_t)site * 2 + (p & 1)) * 9); };
        M3<double> q = m3_mul<false>(m3_load(U + ((size_t)s * 4 + mu) * 9), Dl(s));
        const M3<double> d = Dl(sm), u = m3_load(U + ((size_t)sm * 4 + mu) * 9);
        for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b)
                for (int c = 0; c < 3; ++c) cmac(q.e[a][b], d.e[a][c], u.e[c][b]);
        double* f = &F[p][0][lane];
        for (int a = 0; a < 3; ++a) f[32 * a] = 0.25 * q.e[a][a].y;
        int k = 3;
        for (int a = 0; a < 3; ++a)
            for (int b = a + 1; b < 3; ++b, k += 2) {
                f[32 * k] = 0.125 * (q.e[a][b].x - q.e[b][a].x);
                f[32 * (k + 1)] = 0.125 * (q.e[a][b].y + q.e[b][a].y);
            }
    } else {
        for (int k = 0; k < 9; ++k) F[p][k][lane] = 0.0;
    }
    __syncthreads();
    // items: per chirality the 6 diagonal entries and the 15 above it
    const double hc = 0.5 * csw;
    for (int e = threadIdx.x; e < 32 * 42; e += blockDim.x) {
        const int l = e / 42, r = e - l * 42, chi = r / 21, o = r - chi * 21;
        if (s0 + l >= g.V) continue;
        const double sg = chi ? -1.0 : 1.0;
        // F_p[a][b] of site l
        auto Fab = [&](int pl, int a, int b) {
            if (a == b) return make_double2(0.0, F[pl][a][l]);
            const int k = 1 + 2 * (a + b);   // (0,1), (0,2), (1,2) at 3, 5, 7
            const double re = F[pl][k][l], im = F[pl][k + 1][l];
            return make_double2(a < b ? re : -re, im);
        };
        double* out = A64 + (size_t)(s0 + l) * 72 + 36 * chi;
        float* out32 = A32 + (size_t)(s0 + l) * 72 + 36 * chi;
        if (o < 6) {
            const int a = o % 3;
            const double e3 = sg * F[2][a][l] - F[3][a][l];
            const double v = m0 + 4.0 + (o < 3 ? -hc : hc) * e3;
            out[o] = v;
            out32[o] = (float)v;
        } else {
            int i = 0, k = o - 6;
            while (k >= 5 - i) { k -= 5 - i; ++i; }
            const int j = i + 1 + k, a = i % 3, b = j % 3;
            double2 c;
            if ((i < 3) == (j < 3)) {
                c = sg * Fab(2, a, b) - Fab(3, a, b);
                if (i >= 3) c = -c;
            } else {   // sigma_1 E_1 + sigma_2 E_2 between the spins
                const double2 e1 = sg * Fab(0, a, b) - Fab(5, a, b), e2 = sg * Fab(1, a, b) + Fab(4, a, b);
                c = make_double2(e1.x + e2.y, e1.y - e2.x);
            }
            const int at = herm_off(i, j);
            out[at] = -hc * c.y;
            out[at + 1] = hc * c.x;
            out32[at] = (float)(-hc * c.y);
            out32[at + 1] = (float)(hc * c.x);
        }
    }
}

// ------------------------------------------------------------------ derivative along a link direction
// Links move as U_mu(x) -> exp(i eps X_mu(x)) U_mu(x) (X traceless Hermitian),
// so dU/deps = i X U.  The operator is linear in the links of its hop terms, so
// their derivative is the stencil with dU; the clover leaves are four-link
// products, differentiated factor by factor below.
__global__ void link_tangent_kernel(const double2* __restrict__ U, const double2* __restrict__ X,
                                    double2* __restrict__ dU, int V) {
    const size_t nl = (size_t)V * 4;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < nl; e += (size_t)gridDim.x * blockDim.x) {
        const double2* u = U + e * 9;
        const double2* x = X + e * 9;
        for (int a = 0; a < 3; ++a)
            for (int c = 0; c < 3; ++c) {
                double2 acc = make_double2(0, 0);
                for (int b = 0; b < 3; ++b) cmac(acc, x[a * 3 + b], u[b * 3 + c]);
                dU[e * 9 + a * 3 + c] = make_double2(-acc.y, acc.x);   // i * acc
            }
    }
}

struct M3T { M3<double> m, d; };   // a matrix and its derivative
__device__ __forceinline__ M3T m3t_mul(const M3T& x, const M3T& y) {
    M3T r;
    r.m = m3_mul(x.m, y.m);
    const M3<double> a = m3_mul(x.d, y.m), b = m3_mul(x.m, y.d);
    for (int i = 0; i < 3; ++i) for (int j = 0; j < 3; ++j) r.d.e[i][j] = a.e[i][j] + b.e[i][j];
    return r;
}
__device__ __forceinline__ M3T m3t_dag(const M3T& x) { return M3T{m3_dag(x.m), m3_dag(x.d)}; }

// Packed derivative of the clover blocks (no constant diagonal), same layout
// and conventions as clover_assemble_kernel.
__global__ void clover_tangent_kernel(const double2* __restrict__ U, const double2* __restrict__ dU, Geom g,
                                      double csw, double* __restrict__ dA) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.V) return;
    int x[4];
    site_coords(g, s, x);
    double2 C[2][6][6];
    for (int chi = 0; chi < 2; ++chi)
        for (int i = 0; i < 6; ++i) for (int j = 0; j < 6; ++j) C[chi][i][j] = make_double2(0, 0);
    if (csw != 0.0) {
        for (int mu = 0; mu < 4; ++mu) {
            for (int nu = mu + 1; nu < 4; ++nu) {
                auto L = [&](int site, int d) {
                    return M3T{m3_load(U + ((size_t)site * 4 + d) * 9), m3_load(dU + ((size_t)site * 4 + d) * 9)};
                };
                const M3T Umu = L(s, mu), Unu = L(s, nu);
                const M3T Umu_m = L(shifted(g, x, mu, -1, nu, 0), mu);
                const M3T Unu_m = L(shifted(g, x, mu, 0, nu, -1), nu);
                const M3T l1 = m3t_mul(m3t_mul(Umu, L(shifted(g, x, mu, 1, nu, 0), nu)),
                                       m3t_mul(m3t_dag(L(shifted(g, x, mu, 0, nu, 1), mu)), m3t_dag(Unu)));
                const M3T l2 = m3t_mul(m3t_mul(Unu, m3t_dag(L(shifted(g, x, mu, -1, nu, 1), mu))),
                                       m3t_mul(m3t_dag(L(shifted(g, x, mu, -1, nu, 0), nu)), Umu_m));
                const M3T l3 = m3t_mul(m3t_mul(m3t_dag(Umu_m), m3t_dag(L(shifted(g, x, mu, -1, nu, -1), nu))),
                                       m3t_mul(L(shifted(g, x, mu, -1, nu, -1), mu), Unu_m));
                const M3T l4 = m3t_mul(m3t_mul(m3t_dag(Unu_m), L(shifted(g, x, mu, 0, nu, -1), mu)),
                                       m3t_mul(L(shifted(g, x, mu, 1, nu, -1), nu), m3t_dag(Umu)));
                double2 F[3][3];
                for (int a = 0; a < 3; ++a) for (int b = 0; b < 3; ++b) {
                    const double2 q = l1.d.e[a][b] + l2.d.e[a][b] + l3.d.e[a][b] + l4.d.e[a][b];
                    const double2 qh = conj(l1.d.e[b][a] + l2.d.e[b][a] + l3.d.e[b][a] + l4.d.e[b][a]);
                    F[a][b] = 0.125 * (q - qh);
                }
                for (int chi = 0; chi < 2; ++chi) {
                    double2 S[2][2];
                    sigma_block(mu, nu, chi, S);
                    for (int si = 0; si < 2; ++si) for (int sj = 0; sj < 2; ++sj)
                        for (int a = 0; a < 3; ++a) for (int b = 0; b < 3; ++b)
                            C[chi][si * 3 + a][sj * 3 + b] += S[si][sj] * F[a][b];
                }
            }
        }
    }
    for (int chi = 0; chi < 2; ++chi) {
        double* out = dA + (size_t)s * 72 + 36 * chi;
        for (int i = 0; i < 6; ++i) out[i] = mul_ipow(0.5 * csw * C[chi][i][i], 1).x;
        for (int i = 0; i < 6; ++i) for (int j = i + 1; j < 6; ++j) {
            const double2 v = mul_ipow(0.5 * csw * C[chi][i][j], 1);
            const int o = herm_off(i, j);
            out[o] = v.x;
            out[o + 1] = v.y;
        }
    }
}

// ------------------------------------------------------------------ force: the derivative per link
// F_rho(y) traceless Hermitian with d/d eps sum_k Re <g_k, Q psi_k> = sum
// tr(X_rho(y) F_rho(y)) (links moving as exp(i eps X) U); for g = psi = v that is
// the eigenvalue force times v^H v.  Q' is Hermitian, so the hop terms give
// K = -i U A with the colour outer products A = sum_k (A(psi_k, g_k) +
// A(g_k, psi_k)) / 2, A(a, b) = sum_s ((1 - gamma_rho) a(y + rho))_s (Gamma5
// b)_s(y)^H, and the clover term gives, per plane (rho, nu), (c_sw / 16) (below -
// above): the plaquettes above and below the link with the insertion Bt = B +
// B^H, B = sum_k sum_st sigma_{rho nu, st} psi_t (Gamma5 g)_s^H, placed at each
// corner.  F is the traceless Hermitian part of K.  Both outer products are
// linear in the fields, so a sum over fields needs the plaquette products, 98 %
// of the arithmetic, once.  Everything here is bound by the FP64 pipe (2 fused
// multiply-adds per clock and SM): the kernels are written for the fewest
// operations.  16^4, 8 fields: 8 x (6.54 + 0.82) ms with one thread per link and
// field -> 3.5 ms (plaquettes 1.93, hops 1.0, insertions 0.39, links 0.17).

__device__ __forceinline__ int plane_index(int mu, int nu) {   // mu < nu
    return mu == 0 ? nu - 1 : (mu == 1 ? nu + 1 : 5);
}
__device__ __forceinline__ double2 shfl2(double2 v, int o) {
    return make_double2(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
}

// Bt of the six planes mu < nu: [site][plane][3][3].  Eight lanes per site: lane
// (chi, i, j) sums M = psi_j g_i^H of spins 2 chi + j, 2 chi + i over the fields.
// With T_k = sum_ij (sigma_k)_ij M_ij per chirality, sigma^chi_{0k} = +-sigma_k
// and sigma^chi_{jk} = -eps_jkl sigma_l, and Gamma5 g changes sign with chi, so
// plane (0, k) is T^0_k + T^1_k and plane (j, k) is -eps_jkl (T^0_l - T^1_l): sums
// and differences between lanes.
// only >= 0: that plane alone, [site][3][3].
__global__ void __launch_bounds__(128) clover_insertion_kernel(const double2* __restrict__ psi,
                                                               const double2* __restrict__ gv, int nvec, Geom g, int only,
                                                               double2* __restrict__ Bt) {
    const unsigned tid = blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = (int)(tid >> 3) < g.V;
    const int s = live ? (int)(tid >> 3) : g.V - 1;
    const int chi = (tid >> 2) & 1, i = (tid >> 1) & 1, j = tid & 1;
    const size_t n = (size_t)g.V * 12;
    const double2* p = psi + (size_t)s * 12 + (2 * chi + j) * 3;
    const double2* q = gv + (size_t)s * 12 + (2 * chi + i) * 3;
    double2 M[9], N[9];   // the terms of Re g and of Im g
#pragma unroll
    for (int k = 0; k < 9; ++k) M[k] = N[k] = make_double2(0, 0);
    for (int f = 0; f < nvec; ++f) {
        double2 pv[3], qv[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            pv[c] = __ldg(p + f * n + c);
            qv[c] = __ldg(q + f * n + c);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                double2 &m = M[a * 3 + b], &o = N[a * 3 + b];
                m.x = fma(qv[b].x, pv[a].x, m.x);
                m.y = fma(qv[b].x, pv[a].y, m.y);
                o.x = fma(qv[b].y, pv[a].y, o.x);
                o.y = fma(-qv[b].y, pv[a].x, o.y);
            }
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) M[k] += N[k];
    // lanes (0,0): T_3 = M_00 - M_11; (0,1): T_1 = M_01 + M_10; (1,0): T_2 = -i M_01 + i M_10
    // then over chi: lane chi = 0 the sum (plane 0 k), chi = 1 the difference (spatial plane)
    const int k = i == j ? 3 : (j ? 1 : 2);
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        const double2 o = shfl2(M[e], 3);
        if (k == 1) M[e] = M[e] + o;
        else M[e] = M[e] - o;                               // (1,0): M_10 - M_01
        if (k == 2) M[e] = make_double2(-M[e].y, M[e].x);   // times i
        const double2 t = shfl2(M[e], 4);
        M[e] = chi ? t - M[e] : M[e] + t;
    }
    if (!live || (i && j)) return;
    const int plane = chi ? 6 - k : k - 1;
    const bool minus = chi && k != 2;   // -eps: planes (1,2), (2,3) minus, (1,3) plus
    if (only >= 0 && plane != only) return;
    double2* o = Bt + (only >= 0 ? (size_t)s : (size_t)s * 6 + plane) * 9;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const double2 v = M[a * 3 + b] + conj(M[b * 3 + a]);
            o[a * 3 + b] = minus ? -v : v;
        }
}

__device__ __forceinline__ void m3_store(double2* p, const M3<double>& m) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) p[a * 3 + b] = m.e[a][b];
}

// S + T = A(a, b) of direction rho, added to them unless first: h = up - B dn of
// a(y + rho) (times the boundary sign) against c_k = b_k + (B b_low)_k of b(y): the
// two halves of Gamma5 b meet the same h, so they are added before the product.  S
// takes the terms of Re c, T those of Im c.
template <int rho, bool first>
__device__ __forceinline__ void hop_outer(const double2* __restrict__ an, const double2* __restrict__ bs, double sg,
                                          double2 (&S)[9], double2 (&T)[9]) {
    constexpr SpinMono Bm = kB(rho), BHm = kBH(rho);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        double2 h[3], c[3];
        const int lo = BHm.perm[i];   // spin 2 + lo reads h_i with phase i^ph[lo]
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            h[a] = __ldg(an + i * 3 + a) - mul_ipow(__ldg(an + (2 + Bm.perm[i]) * 3 + a), Bm.ph[i]);
            if (sg < 0) h[a] = -h[a];
            c[a] = __ldg(bs + i * 3 + a) + mul_ipow(__ldg(bs + (2 + lo) * 3 + a), 4 - BHm.ph[lo]);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                double2 &m = S[a * 3 + b], &o = T[a * 3 + b];
                const bool add = !first || i > 0;
                m.x = add ? fma(c[b].x, h[a].x, m.x) : c[b].x * h[a].x;
                m.y = add ? fma(c[b].x, h[a].y, m.y) : c[b].x * h[a].y;
                o.x = add ? fma(c[b].y, h[a].y, o.x) : c[b].y * h[a].y;
                o.y = add ? fma(-c[b].y, h[a].x, o.y) : -c[b].y * h[a].x;
            }
    }
}

// Hop part K = -i U A of every link, summed over the fields; blockIdx.y = rho.
template <int rho>
__device__ __forceinline__ void hop_force(const double2* __restrict__ U, const double2* __restrict__ psi,
                                          const double2* __restrict__ gv, int nvec, const Geom& g, int s,
                                          double2* __restrict__ K) {
    int x[4], neg;
    site_coords(g, s, x);
    const int sf = nb_fwd(g, x, s, rho, neg);
    const double sg = neg ? -1.0 : 1.0;
    const size_t n = (size_t)g.V * 12;
    double2 A[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) A[k] = make_double2(0, 0);
    // a field by itself, then pairs of fields, then their sum: one chain over eight
    // fields had 1.3 times the error of the fields' forces added up
    double2 P[9];
    for (int f = 0; f < nvec; ++f) {
        const double2 *p = psi + f * n, *q = gv + f * n;
        double2 S[9], T[9];
        hop_outer<rho, true>(p + (size_t)sf * 12, q + (size_t)s * 12, sg, S, T);
        if (psi != gv) hop_outer<rho, false>(q + (size_t)sf * 12, p + (size_t)s * 12, sg, S, T);
        const bool pair = f & 1, flush = pair || f + 1 == nvec;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            P[k] = pair ? P[k] + (S[k] + T[k]) : S[k] + T[k];
            if (flush) A[k] += P[k];
        }
    }
    const double c = psi != gv ? 0.5 : 1.0;
    const size_t e = (size_t)s * 4 + rho;
    M3<double> u = m3_load(U + e * 9), Am;
    for (int a = 0; a < 3; ++a) for (int b = 0; b < 3; ++b) Am.e[a][b] = c * A[a * 3 + b];
    const M3<double> UA = m3_mul(u, Am);
    for (int a = 0; a < 3; ++a) for (int b = 0; b < 3; ++b) K[e * 9 + a * 3 + b] = mul_ipow(UA.e[a][b], 3);   // -i U A
}
__global__ void __launch_bounds__(128) hop_force_kernel(const double2* __restrict__ U, const double2* __restrict__ psi,
                                                        const double2* __restrict__ gv, int nvec, Geom g,
                                                        double2* __restrict__ K) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.V) return;
    switch (blockIdx.y) {
        case 0: hop_force<0>(U, psi, gv, nvec, g, s, K); break;
        case 1: hop_force<1>(U, psi, gv, nvec, g, s, K); break;
        case 2: hop_force<2>(U, psi, gv, nvec, g, s, K); break;
        default: hop_force<3>(U, psi, gv, nvec, g, s, K); break;
    }
}

// One thread per plaquette (x; mu < nu) = a b (d c)^H with corners 0..3 at x,
// x + mu, x + mu + nu, x + nu: the clover force on its four links.  With the
// inserted half paths X = a B1 b and Y = d B3 c and the sums over the three
// other insertions S1 = B2 W + Y^H + W B0 (W = (d c)^H), S2 = B0 E + X + E B2
// (E = a b), every link's term closes with one or two products more, because
// the Hermitian B make the sums of the reversed paths S1^H and S2^H:
//   above a = X W + E S1           below c = (B3 d^H E + d^H S2) c^H
//   above d = Y E^H + D S2^H       below b = (B1 a^H D + a^H S1^H) b^H
// 20 products instead of the 36 of one thread per link.  W4: [plane][a, b, c,
// d][site][3][3].
__global__ void __launch_bounds__(128) plaquette_force_kernel(const double2* __restrict__ U,
                                                              const double2* __restrict__ Bt, Geom g, int plane0,
                                                              int only, double2* __restrict__ W4) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.V) return;
    const int pl = plane0 + blockIdx.y;
    const int mu = pl < 3 ? 0 : (pl < 5 ? 1 : 2), nu = pl < 3 ? pl + 1 : (pl < 5 ? pl - 1 : 3);
    int x[4];
    site_coords(g, s, x);
    const int s1 = shifted(g, x, mu, 1, nu, 0), s3 = shifted(g, x, mu, 0, nu, 1), s2 = shifted(g, x, mu, 1, nu, 1);
    auto link = [&](int site, int d) { return m3_load(U + ((size_t)site * 4 + d) * 9); };
    auto ins = [&](int site) { return m3_load(Bt + (only >= 0 ? (size_t)site : (size_t)site * 6 + pl) * 9); };
    double2* out = W4 + (size_t)blockIdx.y * 4 * g.V * 9 + (size_t)s * 9;
    const size_t step = (size_t)g.V * 9;
    M3<double> E, D, X, Y;
    M3<double> aB1, dB3;
    {
        const M3<double> a = link(s, mu), b = link(s1, nu);
        E = m3_mul(a, b);
        aB1 = m3_mul(a, ins(s1));
        X = m3_mul(aB1, b);
    }
    {
        const M3<double> d = link(s, nu), c = link(s3, mu);
        D = m3_mul(d, c);
        dB3 = m3_mul(d, ins(s3));
        Y = m3_mul(dB3, c);
    }
    {
        const M3<double> W = m3_dag(D);
        M3<double> S1 = m3_dag(Y);
        m3_mac(S1, ins(s2), W);
        m3_mac(S1, W, ins(s));
        M3<double> r = m3_mul(X, W);
        m3_mac(r, E, S1);
        m3_store(out, r);                                   // above a
        M3<double> t = m3_mul(m3_dag(aB1), D);
        m3_mac(t, m3_dag(link(s, mu)), m3_dag(S1));
        m3_store(out + step, m3_mul(t, m3_dag(link(s1, nu))));        // below b
    }
    {
        M3<double> S2 = X;
        m3_mac(S2, ins(s), E);
        m3_mac(S2, E, ins(s2));
        M3<double> r = m3_mul(Y, m3_dag(E));
        m3_mac(r, D, m3_dag(S2));
        m3_store(out + 3 * step, r);                        // above d
        M3<double> t = m3_mul(m3_dag(dB3), E);
        m3_mac(t, m3_dag(link(s, nu)), S2);
        m3_store(out + 2 * step, m3_mul(t, m3_dag(link(s3, mu))));    // below c
    }
}

// One thread per link: adds the plaquette terms of planes plane0 .. plane0 +
// nplanes - 1 to K (in F) and, with `last`, leaves F = traceless Hermitian part
// (over nrm, device v^H v, unless null) or, with grad, the link gradient i F U.
__global__ void __launch_bounds__(128) link_force_kernel(const double2* __restrict__ U, const double2* __restrict__ W4,
                                                         const double2* __restrict__ nrm, Geom g, double csw, int plane0,
                                                         int nplanes, int last, int grad, double2* __restrict__ F) {
    const size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (e >= (size_t)g.V * 4) return;
    const int s = (int)(e >> 2), rho = (int)(e & 3);
    int x[4];
    site_coords(g, s, x);
    M3<double> K = m3_load(F + e * 9);
    const size_t step = (size_t)g.V * 9;
    for (int o = 0; o < 4; ++o) {
        if (o == rho || nplanes == 0) continue;
        const int pl = (rho < o ? plane_index(rho, o) : plane_index(o, rho)) - plane0;
        if (pl < 0 || pl >= nplanes) continue;
        // the link is a of the plaquette above and c of the one below in planes
        // (rho, o), d and b in planes (o, rho), where the insertion changes sign
        const double c = (rho < o ? 1.0 : -1.0) * csw / 16.0;
        const double2* up = W4 + (size_t)pl * 4 * step + (rho < o ? 0 : 3) * step + (size_t)s * 9;
        const double2* dn = W4 + (size_t)pl * 4 * step + (rho < o ? 2 : 1) * step +
                            (size_t)shifted(g, x, rho, 0, o, -1) * 9;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const double2 u = up[k], d = dn[k];
            K.e[k / 3][k % 3] += c * (d - u);
        }
    }
    if (!last) {
        m3_store(F + e * 9, K);
        return;
    }
    double inv = 1.0;
    if (nrm != nullptr) {
        const double n = nrm[0].x;
        inv = n > 0 ? 1.0 / n : 0.0;
    }
    M3<double> H;
    for (int a = 0; a < 3; ++a) for (int b = 0; b < 3; ++b) H.e[a][b] = 0.5 * (K.e[a][b] + conj(K.e[b][a]));
    const double tr = (H.e[0][0].x + H.e[1][1].x + H.e[2][2].x) / 3.0;
    for (int a = 0; a < 3; ++a) H.e[a][a].x -= tr;
    // link gradient i F U: the tangent vector whose real inner product with any
    // dU = i X U is tr(X F)
    if (grad) H = m3_mul(H, m3_load(U + e * 9));
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) F[e * 9 + a * 3 + b] = inv * (grad ? mul_ipow(H.e[a][b], 1) : H.e[a][b]);
}

// Planes handled per launch: all six while their terms (3456 bytes per site) stay
// below 1 GB, one at a time on larger lattices and where memory is short (form 1),
// and there the insertions plane by plane too (form 2: 720 bytes per site against
// 1440 and 4320; six insertion passes instead of one).  The terms of a link are added
// in the same order in all forms: the same bits.
size_t force_scratch(const FineOp& f, int form) {
    if (f.csw == 0.0) return 0;
    const size_t per = form == 0 && f.g.V <= 300000 ? 54 + 6 * 36 : (form < 2 ? 54 + 36 : 9 + 36);
    return per * f.g.V * sizeof(double2);
}

void bilinear_force(const FineOp& f, int nvec, const double2* gv, const double2* psi, const double2* nrm, int grad,
                    void* scratch, int form, double2* F, cudaStream_t st) {
    double2* Bt = (double2*)scratch;
    double2* W4 = Bt + (size_t)f.g.V * (form < 2 ? 54 : 9);
    const unsigned sites = (f.g.V + 127) / 128, links = (unsigned)(((size_t)f.g.V * 4 + 127) / 128);
    {
        KTimer kt("hop_force", 0.0, 0.0, st);
        hop_force_kernel<<<dim3(sites, 4), 128, 0, st>>>(f.U64, psi, gv, nvec, f.g, F);
    }
    if (f.csw == 0.0) {
        KTimer kt("link_force", 0.0, 0.0, st);
        link_force_kernel<<<links, 128, 0, st>>>(f.U64, nullptr, nrm, f.g, 0.0, 0, 0, 1, grad, F);
        return;
    }
    const int np = form == 0 && f.g.V <= 300000 ? 6 : 1;
    for (int p0 = 0; p0 < 6; p0 += np) {
        const int only = form < 2 ? -1 : p0;
        if (p0 == 0 || only >= 0) {
            KTimer kt("clover_insertion", 0.0, 0.0, st);
            clover_insertion_kernel<<<(unsigned)(((size_t)f.g.V * 8 + 127) / 128), 128, 0, st>>>(psi, gv, nvec, f.g, only,
                                                                                                 Bt);
        }
        {
            KTimer kt("plaquette_force", 0.0, 0.0, st);
            plaquette_force_kernel<<<dim3(sites, np), 128, 0, st>>>(f.U64, Bt, f.g, p0, only, W4);
        }
        KTimer kt("link_force", 0.0, 0.0, st);
        link_force_kernel<<<links, 128, 0, st>>>(f.U64, W4, nrm, f.g, f.csw, p0, np, p0 + np >= 6, grad, F);
    }
}

// ------------------------------------------------------------------ stencil
// out_j = op(tau_j) in_j, or out_j = b_j - op(tau_j) in_j when b != nullptr.
// op = QCD_OP_D: D - tau Gamma5 ; op = QCD_OP_Q: Gamma5 D - tau.

// sign flip without the FP64 pipe
__device__ __forceinline__ double flip(double v, int mask) {
    return __hiloint2double(__double2hiint(v) ^ mask, __double2loint(v));
}

// FP64 stencil, eight lanes per site: lane q takes the hop of direction
// mu = q / 2 (forward for even q).  FP64 runs at 2 fused multiply-adds per clock
// and SM on this part, so the kernel is bound by that pipe at every size (1248
// operations per site); the eight lanes spread a site over as many warps, which
// fills the chip from a few hundred sites on instead of from a few hundred
// thousand.  Everything that is a sign, a factor i or a permutation of spins
// (lane dependent) is done by integer selects and sign flips.  The twelve rows
// are summed by two exchange-and-halve steps (lane bit 2 ends with chirality
// half, bit 1 with the spin), each lane then adds the clover columns of spin
// (lane bit 0) to its three rows, and one exchange completes the sums.  4^4: 59 us
// with one thread per site (8 warps on two SMs) -> 10 us, mostly the call itself.
__global__ void __launch_bounds__(128) wilson_clover_f64_kernel(
    double2* __restrict__ out, const double2* __restrict__ in, const double2* __restrict__ b,
    const double2* __restrict__ U, const double* __restrict__ A, Geom g, int op, Shifts tau, size_t stride,
    const int* __restrict__ act) {
    const int j = blockIdx.y;
    if (act != nullptr && !act[j]) return;
    const unsigned tid = blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = (int)(tid >> 3) < g.V;
    const int s = live ? (int)(tid >> 3) : g.V - 1;   // idle lanes follow along for the exchanges
    const int q = tid & 7, mu = q >> 1;
    const bool fw = !(q & 1);
    in += j * stride;
    int x[4];
    site_coords(g, s, x);
    int ms = 1, xm = x[3], Lm = g.L[3];
    if (mu == 2) { ms = g.L[3]; xm = x[2]; Lm = g.L[2]; }
    if (mu == 1) { ms = g.L[3] * g.L[2]; xm = x[1]; Lm = g.L[1]; }
    if (mu == 0) { ms = g.L[3] * g.L[2] * g.L[1]; xm = x[0]; Lm = g.L[0]; }
    const bool wraps = fw ? xm == Lm - 1 : xm == 0;
    const int sn = s + (fw ? ms : -ms) * (wraps ? 1 - Lm : 1);
    const bool neg = wraps && mu == 0 && g.antiperiodic;
    const bool swap = mu == 1 || mu == 2, imag = mu & 1;
    constexpr int kSign = (int)0x80000000;

    // h_s = up_s -+ (B dn)_s (- forward): B rows are -1, -i (mu = 0, 1) or
    // -1, +1 / -i, +i (mu = 2, 3), columns swapped for mu = 1, 2
    const double2* nb = in + (size_t)sn * 12;
    const double c0 = fw ? 1.0 : -1.0, c1 = mu < 2 ? c0 : -c0;
    double2 h[2][3];
#pragma unroll
    for (int sp = 0; sp < 2; ++sp) {
        const double2* dn = nb + 6 + (swap ? 1 - sp : sp) * 3;
        const double c = sp ? c1 : c0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double2 u = __ldg(nb + sp * 3 + a), d = __ldg(dn + a);
            h[sp][a].x = fma(imag ? -c : c, imag ? d.y : d.x, u.x);
            h[sp][a].y = fma(c, imag ? d.x : d.y, u.y);
        }
    }
    // o = U h (forward) or U^H h (backward), with the boundary sign
    const double2* ul = U + ((size_t)(fw ? s : sn) * 4 + mu) * 9;
    const int mx = neg ? kSign : 0, my = fw ? mx : mx ^ kSign;
    double2 o[2][3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            double2 e = __ldg(ul + (fw ? a * 3 + c : c * 3 + a));
            e = make_double2(flip(e.x, mx), flip(e.y, my));
#pragma unroll
            for (int sp = 0; sp < 2; ++sp) {
                if (c == 0) o[sp][a] = e * h[sp][0];
                else cmac(o[sp][a], e, h[sp][c]);
            }
        }
    }
    // rows of this hop over -1/2: o_s above, -+ (B^H o)_s below; B^H rows are
    // -1 / i (mu = 0, 1), +1, -1 / i, -i (mu = 2, 3), columns swapped for 1, 2
    const int f0 = (mu == 0) != fw ? kSign : 0, f1 = mu < 2 ? f0 : f0 ^ kSign;
    double2 w[6];   // rows of this lane's chirality half after the exchange
    const bool low = q & 4;
#pragma unroll
    for (int sp = 0; sp < 2; ++sp)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double2 v = swap ? o[1 - sp][a] : o[sp][a];
            const int f = sp ? f1 : f0;
            const double2 d = imag ? make_double2(flip(v.y, f ^ kSign), flip(v.x, f)) : make_double2(flip(v.x, f), flip(v.y, f));
            const double2 keep = low ? d : o[sp][a], send = low ? o[sp][a] : d;
            w[sp * 3 + a] = keep + shfl2(send, 4);
        }
    const bool sp1 = q & 2;
    double2 r[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) r[a] = (sp1 ? w[3 + a] : w[a]) + shfl2(sp1 ? w[a] : w[3 + a], 2);
    // clover block of the chirality: rows 3 sp + a, columns 3 p + c
    const int chi = low, sp = sp1, p = q & 1;
    const double2* pc = in + (size_t)s * 12 + (2 * chi + p) * 3;
    const double* Ab = A + (size_t)s * 72 + 36 * chi;
    double2 psi[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) psi[c] = __ldg(pc + c);
    const double t = tau.t[j];
    const double sg = op != QCD_OP_D && chi ? -1.0 : 1.0, ts = op == QCD_OP_D && chi ? t : -t;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double2 acc = -0.5 * r[a];
#pragma unroll
        for (int cc = 1; cc <= 3; ++cc) {   // the diagonal, the largest term, last
            const int c = (a + cc) % 3;
            const int i = 3 * sp + a, k = 3 * p + c;
            const int lo = min(i, k), hi = max(i, k);
            double2 m;
            if (a == c && sp == p) m = make_double2(__ldg(Ab + i), 0.0);
            else m = __ldg(reinterpret_cast<const double2*>(Ab + herm_off(lo, hi)));
            m.y = flip(m.y, i > k ? kSign : 0);
            // the real diagonal: nothing times its zero (not NaN for an infinite psi)
            const double2 v = psi[c], z = a == c && sp == p ? make_double2(0.0, 0.0) : v;
            acc.x = fma(-m.y, z.y, fma(m.x, v.x, acc.x));
            acc.y = fma(m.y, z.x, fma(m.x, v.y, acc.y));
        }
        r[a] = sg < 0 ? -acc : acc;
    }
    if (sp == p)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            r[a].x = fma(ts, psi[a].x, r[a].x);
            r[a].y = fma(ts, psi[a].y, r[a].y);
        }
#pragma unroll
    for (int a = 0; a < 3; ++a) r[a] += shfl2(r[a], 1);
    if (!live || p) return;
    const size_t row = j * stride + (size_t)s * 12 + (2 * chi + sp) * 3;
#pragma unroll
    for (int a = 0; a < 3; ++a) out[row + a] = b != nullptr ? b[row + a] - r[a] : r[a];
}

// FP64 stencil, one thread per site: 1152 operations per site, 8 % fewer than
// with eight lanes, for lattices that fill the FP64 pipes by themselves (86 %
// busy).  32 x 16^3: 391 -> 289 us, from the fused multiply-adds.
__global__ void __launch_bounds__(128) wilson_clover_f64_site_kernel(
    double2* __restrict__ out, const double2* __restrict__ in, const double2* __restrict__ b,
    const double2* __restrict__ U, const double* __restrict__ A, Geom g, int op, Shifts tau, size_t stride,
    const int* __restrict__ act) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.V) return;
    const int j = blockIdx.y;
    if (act != nullptr && !act[j]) return;
    in += j * stride;
    out += j * stride;
    int x[4];
    site_coords(g, s, x);
    Spinor<double> acc;
    const double2* A2 = reinterpret_cast<const double2*>(A + (size_t)s * 72);
#pragma unroll
    for (int chi = 0; chi < 2; ++chi) {
        double2 psi[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) psi[k] = __ldg(in + (size_t)s * 12 + 6 * chi + k);
        double2* ys = acc.c + 6 * chi;
#pragma unroll
        for (int i = 0; i < 6; ++i)
#pragma unroll
            for (int k = i + 1; k < 6; ++k) {
                const double2 m = __ldg(A2 + 18 * chi + herm_off(i, k) / 2);
                if (i == 0 && k == 1) ys[0] = m * psi[1];
                else cmac(ys[i], m, psi[k]);
                if (i == 0) ys[k] = cmulc(m, psi[0]);
                else cmacc(ys[k], m, psi[i]);
            }
    }
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
#pragma unroll
        for (int dir = 0; dir < 2; ++dir) {
            int neg;
            Spinor<double> nb;
            Link<double> u;
            const int sn = dir == 0 ? nb_fwd(g, x, s, mu, neg) : nb_bwd(g, x, s, mu, neg);
            load_spinor<double>(in + (size_t)sn * 12, nb);
            load_link<double>(U + ((size_t)(dir == 0 ? s : sn) * 4 + mu) * 9, u);
            const double sg = neg ? -1.0 : 1.0;
            if (dir == 0) {
                if (mu == 0) hop_accumulate<double, 0, true>(nb, u, sg, acc);
                if (mu == 1) hop_accumulate<double, 1, true>(nb, u, sg, acc);
                if (mu == 2) hop_accumulate<double, 2, true>(nb, u, sg, acc);
                if (mu == 3) hop_accumulate<double, 3, true>(nb, u, sg, acc);
            } else {
                if (mu == 0) hop_accumulate<double, 0, false>(nb, u, sg, acc);
                if (mu == 1) hop_accumulate<double, 1, false>(nb, u, sg, acc);
                if (mu == 2) hop_accumulate<double, 2, false>(nb, u, sg, acc);
                if (mu == 3) hop_accumulate<double, 3, false>(nb, u, sg, acc);
            }
        }
    }
    const double t = tau.t[j];
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const int chi = k / 6;
        const double2 p = __ldg(in + (size_t)s * 12 + k);
        const double2 d2 = __ldg(A2 + 18 * chi + (k % 6) / 2);
        const double d = k % 2 ? d2.y : d2.x, ts = op == QCD_OP_D && chi ? t : -t;
        double2 v = acc.c[k];
        v.x = fma(d, p.x, v.x);
        v.y = fma(d, p.y, v.y);
        if (op != QCD_OP_D && chi) v = -v;
        v.x = fma(ts, p.x, v.x);
        v.y = fma(ts, p.y, v.y);
        if (b != nullptr) v = b[j * stride + (size_t)s * 12 + k] - v;
        out[(size_t)s * 12 + k] = v;
    }
}

// FP32 stencil with links and clover blocks in site-fastest (SoA) copies:
// Us[(mu * 9 + k) * V + site] (float2) and As[q * V + site] (float4, q < 18),
// so a warp's link and clover loads are contiguous; spinors keep the ABI
// layout.  A thread applies the operator to NR right-hand sides of one site: the
// links and clover block (864 of the 1,728 bytes that a single apply moves into
// the SM) are loaded once for all of them.  Consecutive CTAs take the same 128
// sites for the next NR right-hand sides and find links and clover in L2.  With
// tb > 0 the site blocks are visited time-fastest within bricks of tb time
// slices (block u: t = (u / (tb ns)) tb + u % tb, spatial block (u / tb) % ns of
// ns = L1 L2 L3 / 128), so the neighbours of a block in every direction are
// read by CTAs a few hundred launches apart and still sit in L2.
// Spinors move in 32-byte pieces where the fields are aligned to 32 bytes (W32):
// the L1 pipe, 70 % busy with 16-byte ones (each load instruction of a warp
// touches 24 lines), was what bound several right-hand sides.  64 x 32^3, one
// right-hand side: 318 -> 280 us = 5.75 TB/s (85 % of the copy bandwidth); 32 x
// 16^3, 16 right-hand sides: 245 -> 193 us, now bound by load latency at 16 warps
// per SM (three or five CTAs per SM and four right-hand sides per thread are
// slower).
template <int NR, bool W32, int CTAS = 4>
__global__ void __launch_bounds__(128, CTAS) wilson_clover_soa_kernel(
    float2* __restrict__ out, const float2* __restrict__ in, const float2* __restrict__ b,
    const float2* __restrict__ Us, const float4* __restrict__ As, Geom g, int op, Shifts tau, size_t stride,
    const int* __restrict__ act, int nrhs, int tb) {
    const int groups = (nrhs + NR - 1) / NR;
    const int j0 = (int)(blockIdx.x % groups) * NR;
    const unsigned u = blockIdx.x / groups;
    int s;
    if (tb > 0) {
        const unsigned vs = (unsigned)(g.L[1] * g.L[2] * g.L[3]), ns = vs / 128u;
        const unsigned t = (u / (tb * ns)) * tb + u % tb, sb = (u / tb) % ns;
        s = (int)(t * vs + sb * 128u + threadIdx.x);
    } else {
        s = (int)(u * blockDim.x + threadIdx.x);
    }
    bool on[NR], any = false;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        on[r] = j0 + r < nrhs && (act == nullptr || act[j0 + r]);
        any = any || on[r];
    }
    if (s >= g.V || !any) return;
    in += j0 * stride;
    out += j0 * stride;
    const size_t V = (size_t)g.V;
    int x[4];
    site_coords(g, s, x);
    Spinor<float> acc[NR], psi[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r)
        if (on[r]) load_spinor_w<W32>(in + r * stride + (size_t)s * 12, psi[r]);
#pragma unroll
    for (int chi = 0; chi < 2; ++chi) {
        float ar[36];
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const float4 v = __ldg(As + (size_t)(9 * chi + q) * V + s);
            ar[4 * q] = v.x; ar[4 * q + 1] = v.y; ar[4 * q + 2] = v.z; ar[4 * q + 3] = v.w;
        }
#pragma unroll
        for (int r = 0; r < NR; ++r)
            if (on[r]) herm_off_apply<float>(ar, psi[r].c + 6 * chi, acc[r].c + 6 * chi);
    }
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
#pragma unroll
        for (int dir = 0; dir < 2; ++dir) {
            int neg;
            const int sn = dir == 0 ? nb_fwd(g, x, s, mu, neg) : nb_bwd(g, x, s, mu, neg);
            Link<float> l;
#pragma unroll
            for (int k = 0; k < 9; ++k) l.e[k] = __ldg(Us + (size_t)(mu * 9 + k) * V + (dir == 0 ? s : sn));
            const float sg = neg ? -1.f : 1.f;
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                if (!on[r]) continue;
                Spinor<float> nb;
                load_spinor_w<W32>(in + r * stride + (size_t)sn * 12, nb);
                if (dir == 0) {
                    if (mu == 0) hop_accumulate<float, 0, true>(nb, l, sg, acc[r]);
                    if (mu == 1) hop_accumulate<float, 1, true>(nb, l, sg, acc[r]);
                    if (mu == 2) hop_accumulate<float, 2, true>(nb, l, sg, acc[r]);
                    if (mu == 3) hop_accumulate<float, 3, true>(nb, l, sg, acc[r]);
                } else {
                    if (mu == 0) hop_accumulate<float, 0, false>(nb, l, sg, acc[r]);
                    if (mu == 1) hop_accumulate<float, 1, false>(nb, l, sg, acc[r]);
                    if (mu == 2) hop_accumulate<float, 2, false>(nb, l, sg, acc[r]);
                    if (mu == 3) hop_accumulate<float, 3, false>(nb, l, sg, acc[r]);
                }
            }
        }
    }
    // diagonal of the clover blocks and shift, psi read again (L1) rather than
    // held through the hops
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        if (!on[r]) continue;
        const size_t at = r * stride + (size_t)s * 12;
        load_spinor_w<W32>(in + at, psi[r]);
        const float t = (float)tau.t[j0 + r];
#pragma unroll
        for (int chi = 0; chi < 2; ++chi) {
            const float4 d0 = __ldg(As + (size_t)(9 * chi) * V + s), d1 = __ldg(As + (size_t)(9 * chi + 1) * V + s);
            const float d[6] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y};
            const float sg = op != QCD_OP_D && chi ? -1.f : 1.f, ts = op == QCD_OP_D && chi ? t : -t;
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                float2& v = acc[r].c[6 * chi + k];
                const float2 p = psi[r].c[6 * chi + k];
                v.x = fmaf(ts, p.x, sg * fmaf(d[k], p.x, v.x));
                v.y = fmaf(ts, p.y, sg * fmaf(d[k], p.y, v.y));
            }
        }
        if (b != nullptr) {
            Spinor<float> bb;
            load_spinor<float>(b + j0 * stride + at, bb);
#pragma unroll
            for (int k = 0; k < 12; ++k) acc[r].c[k] = bb.c[k] - acc[r].c[k];
        }
        if constexpr (W32) {
#pragma unroll
            for (int k = 0; k < 3; ++k) store8(out + at + 4 * k, acc[r].c + 4 * k);
        } else {
            store_spinor<float>(out + at, acc[r]);
        }
    }
}

// site-fastest copies of the FP32 links and clover blocks
__global__ void soa_copies_kernel(const float2* __restrict__ U, const float* __restrict__ A, float2* __restrict__ Us,
                                  float4* __restrict__ As, int V) {
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < (size_t)V * 36; e += (size_t)gridDim.x * blockDim.x) {
        const size_t site = e % V;
        const int r = (int)(e / V);   // mu * 9 + k
        Us[e] = U[site * 36 + r];
    }
    const float4* A4 = reinterpret_cast<const float4*>(A);
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < (size_t)V * 18; e += (size_t)gridDim.x * blockDim.x) {
        const size_t site = e % V;
        const int q = (int)(e / V);
        As[e] = A4[site * 18 + q];
    }
}

// ------------------------------------------------------------------ host launchers
// Largest deviation of U U^H from the identity over all links, as the bit
// pattern of a non-negative double (which orders like the value); a
// non-finite entry records +inf.
__global__ void gauge_check_kernel(const double2* __restrict__ U, size_t nlinks, unsigned long long* __restrict__ dev) {
    double worst = 0.0;
    for (size_t l = blockIdx.x * (size_t)blockDim.x + threadIdx.x; l < nlinks; l += (size_t)gridDim.x * blockDim.x) {
        double2 u[9];
        bool fin = true;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            u[k] = U[l * 9 + k];
            fin = fin && isfinite(u[k].x) && isfinite(u[k].y);
        }
        if (!fin) { worst = INFINITY; continue; }
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                double2 acc = make_double2(a == b ? -1.0 : 0.0, 0.0);
#pragma unroll
                for (int c = 0; c < 3; ++c) cmacc(acc, u[b * 3 + c], u[a * 3 + c]);
                worst = fmax(worst, fmax(fabs(acc.x), fabs(acc.y)));
            }
    }
    for (int o = 16; o > 0; o >>= 1) worst = fmax(worst, __shfl_xor_sync(0xffffffffu, worst, o));
    if ((threadIdx.x & 31) == 0) atomicMax(dev, (unsigned long long)__double_as_longlong(worst));
}

double gauge_unitarity_deviation(const double2* U, size_t nlinks, unsigned long long* scratch, cudaStream_t st) {
    cudaMemsetAsync(scratch, 0, sizeof(unsigned long long), st);
    KTimer kt("gauge_check", (double)nlinks * 144, (double)nlinks * 27 * 8, st);
    const int grid = (int)std::min<size_t>((nlinks + 255) / 256, 4096);
    gauge_check_kernel<<<grid, 256, 0, st>>>(U, nlinks, scratch);
    unsigned long long h = 0;
    cudaMemcpyAsync(&h, scratch, sizeof(h), cudaMemcpyDeviceToHost, st);
    if (cudaStreamSynchronize(st) != cudaSuccess) return NAN;
    double d;
    memcpy(&d, &h, sizeof(d));
    return d;
}

// A64, A32 and the FP32 copies of the links from U64.  The staples (864 bytes per
// site) use the buffers of the FP32 links and of the layouts made last.
void launch_clover_build(const FineOp& f, cudaStream_t st) {
    {
        KTimer kt("clover_build", 0.0, 0.0, st);
        const StapleBufs D{{(double2*)f.U32s, (double2*)f.A32s, (double2*)f.U32}};
        if (f.csw != 0.0) clover_staples_kernel<<<dim3((f.g.V + 127) / 128, 6), 128, 0, st>>>(f.U64, f.g, D);
        clover_assemble_kernel<<<(f.g.V + 31) / 32, 192, 0, st>>>(f.U64, f.g, D, f.m0, f.csw, f.A64, f.A32);
    }
    blas_convert(QCD_FP64, f.U64, QCD_FP32, f.U32, (size_t)f.g.V * 36, st);
    soa_copies_kernel<<<1216, 256, 0, st>>>(f.U32, f.A32, f.U32s, f.A32s, f.g.V);
}

static void launch_f64(const FineOp& f, const double2* U, const double* A, int op, int nrhs, const double2* in,
                       double2* out, const double2* b, const Shifts& sh, const int* act, cudaStream_t st) {
    // One thread per site (8 % fewer operations) from the lattice where batches of any
    // size gain more than a single field loses; eight lanes per site below.  The line
    // depends on the lattice only, so a field's result does not depend on the batch it
    // is in.  Measured, eight lanes / one thread, 1, 2 and 8 fields (us):
    //   8^4 16.9 / 45.8, 27 / 46, 85 / 85        12^4 56 / 85, 107 / 126, 390 / 365
    //   16^3 x 8 85 / 85, 157 / 166, 607 / 565   16^3 x 15 151 / 166, 290 / 287, 1133 / 1043
    //   16^4 157 / 167, 308 / 288, 1206 / 1088   32 x 16^3 308 / 290, 607 / 570, 2403 / 2166
    // Batches of four and more lose up to 9 % to one thread between 12^4 and the line.
    if (f.g.V >= 65536) {
        const dim3 grid((f.g.V + 127) / 128, nrhs);
        wilson_clover_f64_site_kernel<<<grid, 128, 0, st>>>(out, in, b, U, A, f.g, op, sh, (size_t)f.g.V * 12, act);
        return;
    }
    const dim3 grid((unsigned)(((size_t)f.g.V * 8 + 127) / 128), nrhs);
    wilson_clover_f64_kernel<<<grid, 128, 0, st>>>(out, in, b, U, A, f.g, op, sh, (size_t)f.g.V * 12, act);
}

static void launch_dirac(const FineOp& f, int prec, int op, int nrhs, const void* in, void* out, const void* b,
                         const double* tau, const int* act, cudaStream_t st) {
    Shifts sh{};
    for (int j = 0; j < nrhs; ++j) sh.t[j] = tau ? tau[j] : 0.0;
    const double bytes = (double)f.g.V * (nrhs * (b ? 72.0 : 48.0) + 144.0) * (prec == QCD_FP64 ? 8 : 4);
    if (prec == QCD_FP64) {
        KTimer kt("wilson_clover_f64", bytes, 1824.0 * f.g.V * nrhs, st);
        launch_f64(f, f.U64, f.A64, op, nrhs, (const double2*)in, (double2*)out, (const double2*)b, sh, act, st);
        return;
    }
    KTimer kt("wilson_clover_f32", bytes, 1824.0 * f.g.V * nrhs, st);
    // several right-hand sides: time-fastest bricks of 8 time slices
    // (needs whole 128-site blocks per time slice and L0 a multiple of 8)
    const int vs = f.g.L[1] * f.g.L[2] * f.g.L[3];
    const int tb = (nrhs > 1 && vs % 128 == 0 && f.g.L[0] % 8 == 0) ? 8 : 0;
    // two right-hand sides per thread once that leaves enough threads: 16 x 8^3
    // with 4 10.3 us against 7.7 with one, 32 x 16^3 with 2 35.4 / 38.9, with 16
    // 193 / 219, 64 x 32^3 with 2 440 / 507
    const int nr = nrhs > 1 && (size_t)f.g.V * nrhs >= 196608 ? 2 : 1;
    const bool w32 = (((uintptr_t)in | (uintptr_t)out) & 31) == 0;
    const unsigned grid = (unsigned)((f.g.V + 127) / 128) * (unsigned)((nrhs + nr - 1) / nr);
    auto kern = nr == 2 ? (w32 ? wilson_clover_soa_kernel<2, true> : wilson_clover_soa_kernel<2, false>)
                        : (w32 ? wilson_clover_soa_kernel<1, true> : wilson_clover_soa_kernel<1, false>);
    // a single right-hand side far past L2: 168 registers, more loads in flight per
    // thread (2^21 sites 281 us against 291, 2^20 146 / 152, 2^19 76.5 / 78.6, 2^18 43.5 /
    // 45.0; 2^17, in L2, 25.0 / 23.3): the line lies inside what was faster
    if (nr == 1 && w32 && f.g.V >= (1 << 20)) kern = wilson_clover_soa_kernel<1, true, 3>;
    kern<<<grid, 128, 0, st>>>((float2*)out, (const float2*)in, (const float2*)b, f.U32s, f.A32s, f.g, op, sh,
                               (size_t)f.g.V * 12, act, nrhs, tb);
}

void tangent_fields(const FineOp& f, const double2* X, double2* dU, double* dA, cudaStream_t st) {
    {
        KTimer kt("link_tangent", 0.0, 0.0, st);
        link_tangent_kernel<<<1216, 256, 0, st>>>(f.U64, X, dU, f.g.V);
    }
    KTimer kt("clover_tangent", 0.0, 0.0, st);
    clover_tangent_kernel<<<(f.g.V + 127) / 128, 128, 0, st>>>(f.U64, dU, f.g, f.csw, dA);
}

void apply_tangent(const FineOp& f, const double2* dU, const double* dA, int nrhs, const double2* in, double2* out,
                   cudaStream_t st) {
    // the hop terms with dU and the clover derivative: the stencil with these
    // fields in place of U and (m0 + 4) + C, shift 0
    Shifts sh{};
    KTimer kt("wilson_tangent_f64", 0.0, 1824.0 * f.g.V * nrhs, st);
    launch_f64(f, dU, dA, QCD_OP_D, nrhs, in, out, nullptr, sh, nullptr, st);
}

void apply_op(const FineOp& f, int prec, int op, int nrhs, const void* in, void* out,
              const double* tau, cudaStream_t st, const int* act) {
    launch_dirac(f, prec, op, nrhs, in, out, nullptr, tau, act, st);
}

void residual_op(const FineOp& f, int prec, int op, int nrhs, const void* b, const void* x, void* r,
                 const double* tau, cudaStream_t st, const int* act) {
    launch_dirac(f, prec, op, nrhs, x, r, b, tau, act, st);
}

}  // namespace qcd
