// Device-resident Krylov control.
//
// (1) The Hessenberg bookkeeping of batched (F)GMRES -- Givens rotations,
//     residual estimates, per-right-hand-side stopping and the final
//     triangular solve -- as tiny kernels, so that a whole (F)GMRES solve is a
//     fixed launch sequence without host round trips (converged right-hand
//     sides are skipped by every kernel through the `active` flags).
// (2) A persistent cooperative kernel that runs a complete batched GMRES on
//     the coarse stencil (the coarse-grid solve to a fixed reduction, Table 2
//     "coarse grid tolerance") in one launch: operator apply, classical
//     Gram-Schmidt applied twice, Givens and the solution update, separated by
//     grid-wide barriers of the cooperative launch.
#include <cooperative_groups.h>

#include <algorithm>
#include <utility>
#include "internal.h"

namespace cg = cooperative_groups;

namespace qcd {

namespace {

__device__ __forceinline__ double cabs2(double2 a) { return a.x * a.x + a.y * a.y; }

// Givens update of column `it` of one right-hand side; h[0..it] is the new
// Hessenberg column, hn its sub-diagonal entry.  Returns |g_{it+1}|.
// (FP64: the host-side FGMRES bookkeeping and FP64 coarse solves.)
__device__ double givens_column(double2* h, double hn, double* cs, double2* sn, double2* g, int it) {
    for (int i = 0; i < it; ++i) {
        double2 a = h[i], c = h[i + 1];
        h[i] = cs[i] * a + sn[i] * c;
        h[i + 1] = cs[i] * c - conj(sn[i]) * a;
    }
    double2 a = h[it];
    double2 c = make_double2(hn, 0.0);
    double aa = sqrt(cabs2(a)), rr = sqrt(aa * aa + hn * hn);
    if (aa > 0) {
        cs[it] = aa / rr;
        sn[it] = (1.0 / rr) * ((1.0 / aa) * a * conj(c));
    } else {
        cs[it] = 0.0;
        sn[it] = make_double2(1, 0);
    }
    h[it] = cs[it] * a + sn[it] * c;
    g[it + 1] = -1.0 * (conj(sn[it]) * g[it]);
    g[it] = cs[it] * g[it];
    return sqrt(cabs2(g[it + 1]));
}

// Same update in the working precision R of a coarse solve (FP32 for the
// mixed-precision path: the coarse system only needs a 0.5 reduction).
template <typename R>
__device__ double givens_column_t(cplx<R>* h, R hn, R* cs, cplx<R>* sn, cplx<R>* g, int it) {
    for (int i = 0; i < it; ++i) {
        cplx<R> a = h[i], c = h[i + 1];
        h[i] = cs[i] * a + sn[i] * c;
        h[i + 1] = cs[i] * c - conj(sn[i]) * a;
    }
    cplx<R> a = h[it];
    cplx<R> c = mk<R>(hn, R(0));
    R aa = sqrt(a.x * a.x + a.y * a.y), rr = sqrt(aa * aa + hn * hn);
    if (aa > R(0)) {
        cs[it] = aa / rr;
        sn[it] = (R(1) / rr) * ((R(1) / aa) * a * conj(c));
    } else {
        cs[it] = R(0);
        sn[it] = mk<R>(R(1), R(0));
    }
    h[it] = cs[it] * a + sn[it] * c;
    g[it + 1] = R(-1) * (conj(sn[it]) * g[it]);
    g[it] = cs[it] * g[it];
    return (double)sqrt(g[it + 1].x * g[it + 1].x + g[it + 1].y * g[it + 1].y);
}

__global__ void kry_init_kernel(KryDev K, const double2* __restrict__ nrm, const int* __restrict__ outer_act) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= K.nrhs) return;
    const double b = sqrt(fmax(nrm[j].x, 0.0));
    const bool on = b > 0.0 && (outer_act == nullptr || outer_act[j] != 0);
    K.beta[j] = b;
    K.g[(size_t)j * (K.maxit + 1)] = make_double2(b, 0.0);
    K.active[j] = on ? 1 : 0;
    K.k[j] = 0;
    K.scale[j] = make_double2(on ? 1.0 / b : 0.0, 0.0);
}

// ------------------------------------------------------------------ Arnoldi step
// One step of batched (F)GMRES in three launches (they were six): inner products
// h1 = V^H w; w -= V h1 with h2 = V^H w of the result; w -= V h2 with ||w||^2 and the
// Givens update.  CTA (x, j) owns a part of the entries of right-hand side j, and a
// thread meets the same entries in both halves of a launch.  Bound by the reads of V
// from L2; 16 inner products per pass over w (4 or 8 in the first steps), whose loads
// overlap and whose sums share one halving reduction of the warp.  One wave of CTAs
// (3 per SM with 16 products; 4 of them in two waves took 18 + 24 us).  16 x 8^3,
// 4 right-hand sides, steps 1 to 20 with the launch records on: 75 -> 54 us (inner
// products 15.6, with the first projection 18.3, second projection, norm and
// rotation 20.3).
template <typename Z, typename R>
__device__ __forceinline__ Z kry_projected(const Z* __restrict__ V, size_t vs, int nv, const Z* cs, Z w, size_t e) {
    Z acc;
    acc.x = 0; acc.y = 0;
    for (int i = 0; i < nv; i += 8) {
        Z x[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            x[q].x = 0; x[q].y = 0;
            if (i + q < nv) x[q] = __ldg(V + (size_t)(i + q) * vs + e);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (i + q < nv) acc += cs[i + q] * x[q];
    }
    w.x -= acc.x;
    w.y -= acc.y;
    return w;
}

// true in the CTA of right-hand side j that finishes last
__device__ __forceinline__ bool kry_last(unsigned* counter) {
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// CTAs per SM that the registers of 2 G sums and G loads leave
template <typename R, int G> __host__ __device__ constexpr int kry_ctas() { return sizeof(R) * G >= 64 ? 3 : 4; }
template <typename Z, typename R, int G, bool kProject>
__global__ void __launch_bounds__(256, kry_ctas<R, G>()) kry_dots_kernel(const Z* __restrict__ V, size_t vs, int nv, Z* w, size_t n,
                                                       int nrhs, const double2* __restrict__ h,
                                                       double* __restrict__ partial, unsigned* __restrict__ counters,
                                                       double2* __restrict__ dots, const int* __restrict__ act) {
    const int j = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, parts = gridDim.x;
    if (!act[j]) return;
    __shared__ Z cs[kMaxKry + 1];
    __shared__ R red[8][2 * G];
    const size_t lo = n * blockIdx.x / parts, hi = n * (blockIdx.x + 1) / parts;
    const Z* Vj = V + (size_t)j * n;
    Z* wj = w + (size_t)j * n;
    if constexpr (kProject) {
        for (int i = threadIdx.x; i < nv; i += blockDim.x) {
            cs[i].x = (R)h[(size_t)i * nrhs + j].x;
            cs[i].y = (R)h[(size_t)i * nrhs + j].y;
        }
        __syncthreads();
        for (size_t e = lo + threadIdx.x; e < hi; e += blockDim.x)
            wj[e] = kry_projected<Z, R>(Vj, vs, nv, cs, wj[e], e);
    }
    double* pj = partial + (size_t)j * nv * 2 * parts;
    for (int i0 = 0; i0 < nv; i0 += G) {
        R acc[2 * G];
#pragma unroll
        for (int q = 0; q < 2 * G; ++q) acc[q] = R(0);
        for (size_t e = lo + threadIdx.x; e < hi; e += blockDim.x) {
            const Z y = wj[e];
            Z x[G];
#pragma unroll
            for (int q = 0; q < G; ++q) {
                x[q].x = 0; x[q].y = 0;
                if (i0 + q < nv) x[q] = __ldg(Vj + (size_t)(i0 + q) * vs + e);
            }
#pragma unroll
            for (int q = 0; q < G; ++q) cdot(acc[2 * q], acc[2 * q + 1], x[q], y);
        }
        int base = 0;
        scatter_sum<2 * G, 16>(acc, lane, base);
        if ((lane & (32 / (2 * G) - 1)) == 0) red[warp][base] = acc[0];
        __syncthreads();
        // the sums of the warps in FP64, as everything across warps
        if (threadIdx.x < 2 * G && i0 + threadIdx.x / 2 < nv) {
            double s = 0.0;
#pragma unroll
            for (int k = 0; k < 8; ++k) s += (double)red[k][threadIdx.x];
            pj[(size_t)(2 * i0 + threadIdx.x) * parts + blockIdx.x] = s;
        }
        __syncthreads();
    }
    if (!kry_last(&counters[j])) return;
    for (int v = warp; v < nv; v += 8) {
        double2 s = make_double2(0.0, 0.0);
        for (int t = lane; t < parts; t += 32) {
            s.x += __ldcg(pj + (size_t)(2 * v) * parts + t);
            s.y += __ldcg(pj + (size_t)(2 * v + 1) * parts + t);
        }
        s.x = warp_sum(s.x);
        s.y = warp_sum(s.y);
        if (lane == 0) dots[(size_t)v * nrhs + j] = s;
    }
    if (threadIdx.x == 0) counters[j] = 0u;
}

// w -= V h2 and, in the CTA that finishes last, ||w|| and the Givens update
template <typename Z, typename R>
__global__ void __launch_bounds__(256) kry_step_kernel(KryDev K, int it, const Z* __restrict__ V, size_t vs, Z* w,
                                                       size_t n, const double2* __restrict__ h1,
                                                       const double2* __restrict__ h2, double* __restrict__ partial,
                                                       unsigned* __restrict__ counters) {
    const int j = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, parts = gridDim.x, nv = it + 1;
    if (!K.active[j]) return;
    __shared__ Z co[kMaxKry + 1];
    __shared__ double red[8];
    const size_t lo = n * blockIdx.x / parts, hi = n * (blockIdx.x + 1) / parts;
    const Z* Vj = V + (size_t)j * n;
    Z* wj = w + (size_t)j * n;
    for (int i = threadIdx.x; i < nv; i += blockDim.x) {
        co[i].x = (R)h2[(size_t)i * K.nrhs + j].x;
        co[i].y = (R)h2[(size_t)i * K.nrhs + j].y;
    }
    __syncthreads();
    R nn = 0;
    for (size_t e = lo + threadIdx.x; e < hi; e += blockDim.x) {
        const Z o = kry_projected<Z, R>(Vj, vs, nv, co, wj[e], e);
        wj[e] = o;
        nn += o.x * o.x + o.y * o.y;
    }
    nn = warp_sum(nn);
    if (lane == 0) red[warp] = (double)nn;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int k = 0; k < 8; ++k) s += red[k];
        partial[(size_t)j * parts + blockIdx.x] = s;
    }
    if (!kry_last(&counters[j])) return;
    // the column, the rotations so far and the norm in shared memory: one thread
    // turns the column in a serial chain of FP64 operations
    __shared__ double2 h[kMaxKry + 1], sn[kMaxKry];
    __shared__ double cs[kMaxKry], norm2;
    for (int i = threadIdx.x; i < nv; i += blockDim.x) h[i] = h1[(size_t)i * K.nrhs + j] + h2[(size_t)i * K.nrhs + j];
    for (int i = threadIdx.x; i < it; i += blockDim.x) {
        cs[i] = K.cs[(size_t)j * K.maxit + i];
        sn[i] = K.sn[(size_t)j * K.maxit + i];
    }
    if (warp == 7) {
        double s = 0.0;
        for (int t = lane; t < parts; t += 32) s += __ldcg(partial + (size_t)j * parts + t);
        s = warp_sum(s);
        if (lane == 0) norm2 = s;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const double hn = sqrt(fmax(norm2, 0.0)), beta = K.beta[j];
        const double res = givens_column(h, hn, cs, sn, K.g + (size_t)j * (K.maxit + 1), it);
        K.cs[(size_t)j * K.maxit + it] = cs[it];
        K.sn[(size_t)j * K.maxit + it] = sn[it];
        K.k[j] = it + 1;
        K.scale[j] = make_double2(hn > 0 ? 1.0 / hn : 0.0, 0.0);
        if (res <= K.tol * beta) K.active[j] = 0;
        K.resid[j] = beta > 0 ? res / beta : 0.0;
        counters[j] = 0u;
    }
    __syncthreads();
    double2* Rj = K.R + (size_t)j * K.maxit * K.maxit;
    for (int i = threadIdx.x; i <= it; i += blockDim.x) Rj[(size_t)i * K.maxit + it] = h[i];
}

// Triangular solve R y = g, one warp per right-hand side: each y_i is taken out of
// the rows above at once (65 us with one thread per right-hand side and 20 steps).
__global__ void __launch_bounds__(32) kry_finish_kernel(KryDev K) {
    const int j = blockIdx.x, lane = threadIdx.x, kd = K.k[j];
    const double2* R = K.R + (size_t)j * K.maxit * K.maxit;
    __shared__ double2 y[kMaxKry];
    for (int i = lane; i < kd; i += 32) y[i] = K.g[(size_t)j * (K.maxit + 1) + i];
    __syncwarp();
    for (int i = kd - 1; i >= 0; --i) {
        const double2 d = R[(size_t)i * K.maxit + i];
        const double den = cabs2(d);
        const double2 v = den > 0 ? (1.0 / den) * cmulc(d, y[i]) : make_double2(0, 0);
        __syncwarp();
        if (lane == 0) y[i] = v;
        for (int l = lane; l < i; l += 32) y[l] -= R[(size_t)l * K.maxit + i] * v;
        __syncwarp();
    }
    for (int i = lane; i < K.maxit; i += 32)
        K.coef[(size_t)i * K.nrhs + j] = i < kd ? y[i] : make_double2(0, 0);
}

// ------------------------------------------------------------------ coarse GMRES
// Each CTA owns the chunk [lo, hi) of every coarse vector.  It keeps its
// chunk of the whole Krylov basis in shared memory; only the newest basis
// vector is published to global memory (double-buffered) for the neighbour
// reads of the stencil.  Inner products are accumulated into FP64 totals
// with atomics, one grid barrier per reduction; the totals are double-
// buffered by iteration parity, so zeroing the next iteration's buffer never
// races with readers of the current one.  Every CTA performs the (tiny)
// Givens updates itself on identical totals.
// Bound by latency: per iteration two or three barriers, the gather of the
// neighbour vectors and the serial bookkeeping.  Stencil blocks (in flight from the
// start to the first apply) and neighbour vectors come by 16-byte asynchronous
// copies; with loads of one entry through registers, a few in flight per thread,
// the 16 x 8^3 hierarchy (512 sites, nc 16, 4 right-hand sides) took 39 us per solve
// in two or three iterations and 148 in twelve, then 26 and 124.  The rotations run
// between arriving at the end-of-iteration barrier and waiting, and the last
// projection writes the next basis vector: 26 and 112.
template <typename Z, typename R>
struct CoarseArgs {
    Geom gc;
    int nc;
    const Z* A;          // [Vc][9][col][row]
    const Z* b;          // nrhs coarse vectors
    Z* x;                // nrhs coarse vectors (output)
    Z* Vg;               // [2][nrhs][nco] newest basis vector, double-buffered
    double2* tot;        // [2 parities][2 passes][npair] FP64 totals
    double2* Rg;         // [nrhs][maxit][maxit] triangular factor (written by CTA 0)
    double2* yv;         // [nrhs][maxit]
    int* iters;          // [nrhs] iterations used (written by CTA 0)
    unsigned long long* counter;   // [2] solves, iterations (accumulated, may be null)
    double* resid;       // [nrhs] relative residual estimates
    int op;
    const double* tau;   // device [nrhs]
    const int* act;      // device [nrhs] or null
    double tol;
    int maxit;
    int nrhs;
    int E;               // chunk length per CTA (= sites per CTA * nc)
    int sps;             // coarse sites per CTA
    int a_smem;          // 1: this CTA's stencil blocks are staged in shared memory
    Z* Vglob;            // non-null: the Krylov basis and w chunks live in global
    Z* wglob;            //   memory ([CTA][(maxit+1)][nrhs][E] and [CTA][nrhs][E])
};

template <typename Z, typename R>
__device__ __forceinline__ void coarse_row(const CoarseArgs<Z, R>& a, const Z* xj, int s, int r, const int c[4], R tj,
                                           Z& out) {
    Z acc; acc.x = 0; acc.y = 0;
    for (int d = 0; d < 9; ++d) {
        int sn = s;
        if (d > 0) {
            int mu = (d - 1) & 3, step = d <= 4 ? 1 : -1;
            int cn[4] = {c[0], c[1], c[2], c[3]};
            cn[mu] = (cn[mu] + step + a.gc.L[mu]) % a.gc.L[mu];
            sn = site_index(a.gc, cn);
        }
        const Z* am = a.A + (((size_t)s * 9 + d) * a.nc) * a.nc + r;
        const Z* xs = xj + (size_t)sn * a.nc;
        Z part; part.x = 0; part.y = 0;   // a direction by itself rounds less than one chain over all
        for (int col = 0; col < a.nc; ++col) cmac(part, am[(size_t)col * a.nc], xs[col]);
        acc += part;
    }
    const R sg = r < a.nc / 2 ? R(1) : R(-1);
    Z xv = xj[(size_t)s * a.nc + r];
    if (a.op == QCD_OP_D) { acc -= (tj * sg) * xv; }
    else { acc = sg * acc; acc -= tj * xv; }
    out = acc;
}

struct CoarseSmem { size_t As, xn, nbr, Vs, ws, hr, hcol, cs, sn, g, beta, hn, live, kd, total; };
// Shared-memory layout of one CTA.  sps = 0: no staged stencil blocks;
// basis_in_smem = false: the Krylov basis and w chunks are in global memory.
template <typename Z>
__host__ __device__ inline CoarseSmem coarse_smem(int nrhs, int maxit, int E, int sps = 0, int nc = 0,
                                                  bool basis_in_smem = true) {
    auto up = [](size_t v) { return (v + 15) & ~size_t(15); };
    const size_t Eb = basis_in_smem ? (size_t)E : 0;
    CoarseSmem L;
    size_t o = 0;
    L.As = o;   o = up(o + sizeof(Z) * (size_t)sps * 9 * nc * nc);
    L.xn = o;   o = up(o + sizeof(Z) * (size_t)nrhs * sps * 9 * nc);
    L.nbr = o;  o = up(o + sizeof(int) * (size_t)sps * 9);
    L.Vs = o;   o = up(o + sizeof(Z) * (size_t)(maxit + 1) * nrhs * Eb);
    L.ws = o;   o = up(o + sizeof(Z) * (size_t)nrhs * Eb);
    L.hr = o;   o = up(o + sizeof(Z) * (size_t)(maxit + 1) * nrhs);
    L.hcol = o; o = up(o + sizeof(Z) * (size_t)(maxit + 1) * nrhs);
    L.cs = o;   o = up(o + sizeof(Z) * (size_t)nrhs * maxit);
    L.sn = o;   o = up(o + sizeof(Z) * (size_t)nrhs * maxit);
    L.g = o;    o = up(o + sizeof(Z) * (size_t)nrhs * (maxit + 1));
    L.beta = o; o = up(o + sizeof(double) * nrhs);
    L.hn = o;   o = up(o + sizeof(Z) * nrhs);
    L.live = o; o = up(o + sizeof(int) * nrhs);
    L.kd = o;   o = up(o + sizeof(int) * nrhs);
    L.total = o;
    return L;
}

// 16 bytes from global memory (through L2: other CTAs may have just written them) to
// shared memory, in flight until the wait
__device__ __forceinline__ void async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

template <typename Z> struct __align__(16) Pair { Z a, b; };

template <typename Z, typename R>
__global__ void __launch_bounds__(256) coarse_gmres_kernel(CoarseArgs<Z, R> a) {
    cg::grid_group grid = cg::this_grid();
    extern __shared__ __align__(16) unsigned char sraw[];
    const int nrhs = a.nrhs, maxit = a.maxit, E = a.E, nc = a.nc;
    const bool gbasis = a.Vglob != nullptr;
    const CoarseSmem LY = coarse_smem<Z>(nrhs, maxit, E, a.a_smem ? a.sps : 0, a.a_smem ? nc : 0, !gbasis);
    Z* As = reinterpret_cast<Z*>(sraw + LY.As);          // [sps][9][col][row] stencil blocks of my sites
    Z* xn = reinterpret_cast<Z*>(sraw + LY.xn);          // [nrhs][sps][9][nc] neighbour vectors
    int* nbr = reinterpret_cast<int*>(sraw + LY.nbr);    // [sps][9] neighbour sites
    // [(maxit+1)][nrhs][E] basis chunk and [nrhs][E] w chunk of this CTA
    Z* Vs = gbasis ? a.Vglob + (size_t)blockIdx.x * (maxit + 1) * nrhs * E : reinterpret_cast<Z*>(sraw + LY.Vs);
    Z* ws = gbasis ? a.wglob + (size_t)blockIdx.x * nrhs * E : reinterpret_cast<Z*>(sraw + LY.ws);
    // the serial per-iteration bookkeeping runs in the working precision R:
    // a dependent chain of FP64 operations is very slow on this part
    Z* hr = reinterpret_cast<Z*>(sraw + LY.hr);               // current-pass coefficients in the working precision
    Z* hcol = reinterpret_cast<Z*>(sraw + LY.hcol);      // [nrhs][maxit+1] column under rotation
    R* cs = reinterpret_cast<R*>(sraw + LY.cs);
    Z* sn = reinterpret_cast<Z*>(sraw + LY.sn);
    Z* g = reinterpret_cast<Z*>(sraw + LY.g);
    double* beta = reinterpret_cast<double*>(sraw + LY.beta);
    int* live = reinterpret_cast<int*>(sraw + LY.live);
    int* kd = reinterpret_cast<int*>(sraw + LY.kd);
    R* hn = reinterpret_cast<R*>(sraw + LY.hn);          // [nrhs] norm of the projected w

    const size_t nco = (size_t)a.gc.V * a.nc;
    const size_t lo = (size_t)blockIdx.x * E;
    const int len = lo >= nco ? 0 : (int)min((size_t)E, nco - lo);
    const int s0 = blockIdx.x * a.sps;
    const int nsl = len / nc;                               // sites owned by this CTA
    if (a.a_smem) {
        // 16-byte copies in flight until the first operator apply (nc is even: blocks
        // and vectors start on 16-byte boundaries)
        const char* src = reinterpret_cast<const char*>(a.A + (size_t)s0 * 9 * nc * nc);
        const size_t bytes = sizeof(Z) * (size_t)nsl * 9 * nc * nc;
        for (size_t t = 16 * (size_t)threadIdx.x; t < bytes; t += 16 * (size_t)blockDim.x)
            async16(reinterpret_cast<char*>(As) + t, src + t);
        async_commit();
        for (int t = threadIdx.x; t < nsl * 9; t += blockDim.x) {
            const int sl = t / 9, d = t % 9;
            int c[4];
            site_coords(a.gc, s0 + sl, c);
            int sn = s0 + sl;
            if (d > 0) {
                int mu = (d - 1) & 3, step = d <= 4 ? 1 : -1;
                c[mu] = (c[mu] + step + a.gc.L[mu]) % a.gc.L[mu];
                sn = site_index(a.gc, c);
            }
            nbr[t] = sn;
        }
    }
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const int npair = (maxit + 2) * nrhs;
    auto TOT = [&](int parity, int pass) { return a.tot + ((size_t)parity * 2 + pass) * npair; };
    auto VS = [&](int i, int j) { return Vs + ((size_t)i * nrhs + j) * E; };

    // partial inner products of this chunk: <Vs_i[j], ws[j]> for i < ni (+ ||ws_j||^2), added to `tot`
    auto dots = [&](double2* tot, int ni, bool with_norm, const Z* Y) {
        const int np = ni * nrhs + (with_norm ? nrhs : 0);
        // two pairs per warp and round (independent shuffle chains overlap);
        // this CTA's share in the working precision R, only the cross-CTA
        // totals are FP64 (FP64 throughput per SM is tiny on this part)
        for (int p0 = 2 * warp; p0 < np; p0 += 2 * nw) {
            R re[2] = {0, 0}, im[2] = {0, 0};
            int slot[2] = {-1, -1};
            for (int q = 0; q < 2; ++q) {
                const int p = p0 + q;
                if (p >= np) break;
                int j;
                const Z* xa;
                if (p < ni * nrhs) { j = p % nrhs; xa = VS(p / nrhs, j); }
                else { j = p - ni * nrhs; xa = Y + (size_t)j * E; }
                if (!live[j]) continue;
                const Z* ya = Y + (size_t)j * E;
                for (int e = lane; e < len; e += 32) {
                    Z u = xa[e], v = ya[e];
                    cdot(re[q], im[q], u, v);
                }
                slot[q] = p < ni * nrhs ? p : (maxit + 1) * nrhs + j;
            }
            for (int o = 16; o > 0; o >>= 1) {
                re[0] += __shfl_xor_sync(0xffffffffu, re[0], o);
                im[0] += __shfl_xor_sync(0xffffffffu, im[0], o);
                re[1] += __shfl_xor_sync(0xffffffffu, re[1], o);
                im[1] += __shfl_xor_sync(0xffffffffu, im[1], o);
            }
            if (lane == 0 && len > 0)
                for (int q = 0; q < 2; ++q)
                    if (slot[q] >= 0) {
                        atomicAdd(&tot[slot[q]].x, (double)re[q]);
                        atomicAdd(&tot[slot[q]].y, (double)im[q]);
                    }
        }
    };
    // put(j, e, ws[j][e] - sum_i hr[i][j] Vs_i[j][e])
    auto project = [&](int ni, auto put) {
        for (int t = tid; t < nrhs * len; t += blockDim.x) {
            const int j = t / len, e = t % len;
            if (!live[j]) continue;
            Z acc = ws[(size_t)j * E + e];
            const Z* v = VS(0, j) + e;
#pragma unroll 4
            for (int i = 0; i < ni; ++i, v += (size_t)nrhs * E) acc -= hr[i * nrhs + j] * *v;
            put(j, e, acc);
        }
    };
    // coefficients of a Gram-Schmidt pass from its totals (hr; added to hcol), one
    // warp per right-hand side, and hn = ||w|| after it; 1 where another is needed
    auto column = [&](int parity, int pass, int it) {
        int again = 0;
        for (int j = warp; j < nrhs; j += nw) {
            if (!live[j]) continue;
            const double2* tot = TOT(parity, pass);
            R sq = 0;
            for (int i = lane; i <= it; i += 32) {
                const double2 v = tot[i * nrhs + j];
                const Z c = mk<R>((R)v.x, (R)v.y);
                Z* h = hcol + (size_t)j * (maxit + 1) + i;
                hr[i * nrhs + j] = c;
                *h = pass == 0 ? c : *h + c;
                sq += c.x * c.x + c.y * c.y;
            }
            const R before = (R)tot[(maxit + 1) * nrhs + j].x;
            const R rest = before - warp_sum(sq);
            if (lane == 0) hn[j] = rest > R(0) ? sqrt(rest) : R(0);
            again |= rest < R(0.1) * before;
        }
        return again;
    };

    // ---- load b, beta = ||b||
    for (int j = tid; j < nrhs; j += blockDim.x) live[j] = (a.act == nullptr || a.act[j]) ? 1 : 0;
    for (int t = tid; t < nrhs * len; t += blockDim.x) {
        const int j = t / len, e = t % len;
        ws[(size_t)j * E + e] = a.b[(size_t)j * nco + lo + e];
    }
    __syncthreads();
    dots(TOT(1, 1), 0, true, ws);           // parity 1 pass 1 region: unused by iteration 0
    grid.sync();
    for (int j = tid; j < nrhs; j += blockDim.x) {
        const double bb = live[j] ? sqrt(fmax(TOT(1, 1)[(maxit + 1) * nrhs + j].x, 0.0)) : 0.0;
        beta[j] = bb;
        if (!(bb > 0)) live[j] = 0;
        kd[j] = 0;
        g[(size_t)j * (maxit + 1)] = mk<R>((R)bb, R(0));
    }
    __syncthreads();
    for (int t = tid; t < nrhs * len; t += blockDim.x) {
        const int j = t / len, e = t % len;
        const R ib = live[j] ? (R)(1.0 / beta[j]) : R(0);
        Z v = ws[(size_t)j * E + e];
        v.x *= ib; v.y *= ib;
        VS(0, j)[e] = v;
        a.Vg[(size_t)j * nco + lo + e] = v;
    }
    grid.sync();
    for (int it = 0; it < maxit; ++it) {
        int any = 0;
        for (int j = 0; j < nrhs; ++j) any |= live[j];
        if (!any) break;
        const int par = it & 1;
        // zero the other parity's totals: every CTA has passed the barrier, so
        // nobody still reads them (they held the previous iteration's sums, or
        // beta in iteration 0), and the next atomics into them follow the
        // next barrier
        if (blockIdx.x == 0)
            for (int t = tid; t < 2 * npair; t += blockDim.x) a.tot[(size_t)(par ^ 1) * 2 * npair + t] = make_double2(0, 0);
        // w = A v_it on this chunk
        const Z* Vit = a.Vg + (size_t)par * nrhs * nco;
        if (a.a_smem) {
            // gather the 9 neighbour blocks of every owned site, then multiply from shared memory
            constexpr int E16 = 16 / sizeof(Z);   // entries per copy
            const int pc = nc / E16, np = nsl * 9 * pc;
            for (int j = 0; j < nrhs; ++j) {
                if (!live[j]) continue;
                const Z* vj = Vit + (size_t)j * nco;
                for (int t = tid; t < np; t += blockDim.x) {
                    const int b = t / pc, q = (t - b * pc) * E16;
                    async16(xn + ((size_t)j * nsl * 9 + b) * nc + q, vj + (size_t)nbr[b] * nc + q);
                }
            }
            async_commit();
            async_wait_all();
            __syncthreads();
            // Tiles of two rows by two right-hand sides, the columns dealt to four
            // lanes: per column one load of two block entries and two of vector
            // entries feed four products.  The eight tiles of a warp cover
            // consecutive rows (conflict-free), and the sums over the four lanes
            // leave one of the four results in each.
            const int rp = len / 2, tiles = rp * ((nrhs + 1) / 2), g8 = 8 * warp + (lane & 7), sub = lane >> 3;
            for (int t0 = 0; t0 < tiles; t0 += 8 * nw) {
                const int t = min(t0 + g8, tiles - 1);
                const int e = t % rp * 2, j = t / rp * 2, j1 = min(j + 1, nrhs - 1), sl = e / nc, r = e - sl * nc;
                const Z* am = As + (size_t)sl * 9 * nc * nc + r;
                const Z* x0 = xn + ((size_t)j * nsl + sl) * 9 * nc;
                const Z* x1 = xn + ((size_t)j1 * nsl + sl) * 9 * nc;
                Z acc[2][2];   // [rhs][row]
#pragma unroll
                for (int q = 0; q < 4; ++q) { acc[q >> 1][q & 1].x = 0; acc[q >> 1][q & 1].y = 0; }
                const Pair<Z>* ap = reinterpret_cast<const Pair<Z>*>(am + (size_t)sub * nc);
                // two columns are summed before they join the running sum: a chain of
                // fused multiply-adds over all of them would round it twice per column
                int dc = sub;
                auto add = [](Z& s, Z m, Z u, Z m2, Z u2) {
                    Z t = m * u;
                    cmac(t, m2, u2);
                    s += t;
                };
#pragma unroll 2
                for (; dc + 4 < 9 * nc; dc += 8, ap += 4 * nc) {
                    const Pair<Z> m = ap[0], m2 = ap[2 * nc];
                    const Z u0 = x0[dc], u1 = x1[dc], v0 = x0[dc + 4], v1 = x1[dc + 4];
                    add(acc[0][0], m.a, u0, m2.a, v0);
                    add(acc[0][1], m.b, u0, m2.b, v0);
                    add(acc[1][0], m.a, u1, m2.a, v1);
                    add(acc[1][1], m.b, u1, m2.b, v1);
                }
                if (dc < 9 * nc) {
                    const Pair<Z> m = *ap;
                    const Z u0 = x0[dc], u1 = x1[dc];
                    acc[0][0] += m.a * u0;
                    acc[0][1] += m.b * u0;
                    acc[1][0] += m.a * u1;
                    acc[1][1] += m.b * u1;
                }
                const bool hi = sub & 2, odd = sub & 1;   // lane bits 16 and 8
                Z k0 = hi ? acc[1][0] : acc[0][0], k1 = hi ? acc[1][1] : acc[0][1];
                const Z g0 = hi ? acc[0][0] : acc[1][0], g1 = hi ? acc[0][1] : acc[1][1];
                k0.x += __shfl_xor_sync(0xffffffffu, g0.x, 16);
                k0.y += __shfl_xor_sync(0xffffffffu, g0.y, 16);
                k1.x += __shfl_xor_sync(0xffffffffu, g1.x, 16);
                k1.y += __shfl_xor_sync(0xffffffffu, g1.y, 16);
                Z o = odd ? k1 : k0;
                const Z gv = odd ? k0 : k1;
                o.x += __shfl_xor_sync(0xffffffffu, gv.x, 8);
                o.y += __shfl_xor_sync(0xffffffffu, gv.y, 8);
                const int jo = j + (hi ? 1 : 0), eo = e + (odd ? 1 : 0), ro = r + (odd ? 1 : 0);
                if (t0 + g8 < tiles && jo < nrhs && live[jo]) {
                    const R sg = ro < nc / 2 ? R(1) : R(-1);
                    const R tj = (R)a.tau[jo];
                    const Z xv = (hi ? x1 : x0)[ro];      // direction 0 is the site itself
                    if (a.op == QCD_OP_D) { o -= (tj * sg) * xv; }
                    else { o = sg * o; o -= tj * xv; }
                    ws[(size_t)jo * E + eo] = o;
                }
            }
        } else {
            for (int t = tid; t < nrhs * len; t += blockDim.x) {
                const int j = t / len, e = t % len;
                if (!live[j]) continue;
                const size_t ge = lo + e;
                const int s = (int)(ge / a.nc), r = (int)(ge % a.nc);
                int c[4];
                site_coords(a.gc, s, c);
                Z out;
                coarse_row<Z, R>(a, Vit + (size_t)j * nco, s, r, c, (R)a.tau[j], out);
                ws[(size_t)j * E + e] = out;
            }
        }
        __syncthreads();
        // classical Gram-Schmidt, pass 1, with ||w||^2 before the projection
        dots(TOT(par, 0), it + 1, true, ws);
        grid.sync();
        // second pass only if some right-hand side lost more than 90% of its
        // squared norm in the first (a Kahan-Parlett test, loosened for a
        // solve that only needs a 0.5 reduction); every CTA takes the same
        // decision from the same totals.  Without it ||w||^2 is by Pythagoras.
        const bool again = __syncthreads_or(column(par, 0, it));
        if (again) {
            project(it + 1, [&](int j, int e, Z v) { ws[(size_t)j * E + e] = v; });
            __syncthreads();
            dots(TOT(par, 1), it + 1, true, ws);
            grid.sync();
            column(par, 1, it);
            __syncthreads();
        }
        // v_{it+1} = w / ||w||, w projected for the last time
        project(it + 1, [&](int j, int e, Z v) {
            const R ih = hn[j] > R(0) ? R(1) / hn[j] : R(0);
            v.x *= ih; v.y *= ih;
            VS(it + 1, j)[e] = v;
            a.Vg[((size_t)(par ^ 1) * nrhs + j) * nco + lo + e] = v;
        });
        // the rotations, a serial chain, while the other CTAs arrive
        __syncthreads();
        auto token = grid.barrier_arrive();
        if (tid < nrhs && live[tid]) {
            const int j = tid;
            Z* h = hcol + (size_t)j * (maxit + 1);
            const double res = givens_column_t<R>(h, hn[j], cs + (size_t)j * maxit, sn + (size_t)j * maxit,
                                                  g + (size_t)j * (maxit + 1), it);
            if (blockIdx.x == 0) {
                Z* Rj = reinterpret_cast<Z*>(a.Rg) + (size_t)j * maxit * maxit;
                for (int i = 0; i <= it; ++i) Rj[(size_t)i * maxit + it] = h[i];
                a.resid[j] = beta[j] > 0 ? res / beta[j] : 0.0;
            }
            kd[j] = it + 1;
            if (res <= a.tol * beta[j]) live[j] = 0;   // converged
        }
        grid.barrier_wait(std::move(token));
        __syncthreads();
    }
    async_wait_all();   // the staged blocks, when no iteration ran
    // triangular solve (CTA 0) and x = V y
    if (blockIdx.x == 0 && tid < nrhs) {
        const int j = tid, k = kd[j];
        const Z* Rj = reinterpret_cast<const Z*>(a.Rg) + (size_t)j * maxit * maxit;
        const Z* gj = g + (size_t)j * (maxit + 1);
        Z* y = reinterpret_cast<Z*>(a.yv) + (size_t)j * maxit;
        for (int i = k - 1; i >= 0; --i) {
            Z sacc = gj[i];
            for (int l = i + 1; l < k; ++l) sacc -= Rj[(size_t)i * maxit + l] * y[l];
            const Z d = Rj[(size_t)i * maxit + i];
            const R den = d.x * d.x + d.y * d.y;
            y[i] = den > R(0) ? (R(1) / den) * cmulc(d, sacc) : mk<R>(R(0), R(0));
        }
        a.iters[j] = k;
        if (a.counter != nullptr && (a.act == nullptr || a.act[j])) {
            atomicAdd(a.counter, 1ull);
            atomicAdd(a.counter + 1, (unsigned long long)k);
        }
    }
    grid.sync();
    for (int t = tid; t < nrhs * len; t += blockDim.x) {
        const int j = t / len, e = t % len;
        if (a.act != nullptr && !a.act[j]) continue;
        const int k = kd[j];
        const Z* y = reinterpret_cast<const Z*>(a.yv) + (size_t)j * maxit;
        Z o; o.x = 0; o.y = 0;
        for (int i = 0; i < k; ++i) o += y[i] * VS(i, j)[e];
        a.x[(size_t)j * nco + lo + e] = o;
    }
}

}  // namespace

size_t kry_bytes(int nrhs, int maxit) {
    return sizeof(double) * nrhs * 2 + sizeof(int) * nrhs * 2 + sizeof(double) * (size_t)nrhs * maxit +
           sizeof(double2) * ((size_t)nrhs * maxit + (size_t)nrhs * (maxit + 1) + (size_t)nrhs * maxit * maxit +
                              (size_t)maxit * nrhs + nrhs) + 256;
}

KryDev kry_layout(void* buf, int nrhs, int maxit, double tol) {
    KryDev K;
    K.nrhs = nrhs;
    K.maxit = maxit;
    K.tol = tol;
    char* p = (char*)buf;
    auto take = [&](size_t bytes) { char* q = p; p += (bytes + 15) & ~size_t(15); return (void*)q; };
    K.g = (double2*)take(sizeof(double2) * (size_t)nrhs * (maxit + 1));
    K.sn = (double2*)take(sizeof(double2) * (size_t)nrhs * maxit);
    K.R = (double2*)take(sizeof(double2) * (size_t)nrhs * maxit * maxit);
    K.coef = (double2*)take(sizeof(double2) * (size_t)maxit * nrhs);
    K.scale = (double2*)take(sizeof(double2) * nrhs);
    K.cs = (double*)take(sizeof(double) * (size_t)nrhs * maxit);
    K.beta = (double*)take(sizeof(double) * nrhs);
    K.resid = (double*)take(sizeof(double) * nrhs);
    K.active = (int*)take(sizeof(int) * nrhs);
    K.k = (int*)take(sizeof(int) * nrhs);
    return K;
}

void kry_init(const KryDev& K, const double2* nrm, const int* outer_act, cudaStream_t st) {
    KTimer kt("kry_init", 0.0, 0.0, st);
    kry_init_kernel<<<1, 64, 0, st>>>(K, nrm, outer_act);
}
int coarse_gmres_grid() {
    static int nct = 0;
    if (nct == 0) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        nct = sms > 0 ? sms : 1;
    }
    return nct;
}

template <typename Z, typename R, int G, bool kProject>
static void launch_kry_dots(const KryDev& K, const Z* V, size_t vs, size_t n, int nv, Z* w, const double2* h,
                            double* partial, unsigned* counters, double2* dots, dim3 grid, cudaStream_t st) {
    KTimer kt(std::is_same<R, double>::value ? (kProject ? "kry_project_f64" : "kry_dots_f64")
                                             : (kProject ? "kry_project_f32" : "kry_dots_f32"),
              (double)(nv + (kProject ? 2 : 1)) * K.nrhs * n * sizeof(Z), (kProject ? 16.0 : 8.0) * nv * K.nrhs * n, st);
    kry_dots_kernel<Z, R, G, kProject><<<grid, 256, 0, st>>>(V, vs, nv, w, n, K.nrhs, h, partial, counters, dots, K.active);
}
// parts per right-hand side: one wave over all of them, at least 256 entries each
static dim3 kry_grid(int nrhs, size_t n, int ctas) {
    const size_t parts = std::max<size_t>(1, (size_t)ctas * coarse_gmres_grid() / nrhs);
    return dim3((unsigned)std::min({parts, std::max<size_t>(1, n / 256), (size_t)kKryParts}), nrhs);
}
template <typename Z, typename R, int G>
static void arnoldi_passes(const KryDev& K, const Z* V, size_t vs, size_t n, int nv, Z* w, double2* h1, double2* h2,
                           double* partial, unsigned* counters, cudaStream_t st) {
    const dim3 grid = kry_grid(K.nrhs, n, kry_ctas<R, G>());
    launch_kry_dots<Z, R, G, false>(K, V, vs, n, nv, w, nullptr, partial, counters, h1, grid, st);
    launch_kry_dots<Z, R, G, true>(K, V, vs, n, nv, w, h1, partial, counters, h2, grid, st);
}
template <typename Z, typename R, int GMAX>
static void arnoldi(const KryDev& K, const Z* V, size_t vs, size_t n, int it, Z* w, double2* h1, double2* h2,
                    double* partial, unsigned* counters, cudaStream_t st) {
    const int nv = it + 1;
    if (nv <= 4) arnoldi_passes<Z, R, 4>(K, V, vs, n, nv, w, h1, h2, partial, counters, st);
    else if (nv <= 8 || GMAX == 8) arnoldi_passes<Z, R, 8>(K, V, vs, n, nv, w, h1, h2, partial, counters, st);
    else arnoldi_passes<Z, R, GMAX>(K, V, vs, n, nv, w, h1, h2, partial, counters, st);
    KTimer kt("kry_step", (double)(nv + 2) * K.nrhs * n * sizeof(Z), 8.0 * nv * K.nrhs * n, st);
    kry_step_kernel<Z, R><<<kry_grid(K.nrhs, n, 4), 256, 0, st>>>(K, it, V, vs, w, n, h1, h2, partial, counters);
}
void kry_arnoldi(const KryDev& K, int prec, const void* V, size_t vs, size_t n, int it, void* w, double2* h1, double2* h2,
                 void* partial, unsigned* counters, cudaStream_t st) {
    if (prec == QCD_FP64)
        arnoldi<double2, double, 8>(K, (const double2*)V, vs, n, it, (double2*)w, h1, h2, (double*)partial, counters, st);
    else
        arnoldi<float2, float, 16>(K, (const float2*)V, vs, n, it, (float2*)w, h1, h2, (double*)partial, counters, st);
}
void kry_finish(const KryDev& K, cudaStream_t st) {
    KTimer kt("kry_finish", 0.0, 0.0, st);
    kry_finish_kernel<<<K.nrhs, 32, 0, st>>>(K);
}


// Site-based partition: each CTA owns `sps` consecutive coarse sites.
static void coarse_partition(const Coarse& c, int& sps, int& nblk) {
    const int nct = c.ctas > 0 ? std::min(c.ctas, coarse_gmres_grid()) : coarse_gmres_grid();
    sps = (c.gc.V + nct - 1) / nct;
    nblk = (c.gc.V + sps - 1) / sps;
}
constexpr size_t kCoarseSmemCap = 200 * 1024;

// Where the cooperative kernel keeps its data, in order of preference:
// stencil blocks and Krylov basis in shared memory (layout 1), basis only
// (layout 2), basis in global memory (layout 3).  `want` = 0 picks the first
// that fits; 1..3 forces one (it must fit).
struct CoarseMode {
    int layout = 0;       // 1, 2, 3; 0: nothing fits
    size_t smem = 0;
};
static CoarseMode coarse_mode(const Coarse& c, int prec, int nrhs, int maxit, int want) {
    int sps, nblk;
    coarse_partition(c, sps, nblk);
    const int E = sps * c.nc;
    CoarseMode m;
    for (int layout = 1; layout <= 3; ++layout) {
        if (want != 0 && layout != want) continue;
        const int s = layout == 1 ? sps : 0, nc = layout == 1 ? c.nc : 0;
        const bool smem_basis = layout != 3;
        const size_t t = prec == QCD_FP64 ? coarse_smem<double2>(nrhs, maxit, E, s, nc, smem_basis).total
                                          : coarse_smem<float2>(nrhs, maxit, E, s, nc, smem_basis).total;
        if (t <= kCoarseSmemCap) {
            m.layout = layout;
            m.smem = t;
            return m;
        }
    }
    return m;
}

size_t coarse_gmres_scratch(const Coarse& c, int prec, int nrhs, int maxit, int want_layout) {
    const size_t nco = (size_t)c.gc.V * c.nc;
    const size_t es = prec == QCD_FP64 ? sizeof(double2) : sizeof(float2);
    const size_t npair = (size_t)(maxit + 2) * nrhs;
    size_t bytes = es * nco * nrhs * 2 + sizeof(double2) * (4 * npair + (size_t)nrhs * maxit * maxit + (size_t)nrhs * maxit) +
                   4096;
    if (coarse_mode(c, prec, nrhs, maxit, want_layout).layout == 3) {
        int sps, nblk;
        coarse_partition(c, sps, nblk);
        const size_t E = (size_t)sps * c.nc;
        bytes += es * nblk * E * nrhs * (size_t)(maxit + 2) + 1024;
    }
    return bytes;
}

// Right-hand sides per launch: the library's cap whenever some layout fits
// (the global-memory basis always does unless the bookkeeping alone is too big).
int coarse_gmres_group(const Coarse& c, int prec, int maxit, int want_layout) {
    for (int g = kMaxCoarseRhs; g >= 1; --g)
        if (coarse_mode(c, prec, g, maxit, want_layout).layout != 0) return g;
    return 0;
}

int coarse_gmres_layout(const Coarse& c, int prec, int nrhs, int maxit, int want_layout) {
    return coarse_mode(c, prec, nrhs, maxit, want_layout).layout;
}

template <typename Z, typename R>
static int launch_coarse(const Coarse& c, int op, int nrhs, const void* b, void* x, const double* tau_dev,
                         const int* act, double tol, int maxit, void* scratch, int* iters, double* resid,
                         unsigned long long* counter, int want_layout, cudaStream_t st) {
    const size_t nco = (size_t)c.gc.V * c.nc;
    int sps, nblk;
    coarse_partition(c, sps, nblk);
    const int E = sps * c.nc;
    const CoarseMode md = coarse_mode(c, std::is_same<R, double>::value ? QCD_FP64 : QCD_FP32, nrhs, maxit,
                                      want_layout);
    if (md.layout == 0) return -4;
    const size_t npair = (size_t)(maxit + 2) * nrhs;
    char* p = (char*)scratch;
    auto take = [&](size_t bytes) { char* q = p; p += (bytes + 255) & ~size_t(255); return (void*)q; };
    CoarseArgs<Z, R> a;
    a.gc = c.gc;
    a.nc = c.nc;
    a.A = std::is_same<R, double>::value ? (const Z*)c.A64 : (const Z*)c.A32;
    a.b = (const Z*)b;
    a.x = (Z*)x;
    a.Vg = (Z*)take(sizeof(Z) * nco * nrhs * 2);
    a.tot = (double2*)take(sizeof(double2) * 4 * npair);
    a.Rg = (double2*)take(sizeof(double2) * (size_t)nrhs * maxit * maxit);
    a.yv = (double2*)take(sizeof(double2) * (size_t)nrhs * maxit);
    a.Vglob = nullptr;
    a.wglob = nullptr;
    if (md.layout == 3) {
        a.Vglob = (Z*)take(sizeof(Z) * (size_t)nblk * (maxit + 1) * nrhs * E);
        a.wglob = (Z*)take(sizeof(Z) * (size_t)nblk * nrhs * E);
    }
    a.iters = iters;
    a.counter = counter;
    a.resid = resid;
    a.op = op;
    a.tau = tau_dev;
    a.act = act;
    a.tol = tol;
    a.maxit = maxit;
    a.nrhs = nrhs;
    a.E = E;
    a.sps = sps;
    a.a_smem = md.layout == 1 ? 1 : 0;
    cudaMemsetAsync(a.tot, 0, sizeof(double2) * 4 * npair, st);
    auto kern = coarse_gmres_kernel<Z, R>;
    const size_t sm = md.smem;
    if (sm + 1024 > 48 * 1024) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 256, sm);
    if (per_sm < 1) return -1;
    void* args[] = {&a};
    const double es = sizeof(Z);
    KTimer kt(std::is_same<R, double>::value ? "coarse_gmres_f64" : "coarse_gmres_f32",
              es * ((double)c.gc.V * 9 * c.nc * c.nc + 4.0 * nrhs * nco), 0.0, st);
    cudaError_t e = cudaLaunchCooperativeKernel((void*)kern, dim3(nblk), dim3(256), args, sm, st);
    return e == cudaSuccess ? 0 : -2;
}

int coarse_gmres(const Coarse& c, int prec, int op, int nrhs, const void* b, void* x, const double* tau_dev,
                 const int* act, double tol, int maxit, void* scratch, int* iters, double* resid,
                 unsigned long long* counter, int want_layout, cudaStream_t st) {
    if (nrhs < 1 || nrhs > kMaxCoarseRhs || maxit < 1 || maxit > kMaxCoarse) return -3;
    if (prec == QCD_FP64)
        return launch_coarse<double2, double>(c, op, nrhs, b, x, tau_dev, act, tol, maxit, scratch, iters, resid,
                                              counter, want_layout, st);
    return launch_coarse<float2, float>(c, op, nrhs, b, x, tau_dev, act, tol, maxit, scratch, iters, resid, counter,
                                        want_layout, st);
}

}  // namespace qcd
