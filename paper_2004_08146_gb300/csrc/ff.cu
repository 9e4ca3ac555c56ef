// Double-float ("ff") vector kernels for the Davidson basis (Sec. 3,
// Algorithm 2: Gram-Schmidt against [V X], the basis combinations u = V s,
// W s, the thick-restart transform and the lock-time deflation).
//
// A complex number is stored as two FP32 pairs, hi + lo (16 bytes, the size
// of a complex128), good to about 2^-48 relative.  Products and sums use the
// error-free transformations of Dekker and Knuth on the FP32 units:
//   two_prod(a, b) = (a*b, fma(a, b, -a*b))        exact product,
//   two_sum(a, b)  = (a+b, rounding error of a+b)   exact sum (6 flops).
// On this part FP32 FMA throughput is about 60x the FP64 rate, so these
// operations run at HBM speed where the FP64 forms were bound by the FP64
// pipe.  Results of inner products are returned in FP64.
#include <algorithm>

#include "ffsum.cuh"
#include "internal.h"

namespace qcd {

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ ffr two_prod(float a, float b) {
    const float p = a * b;
    return {p, fmaf(a, b, -p)};
}
__device__ __forceinline__ ffr split(double d) {
    const float h = (float)d;
    return {h, (float)(d - (double)h)};
}
__device__ __forceinline__ double join(ffr a) { return (double)a.h + (double)a.l; }

// accumulator: acc += a * b with a = (ah, al), b = (bh, bl): the exact
// product of the high parts and the exact sum into the running high part,
// the rounding errors and cross terms into the low part, renormalised every
// step so that the low part stays below half an ulp of the high part
// (sums of a few thousand terms stay at ~1e-16 relative).
struct acc_t {
    float h = 0.f, l = 0.f;
    __device__ __forceinline__ void mac(float ah, float al, float bh, float bl) {
        const ffr p = two_prod(ah, bh);
        const ffr s = two_sum(h, p.h);
        const ffr r = fast_two_sum(s.h, l + (s.l + p.l + fmaf(ah, bl, al * bh)));
        h = r.h;
        l = r.l;
    }
    __device__ __forceinline__ void msub(float ah, float al, float bh, float bl) { mac(-ah, -al, bh, bl); }
    __device__ __forceinline__ ffr get() const { return fast_two_sum(h, l); }
};

// ---- element access: float4 = (re.h, im.h, re.l, im.l)
__device__ __forceinline__ float4 pack(ffr re, ffr im) { return make_float4(re.h, im.h, re.l, im.l); }

__global__ void ff_from_fp64_kernel(const double2* __restrict__ x, float4* __restrict__ y, size_t n) {
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x) {
        const double2 v = x[t];
        y[t] = pack(split(v.x), split(v.y));
    }
}
__global__ void ff_to_fp64_kernel(const float4* __restrict__ x, double2* __restrict__ y, size_t n) {
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x) {
        const float4 v = x[t];
        y[t] = make_double2((double)v.x + (double)v.z, (double)v.y + (double)v.w);
    }
}
__global__ void ff_to_fp32_kernel(const float4* __restrict__ x, float2* __restrict__ y, size_t n) {
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x) {
        const float4 v = x[t];
        y[t] = make_float2(v.x + v.z, v.y + v.w);
    }
}
__global__ void ff_from_fp32_kernel(const float2* __restrict__ x, float4* __restrict__ y, size_t n) {
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x) {
        const float2 v = x[t];
        y[t] = make_float4(v.x, v.y, 0.f, 0.f);
    }
}

// (re, im) accumulators of conj(a) b and of c a
struct acc2_t {
    acc_t re, im;
    __device__ __forceinline__ void dot(const float4& a, const float4& b) {
        re.mac(a.x, a.z, b.x, b.z);
        im.mac(a.x, a.z, b.y, b.w);
        re.mac(a.y, a.w, b.y, b.w);
        im.msub(a.y, a.w, b.x, b.z);
    }
    __device__ __forceinline__ void axpy(const float4& c, const float4& a) {
        re.mac(c.x, c.z, a.x, a.z);
        re.msub(c.y, c.w, a.y, a.w);
        im.mac(c.x, c.z, a.y, a.w);
        im.mac(c.y, c.w, a.x, a.z);
    }
};

// sums over the lanes of a warp, the same in all of them
__device__ __forceinline__ void add_lane(sum3_t& t, int o) {
    t.add(sum3_t(__shfl_xor_sync(0xffffffffu, t.a, o), __shfl_xor_sync(0xffffffffu, t.b, o),
                 __shfl_xor_sync(0xffffffffu, t.c, o)));
}
__device__ __forceinline__ sum3_t ff_warp_sum(sum3_t t) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) add_lane(t, o);
    return t;
}
// both sums of a complex number, (re, im) in lanes 0 and 16: the halves of the warp
// share them first
__device__ __forceinline__ sum3_t ff_warp_sum2(ffr re, ffr im, int lane) {
    const bool up = lane & 16;
    const ffr k = up ? im : re, s = up ? re : im;
    sum3_t t(k.h, k.l);
    t.add(__shfl_xor_sync(0xffffffffu, s.h, 16), __shfl_xor_sync(0xffffffffu, s.l, 16));
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) add_lane(t, o);
    return t;
}
// a partial sum in memory: 16 bytes
__device__ __forceinline__ float4 pack3(const sum3_t& t) { return make_float4(t.a, t.b, t.c, 0.f); }
__device__ __forceinline__ sum3_t unpack3(const float4& v) { return sum3_t(v.x, v.y, v.z); }

// Dot products of up to two vectors y with the na vectors of set A and the nb of
// set B (Gram-Schmidt against [V X]; the Gram columns W^H W_m, W^H V_m).  A warp
// owns Q vectors over a part of the entries, so every y entry it reads serves Q
// products and 2 Q + 2 loads are in flight; the eight warps of a CTA take
// neighbouring parts for the same vectors and leave one partial, and the CTA that
// finishes a set of vectors last adds them, one sum per warp.  Products
// are 16 FP32 operations each, so warps in flight count: four CTAs per SM with Q = 4
// (Q = 2 for two vectors y), one wave.  16 x 8^3, about 40 vectors: 31 us with idle
// warps in the last set and three CTAs, 21 us now (two y: 40 with Q = 4 and two CTAs,
// 30 now).
struct GramOut {
    double2 *G, *H;   // null: dots only
    int ld, m;
};
template <int Q, int NY>
__global__ void __launch_bounds__(256, 4) ff_dots_kernel(const float4* __restrict__ A, int na, const float4* __restrict__ B,
                                                      int nb, size_t n, const float4* __restrict__ y0,
                                                      const float4* __restrict__ y1,
                                                      float4* __restrict__ partial, unsigned* __restrict__ counters,
                                                      double2* __restrict__ d0, double2* __restrict__ d1, GramOut go) {
    __shared__ float4 red[8][2 * NY * Q];   // re and im of each sum
    __shared__ bool last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nv = na + nb, v0 = blockIdx.y * Q;
    const int part = blockIdx.x * 8 + warp, parts = gridDim.x * 8;
    const size_t lo = n * part / parts, hi = n * (part + 1) / parts;
    const float4* x[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int v = min(v0 + q, nv - 1);   // past the last: read like the last, not kept
        x[q] = v < na ? A + (size_t)v * n : B + (size_t)(v - na) * n;
    }
    acc2_t acc[NY][Q];
    size_t e = lo + lane;
    for (; e + 32 < hi; e += 64) {
        float4 a[Q], b[Q], y[2][NY];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            a[q] = __ldg(x[q] + e);
            b[q] = __ldg(x[q] + e + 32);
        }
        y[0][0] = __ldg(y0 + e);
        y[1][0] = __ldg(y0 + e + 32);
        if constexpr (NY == 2) {
            y[0][1] = __ldg(y1 + e);
            y[1][1] = __ldg(y1 + e + 32);
        }
#pragma unroll
        for (int k = 0; k < NY; ++k)
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                acc[k][q].dot(a[q], y[0][k]);
                acc[k][q].dot(b[q], y[1][k]);
            }
    }
    if (e < hi) {
        float4 y[NY];
        y[0] = __ldg(y0 + e);
        if constexpr (NY == 2) y[1] = __ldg(y1 + e);
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const float4 a = __ldg(x[q] + e);
#pragma unroll
            for (int k = 0; k < NY; ++k) {
                acc[k][q].dot(a, y[k]);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < NY; ++k)
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const sum3_t r = ff_warp_sum2(acc[k][q].re.get(), acc[k][q].im.get(), lane);
            if ((lane & 15) == 0) red[warp][2 * (k * Q + q) + (lane >> 4)] = pack3(r);
        }
    __syncthreads();
    if (warp == 0) {
        if (lane < 2 * NY * Q) {
            sum3_t t;
#pragma unroll
            for (int w = 0; w < 8; ++w) t.add(unpack3(red[w][lane]));
            partial[((size_t)blockIdx.y * 2 * NY * Q + lane) * gridDim.x + blockIdx.x] = pack3(t);
            __threadfence();
        }
        __syncwarp();
        if (lane == 0) last = atomicAdd(&counters[blockIdx.y], 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int k = warp / Q, v = v0 + warp % Q;
    if (warp < NY * Q && v < nv) {
        sum3_t re, im;
        for (unsigned t = lane; t < gridDim.x; t += 32) {
            const float4* p = partial + ((size_t)blockIdx.y * 2 * NY * Q + 2 * warp) * gridDim.x + t;
            re.add(unpack3(__ldcg(p)));
            im.add(unpack3(__ldcg(p + gridDim.x)));
        }
        const double2 d = make_double2(ff_warp_sum(re).value(), ff_warp_sum(im).value());
        if (lane == 0) {
            (k == 0 ? d0 : d1)[v] = d;
            // new column and row of G = W^H W and H = W^H V (Hermitian)
            if (NY == 2 && go.G != nullptr) {
                double2* M = k == 0 ? go.G : go.H;
                M[(size_t)go.m * go.ld + v] = d;
                M[(size_t)v * go.ld + go.m] = conj(d);
            }
        }
    }
    if (threadIdx.x == 0) counters[blockIdx.y] = 0u;
}

constexpr int kFFCoef = 512;   // coefficients staged at a time, a multiple of 8

// acc += sign * sum_i c_i X_i[k]; eight loads in flight; a zero coefficient leaves
// its vector unread (unused basis slots may hold anything).  All threads of the CTA
// take part, in = false without an entry.
__device__ __forceinline__ void ff_accumulate(acc2_t& acc, const float4* __restrict__ X, int nv, size_t n,
                                              const double2* __restrict__ c, double sign, size_t k, bool in,
                                              float4* cs) {
    for (int i0 = 0; i0 < nv; i0 += kFFCoef) {
        const int cnt = min(kFFCoef, nv - i0), pad = (cnt + 7) & ~7;
        __syncthreads();
        for (int e = threadIdx.x; e < pad; e += blockDim.x) {
            const double2 v = e < cnt ? c[i0 + e] : make_double2(0.0, 0.0);
            cs[e] = pack(split(sign * v.x), split(sign * v.y));
        }
        __syncthreads();
        if (!in) continue;
        const float4* x = X + (size_t)i0 * n + k;
        for (int i = 0; i < cnt; i += 8) {
            float4 a[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                a[q] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (cs[i + q].x != 0.f || cs[i + q].y != 0.f) a[q] = __ldg(x + (size_t)(i + q) * n);
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) acc.axpy(cs[i + q], a[q]);
        }
    }
}

// w -= sum_i ca_i A_i + sum_i cb_i B_i.  One thread per entry: the vectors are read
// once and w once, where a chain of updates would pass over w for each.  Six CTAs
// per SM keep 24 warps of eight loads in flight; four quarter sums per entry (32
// warps) gained nothing: 27.6 against 25.0 us.  16 x 8^3, about 50 vectors: 34 -> 25 us.
__global__ void __launch_bounds__(128, 6) ff_project_kernel(const float4* __restrict__ A, int na,
                                                            const double2* __restrict__ ca,
                                                            const float4* __restrict__ B, int nb,
                                                            const double2* __restrict__ cb, float4* __restrict__ w,
                                                            size_t n) {
    __shared__ float4 cs[kFFCoef];
    const size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    const bool in = k < n;
    acc2_t acc;
    if (in) {
        const float4 w0 = w[k];
        acc.re.h = w0.x; acc.re.l = w0.z;
        acc.im.h = w0.y; acc.im.l = w0.w;
    }
    ff_accumulate(acc, A, na, n, ca, -1.0, k, in, cs);
    ff_accumulate(acc, B, nb, n, cb, -1.0, k, in, cs);
    if (in) w[k] = pack(acc.re.get(), acc.im.get());
}

// Sums of NV double-float values over all threads of the grid, NV <= 2: one
// partial per CTA, the last CTA adds them; FP64 results in out[v].x.
template <int NV>
__device__ __forceinline__ void ff_grid_sum(ffr (&v)[NV], float4* partial, unsigned* counter, double2* out) {
    __shared__ float4 red[NV][32];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        const sum3_t r = ff_warp_sum(sum3_t(v[q].h, v[q].l));
        if (lane == 0) red[q][warp] = pack3(r);
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const sum3_t s = ff_warp_sum(lane < nw ? unpack3(red[q][lane]) : sum3_t());
            if (lane == 0) partial[(size_t)q * gridDim.x + blockIdx.x] = pack3(s);
        }
    }
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        if (warp != q) continue;   // NV <= warps of the CTA
        sum3_t a;
        for (unsigned t = lane; t < gridDim.x; t += 32) a.add(unpack3(__ldcg(&partial[(size_t)q * gridDim.x + t])));
        const double s = ff_warp_sum(a).value();
        if (lane == 0) out[q] = make_double2(s, 0.0);
    }
    if (threadIdx.x == 0) *counter = 0u;
}

// u = V s, Qu = W s (m vectors each) and d = (u^H u, Re u^H Qu) in one pass; bound
// by the reads of V and W at 24 warps per SM (see above).  16 x 8^3: 56 -> 42 us.
__global__ void __launch_bounds__(128, 6) ff_ritz_kernel(const float4* __restrict__ V, const float4* __restrict__ W,
                                                         int m, size_t n, const double2* __restrict__ s,
                                                         float4* __restrict__ u, float4* __restrict__ Qu,
                                                         float4* __restrict__ partial, unsigned* __restrict__ counter,
                                                         double2* __restrict__ d) {
    __shared__ float4 cs[kFFCoef];
    acc_t uu, uq;
    const size_t step = (size_t)gridDim.x * blockDim.x;
    for (size_t k0 = blockIdx.x * (size_t)blockDim.x; k0 < n; k0 += step) {
        const size_t k = k0 + threadIdx.x;
        const bool in = k < n;
        acc2_t a, b;
        ff_accumulate(a, V, m, n, s, 1.0, k, in, cs);
        ff_accumulate(b, W, m, n, s, 1.0, k, in, cs);
        if (!in) continue;
        const float4 x = pack(a.re.get(), a.im.get()), y = pack(b.re.get(), b.im.get());
        u[k] = x;
        Qu[k] = y;
        uu.mac(x.x, x.z, x.x, x.z);
        uu.mac(x.y, x.w, x.y, x.w);
        uq.mac(x.x, x.z, y.x, y.z);
        uq.mac(x.y, x.w, y.y, y.w);
    }
    ffr v[2] = {uu.get(), uq.get()};
    ff_grid_sum<2>(v, partial, counter, d);
}

// With d = (u^H u, Re u^H Qu) of the kernel above: r = (Qu - rho u) / ||u|| in
// FP64 (rho the Rayleigh quotient), u <- u / ||u||, and rr = r^H r.
__global__ void __launch_bounds__(256) ff_residual_kernel(float4* __restrict__ u, const float4* __restrict__ Qu,
                                                          const double2* __restrict__ d, size_t n,
                                                          double2* __restrict__ r, float4* __restrict__ partial,
                                                          unsigned* __restrict__ counter, double2* __restrict__ rr) {
    __shared__ float4 cf;   // iu and -rho iu
    if (threadIdx.x == 0) {
        const double uu = d[0].x, rho = d[1].x / uu, iu = 1.0 / sqrt(uu);
        cf = pack(split(iu), split(-rho * iu));
    }
    __syncthreads();
    const float4 c = cf;
    acc_t sum;
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x) {
        const float4 x = u[k], y = Qu[k];
        acc_t re, im, ur, ui;
        re.mac(c.y, c.w, x.x, x.z);
        re.mac(c.x, c.z, y.x, y.z);
        im.mac(c.y, c.w, x.y, x.w);
        im.mac(c.x, c.z, y.y, y.w);
        const ffr a = re.get(), b = im.get();
        r[k] = make_double2(join(a), join(b));
        sum.mac(a.h, a.l, a.h, a.l);
        sum.mac(b.h, b.l, b.h, b.l);
        ur.mac(c.x, c.z, x.x, x.z);
        ui.mac(c.x, c.z, x.y, x.w);
        u[k] = pack(ur.get(), ui.get());
    }
    ffr v[1] = {sum.get()};
    ff_grid_sum<1>(v, partial, counter, rr);
}

// v <- a v (double-float) and y = v in FP64
__global__ void ff_scale_out_kernel(float4* __restrict__ v, double a, double2* __restrict__ y, size_t n) {
    const ffr s = split(a);
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x) {
        const float4 x = v[t];
        acc_t re, im;
        re.mac(s.h, s.l, x.x, x.z);
        im.mac(s.h, s.l, x.y, x.w);
        const ffr a0 = re.get(), b0 = im.get();
        v[t] = pack(a0, b0);
        y[t] = make_double2(join(a0), join(b0));
    }
}

// In-place tall-skinny transform A[j] <- sum_i C[i + j m] A[i], j < p <= m
// (thick restart): each CTA stages kTile rows of all m vectors in shared
// memory and overwrites them with the p new rows; a warp computes one output
// vector for the tile's rows (one row per lane), so each coefficient is a
// warp-wide broadcast.  Coefficients pre-split to double-float in Cf.
constexpr int kTile = 32;
__global__ void __launch_bounds__(256) ff_transform_kernel(float4* __restrict__ A, int m, const float4* __restrict__ Cf,
                                                           int p, size_t n) {
    extern __shared__ float4 tile[];   // [m][kTile]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const size_t ntiles = (n + kTile - 1) / kTile;
    for (size_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const size_t k0 = t * kTile;
        const int rows = (int)min((size_t)kTile, n - k0);
        for (int e = threadIdx.x; e < m * kTile; e += blockDim.x) {
            const int i = e / kTile, r = e % kTile;
            tile[e] = r < rows ? A[(size_t)i * n + k0 + r] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        __syncthreads();
        for (int j = warp; j < p; j += nw) {
            acc_t re, im;
            for (int i = 0; i < m; ++i) {
                const float4 c = __ldg(&Cf[(size_t)j * m + i]);
                const float4 a = tile[i * kTile + lane];
                re.mac(c.x, c.z, a.x, a.z);
                re.msub(c.y, c.w, a.y, a.w);
                im.mac(c.x, c.z, a.y, a.w);
                im.mac(c.y, c.w, a.x, a.z);
            }
            if (lane < rows) A[(size_t)j * n + k0 + lane] = pack(re.get(), im.get());
        }
        __syncthreads();
    }
}

__global__ void ff_split_kernel(const double2* __restrict__ c, float4* __restrict__ cf, int cnt, double scale) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < cnt; e += gridDim.x * blockDim.x) {
        const double2 v = c[e];
        cf[e] = pack(split(scale * v.x), split(scale * v.y));
    }
}

// Lock-time deflation A[j-1] <- A[j] - conj(w_j) f (sum_i w_i A[i]), j = 1..m-1,
// for the pair (V, W) selected by blockIdx.y; w (m entries) and f = w[m].x
// pre-split in wf.  Row k of the result depends on row k of A only, so each
// thread finishes its rows in place.
__global__ void ff_deflate_kernel(float4* __restrict__ A0, float4* __restrict__ A1, int m, size_t n,
                                  const float4* __restrict__ wf) {
    __shared__ float4 w[kMaxBasis + 1];
    for (int i = threadIdx.x; i <= m; i += blockDim.x) w[i] = wf[i];
    __syncthreads();
    float4* A = blockIdx.y ? A1 : A0;
    const float4 f = w[m];
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x) {
        acc_t yr, yi;
        for (int i = 0; i < m; ++i) {
            const float4 c = w[i], a = A[(size_t)i * n + k];
            yr.mac(c.x, c.z, a.x, a.z);
            yr.msub(c.y, c.w, a.y, a.w);
            yi.mac(c.x, c.z, a.y, a.w);
            yi.mac(c.y, c.w, a.x, a.z);
        }
        // y <- f y (f real)
        const ffr y0r = yr.get(), y0i = yi.get();
        acc_t fr, fi;
        fr.mac(f.x, f.z, y0r.h, y0r.l);
        fi.mac(f.x, f.z, y0i.h, y0i.l);
        const ffr yR = fr.get(), yI = fi.get();
        for (int j = 1; j < m; ++j) {
            const float4 c = w[j], a = A[(size_t)j * n + k];
            // a - conj(c) y: re = ar - (cr yr + ci yi), im = ai - (cr yi - ci yr)
            acc_t re, im;
            re.h = a.x; re.l = a.z;
            im.h = a.y; im.l = a.w;
            re.msub(c.x, c.z, yR.h, yR.l);
            re.msub(c.y, c.w, yI.h, yI.l);
            im.msub(c.x, c.z, yI.h, yI.l);
            im.mac(c.y, c.w, yR.h, yR.l);
            A[(size_t)(j - 1) * n + k] = pack(re.get(), im.get());
        }
    }
}

inline int grid_for(size_t n, int th = kThreads) {
    size_t g = (n + th - 1) / th;
    return (int)(g > 1048576 ? 1048576 : (g == 0 ? 1 : g));
}
int sm_count() {
    static int sms = 0;
    if (sms == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 1;
    }
    return sms;
}

}  // namespace

void ff_convert(int prec_in, const void* x, int prec_out, void* y, size_t n, cudaStream_t st) {
    KTimer kt("ff_convert", (double)n * 24, 0.0, st);
    if (prec_in == QCD_FP64 && prec_out == QCD_FF)
        ff_from_fp64_kernel<<<grid_for(n), kThreads, 0, st>>>((const double2*)x, (float4*)y, n);
    else if (prec_in == QCD_FF && prec_out == QCD_FP64)
        ff_to_fp64_kernel<<<grid_for(n), kThreads, 0, st>>>((const float4*)x, (double2*)y, n);
    else if (prec_in == QCD_FF && prec_out == QCD_FP32)
        ff_to_fp32_kernel<<<grid_for(n), kThreads, 0, st>>>((const float4*)x, (float2*)y, n);
    else
        ff_from_fp32_kernel<<<grid_for(n), kThreads, 0, st>>>((const float2*)x, (float4*)y, n);
}

// A partial sum is 16 bytes.  launch_dots: at most 16 sums (8 complex) per set of
// vectors and CTA, one wave of CTAs or one CTA per set; ff_ritz: two per CTA.
constexpr int kRitzCtas = 4096;
size_t ff_part_bytes(int nvec) {
    return sizeof(float4) * (size_t)std::max(16 * std::max(4 * sm_count(), nvec), 2 * kRitzCtas);
}

// CTAs: one wave over all sets of vectors, at least 64 entries per warp
template <int Q, int NY>
static void launch_dots(const void* A, int na, const void* B, int nb, size_t n, const void* y0, const void* y1,
                        double2* d0, double2* d1, void* partial, unsigned* counters, GramOut go, cudaStream_t st) {
    static_assert(Q * NY <= 8, "one warp per sum");
    const int sets = (na + nb + Q - 1) / Q;
    size_t gx = std::max(1, 4 * sm_count() / sets);
    gx = std::min(gx, std::max<size_t>(1, n / 512));
    ff_dots_kernel<Q, NY><<<dim3((unsigned)gx, sets), 256, 0, st>>>(
        (const float4*)A, na, (const float4*)B, nb, n, (const float4*)y0, (const float4*)y1, (float4*)partial,
        counters, d0, d1, go);
}

void ff_dots(const void* A, int na, const void* B, int nb, size_t n, const void* y, double2* dots, void* partial,
             unsigned* counters, cudaStream_t st) {
    const int nv = na + nb;
    if (nv <= 0) return;
    KTimer kt("dots_ff", (double)(nv + 1) * n * 16, 8.0 * nv * n, st);
    const GramOut go{};
    if (nv <= 8) launch_dots<1, 1>(A, na, B, nb, n, y, nullptr, dots, nullptr, partial, counters, go, st);
    else if (nv <= 16) launch_dots<2, 1>(A, na, B, nb, n, y, nullptr, dots, nullptr, partial, counters, go, st);
    else launch_dots<4, 1>(A, na, B, nb, n, y, nullptr, dots, nullptr, partial, counters, go, st);
}

void ff_gram_column(const void* W, int m, size_t n, const void* w, const void* v, double2* dots, double2* G, double2* H,
                    int ld, void* partial, unsigned* counters, cudaStream_t st) {
    KTimer kt("gram_column_ff", (double)(m + 3) * n * 16, 16.0 * (m + 1) * n, st);
    const GramOut go{G, H, ld, m};
    if (m < 8) launch_dots<1, 2>(W, m + 1, nullptr, 0, n, w, v, dots, dots + m + 1, partial, counters, go, st);
    else launch_dots<2, 2>(W, m + 1, nullptr, 0, n, w, v, dots, dots + m + 1, partial, counters, go, st);
}

void ff_project(const void* A, int na, const double2* ca, const void* B, int nb, const double2* cb, void* w, size_t n,
                cudaStream_t st) {
    if (na + nb <= 0) return;
    KTimer kt("project_ff", (double)(na + nb + 2) * n * 16, 8.0 * (na + nb) * n, st);
    ff_project_kernel<<<(unsigned)((n + 127) / 128), 128, 0, st>>>((const float4*)A, na, ca, (const float4*)B, nb, cb,
                                                                   (float4*)w, n);
}

void ff_ritz(const void* V, const void* W, int m, size_t n, const double2* s, void* u, void* Qu, double2* r, double2* d,
             void* partial, unsigned* counters, cudaStream_t st) {
    {
        KTimer kt("ritz_ff", (double)(2 * m + 2) * n * 16, 16.0 * m * n, st);
        const unsigned grid = (unsigned)std::min<size_t>((n + 127) / 128, kRitzCtas);
        ff_ritz_kernel<<<grid, 128, 0, st>>>((const float4*)V, (const float4*)W, m, n, s, (float4*)u, (float4*)Qu,
                                             (float4*)partial, counters, d);
    }
    KTimer kt("residual_ff", (double)n * 64, 0.0, st);
    const unsigned grid = (unsigned)std::min<size_t>((n + 255) / 256, (size_t)sm_count() * 4);
    ff_residual_kernel<<<grid, 256, 0, st>>>((float4*)u, (const float4*)Qu, d, n, r, (float4*)partial, counters, d + 2);
}

void ff_scale_out(void* v, double a, double2* y, size_t n, cudaStream_t st) {
    KTimer kt("ff_scale_out", (double)n * 48, 0.0, st);
    ff_scale_out_kernel<<<grid_for(n), kThreads, 0, st>>>((float4*)v, a, y, n);
}

void ff_transform_inplace(void* A, int m, const double2* C, int p, size_t n, void* cf_scratch, cudaStream_t st) {
    float4* Cf = (float4*)cf_scratch;
    ff_split_kernel<<<(m * p + 255) / 256, 256, 0, st>>>(C, Cf, m * p, 1.0);
    const size_t sm = (size_t)m * kTile * sizeof(float4);
    if (sm + 1024 > 48 * 1024)
        cudaFuncSetAttribute(ff_transform_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    const size_t ntiles = (n + kTile - 1) / kTile;
    const int grid = (int)std::min<size_t>(ntiles, (size_t)sm_count() * 4);
    KTimer kt("basis_transform_ff", (double)(m + p) * n * 16, 8.0 * m * p * n, st);
    ff_transform_kernel<<<grid, 256, sm, st>>>((float4*)A, m, Cf, p, n);
}

void ff_deflate(void* A0, void* A1, int m, size_t n, const double2* hw, void* wf_scratch, cudaStream_t st) {
    float4* wf = (float4*)wf_scratch;
    ff_split_kernel<<<1, 128, 0, st>>>(hw, wf, m + 1, 1.0);
    const int gx = (int)std::min<size_t>((n + 255) / 256, (size_t)sm_count() * 8);
    KTimer kt("householder_deflate_ff", (double)(4 * m - 2) * n * 16, 16.0 * m * n * 2, st);
    ff_deflate_kernel<<<dim3(gx, 2), 256, 0, st>>>((float4*)A0, (float4*)A1, m, n, wf);
}

}  // namespace qcd
