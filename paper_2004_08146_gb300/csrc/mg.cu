// Multigrid kernels: chirality-split aggregation P (Sec. 2, above Eq. 2.9),
// restriction P^H and prolongation P (Eq. 2.8), the Galerkin coarse stencil
// D_c = P^H D P (Eq. 2.8, 2.9) and the SAP block solves of Eq. 2.10.
#include <algorithm>

#include <cuda_fp16.h>

#include "internal.h"
#include "dirac.cuh"

namespace qcd {

namespace {

// Work counters of the SAP block solves (for the FP32-ALU roofline): [0] sums
// block sites x GMRES steps, [1] block sites x k (k + 1) / 2 over all block
// solves; 64 slots per counter spread the atomics of one launch.
__device__ unsigned long long g_sap_work[2][64];

__device__ __forceinline__ void count_sap_work(int bs, int kdim) {
    const int slot = (blockIdx.x + 7 * blockIdx.y) & 63;
    atomicAdd(&g_sap_work[0][slot], (unsigned long long)bs * kdim);
    atomicAdd(&g_sap_work[1][slot], (unsigned long long)bs * kdim * (kdim + 1) / 2);
}

// sum of a double2 over the first blockDim.x (power of two) threads
__device__ __forceinline__ double2 block_sum2(double2 v, double2* red) {
    const int t = threadIdx.x;
    red[t] = v;
    __syncthreads();
    for (int s = blockDim.x >> 1; s > 0; s >>= 1) {
        if (t < s) red[t] += red[t + s];
        __syncthreads();
    }
    double2 r = red[0];
    __syncthreads();
    return r;
}

__device__ __forceinline__ void block_coords(const Blocking& B, int blk, int c[4]) {
    int t = blk;
    c[3] = t % B.cd[3]; t /= B.cd[3];
    c[2] = t % B.cd[2]; t /= B.cd[2];
    c[1] = t % B.cd[1]; c[0] = t / B.cd[1];
}
__device__ __forceinline__ void local_coords(const Blocking& B, int l, int o[4]) {
    int t = l;
    o[3] = t % B.b[3]; t /= B.b[3];
    o[2] = t % B.b[2]; t /= B.b[2];
    o[1] = t % B.b[1]; o[0] = t / B.b[1];
}
__device__ __forceinline__ int coarse_index(const Blocking& B, const int c[4]) {
    return ((c[0] * B.cd[1] + c[1]) * B.cd[2] + c[2]) * B.cd[3] + c[3];
}
__device__ __forceinline__ int local_index(const Blocking& B, const int o[4]) {
    return ((o[0] * B.b[1] + o[1]) * B.b[2] + o[2]) * B.b[3] + o[3];
}

// ------------------------------------------------------------------ P build
// One CTA per (coarse site, chirality): gather the nvec restricted test vectors,
// then modified Gram-Schmidt applied twice (FP64), in the order that takes a
// finished vector out of all later ones: a warp projects one later vector at a time,
// the warp of the next vector normalises it, and one barrier per vector is left.
// Vectors in shared memory where they fit.  Bound by the FP64 pipe (a third of it
// sums over lanes).  16 x 8^3, 2^4 aggregates, 8 vectors: 822 us with one inner
// product per block-wide reduction, 201 now.
__global__ void __launch_bounds__(256) build_P_kernel(Geom g, Blocking B, int nv, const double2* __restrict__ vecs,
                                                      double2* P64, float2* __restrict__ P32, int in_smem) {
    extern __shared__ double2 pvs[];
    const int blk = blockIdx.x, chi = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nloc = B.bs * 6;
    double2* Pb = P64 + ((size_t)blk * 2 + chi) * nv * nloc;
    double2* v = in_smem ? pvs : Pb;
    for (int d = threadIdx.x; d < nloc; d += blockDim.x) {
        const int l = d / 6, sc = d % 6;
        const double2* src = vecs + (size_t)block_fine_site(g, B, blk, l) * 12 + 6 * chi + sc;
        for (int i = 0; i < nv; ++i) v[(size_t)i * nloc + d] = src[(size_t)i * g.V * 12];
    }
    __syncthreads();
    auto normalise = [&](double2* p) {   // one warp
        double nn = 0.0;
        for (int d = lane; d < nloc; d += 32) nn += p[d].x * p[d].x + p[d].y * p[d].y;
        nn = warp_sum(nn);
        const double inv = nn > 0 ? 1.0 / sqrt(nn) : 0.0;
        for (int d = lane; d < nloc; d += 32) p[d] = inv * p[d];
    };
    for (int pass = 0; pass < 2; ++pass) {
        if (warp == 0) normalise(v);
        __syncthreads();
        for (int j = 0; j + 1 < nv; ++j) {
            const double2* pj = v + (size_t)j * nloc;
            for (int i = j + 1 + warp; i < nv; i += 8) {
                double2* pi = v + (size_t)i * nloc;
                // h: the products with Re p and with Im p in sums of their own, and the
                // update rounds the vector once (fused into it twice: P 2.4e-16 from
                // the exact one at 20 vectors against 1.8e-16)
                double2 h = make_double2(0, 0), hi = make_double2(0, 0);
                for (int d = lane; d < nloc; d += 32) {
                    const double2 p = pj[d], q = pi[d];
                    h.x = fma(p.x, q.x, h.x);
                    h.y = fma(p.x, q.y, h.y);
                    hi.x = fma(p.y, q.y, hi.x);
                    hi.y = fma(-p.y, q.x, hi.y);
                }
                h += hi;
                // the halves of the warp share the two sums
                const bool up = lane & 16;
                double k = up ? h.y : h.x;
                k += __shfl_xor_sync(0xffffffffu, up ? h.x : h.y, 16);
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
                h = make_double2(__shfl_sync(0xffffffffu, k, 0), __shfl_sync(0xffffffffu, k, 16));
                for (int d = lane; d < nloc; d += 32) pi[d] -= h * pj[d];
                if (i == j + 1) normalise(pi);
            }
            __syncthreads();
        }
    }
    float2* Pb32 = P32 + ((size_t)blk * 2 + chi) * nv * nloc;
    for (int d = threadIdx.x; d < nv * nloc; d += blockDim.x) {
        const double2 x = v[d];
        if (in_smem) Pb[d] = x;
        Pb32[d] = cvt<float2>(x);
    }
}

// ------------------------------------------------------------------ restrict / prolong
// E consecutive complex numbers loaded at once: two complex64 (16-byte aligned
// fields), one complex64 (fields aligned to 8 bytes only) or one complex128
template <typename R, int E> struct Piece;
template <> struct Piece<float, 2> {
    float4 v;
    __device__ __forceinline__ float2 at(int k) const { return k ? make_float2(v.z, v.w) : make_float2(v.x, v.y); }
};
template <> struct Piece<float, 1> {
    float2 v;
    __device__ __forceinline__ float2 at(int) const { return v; }
};
template <> struct Piece<double, 1> {
    double2 v;
    __device__ __forceinline__ double2 at(int) const { return v; }
};
template <typename R, int E> __device__ __forceinline__ Piece<R, E> load_piece(const cplx<R>* p) {
    Piece<R, E> o;
    o.v = __ldg(reinterpret_cast<const decltype(o.v)*>(p));
    return o;
}

// copy of one piece to shared memory behind the loads of other stages; take =
// false writes zeros
template <typename R, int E> __device__ __forceinline__ void async_piece(Piece<R, E>* dst, const cplx<R>* src, bool take) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    constexpr int n = sizeof(Piece<R, E>);
    const int bytes = take ? n : 0;
    if constexpr (n == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// x_c = P^H r: per (aggregate, chirality) the product of the nv x nloc rows of P
// with the nloc x nrhs fine entries (nloc = 6 x aggregate sites).  A warp owns a
// 4 x TJ tile of results, its lanes run along nloc in pieces of E entries (P rows
// and the 48 bytes of a site's chirality half are contiguous), so 4 + TJ loads
// feed 4 TJ products per entry, and the lanes are summed once at the end.  The
// warps of a CTA cover all tiles of the aggregate and up to kTransferRhs
// right-hand sides: P and r come from memory once, kStage pieces of every row per
// stage, through a ring of kRing stages of asynchronous copies (loading into
// registers kept one stage, 18 KB per SM, in flight and ran at 1.6 TB/s).
// 32 x 16^3, 4^4 aggregates, nv 20, 16 right-hand sides: 786 us with
// one chunk of 8 per pass and one warp per vector -> 154 us (3.0 TB/s; prologue of a
// single resident CTA per SM not hidden); 143 us with one chain of fused
// multiply-adds per sum.
// FP64 is bound by its pipe (2 operations per clock and SM, a quarter of them for each
// quarter of the warps): smaller tiles without rows of padding, at least four warps
// where there is work for them, and the terms with Re P and with Im P in sums of their
// own, which costs registers instead of operations.
template <typename R> constexpr int kTransferRhs = sizeof(R) == 4 ? 16 : 4;
template <typename R, int TI, int TJ> constexpr int kRestrictThreads =
    sizeof(R) == 4 ? (TJ == 4 ? 640 : 512) : (TI * TJ <= 2 ? 1024 : (TI * TJ == 4 ? 768 : 512));
constexpr int kRing = 4, kStage = 64;   // a stage: two pieces of a row per lane
constexpr int kSiteTable = 1024;   // aggregates up to this size look their entries up
template <typename R, int E, int TI, int TJ>
__global__ void __launch_bounds__(kRestrictThreads<R, TI, TJ>) restrict_tile_kernel(
    Geom g, Blocking B, int nv, const cplx<R>* __restrict__ P, const cplx<R>* __restrict__ r, cplx<R>* __restrict__ xc,
    int nrhs, int chunk, int ring, const int* __restrict__ act) {
    constexpr bool kTwo = sizeof(R) == 8;
    using Pc = Piece<R, E>;
    extern __shared__ __align__(16) unsigned char rsm[];
    const int nc = 2 * nv, nloc = B.bs * 6, np = nloc / E;
    const bool table = B.bs <= kSiteTable;
    const int blk = blockIdx.x >> 1, chi = blockIdx.x & 1;
    const int jc = blockIdx.y * chunk, nr = min(nrhs - jc, chunk), rows = nv + nr;
    Pc* stage = reinterpret_cast<Pc*>(rsm);                                       // [ring][rows][kStage]
    int* entry = reinterpret_cast<int*>(stage + (size_t)ring * rows * kStage);    // fine entry of a piece
    auto entry_of = [&](int e) { return block_fine_site(g, B, blk, e * E / 6) * 12 + e * E % 6 + 6 * chi; };
    if (table) {
        for (int e = threadIdx.x; e < np; e += blockDim.x) entry[e] = entry_of(e);
        __syncthreads();
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const size_t fstride = (size_t)g.V * 12;
    const cplx<R>* Pb = P + ((size_t)blk * 2 + chi) * nv * nloc;
    const cplx<R>* rb = r + (size_t)jc * fstride;
    const int nst = (np + kStage - 1) / kStage, slots = rows * kStage;
    auto fill = [&](int st, int at) {   // one commit group per stage, empty past the last
        if (st < nst) {
#pragma unroll
            for (int h = 0; h < kStage; h += 32) {
                const int e = st * kStage + h + lane;
                const bool in = e < np;
                const int ee = in ? e : 0;
                Pc* dst = stage + at + h + lane;
                const cplx<R>* ps = Pb + ee * E;
                const cplx<R>* rs = rb + (table ? entry[ee] : entry_of(ee));
                int q = warp;
                for (; q < nv; q += nw) async_piece<R, E>(dst + q * kStage, ps + (size_t)q * nloc, in);
                for (; q < rows; q += nw) async_piece<R, E>(dst + q * kStage, rs + (size_t)(q - nv) * fstride, in);
            }
        }
        async_commit();
    };
#pragma unroll
    for (int st = 0; st < kRing - 1; ++st) fill(st, st * slots);
    const int nit = (nv + TI - 1) / TI;
    const int i0 = (warp % nit) * TI, j0 = (warp / nit) * TJ;
    const bool idle = j0 >= nr;   // the last chunk may need fewer warps
    R acc[TI * TJ * 2], acc2[kTwo ? TI * TJ * 2 : 1];
#pragma unroll
    for (int q = 0; q < TI * TJ * 2; ++q) {
        acc[q] = R(0);
        if constexpr (kTwo) acc2[q] = R(0);
    }
    // rows past the last are read like the last and not written
    int ra[TI], ru[TJ];
#pragma unroll
    for (int q = 0; q < TI; ++q) ra[q] = min(i0 + q, nv - 1) * kStage + lane;
#pragma unroll
    for (int u = 0; u < TJ; ++u) ru[u] = (nv + min(j0 + u, nr - 1)) * kStage + lane;
    int cur = 0, next = (kRing - 1) * slots;
    for (int st = 0; st < nst; ++st) {
        async_wait<kRing - 2>();
        __syncthreads();   // stage st has arrived for all, stage st - 1 is read
        fill(st + kRing - 1, next);
        next = cur;
        const Pc* sp = stage + cur;
        cur = cur + slots == kRing * slots ? 0 : cur + slots;
        if (idle) continue;
        // FP32: the products of a stage by themselves, then into the running sum, which
        // so rounds once in 2 E products (in the chain of all of them it rounds twice in
        // each; 4^4 aggregates: 1.1e-7 from the exact sum against 1.9e-7)
        Pc a[2][TI];
#pragma unroll
        for (int q = 0; q < TI; ++q) {
            a[0][q] = sp[ra[q]];
            a[1][q] = sp[ra[q] + 32];
        }
#pragma unroll
        for (int u = 0; u < TJ; ++u) {
            const Pc b[2] = {sp[ru[u]], sp[ru[u] + 32]};
#pragma unroll
            for (int q = 0; q < TI; ++q) {
                R &re = acc[(q * TJ + u) * 2], &im = acc[(q * TJ + u) * 2 + 1];
                if constexpr (kTwo) {
                    R &re2 = acc2[(q * TJ + u) * 2], &im2 = acc2[(q * TJ + u) * 2 + 1];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const cplx<R> m = a[h][q].at(0), v = b[h].at(0);
                        re = fma(m.x, v.x, re);
                        im = fma(m.x, v.y, im);
                        re2 = fma(m.y, v.y, re2);
                        im2 = fma(m.y, v.x, im2);
                    }
                } else {
                    cplx<R> t = cmulc(a[0][q].at(0), b[0].at(0));
#pragma unroll
                    for (int k = 1; k < 2 * E; ++k) cmacc(t, a[k / E][q].at(k % E), b[k / E].at(k % E));
                    re += t.x;
                    im += t.y;
                }
            }
        }
    }
    if constexpr (kTwo)
#pragma unroll
        for (int q = 0; q < TI * TJ * 2; q += 2) {
            acc[q] += acc2[q];
            acc[q + 1] -= acc2[q + 1];
        }
    constexpr int N = TI * TJ * 2, keep = N / 32 > 1 ? N / 32 : 1, dup = N < 32 ? 32 / N : 1;
    int base = 0;
    scatter_sum<N, 16>(acc, lane, base);
    if (lane % dup) return;
    R* out = reinterpret_cast<R*>(xc);
#pragma unroll
    for (int k = 0; k < keep; ++k) {
        const int e = base + k, i = i0 + e / 2 / TJ, u = j0 + e / 2 % TJ, j = jc + u;
        if (i < nv && u < nr && (act == nullptr || act[j]))
            out[((size_t)j * B.nb * nc + (size_t)blk * nc + chi * nv + i) * 2 + e % 2] = acc[k];
    }
}

// x = P x_c: a thread takes two pieces of E entries of an aggregate's fine
// entries (a warp's pieces are whole sites) and TJ right-hand sides, whose
// coarse entries are broadcast from shared memory ([chirality][i][rhs], the two
// halves in different banks).  A broadcast costs as much shared-memory bandwidth
// as any other load of its width, so the tile is 2 E x TJ instead of E x 2 TJ;
// the CTAs of the other right-hand sides follow in launch order and find P in
// L2.  P comes by asynchronous copies kAhead rows ahead into a ring that each
// thread fills and reads for itself (no barrier).
// 32 x 16^3, 4^4 aggregates, nv 20, 16 right-hand sides: 339 us ->
// 153 us (3.0 TB/s) at five CTAs per SM; 145 us with one chain of fused multiply-adds
// per sum, four or six CTAs 165 / 158 us.  FP64 takes one piece per thread and at most
// two right-hand sides: what counts there are the operations on padding.
constexpr int kAhead = 8;
constexpr int kProlongT = 96;   // whole warps and whole sites: both pieces lie at the same place of a site
template <typename R, int E, int TJ>
__global__ void __launch_bounds__(kProlongT, 5) prolong_tile_kernel(Geom g, Blocking B, int nv,
                                                                 const cplx<R>* __restrict__ P,
                                                                 const cplx<R>* __restrict__ xc, cplx<R>* __restrict__ x,
                                                                 int nrhs, int parts, const int* __restrict__ act) {
    constexpr bool kTwo = sizeof(R) == 8;
    constexpr int NP = kTwo ? 1 : 2;   // pieces of a thread
    constexpr int kPer = 12 / E, T = kProlongT, kStep = T / kPer;   // pieces per site, sites between the two pieces
    static_assert(T % kPer == 0 && T % 32 == 0, "CTA of whole warps and whole sites");
    using Pc = Piece<R, E>;
    extern __shared__ __align__(16) unsigned char psm[];
    Pc* ring = reinterpret_cast<Pc*>(psm) + threadIdx.x;   // [kAhead][NP][T]
    cplx<R>* cs = reinterpret_cast<cplx<R>*>(psm + sizeof(Pc) * kAhead * NP * T);
    const int nc = 2 * nv, nloc = B.bs * 6, half = (nv + (nv & 1)) * TJ + 2;
    const int groups = (nrhs + TJ - 1) / TJ;
    const int j0 = (blockIdx.x % groups) * TJ, part = (blockIdx.x / groups) % parts, blk = blockIdx.x / groups / parts;
    const int l = NP * part * kStep + threadIdx.x / kPer, w = threadIdx.x % kPer;
    const int chi = w / (kPer / 2), s = (w % (kPer / 2)) * E;
    // aggregates that one piece per thread covers: the second repeats the first and is
    // multiplied for nothing (16 sites, 16 x 8^3, 4 right-hand sides: 9 us, launch and
    // latency, not arithmetic)
    const bool two = NP == 2 && B.bs > kStep;
    const cplx<R>* p = P + ((size_t)blk * 2 + chi) * nv * nloc + s;
    auto fill = [&](int i) {
        if (i < nv)
#pragma unroll
            for (int h = 0; h < NP; ++h) {
                const int lh = l + h * kStep;
                const bool in = lh < B.bs;
                if (h == 0 || two)
                    async_piece<R, E>(ring + ((i % kAhead) * NP + h) * T, p + (size_t)i * nloc + (in ? lh * 6 : 0), in);
            }
        async_commit();
    };
#pragma unroll
    for (int i = 0; i < kAhead - 2; ++i) fill(i);
    for (int e = threadIdx.x; e < nc * TJ; e += T) {
        const int i = e % nc, u = e / nc;
        cplx<R> v = czero<R>();
        if (j0 + u < nrhs) v = xc[(size_t)(j0 + u) * B.nb * nc + (size_t)blk * nc + i];
        cs[(i / nv) * half + (i % nv) * TJ + u] = v;
    }
    if ((nv & 1) && threadIdx.x < 2 * TJ) cs[threadIdx.x / TJ * half + nv * TJ + threadIdx.x % TJ] = czero<R>();
    __syncthreads();
    const cplx<R>* c = cs + chi * half;
    cplx<R> acc[NP][TJ][E], acc2[kTwo ? TJ : 1];
#pragma unroll
    for (int u = 0; u < TJ; ++u) {
        if constexpr (kTwo) acc2[u] = czero<R>();
#pragma unroll
        for (int h = 0; h < NP; ++h)
#pragma unroll
            for (int k = 0; k < E; ++k) acc[h][u][k] = czero<R>();
    }
    // FP32: two rows at a time, summed by themselves before they join the running sum
    // (one chain over all rows: 1.14e-7 from the exact sum against 7.4e-8 at nv 20)
    const int second = two ? T : 0;
    for (int i = 0; i < nv; i += 2) {
        async_wait<kAhead - 4>();
        // past the last of an odd number: the same row again, times the zeros behind it
        const bool pair = i + 1 < nv;
        const Pc *r0 = ring + (i % kAhead) * NP * T, *r1 = pair ? ring + ((i + 1) % kAhead) * NP * T : r0;
        const Pc a[2][2] = {{r0[0], r0[second]}, {r1[0], r1[second]}};   // [row][piece]
        fill(i + kAhead - 2);
        fill(i + kAhead - 1);
#pragma unroll
        for (int u = 0; u < TJ; ++u) {
            const cplx<R> v = c[i * TJ + u], w = c[(i + 1) * TJ + u];
            if constexpr (kTwo) {
                cplx<R>&s1 = acc[0][u][0], &s2 = acc2[u];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const cplx<R> m = a[q][0].at(0), z = q ? w : v;
                    s1.x = fma(m.x, z.x, s1.x);
                    s1.y = fma(m.x, z.y, s1.y);
                    s2.x = fma(m.y, z.y, s2.x);
                    s2.y = fma(m.y, z.x, s2.y);
                }
            } else {
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int k = 0; k < E; ++k) {
                        cplx<R> t = a[0][h].at(k) * v;
                        cmac(t, a[1][h].at(k), w);
                        acc[h][u][k] += t;
                    }
            }
        }
    }
    if constexpr (kTwo)
#pragma unroll
        for (int u = 0; u < TJ; ++u) acc[0][u][0] = mk<R>(acc[0][u][0].x - acc2[u].x, acc[0][u][0].y + acc2[u].y);
#pragma unroll
    for (int h = 0; h < NP; ++h) {
        const int lh = l + h * kStep;
        if (lh >= B.bs) continue;
        cplx<R>* o = x + (size_t)block_fine_site(g, B, blk, lh) * 12 + 6 * chi + s;
#pragma unroll
        for (int u = 0; u < TJ; ++u) {
            const int j = j0 + u;
            if (j >= nrhs || (act != nullptr && !act[j])) continue;
            cplx<R>* q = o + (size_t)j * g.V * 12;
            if constexpr (E == 2)
                *reinterpret_cast<float4*>(q) = make_float4(acc[h][u][0].x, acc[h][u][0].y, acc[h][u][1].x, acc[h][u][1].y);
            else
                *q = acc[h][u][0];
        }
    }
}

// ------------------------------------------------------------------ coarse build
// CTA (coarse site blk, direction d): column by column, h(l) = the part of
// (D P e_col)(y_l) that D couples from block blk + d (d = 0: site-diagonal and
// in-block hops), then A[blk][d][col][row] = P_blk[row]^H h.
template <typename R>
__device__ __forceinline__ void P_spinor(const cplx<R>* __restrict__ P, int nv, int nloc, int blk, int chi, int i, int l,
                                         Spinor<R>& s) {
#pragma unroll
    for (int k = 0; k < 12; ++k) s.c[k] = czero<R>();
    const cplx<R>* p = P + (((size_t)blk * 2 + chi) * nv + i) * nloc + (size_t)l * 6;
#pragma unroll
    for (int k = 0; k < 6; ++k) s.c[6 * chi + k] = p[k];
}

template <bool fwd, typename R>
__device__ __forceinline__ void hop_dispatch(int mu, const Spinor<R>& psi, const Link<R>& u, R sg, Spinor<R>& acc) {
    switch (mu) {
        case 0: hop_accumulate<R, 0, fwd>(psi, u, sg, acc); break;
        case 1: hop_accumulate<R, 1, fwd>(psi, u, sg, acc); break;
        case 2: hop_accumulate<R, 2, fwd>(psi, u, sg, acc); break;
        default: hop_accumulate<R, 3, fwd>(psi, u, sg, acc); break;
    }
}

// Sites of block blk that direction d draws from: all bs for d = 0, the
// sites on the face towards block blk + d otherwise (none when the block grid
// has extent 1 in that direction, whose hops wrap into d = 0).
__device__ __forceinline__ bool coarse_active(const Blocking& B, int d, const int o[4]) {
    if (d == 0) return true;
    const bool fw = d <= 4;
    const int mu = (d - 1) % 4;
    return (fw ? o[mu] == B.b[mu] - 1 : o[mu] == 0) && B.cd[mu] > 1;
}

// Columns col0 .. col0+nch-1 at a time: every thread takes (column, active
// site) tasks and leaves h in shared memory ([column][active site][12]);
// then one warp per (column, row) entry forms P_blk[row]^H h over the active
// sites only.
template <typename R>
__global__ void __launch_bounds__(256) build_coarse_kernel(Geom g, Blocking B, int nv, const cplx<R>* __restrict__ U,
                                                          const R* __restrict__ A, const cplx<R>* __restrict__ P,
                                                          cplx<R>* __restrict__ Ac, int chunk) {
    extern __shared__ __align__(16) unsigned char hraw[];
    cplx<R>* hsm = reinterpret_cast<cplx<R>*>(hraw);   // [chunk][na][12], then na ints
    int* lst = reinterpret_cast<int*>(hsm + (size_t)chunk * B.bs * 12);
    __shared__ int na_s;
    const int blk = blockIdx.x, d = blockIdx.y;
    const int nc = 2 * nv, nloc = B.bs * 6;
    int cb[4];
    block_coords(B, blk, cb);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    if (threadIdx.x == 0) {
        int c = 0;
        for (int l = 0; l < B.bs; ++l) {
            int o[4];
            local_coords(B, l, o);
            if (coarse_active(B, d, o)) lst[c++] = l;
        }
        na_s = c;
    }
    __syncthreads();
    const int na = na_s;
    for (int col0 = 0; col0 < nc; col0 += chunk) {
        const int nch = min(chunk, nc - col0);
        for (int t = threadIdx.x; t < nch * na; t += blockDim.x) {
            const int cc = t / na, a = t % na;
            const int col = col0 + cc, l = lst[a];
            const int chic = col / nv, ic = col % nv;
            int o[4], x[4];
            local_coords(B, l, o);
            for (int mu = 0; mu < 4; ++mu) x[mu] = cb[mu] * B.b[mu] + o[mu];
            const int y = site_index(g, x);
            Spinor<R> acc;
#pragma unroll
            for (int k = 0; k < 12; ++k) acc.c[k] = czero<R>();
            if (d == 0) {
                Spinor<R> ps;
                P_spinor<R>(P, nv, nloc, blk, chic, ic, l, ps);
                clover_apply<R>(A + (size_t)y * 72, ps, acc);
            }
            for (int mu = 0; mu < 4; ++mu) {
                for (int dir = 0; dir < 2; ++dir) {
                    const bool fw = dir == 0;
                    const bool face = (fw ? (o[mu] == B.b[mu] - 1) : (o[mu] == 0)) && B.cd[mu] > 1;
                    const int want = face ? (fw ? 1 + mu : 5 + mu) : 0;
                    if (want != d) continue;
                    int neg;
                    const int yn = fw ? nb_fwd(g, x, y, mu, neg) : nb_bwd(g, x, y, mu, neg);
                    int xn[4];
                    site_coords(g, yn, xn);
                    int cn[4], on[4];
                    for (int k = 0; k < 4; ++k) { cn[k] = xn[k] / B.b[k]; on[k] = xn[k] % B.b[k]; }
                    Spinor<R> ps;
                    P_spinor<R>(P, nv, nloc, coarse_index(B, cn), chic, ic, local_index(B, on), ps);
                    Link<R> u;
                    load_link<R>(U + ((size_t)(fw ? y : yn) * 4 + mu) * 9, u);
                    if (fw) hop_dispatch<true, R>(mu, ps, u, neg ? R(-1) : R(1), acc);
                    else hop_dispatch<false, R>(mu, ps, u, neg ? R(-1) : R(1), acc);
                }
            }
            cplx<R>* h = hsm + ((size_t)cc * na + a) * 12;
#pragma unroll
            for (int k = 0; k < 12; ++k) h[k] = acc.c[k];
        }
        __syncthreads();
        for (int e = warp; e < nch * nc; e += nwarps) {
            const int cc = e / nc, row = e % nc;
            const int chir = row / nv, ir = row % nv;
            const cplx<R>* pr = P + (((size_t)blk * 2 + chir) * nv + ir) * nloc;
            const cplx<R>* h = hsm + (size_t)cc * na * 12 + 6 * chir;
            R re = 0, im = 0;
            for (int q = lane; q < na * 6; q += 32) {
                const int a = q / 6, sc = q % 6;
                const cplx<R> pv = pr[lst[a] * 6 + sc], hv = h[a * 12 + sc];
                cdot(re, im, pv, hv);
            }
            re = warp_sum(re);
            im = warp_sum(im);
            if (lane == 0) Ac[(((size_t)blk * 9 + d) * nc + col0 + cc) * nc + row] = mk<R>(re, im);
        }
        __syncthreads();
    }
}

__global__ void narrow_kernel(const double2* __restrict__ a, float2* __restrict__ b, size_t n) {
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
        b[t] = cvt<float2>(a[t]);
}

// ------------------------------------------------------------------ coarse apply
// Multi-right-hand-side coarse stencil: one CTA per (coarse site, chunk of
// up to kCoarseRC right-hand sides).  The 9 neighbour vectors of the chunk
// are staged in shared memory ([d][col][rhs]); every stencil block entry is
// then loaded once per chunk (coalesced: consecutive threads take consecutive
// rows of the column-major blocks) and multiplied into kCoarseRPT
// right-hand sides held in registers, so the (2 Nv)^2 x 9 blocks -- the bulk
// of the bytes -- are read once per chunk instead of once per right-hand side.
constexpr int kCoarseRC = 16;
constexpr int kCoarseRPT = 4;
template <typename Z, typename R>
__global__ void coarse_apply_mrhs_kernel(Geom gc, int nc, const Z* __restrict__ A, const Z* __restrict__ x,
                                         Z* __restrict__ y, int op, Shifts tau, int nrhs, int rc) {
    extern __shared__ __align__(16) unsigned char craw[];
    Z* xs = reinterpret_cast<Z*>(craw);                 // [9][nc][rc]
    __shared__ int nbr[9];
    const int s = blockIdx.x;
    const int j0 = blockIdx.y * rc;
    const size_t vstride = (size_t)gc.V * nc;
    for (int d = threadIdx.x; d < 9; d += blockDim.x) {   // small blocks: fewer than nine threads
        int c[4];
        site_coords(gc, s, c);
        int sn = s;
        if (d > 0) {
            const int mu = (d - 1) & 3, step = d <= 4 ? 1 : -1;
            c[mu] = (c[mu] + step + gc.L[mu]) % gc.L[mu];
            sn = site_index(gc, c);
        }
        nbr[d] = sn;
    }
    __syncthreads();
    const int nstage = 9 * nc * rc;
    for (int e0 = threadIdx.x; e0 < nstage; e0 += 8 * blockDim.x) {
        Z v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int e = e0 + q * blockDim.x;
            v[q].x = 0; v[q].y = 0;
            if (e < nstage) {
                const int col = e % nc, jj = (e / nc) % rc, d = e / (nc * rc);
                if (j0 + jj < nrhs) v[q] = __ldg(x + (size_t)(j0 + jj) * vstride + (size_t)nbr[d] * nc + col);
            }
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int e = e0 + q * blockDim.x;
            if (e < nstage) {
                const int col = e % nc, jj = (e / nc) % rc, d = e / (nc * rc);
                xs[((size_t)d * nc + col) * rc + jj] = v[q];
            }
        }
    }
    __syncthreads();
    const int r = threadIdx.x % nc, grp = threadIdx.x / nc;
    if (grp * kCoarseRPT >= rc) return;
    Z acc[kCoarseRPT];
#pragma unroll
    for (int k = 0; k < kCoarseRPT; ++k) { acc[k].x = 0; acc[k].y = 0; }
    const Z* As = A + (size_t)s * 9 * nc * nc + r;
    for (int d = 0; d < 9; ++d) {
        const Z* Ad = As + (size_t)d * nc * nc;
        const Z* xd = xs + (size_t)d * nc * rc + grp * kCoarseRPT;
        // a direction by itself: one chain over all nine was 1.35 times as far from
        // the exact sum as products added one by one, this is less than half as far
        Z part[kCoarseRPT];
#pragma unroll
        for (int k = 0; k < kCoarseRPT; ++k) { part[k].x = 0; part[k].y = 0; }
#pragma unroll 4
        for (int col = 0; col < nc; ++col) {
            const Z a = __ldg(Ad + (size_t)col * nc);
            const Z* xv = xd + (size_t)col * rc;
#pragma unroll
            for (int k = 0; k < kCoarseRPT; ++k) cmac(part[k], a, xv[k]);
        }
#pragma unroll
        for (int k = 0; k < kCoarseRPT; ++k) acc[k] += part[k];
    }
    const R sg = r < nc / 2 ? R(1) : R(-1);
#pragma unroll
    for (int k = 0; k < kCoarseRPT; ++k) {
        const int jj = grp * kCoarseRPT + k, j = j0 + jj;
        if (j >= nrhs) break;
        const R tj = (R)tau.t[j];
        const Z xv = xs[(size_t)r * rc + jj];        // direction 0 is the site itself
        Z o = acc[k];
        if (op == QCD_OP_D) { o -= (tj * sg) * xv; }
        else { o = sg * o; o -= tj * xv; }
        y[(size_t)j * vstride + (size_t)s * nc + r] = o;
    }
}

// ---- a wait on an mbarrier, bounded in time, for the self-test below: one that gives
// up counts itself in g_wait_timeouts.
__device__ unsigned long long g_wait_timeouts;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* bar, unsigned parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// wait for phase `parity` of the barrier, giving up after `limit` clocks
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity, long long limit) {
    if (mbar_try(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try(bar, parity)) {
        if (clock64() - t0 > limit) {
            atomicAdd(&g_wait_timeouts, 1ull);
            return false;
        }
    }
    return true;
}

// Self-test of the bounded wait: one warp waits on an mbarrier that nothing
// arrives at, gives up after `limit` clocks, counts itself and returns.
__global__ void wait_probe_kernel(long long limit) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) mbar_wait(&bar, 0, limit);
}

// FP32 coarse stencil, one CTA per (coarse site, 2 J right-hand sides), one warp
// per direction.  A warp streams its block A_d and its neighbour's vectors in
// stages of eight columns through a ring of its own (asynchronous copies of 16
// bytes per lane, three stages), so no barrier of the CTA stands between the nine
// streams and two CTAs keep up to 220 KB per SM in flight.  Lane (r, h) holds rows
// r, r + 16, .. of y for J right-hand sides: per pair of columns 2 R + J loads from
// shared memory feed 8 R J FMAs (one row and eight right-hand sides per thread, as
// before, are bound by the shared-memory loads).  The nine partial results are
// added through shared memory at the end.  Bound by the FMA pipe and the issue slots
// at 16 right-hand sides and by HBM below about 6.  Nv = 24: 8^4 sites, 16
// right-hand sides 280 -> 253 us (43 TFLOP/s); 8 x 4^3 sites, 4 right-hand sides
// 33 -> 18 us, 1: 31 -> 16.5 us (86 MB: 5.2 TB/s).  Blocks by cp.async.bulk (one
// copy per stage and an mbarrier) 262 us, fma.f32x2 302 us.
constexpr int kStageCols = 8;     // columns per stage
constexpr int kStages = 3;
// one warp's stages: kStageCols columns of A_d and of the W vectors; the sums of the
// result reuse them, rows of W + 2
__host__ __device__ constexpr size_t coarse_stage_bytes(int nc, int W) {
    return sizeof(float2) * (size_t)kStageCols * (nc + W);
}
__host__ __device__ inline size_t coarse_ring_bytes(int nc, int W) {
    const size_t ring = kStages * coarse_stage_bytes(nc, W), sums = sizeof(float2) * (size_t)nc * (W + 2);
    return ring > sums ? ring : sums;
}
template <int R, int J>
__global__ void __launch_bounds__(288, 2) coarse_apply_staged_kernel(Geom gc, int nc, const float2* __restrict__ A,
                                                                  const float2* __restrict__ x,
                                                                  float2* __restrict__ y, int op, Shifts tau,
                                                                  int nrhs) {
    constexpr int W = 2 * J, RS = W + 2;   // right-hand sides per CTA; row stride of the sums (16 bytes of padding)
    extern __shared__ __align__(16) unsigned char dsm[];
    const int lane = threadIdx.x & 31, d = threadIdx.x >> 5;
    const int s = blockIdx.x, j0 = blockIdx.y * W;
    const size_t vstride = (size_t)gc.V * nc, wbytes = coarse_ring_bytes(nc, W);
    unsigned char* ring = dsm + d * wbytes;
    const size_t stage = coarse_stage_bytes(nc, W);
    int c[4];
    site_coords(gc, s, c);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {   // no indexed array: c stays in registers
        if (d == mu + 1) c[mu] = c[mu] + 1 == gc.L[mu] ? 0 : c[mu] + 1;
        if (d == mu + 5) c[mu] = c[mu] == 0 ? gc.L[mu] - 1 : c[mu] - 1;
    }
    const int sn = site_index(gc, c);
    // 16-byte pieces: the columns of A_d are contiguous, two columns of a vector each
    const int live = min(W, nrhs - j0), nst = (nc + kStageCols - 1) / kStageCols;
    constexpr int XP = (W * kStageCols / 2 + 31) / 32;   // pieces of the vectors per lane and stage
    const float2* pa = A + ((size_t)s * 9 + d) * nc * nc + 2 * lane;
    const float2* px[XP];
#pragma unroll
    for (int i = 0; i < XP; ++i) {
        const int e = lane + 32 * i, j = min(e / (kStageCols / 2), live - 1);
        px[i] = x + (size_t)(j0 + j) * vstride + (size_t)sn * nc + e % (kStageCols / 2) * 2;
    }
    int filled = 0;
    unsigned char* fbuf = ring;
    auto fill = [&]() {
        if (filled < nst) {
            const int cols = min(kStageCols, nc - filled * kStageCols), np = cols * nc / 2;
            Piece<float, 2>* o = reinterpret_cast<Piece<float, 2>*>(fbuf) + lane;
            const float2* src = pa;
#pragma unroll 2
            for (int e = lane; e < np; e += 32, o += 32, src += 64) async_piece<float, 2>(o, src, true);
            pa += kStageCols * nc;
            o = reinterpret_cast<Piece<float, 2>*>(fbuf) + kStageCols / 2 * nc + lane;
#pragma unroll
            for (int i = 0; i < XP; ++i) {
                const int e = lane + 32 * i;
                if (e < live * (kStageCols / 2) && e % (kStageCols / 2) * 2 < cols) async_piece<float, 2>(o + 32 * i, px[i], true);
                px[i] += kStageCols;
            }
            ++filled;
            fbuf = filled % kStages == 0 ? ring : fbuf + stage;
        }
        async_commit();
    };
#pragma unroll
    for (int i = 0; i < kStages - 1; ++i) fill();
    const int r0 = lane & 15, h = lane >> 4;
    float2 acc[R][J];
#pragma unroll
    for (int q = 0; q < R; ++q)
#pragma unroll
        for (int k = 0; k < J; ++k) acc[q][k] = make_float2(0.f, 0.f);
    const unsigned char* buf = ring;
    for (int i = 0; i < nst; ++i) {
        fill();
        async_wait<kStages - 1>();
        __syncwarp();
        // rows past the last read the next column (after the last the vectors): not kept
        const float2* ap = reinterpret_cast<const float2*>(buf) + r0;
        const float2* Xs = reinterpret_cast<const float2*>(buf) + (size_t)kStageCols * nc + h * J * kStageCols;
        auto two = [&](const float2* xc) {
            float2 a0[R], a1[R];
#pragma unroll
            for (int q = 0; q < R; ++q) {
                a0[q] = ap[16 * q];
                a1[q] = ap[nc + 16 * q];
            }
            ap += 2 * nc;
#pragma unroll
            for (int k = 0; k < J; ++k) {
                const float4 v = *reinterpret_cast<const float4*>(xc + k * kStageCols);
#pragma unroll
                for (int q = 0; q < R; ++q) cmac(acc[q][k], a0[q], make_float2(v.x, v.y));
#pragma unroll
                for (int q = 0; q < R; ++q) cmac(acc[q][k], a1[q], make_float2(v.z, v.w));
            }
        };
        const int cols = nc - i * kStageCols;
        if (cols >= kStageCols) {
#pragma unroll
            for (int col = 0; col < kStageCols; col += 2) two(Xs + col);
        } else {
            for (int col = 0; col < cols; col += 2) two(Xs + col);
        }
        buf = (i + 1) % kStages == 0 ? ring : buf + stage;
        __syncwarp();   // stage read: filled again next
    }
#pragma unroll
    for (int q = 0; q < R; ++q) {
        const int row = r0 + 16 * q;
        if (row < nc) {
            float4* o = reinterpret_cast<float4*>(reinterpret_cast<float2*>(ring) + (size_t)row * RS + h * J);
#pragma unroll
            for (int k = 0; k < J; k += 2)
                o[k / 2] = make_float4(acc[q][k].x, acc[q][k].y, acc[q][k + 1].x, acc[q][k + 1].y);
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < nc * J; e += blockDim.x) {
        const int row = e % nc, k = e / nc * 2;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int dd = 0; dd < 9; ++dd) {
            const float4 v = *reinterpret_cast<const float4*>(dsm + dd * wbytes + sizeof(float2) * ((size_t)row * RS + k));
            o.x += v.x;
            o.y += v.y;
            o.z += v.z;
            o.w += v.w;
        }
        const float sg = row < nc / 2 ? 1.f : -1.f;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int j = j0 + k + i;
            if (j >= nrhs) break;
            const size_t at = (size_t)j * vstride + (size_t)s * nc + row;
            const float tj = (float)tau.t[j];
            const float2 xv = __ldg(x + at);
            float2 r = i ? make_float2(o.z, o.w) : make_float2(o.x, o.y);
            if (op == QCD_OP_D) { r -= (tj * sg) * xv; }
            else { r = sg * r; r -= tj * xv; }
            y[at] = r;
        }
    }
}

template <int R, int J>
static void launch_coarse_staged(const Coarse& c, int op, int nrhs, const float2* x, float2* y, const Shifts& sh,
                              cudaStream_t st) {
    const size_t sm = 9 * coarse_ring_bytes(c.nc, 2 * J);
    if (sm > 48 * 1024)
        cudaFuncSetAttribute(coarse_apply_staged_kernel<R, J>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    coarse_apply_staged_kernel<R, J><<<dim3(c.gc.V, (nrhs + 2 * J - 1) / (2 * J)), 288, sm, st>>>(c.gc, c.nc, c.A32, x, y,
                                                                                               op, sh, nrhs);
}
// J: the fewest chunks of at most 16, evenly filled (20 right-hand sides: two of 12,
// 47 us against 65 with 16 + 4 at 8 x 4^3 sites, Nv = 20)
template <int R>
static void coarse_staged_rows(const Coarse& c, int op, int nrhs, const float2* x, float2* y, const Shifts& sh,
                             cudaStream_t st) {
    const int chunks = (nrhs + 15) / 16, j = (nrhs + 2 * chunks - 1) / (2 * chunks);
    if (j <= 2) launch_coarse_staged<R, 2>(c, op, nrhs, x, y, sh, st);
    else if (j <= 4) launch_coarse_staged<R, 4>(c, op, nrhs, x, y, sh, st);
    else if (j <= 6) launch_coarse_staged<R, 6>(c, op, nrhs, x, y, sh, st);
    else launch_coarse_staged<R, 8>(c, op, nrhs, x, y, sh, st);
}

// Tensor-core coarse stencil (FP32 data, 3xTF32 products): per coarse site
// and chunk of kTcR right-hand sides, the stencil is one real GEMM
//   [Re y; Im y] (2nc x R) = sum_d [[Re A_d, -Im A_d], [Im A_d, Re A_d]] (2nc x 2nc)
//                            [Re x_d; Im x_d] (2nc x R),
// x_d the neighbour in direction d.  Each warp owns a 16-row tile of the
// result and runs mma.sync m16n8k8 (TF32 in, FP32 accumulate) over K = 9 x 2nc;
// every operand is split as big + small TF32 parts and the three products
// small*big + big*small + big*big keep FP32-level accuracy.  The neighbour
// vectors are staged once ([d][k][r], padded rows: conflict-free fragment
// loads); the blocks A_d one direction at a time.  Needs nc % 8 == 0.
constexpr int kTcR = 16;
constexpr int kTcXs = 24;   // padded row stride of the staged vectors (floats)
constexpr int kTcPre = 16;  // prefetched block entries per thread: nc^2 <= 16 x 32 (nc / 8)

__device__ __forceinline__ uint32_t tf32_of(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ void tf32_split(float x, uint32_t& big, uint32_t& small) {
    big = tf32_of(x);
    small = tf32_of(x - __uint_as_float(big));
}
__device__ __forceinline__ void mma_tf32(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// column stride of the staged block (complex entries): 2 x stride = 16 mod 32
// words, so the four columns of a fragment load fall on disjoint bank halves
__host__ __device__ inline int tc_astride(int nc) { return nc + (24 - nc % 16) % 16; }

__global__ void coarse_apply_tc_kernel(Geom gc, int nc, const float2* __restrict__ A, const float2* __restrict__ x,
                                       float2* __restrict__ y, int op, Shifts tau, int nrhs) {
    extern __shared__ __align__(16) float tsm[];
    const int n2 = 2 * nc, astride = tc_astride(nc);
    float* Xs = tsm;                                               // [9][2nc][kTcXs]
    float2* As = reinterpret_cast<float2*>(Xs + (size_t)9 * n2 * kTcXs);   // [nc cols][astride]
    float* Ys = reinterpret_cast<float*>(As);                      // [2nc][kTcR], after the last direction
    __shared__ int nbr[9];
    const int s = blockIdx.x, j0 = blockIdx.y * kTcR;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t = lane & 3;
    const size_t vstride = (size_t)gc.V * nc;
    if (tid < 9) {
        int c[4];
        site_coords(gc, s, c);
        int sn = s;
        if (tid > 0) {
            const int mu = (tid - 1) & 3, step = tid <= 4 ? 1 : -1;
            c[mu] = (c[mu] + step + gc.L[mu]) % gc.L[mu];
            sn = site_index(gc, c);
        }
        nbr[tid] = sn;
    }
    __syncthreads();
    // stage the neighbour vectors: batches of 8 loads in flight per thread
    const int nstage = 9 * nc * kTcR;
    for (int e0 = tid; e0 < nstage; e0 += 8 * blockDim.x) {
        float2 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int e = e0 + q * blockDim.x;
            v[q] = make_float2(0.f, 0.f);
            if (e < nstage) {
                const int col = e % nc, r = (e / nc) % kTcR, d = e / (nc * kTcR);
                if (j0 + r < nrhs) v[q] = __ldg(x + (size_t)(j0 + r) * vstride + (size_t)nbr[d] * nc + col);
            }
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int e = e0 + q * blockDim.x;
            if (e < nstage) {
                const int col = e % nc, r = (e / nc) % kTcR, d = e / (nc * kTcR);
                Xs[((size_t)d * n2 + col) * kTcXs + r] = v[q].x;
                Xs[((size_t)d * n2 + nc + col) * kTcXs + r] = v[q].y;
            }
        }
    }
    // the stencil block of the next direction is loaded into registers while
    // the current one is multiplied (up to kTcPre entries per thread)
    const int nblk = nc * nc;
    float2 pre[kTcPre];
    auto prefetch = [&](int d) {
        const float2* Ad = A + ((size_t)s * 9 + d) * nblk;
#pragma unroll
        for (int q = 0; q < kTcPre; ++q) {
            const int e = tid + q * blockDim.x;
            pre[q] = e < nblk ? __ldg(Ad + e) : make_float2(0.f, 0.f);
        }
    };
    prefetch(0);
    float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    const int row0 = 16 * warp;
    for (int d = 0; d < 9; ++d) {
        __syncthreads();   // staging done / previous block no longer read
#pragma unroll
        for (int q = 0; q < kTcPre; ++q) {
            const int e = tid + q * blockDim.x;
            if (e < nblk) As[(e / nc) * astride + (e % nc)] = pre[q];
        }
        __syncthreads();
        if (d + 1 < 9) prefetch(d + 1);
        const float* Xd = Xs + (size_t)d * n2 * kTcXs;
        for (int k0 = 0; k0 < n2; k0 += 8) {
            uint32_t ab[4], as_[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int rho = row0 + g + (i & 1) * 8, kap = k0 + t + (i >> 1) * 4;
                const bool rim = rho >= nc, kim = kap >= nc;
                const float2 v = As[(kim ? kap - nc : kap) * astride + (rim ? rho - nc : rho)];
                const float val = rim == kim ? v.x : (rim ? v.y : -v.y);
                tf32_split(val, ab[i], as_[i]);
            }
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
                uint32_t bb0, bs0, bb1, bs1;
                tf32_split(Xd[(size_t)(k0 + t) * kTcXs + 8 * nt + g], bb0, bs0);
                tf32_split(Xd[(size_t)(k0 + t + 4) * kTcXs + 8 * nt + g], bb1, bs1);
                mma_tf32(acc[nt], as_, bb0, bb1);
                mma_tf32(acc[nt], ab, bs0, bs1);
                mma_tf32(acc[nt], ab, bb0, bb1);
            }
        }
    }
    __syncthreads();   // the last block is no longer read: Ys reuses its space
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int rho = row0 + g + (i >> 1) * 8, col = 8 * nt + 2 * t + (i & 1);
            Ys[rho * kTcR + col] = acc[nt][i];
        }
    __syncthreads();
    for (int e = tid; e < nc * kTcR; e += blockDim.x) {
        const int row = e % nc, r = e / nc, j = j0 + r;
        if (j >= nrhs) continue;
        float2 o = make_float2(Ys[row * kTcR + r], Ys[(row + nc) * kTcR + r]);
        const float2 xv = make_float2(Xs[(size_t)row * kTcXs + r], Xs[(size_t)(nc + row) * kTcXs + r]);
        const float sg = row < nc / 2 ? 1.f : -1.f;
        const float tj = (float)tau.t[j];
        if (op == QCD_OP_D) { o -= (tj * sg) * xv; }
        else { o = sg * o; o -= tj * xv; }
        y[(size_t)j * vstride + (size_t)s * nc + row] = o;
    }
}

size_t coarse_tc_smem(int nc) {
    // the block region also holds the 2nc x kTcR results at the end
    const size_t ablk = std::max(sizeof(float2) * (size_t)nc * tc_astride(nc), sizeof(float) * (size_t)2 * nc * kTcR);
    return sizeof(float) * (size_t)9 * 2 * nc * kTcXs + ablk;
}

// ------------------------------------------------------------------ SAP block solves
// One CTA per (block of one colour, rhs), one thread per block site; GMRES
// from zero on the Dirichlet block operator (hops leaving the block dropped),
// Arnoldi by modified Gram-Schmidt, Krylov vectors in global scratch.
template <typename R>
__device__ __forceinline__ void block_op(const Geom& g, const Blocking& B, const cplx<R>* __restrict__ U,
                                         const R* __restrict__ A, int y, int l, const int o[4],
                                         const cplx<R>* vsm, int op, R t, Spinor<R>& acc) {
    Spinor<R> psi;
#pragma unroll
    for (int k = 0; k < 12; ++k) psi.c[k] = vsm[l * 12 + k];
    clover_apply<R>(A + (size_t)y * 72, psi, acc);
    int lstride = 1;
#pragma unroll
    for (int mu = 3; mu >= 0; --mu) {
        Link<R> u;
        Spinor<R> nb;
        if (o[mu] < B.b[mu] - 1) {
            const int ln = l + lstride;
#pragma unroll
            for (int k = 0; k < 12; ++k) nb.c[k] = vsm[ln * 12 + k];
            load_link<R>(U + ((size_t)y * 4 + mu) * 9, u);
            switch (mu) {
                case 0: hop_accumulate<R, 0, true>(nb, u, R(1), acc); break;
                case 1: hop_accumulate<R, 1, true>(nb, u, R(1), acc); break;
                case 2: hop_accumulate<R, 2, true>(nb, u, R(1), acc); break;
                default: hop_accumulate<R, 3, true>(nb, u, R(1), acc); break;
            }
        }
        if (o[mu] > 0) {
            const int ln = l - lstride;
#pragma unroll
            for (int k = 0; k < 12; ++k) nb.c[k] = vsm[ln * 12 + k];
            int xb[4];
            site_coords(g, y, xb);
            xb[mu] -= 1;
            load_link<R>(U + ((size_t)site_index(g, xb) * 4 + mu) * 9, u);
            switch (mu) {
                case 0: hop_accumulate<R, 0, false>(nb, u, R(1), acc); break;
                case 1: hop_accumulate<R, 1, false>(nb, u, R(1), acc); break;
                case 2: hop_accumulate<R, 2, false>(nb, u, R(1), acc); break;
                default: hop_accumulate<R, 3, false>(nb, u, R(1), acc); break;
            }
        }
        lstride *= B.b[mu];
    }
    if (op == QCD_OP_D) {
#pragma unroll
        for (int k = 0; k < 6; ++k) acc.c[k] -= t * psi.c[k];
#pragma unroll
        for (int k = 6; k < 12; ++k) acc.c[k] += t * psi.c[k];
    } else {
#pragma unroll
        for (int k = 0; k < 6; ++k) acc.c[k] -= t * psi.c[k];
#pragma unroll
        for (int k = 6; k < 12; ++k) acc.c[k] = -acc.c[k] - t * psi.c[k];
    }
}

template <typename R>
__global__ void sap_block_kernel(Geom g, Blocking B, const cplx<R>* __restrict__ U, const R* __restrict__ A,
                                 const int* __restrict__ blocks, int op, Shifts tau, const cplx<R>* __restrict__ r,
                                 cplx<R>* __restrict__ x, int iters, double tol, cplx<R>* __restrict__ scratch,
                                 const int* __restrict__ act) {
    extern __shared__ double2 sm[];
    const int bs = B.bs;
    cplx<R>* vsm = reinterpret_cast<cplx<R>*>(sm);                       // [bs][12]
    double2* red = reinterpret_cast<double2*>(vsm + (size_t)bs * 12);    // [bs]
    double2* H = red + bs;                              // [(iters+1) * iters]
    double2* gv = H + (iters + 1) * iters;              // [iters + 1]
    double2* sn = gv + iters + 1;                       // [iters]
    double2* yv = sn + iters;                           // [iters]
    double* cs = reinterpret_cast<double*>(yv + iters); // [iters]
    int* flag = reinterpret_cast<int*>(cs + iters);     // [4]

    const int j = blockIdx.y;
    if (act != nullptr && !act[j]) return;
    const int blk = blocks[blockIdx.x];
    const int l = threadIdx.x;
    const size_t fstride = (size_t)g.V * 12;
    r += j * fstride;
    x += j * fstride;
    cplx<R>* kv = scratch + ((size_t)j * gridDim.x + blockIdx.x) * (size_t)(iters + 1) * bs * 12;
    const R t = (R)tau.t[j];

    int o[4];
    local_coords(B, l, o);
    const int y = block_fine_site(g, B, blk, l);

    Spinor<R> w;
    load_spinor<R>(r + (size_t)y * 12, w);
    double2 nn = make_double2(0, 0);
#pragma unroll
    for (int k = 0; k < 12; ++k) nn.x += (double)w.c[k].x * w.c[k].x + (double)w.c[k].y * w.c[k].y;
    nn = block_sum2(nn, red);
    const double beta = sqrt(nn.x);
    if (!(beta > 0.0)) return;
    {
        const R ib = (R)(1.0 / beta);
#pragma unroll
        for (int k = 0; k < 12; ++k) { w.c[k] = ib * w.c[k]; kv[(size_t)l * 12 + k] = w.c[k]; vsm[l * 12 + k] = w.c[k]; }
    }
    if (l == 0) { gv[0] = make_double2(beta, 0); flag[0] = 0; }
    int kdim = 0;
    for (int jj = 0; jj < iters; ++jj) {
        __syncthreads();
        block_op<R>(g, B, U, A, y, l, o, vsm, op, t, w);
        for (int i = 0; i <= jj; ++i) {
            const cplx<R>* vi = kv + (size_t)i * bs * 12 + (size_t)l * 12;
            double2 h = make_double2(0, 0);
#pragma unroll
            for (int k = 0; k < 12; ++k) {
                cplx<R> a = vi[k];
                h.x += (double)a.x * w.c[k].x + (double)a.y * w.c[k].y;
                h.y += (double)a.x * w.c[k].y - (double)a.y * w.c[k].x;
            }
            h = block_sum2(h, red);
            const cplx<R> hr = mk<R>((R)h.x, (R)h.y);
#pragma unroll
            for (int k = 0; k < 12; ++k) cmsub(w.c[k], hr, vi[k]);
            if (l == 0) H[i * iters + jj] = h;
        }
        double2 hn2 = make_double2(0, 0);
#pragma unroll
        for (int k = 0; k < 12; ++k) hn2.x += (double)w.c[k].x * w.c[k].x + (double)w.c[k].y * w.c[k].y;
        hn2 = block_sum2(hn2, red);
        const double hn = sqrt(hn2.x);
        {
            const R ih = hn > 0 ? (R)(1.0 / hn) : R(0);
#pragma unroll
            for (int k = 0; k < 12; ++k) {
                w.c[k] = ih * w.c[k];
                kv[(size_t)(jj + 1) * bs * 12 + (size_t)l * 12 + k] = w.c[k];
                vsm[l * 12 + k] = w.c[k];
            }
        }
        if (l == 0) {
            H[(jj + 1) * iters + jj] = make_double2(hn, 0);
            for (int i = 0; i < jj; ++i) {
                double2 a = H[i * iters + jj], c = H[(i + 1) * iters + jj];
                H[i * iters + jj] = cs[i] * a + sn[i] * c;
                H[(i + 1) * iters + jj] = cs[i] * c - conj(sn[i]) * a;
            }
            double2 a = H[jj * iters + jj];
            double2 c = H[(jj + 1) * iters + jj];
            double aa = sqrt(a.x * a.x + a.y * a.y), rr = sqrt(aa * aa + c.x * c.x + c.y * c.y);
            if (aa > 0) {
                cs[jj] = aa / rr;
                sn[jj] = (1.0 / aa) * a * conj(c);
                sn[jj] = (1.0 / rr) * sn[jj];
            } else {
                cs[jj] = 0.0;
                sn[jj] = make_double2(1, 0);
            }
            H[jj * iters + jj] = cs[jj] * a + sn[jj] * c;
            gv[jj + 1] = -1.0 * (conj(sn[jj]) * gv[jj]);
            gv[jj] = cs[jj] * gv[jj];
            const double res = sqrt(gv[jj + 1].x * gv[jj + 1].x + gv[jj + 1].y * gv[jj + 1].y);
            flag[0] = (tol >= 0.0 && res <= tol * beta) ? 1 : 0;
        }
        __syncthreads();
        kdim = jj + 1;
        if (flag[0]) break;
    }
    if (l == 0) {
        count_sap_work(bs, kdim);
        for (int i = kdim - 1; i >= 0; --i) {
            double2 s = gv[i];
            for (int k = i + 1; k < kdim; ++k) s -= H[i * iters + k] * yv[k];
            double2 dd = H[i * iters + i];
            double den = dd.x * dd.x + dd.y * dd.y;
            yv[i] = den > 0 ? (1.0 / den) * cmulc(dd, s) : make_double2(0, 0);
        }
    }
    __syncthreads();
    Spinor<R> e;
    load_spinor<R>(x + (size_t)y * 12, e);
    for (int i = 0; i < kdim; ++i) {
        const cplx<R> yi = mk<R>((R)yv[i].x, (R)yv[i].y);
        const cplx<R>* vi = kv + (size_t)i * bs * 12 + (size_t)l * 12;
#pragma unroll
        for (int k = 0; k < 12; ++k) cmac(e.c[k], yi, vi[k]);
    }
    store_spinor<R>(x + (size_t)y * 12, e);
}

// ------------------------------------------------------------------ SAP, small blocks
// Blocks of BS <= 32 sites: each SAP block is a BS-lane segment of one warp
// (32 / BS blocks per CTA of one warp).  The block's links and clover and the
// whole Krylov basis live in shared memory; inner products are reduced with
// xor-shuffles inside the segment; Arnoldi by modified Gram-Schmidt, as in the
// 256-site path.  Only __syncwarp() orders shared-memory traffic.
struct SapSmemLayout {
    size_t basis, links, clover, H, g, sn, y, cs, flag, total;
};
template <typename R>
__host__ __device__ inline SapSmemLayout sap_layout(int BS, int iters, size_t basis_elem = sizeof(cplx<R>)) {
    auto up = [](size_t v) { return (v + 15) & ~size_t(15); };
    SapSmemLayout L;
    size_t o = 0;
    L.basis = o;  o = up(o + (size_t)(iters + 1) * BS * 12 * basis_elem);
    L.links = o;  o = up(o + (size_t)BS * 36 * sizeof(cplx<R>));
    L.clover = o; o = up(o + (size_t)BS * 72 * sizeof(R));
    L.H = o;      o = up(o + (size_t)(iters + 1) * iters * sizeof(cplx<R>));
    L.g = o;      o = up(o + (size_t)(iters + 1) * sizeof(cplx<R>));
    L.sn = o;     o = up(o + (size_t)iters * sizeof(cplx<R>));
    L.y = o;      o = up(o + (size_t)iters * sizeof(cplx<R>));
    L.cs = o;     o = up(o + (size_t)iters * sizeof(R));
    L.flag = o;   o = up(o + 4 * sizeof(int));
    L.total = o;
    return L;
}

// Shared memory of the chirality-split kernel with rw right-hand sides per
// CTA: the block's links and clover once, then per warp its Krylov basis and
// GMRES scalars.
struct ChiLayout {
    size_t links, clover, shared, basis, H, g, sn, y, cs, flag, perwarp, total;
};
template <typename R>
__host__ __device__ inline ChiLayout chi_layout(int iters, size_t basis_elem, int rw) {
    auto up = [](size_t v) { return (v + 15) & ~size_t(15); };
    ChiLayout L;
    size_t o = 0;
    L.links = o;  o = up(o + (size_t)16 * 36 * sizeof(cplx<R>));
    L.clover = o; o = up(o + (size_t)16 * 72 * sizeof(R));
    L.shared = o;
    size_t w = 0;
    L.basis = w;  w = up(w + (size_t)(iters + 1) * 16 * 12 * basis_elem);
    L.H = w;      w = up(w + (size_t)(iters + 1) * iters * sizeof(cplx<R>));
    L.g = w;      w = up(w + (size_t)(iters + 1) * sizeof(cplx<R>));
    L.sn = w;     w = up(w + (size_t)iters * sizeof(cplx<R>));
    L.y = w;      w = up(w + (size_t)iters * sizeof(cplx<R>));
    L.cs = w;     w = up(w + (size_t)iters * sizeof(R));
    L.flag = w;   w = up(w + 4 * sizeof(int));
    L.perwarp = w;
    L.total = L.shared + (size_t)rw * w;
    return L;
}

template <int BS, typename T>
__device__ __forceinline__ T seg_sum(T v) {
#pragma unroll
    for (int o = BS / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <typename R, int BS>
__global__ void __launch_bounds__(32) sap_warp_kernel(Geom g, Blocking B, const cplx<R>* __restrict__ U,
                                                      const R* __restrict__ A, const int* __restrict__ blocks, int ncol,
                                                      int op, Shifts tau, const cplx<R>* __restrict__ r,
                                                      cplx<R>* __restrict__ x, int iters, double tol,
                                                      const int* __restrict__ act) {
    constexpr int SPW = 32 / BS;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int lane = threadIdx.x;
    const int seg = lane / BS, l = lane % BS;
    const SapSmemLayout LY = sap_layout<R>(BS, iters);
    unsigned char* base = smraw + (size_t)seg * LY.total;
    cplx<R>* basis = reinterpret_cast<cplx<R>*>(base + LY.basis);
    cplx<R>* slink = reinterpret_cast<cplx<R>*>(base + LY.links);
    R* sclov = reinterpret_cast<R*>(base + LY.clover);
    // Hessenberg bookkeeping by lane 0 in the working precision (a dependent
    // FP64 chain is very slow on this part)
    cplx<R>* H = reinterpret_cast<cplx<R>*>(base + LY.H);
    cplx<R>* gv = reinterpret_cast<cplx<R>*>(base + LY.g);
    cplx<R>* sn = reinterpret_cast<cplx<R>*>(base + LY.sn);
    cplx<R>* yv = reinterpret_cast<cplx<R>*>(base + LY.y);
    R* cs = reinterpret_cast<R*>(base + LY.cs);
    int* flag = reinterpret_cast<int*>(base + LY.flag);

    const int j = blockIdx.y;
    if (act != nullptr && !act[j]) return;
    const int bidx = blockIdx.x * SPW + seg;
    const bool valid = bidx < ncol;
    const int blk = valid ? blocks[bidx] : blocks[0];
    const size_t fstride = (size_t)g.V * 12;
    r += j * fstride;
    x += j * fstride;
    const R t = (R)tau.t[j];
    int o[4];
    {
        int tt = l;
        o[3] = tt % B.b[3]; tt /= B.b[3];
        o[2] = tt % B.b[2]; tt /= B.b[2];
        o[1] = tt % B.b[1]; o[0] = tt / B.b[1];
    }
    const int y = block_fine_site(g, B, blk, l);
    // stage links (forward, this site) and clover
#pragma unroll
    for (int k = 0; k < 36; ++k) slink[l * 36 + k] = __ldg(U + (size_t)y * 36 + k);
#pragma unroll 8
    for (int k = 0; k < 72; ++k) sclov[l * 72 + k] = __ldg(A + (size_t)y * 72 + k);
    Spinor<R> w;
    load_spinor<R>(r + (size_t)y * 12, w);
    R nn = 0;
#pragma unroll
    for (int k = 0; k < 12; ++k) nn += w.c[k].x * w.c[k].x + w.c[k].y * w.c[k].y;
    nn = seg_sum<BS>(nn);
    const R beta = valid ? sqrt(nn) : R(0);
    {
        const R ib = beta > R(0) ? R(1) / beta : R(0);
#pragma unroll
        for (int k = 0; k < 12; ++k) basis[l * 12 + k] = ib * w.c[k];
    }
    if (l == 0) { gv[0] = mk<R>(beta, R(0)); flag[0] = beta > R(0) ? 0 : 1; flag[1] = 0; }
    __syncwarp();
    int lstride[4];
    lstride[3] = 1;
    lstride[2] = B.b[3];
    lstride[1] = B.b[3] * B.b[2];
    lstride[0] = B.b[3] * B.b[2] * B.b[1];
    for (int jj = 0; jj < iters; ++jj) {
        const bool active = flag[0] == 0;
        if (__all_sync(0xffffffffu, !active)) break;
        const cplx<R>* vj = basis + (size_t)jj * BS * 12;
        // w = A_block v_j
        Spinor<R> psi, acc;
#pragma unroll
        for (int k = 0; k < 12; ++k) psi.c[k] = vj[l * 12 + k];
        clover_apply_smem<R>(sclov + l * 72, psi, acc);
        // Dirichlet block: per mu one neighbour inside the block on the
        // forward side if there is one, else on the backward side (a 2-site
        // extent has exactly one), taken by all lanes together; interior
        // sites of wider blocks add their backward neighbour afterwards
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
            Spinor<R> nb;
            Link<R> u;
            const bool fw = o[mu] < B.b[mu] - 1;
            if (fw || o[mu] > 0) {
                const int ln = fw ? l + lstride[mu] : l - lstride[mu];
#pragma unroll
                for (int k = 0; k < 12; ++k) nb.c[k] = vj[ln * 12 + k];
                const cplx<R>* lk = slink + (fw ? l : ln) * 36 + mu * 9;
#pragma unroll
                for (int k = 0; k < 9; ++k) u.e[k] = lk[k];
                switch (mu) {
                    case 0: hop_accumulate_dir<R, 0>(nb, u, R(1), fw, acc); break;
                    case 1: hop_accumulate_dir<R, 1>(nb, u, R(1), fw, acc); break;
                    case 2: hop_accumulate_dir<R, 2>(nb, u, R(1), fw, acc); break;
                    default: hop_accumulate_dir<R, 3>(nb, u, R(1), fw, acc); break;
                }
            }
            const bool both = fw && o[mu] > 0;
            if (__any_sync(0xffffffffu, both) && both) {
                const int ln = l - lstride[mu];
#pragma unroll
                for (int k = 0; k < 12; ++k) nb.c[k] = vj[ln * 12 + k];
#pragma unroll
                for (int k = 0; k < 9; ++k) u.e[k] = slink[ln * 36 + mu * 9 + k];
                switch (mu) {
                    case 0: hop_accumulate<R, 0, false>(nb, u, R(1), acc); break;
                    case 1: hop_accumulate<R, 1, false>(nb, u, R(1), acc); break;
                    case 2: hop_accumulate<R, 2, false>(nb, u, R(1), acc); break;
                    default: hop_accumulate<R, 3, false>(nb, u, R(1), acc); break;
                }
            }
        }
        if (op == QCD_OP_D) {
#pragma unroll
            for (int k = 0; k < 6; ++k) acc.c[k] -= t * psi.c[k];
#pragma unroll
            for (int k = 6; k < 12; ++k) acc.c[k] += t * psi.c[k];
        } else {
#pragma unroll
            for (int k = 0; k < 6; ++k) acc.c[k] -= t * psi.c[k];
#pragma unroll
            for (int k = 6; k < 12; ++k) acc.c[k] = -acc.c[k] - t * psi.c[k];
        }
        // modified Gram-Schmidt against v_0 .. v_jj
        for (int i = 0; i <= jj; ++i) {
            const cplx<R>* vi = basis + (size_t)i * BS * 12 + l * 12;
            R hr = 0, hi = 0;
#pragma unroll
            for (int k = 0; k < 12; ++k) {
                cdot(hr, hi, vi[k], acc.c[k]);
            }
            hr = seg_sum<BS>(hr);
            hi = seg_sum<BS>(hi);
            const cplx<R> h = mk<R>(hr, hi);
#pragma unroll
            for (int k = 0; k < 12; ++k) cmsub(acc.c[k], h, vi[k]);
            if (l == 0 && active) H[i * iters + jj] = mk<R>(hr, hi);
        }
        R hn2 = 0;
#pragma unroll
        for (int k = 0; k < 12; ++k) hn2 += acc.c[k].x * acc.c[k].x + acc.c[k].y * acc.c[k].y;
        hn2 = seg_sum<BS>(hn2);
        const R hn = sqrt(hn2);
        {
            const R ih = hn > R(0) ? R(1) / hn : R(0);
            cplx<R>* vn = basis + (size_t)(jj + 1) * BS * 12 + l * 12;
#pragma unroll
            for (int k = 0; k < 12; ++k) vn[k] = ih * acc.c[k];
        }
        if (l == 0 && active) {
            H[(jj + 1) * iters + jj] = mk<R>(hn, R(0));
            for (int i = 0; i < jj; ++i) {
                cplx<R> a = H[i * iters + jj], c = H[(i + 1) * iters + jj];
                H[i * iters + jj] = cs[i] * a + sn[i] * c;
                H[(i + 1) * iters + jj] = cs[i] * c - conj(sn[i]) * a;
            }
            cplx<R> a = H[jj * iters + jj];
            cplx<R> c = H[(jj + 1) * iters + jj];
            R aa = sqrt(a.x * a.x + a.y * a.y), rr = sqrt(aa * aa + c.x * c.x + c.y * c.y);
            if (aa > R(0)) {
                cs[jj] = aa / rr;
                sn[jj] = (R(1) / rr) * ((R(1) / aa) * a * conj(c));
            } else {
                cs[jj] = R(0);
                sn[jj] = mk<R>(R(1), R(0));
            }
            H[jj * iters + jj] = cs[jj] * a + sn[jj] * c;
            gv[jj + 1] = R(-1) * (conj(sn[jj]) * gv[jj]);
            gv[jj] = cs[jj] * gv[jj];
            const R res = sqrt(gv[jj + 1].x * gv[jj + 1].x + gv[jj + 1].y * gv[jj + 1].y);
            flag[1] = jj + 1;
            if (tol >= 0.0 && (double)res <= tol * (double)beta) flag[0] = 1;
        }
        __syncwarp();
    }
    const int kdim = flag[1];
    if (l == 0) {
        if (valid) count_sap_work(BS, kdim);
        for (int i = kdim - 1; i >= 0; --i) {
            cplx<R> sacc = gv[i];
            for (int k = i + 1; k < kdim; ++k) sacc -= H[i * iters + k] * yv[k];
            cplx<R> dd = H[i * iters + i];
            R den = dd.x * dd.x + dd.y * dd.y;
            yv[i] = den > R(0) ? (R(1) / den) * cmulc(dd, sacc) : mk<R>(R(0), R(0));
        }
    }
    __syncwarp();
    if (!valid || kdim == 0) return;
    Spinor<R> e;
    load_spinor<R>(x + (size_t)y * 12, e);
    for (int i = 0; i < kdim; ++i) {
        const cplx<R> yi = yv[i];
        const cplx<R>* vi = basis + (size_t)i * BS * 12 + l * 12;
#pragma unroll
        for (int k = 0; k < 12; ++k) cmac(e.c[k], yi, vi[k]);
    }
    store_spinor<R>(x + (size_t)y * 12, e);
}

// Storage of the SAP block Krylov basis: the working precision, or FP16
// pairs for FP32 solves (the basis then takes half the shared memory, so more
// block solves are resident per SM; the block solves only need a 1e-1
// reduction).
__device__ __forceinline__ float2 bload(const float2* p) { return *p; }
__device__ __forceinline__ double2 bload(const double2* p) { return *p; }
__device__ __forceinline__ float2 bload(const __half2* p) { return __half22float2(*p); }
__device__ __forceinline__ void bstore(float2* p, float2 v) { *p = v; }
__device__ __forceinline__ void bstore(double2* p, double2 v) { *p = v; }
__device__ __forceinline__ void bstore(__half2* p, float2 v) { *p = __float22half2_rn(v); }

// the value a stored entry reads back as
template <typename BT> __device__ __forceinline__ float2 bround(float2 v) {
    if constexpr (sizeof(BT) == 4) return __half22float2(__float22half2_rn(v));
    else return v;
}
template <typename BT> __device__ __forceinline__ double2 bround(double2 v) { return v; }

// Copy N 16-byte words from global to shared memory with all N loads in
// flight before the first store (staging without a round trip per word).
template <int N>
__device__ __forceinline__ void stage16(void* __restrict__ dst, const void* __restrict__ src) {
    const int4* s4 = reinterpret_cast<const int4*>(src);
    int4* d4 = reinterpret_cast<int4*>(dst);
    int4 v[N];
#pragma unroll
    for (int q = 0; q < N; ++q) v[q] = __ldg(s4 + q);
#pragma unroll
    for (int q = 0; q < N; ++q) d4[q] = v[q];
}

// SAP block solve for 16-site blocks with two lanes per site: lane
// chi * 16 + l holds chirality half chi (spins 2chi, 2chi+1) of site l, so one
// warp solves one block.  The clover term is block diagonal in chirality; in a
// hop each lane forms the projected half-spinor h_s for s = chi, multiplies it
// by the link (9 complex products instead of 18) and takes the other s from
// the partner lane (lane ^ 16) before it reconstructs its own half.  Same
// GMRES as sap_warp_kernel (modified Gram-Schmidt, Givens by lane 0).
template <typename R, typename BT>
__global__ void __launch_bounds__(128) sap_chi_kernel(Geom g, Blocking B, const cplx<R>* __restrict__ U,
                                                      const R* __restrict__ A, const int* __restrict__ blocks,
                                                      int ncol, int op, Shifts tau, const cplx<R>* __restrict__ r,
                                                      cplx<R>* __restrict__ x, int iters, double tol,
                                                      const int* __restrict__ act, int nrhs) {
    constexpr int BS = 16;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, rw = blockDim.x >> 5;
    const int chi = lane >> 4, l = lane & 15;
    const ChiLayout LY = chi_layout<R>(iters, sizeof(BT), rw);
    unsigned char* wbase = smraw + LY.shared + (size_t)wid * LY.perwarp;
    BT* basis = reinterpret_cast<BT*>(wbase + LY.basis);
    cplx<R>* slink = reinterpret_cast<cplx<R>*>(smraw + LY.links);
    R* sclov = reinterpret_cast<R*>(smraw + LY.clover);
    cplx<R>* H = reinterpret_cast<cplx<R>*>(wbase + LY.H);
    cplx<R>* gv = reinterpret_cast<cplx<R>*>(wbase + LY.g);
    cplx<R>* sn = reinterpret_cast<cplx<R>*>(wbase + LY.sn);
    cplx<R>* yv = reinterpret_cast<cplx<R>*>(wbase + LY.y);
    R* cs = reinterpret_cast<R*>(wbase + LY.cs);
    int* flag = reinterpret_cast<int*>(wbase + LY.flag);

    // warp w of the CTA solves the block for right-hand side blockIdx.y * rw + w;
    // the block's links and clover are staged once for all of them
    const int j = blockIdx.y * rw + wid;
    const int blk = blocks[blockIdx.x];
    int o[4];
    {
        int tt = l;
        o[3] = tt % B.b[3]; tt /= B.b[3];
        o[2] = tt % B.b[2]; tt /= B.b[2];
        o[1] = tt % B.b[1]; o[0] = tt / B.b[1];
    }
    const int y = block_fine_site(g, B, blk, l);
    // stage links and clover of the 16 sites (warp 0): lane chi copies half
    // of its site's links and its own chirality block of the clover term
    // (16-byte words, every load in flight at once)
    constexpr int kHalf = 18 * (int)sizeof(cplx<R>) / 16;   // 16-byte words in 18 complex / 36 reals
    if (wid == 0) {
        stage16<kHalf>(slink + l * 36 + 18 * chi, U + (size_t)y * 36 + 18 * chi);
        stage16<kHalf>(sclov + l * 72 + 36 * chi, A + (size_t)y * 72 + 36 * chi);
    }
    const bool mine = j < nrhs && (act == nullptr || act[j]);
    const size_t fstride = (size_t)g.V * 12;
    cplx<R> w[6];
    if (mine) {
        r += j * fstride;
        x += j * fstride;
#pragma unroll
        for (int k = 0; k < 6; ++k) w[k] = __ldg(r + (size_t)y * 12 + 6 * chi + k);
    }
    __syncthreads();
    if (!mine) return;
    const R t = (R)tau.t[j];
    R nn = 0;
#pragma unroll
    for (int k = 0; k < 6; ++k) nn += w[k].x * w[k].x + w[k].y * w[k].y;
    nn = warp_sum(nn);
    const R beta = sqrt(nn);
    {
        const R ib = beta > R(0) ? R(1) / beta : R(0);
#pragma unroll
        for (int k = 0; k < 6; ++k) bstore(basis + l * 12 + 6 * chi + k, ib * w[k]);
    }
    if (lane == 0) { gv[0] = mk<R>(beta, R(0)); flag[0] = beta > R(0) ? 0 : 1; flag[1] = 0; }
    __syncwarp();
    int lstride[4];
    lstride[3] = 1;
    lstride[2] = B.b[3];
    lstride[1] = B.b[3] * B.b[2];
    lstride[0] = B.b[3] * B.b[2] * B.b[1];
    for (int jj = 0; jj < iters; ++jj) {
        const bool active = flag[0] == 0;
        if (!active) break;   // flag is shared by the whole warp
        const BT* vj = basis + (size_t)jj * BS * 12;
        cplx<R> psi[6], acc[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) psi[k] = bload(vj + l * 12 + 6 * chi + k);
        // clover block chi of site l
        {
            const R* a = sclov + l * 72 + 36 * chi;
#pragma unroll
            for (int i = 0; i < 6; ++i) acc[i] = a[i] * psi[i];
#pragma unroll
            for (int i = 0; i < 6; ++i) {
#pragma unroll
                for (int jc = i + 1; jc < 6; ++jc) {
                    const int oo = herm_off(i, jc);
                    const cplx<R> aij = mk<R>(a[oo], a[oo + 1]);
                    cmac(acc[i], aij, psi[jc]);
                    cmacc(acc[jc], aij, psi[i]);
                }
            }
        }
        // hops inside the block (Dirichlet): per mu the forward neighbour if it
        // is inside, else the backward one; interior sites of wider blocks
        // add their backward neighbour in a second round
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
            const SpinMono Bm = kB(mu), BHm = kBH(mu);
            for (int round = 0; round < 2; ++round) {
                const bool fw = round == 0 ? (o[mu] < B.b[mu] - 1) : false;
                const bool has = round == 0 ? (fw || o[mu] > 0) : (o[mu] < B.b[mu] - 1 && o[mu] > 0);
                if (round == 1 && !__any_sync(0xffffffffu, has)) break;
                const int ln = has ? (fw ? l + lstride[mu] : l - lstride[mu]) : l;
                const BT* nb = vj + ln * 12;
                const R pm = fw ? R(-1) : R(1);
                // h_s for s = chi: up_s + pm i^{ph_s} dn_{perm_s}
                const int sp = Bm.perm[chi], ph = Bm.ph[chi];
                cplx<R> h[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) h[a] = bload(nb + chi * 3 + a) + pm * mul_ipow(bload(nb + (2 + sp) * 3 + a), ph);
                const cplx<R>* lk = slink + (fw ? l : ln) * 36 + mu * 9;
                cplx<R> os[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    cplx<R> v = czero<R>();
#pragma unroll
                    for (int b = 0; b < 3; ++b) cmac(v, fw ? lk[a * 3 + b] : conj(lk[b * 3 + a]), h[b]);
                    os[a] = has ? v : czero<R>();
                }
                cplx<R> ot[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    ot[a].x = __shfl_xor_sync(0xffffffffu, os[a].x, 16);
                    ot[a].y = __shfl_xor_sync(0xffffffffu, os[a].y, 16);
                }
                // o[0], o[1] of the site; reconstruct this lane's half
                const R half = R(-0.5);
#pragma unroll
                for (int s2 = 0; s2 < 2; ++s2) {
                    const int src = chi ? BHm.perm[s2] : s2;
                    const int php = chi ? BHm.ph[s2] : 0;
                    const R c = chi ? pm * half : half;
                    const bool mine = src == chi;
#pragma unroll
                    for (int a = 0; a < 3; ++a) acc[s2 * 3 + a] += c * mul_ipow(mine ? os[a] : ot[a], php);
                }
            }
        }
        // shift: D - tau Gamma5 (op D) or Gamma5 D - tau (op Q)
        {
            const R g5 = chi ? R(-1) : R(1);
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                if (op == QCD_OP_D) acc[k] -= (t * g5) * psi[k];
                else acc[k] = g5 * acc[k] - t * psi[k];
            }
        }
        // modified Gram-Schmidt against v_0 .. v_jj
        for (int i = 0; i <= jj; ++i) {
            const BT* vi = basis + (size_t)i * BS * 12 + l * 12 + 6 * chi;
            R hr = 0, hi = 0;
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                cdot(hr, hi, bload(vi + k), acc[k]);
            }
            hr = warp_sum(hr);
            hi = warp_sum(hi);
            const cplx<R> h = mk<R>(hr, hi);
#pragma unroll
            for (int k = 0; k < 6; ++k) cmsub(acc[k], h, bload(vi + k));
            if (lane == 0) H[i * iters + jj] = h;
        }
        R hn2 = 0;
#pragma unroll
        for (int k = 0; k < 6; ++k) hn2 += acc[k].x * acc[k].x + acc[k].y * acc[k].y;
        hn2 = warp_sum(hn2);
        const R hn = sqrt(hn2);
        {
            const R ih = hn > R(0) ? R(1) / hn : R(0);
            BT* vn = basis + (size_t)(jj + 1) * BS * 12 + l * 12 + 6 * chi;
#pragma unroll
            for (int k = 0; k < 6; ++k) bstore(vn + k, ih * acc[k]);
        }
        if (lane == 0) {
            H[(jj + 1) * iters + jj] = mk<R>(hn, R(0));
            for (int i = 0; i < jj; ++i) {
                cplx<R> a = H[i * iters + jj], c = H[(i + 1) * iters + jj];
                H[i * iters + jj] = cs[i] * a + sn[i] * c;
                H[(i + 1) * iters + jj] = cs[i] * c - conj(sn[i]) * a;
            }
            cplx<R> a = H[jj * iters + jj];
            cplx<R> c = H[(jj + 1) * iters + jj];
            R aa = sqrt(a.x * a.x + a.y * a.y), rr = sqrt(aa * aa + c.x * c.x + c.y * c.y);
            if (aa > R(0)) {
                cs[jj] = aa / rr;
                sn[jj] = (R(1) / rr) * ((R(1) / aa) * a * conj(c));
            } else {
                cs[jj] = R(0);
                sn[jj] = mk<R>(R(1), R(0));
            }
            H[jj * iters + jj] = cs[jj] * a + sn[jj] * c;
            gv[jj + 1] = R(-1) * (conj(sn[jj]) * gv[jj]);
            gv[jj] = cs[jj] * gv[jj];
            const R res = sqrt(gv[jj + 1].x * gv[jj + 1].x + gv[jj + 1].y * gv[jj + 1].y);
            flag[1] = jj + 1;
            if (tol >= 0.0 && (double)res <= tol * (double)beta) flag[0] = 1;
        }
        __syncwarp();
    }
    const int kdim = flag[1];
    if (lane == 0) {
        count_sap_work(BS, kdim);
        for (int i = kdim - 1; i >= 0; --i) {
            cplx<R> sacc = gv[i];
            for (int k = i + 1; k < kdim; ++k) sacc -= H[i * iters + k] * yv[k];
            cplx<R> dd = H[i * iters + i];
            R den = dd.x * dd.x + dd.y * dd.y;
            yv[i] = den > R(0) ? (R(1) / den) * cmulc(dd, sacc) : mk<R>(R(0), R(0));
        }
    }
    __syncwarp();
    if (kdim == 0) return;
    cplx<R> e[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) e[k] = x[(size_t)y * 12 + 6 * chi + k];
    for (int i = 0; i < kdim; ++i) {
        const cplx<R> yi = yv[i];
        const BT* vi = basis + (size_t)i * BS * 12 + l * 12 + 6 * chi;
#pragma unroll
        for (int k = 0; k < 6; ++k) cmac(e[k], yi, bload(vi + k));
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) x[(size_t)y * 12 + 6 * chi + k] = e[k];
}

#include "sap_cube.cuh"

inline int grid_for(size_t n, int th = 256) {
    size_t gsz = (n + th - 1) / th;
    return (int)(gsz > 1048576 ? 1048576 : (gsz == 0 ? 1 : gsz));
}

}  // namespace

// ------------------------------------------------------------------ host launchers
void mg_build_P(const FineOp& f, Coarse& c, const double2* vecs, int nvec, cudaStream_t st) {
    dim3 grid(c.B.nb, 2);
    KTimer kt("build_P", 0.0, 0.0, st);
    // up to 48 KB of vectors (four CTAs per SM) in shared memory
    const size_t sm = sizeof(double2) * (size_t)nvec * c.B.bs * 6;
    const int in_smem = sm <= 48 * 1024;
    build_P_kernel<<<grid, 256, in_smem ? sm : 0, st>>>(f.g, c.B, nvec, vecs, c.P64, c.P32, in_smem);
}

void mg_build_coarse(const FineOp& f, Coarse& c, cudaStream_t st, bool fp32_only) {
    dim3 grid(c.B.nb, 9);
    // columns per pass: h of a pass within about 96 KB of shared memory
    const size_t es = fp32_only ? sizeof(float2) : sizeof(double2);
    const size_t per_col = (size_t)c.B.bs * 12 * es;
    const int chunk = (int)std::max<size_t>(1, std::min<size_t>(c.nc, (96u << 10) / per_col));
    const size_t sm = chunk * per_col + (size_t)c.B.bs * sizeof(int);
    if (fp32_only) {
        // the FP32 operator straight from P32, U32 and the FP32 clover; the
        // FP64 one is rebuilt on demand (Coarse::a64_stale)
        if (sm + 1024 > 48 * 1024)
            cudaFuncSetAttribute(build_coarse_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        KTimer kt("build_coarse_f32", 0.0, 0.0, st);
        build_coarse_kernel<float><<<grid, 256, sm, st>>>(f.g, c.B, c.nv, f.U32, f.A32, c.P32, c.A32, chunk);
        c.a64_stale = true;
        return;
    }
    if (sm + 1024 > 48 * 1024)
        cudaFuncSetAttribute(build_coarse_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    KTimer kt("build_coarse", 0.0, 0.0, st);
    build_coarse_kernel<double><<<grid, 256, sm, st>>>(f.g, c.B, c.nv, f.U64, f.A64, c.P64, c.A64, chunk);
    size_t n = (size_t)c.B.nb * 9 * c.nc * c.nc;
    KTimer kt2("narrow", (double)n * 24, 0.0, st);
    narrow_kernel<<<grid_for(n), 256, 0, st>>>(c.A64, c.A32, n);
    c.a64_stale = false;
}

template <typename R, int E, int TI, int TJ>
static void launch_restrict(const FineOp& f, const Coarse& c, int nrhs, int chunk, const cplx<R>* P, const void* r,
                            void* xc, cudaStream_t st, const int* act) {
    const int warps = (c.nv + TI - 1) / TI * ((chunk + TJ - 1) / TJ);
    const dim3 grid(c.B.nb * 2, (nrhs + chunk - 1) / chunk);
    const int ring = std::min(kRing, (c.B.bs * 6 / E + kStage - 1) / kStage);   // no more stages than there are
    const size_t sm = (size_t)ring * (c.nv + chunk) * kStage * sizeof(Piece<R, E>) +
                      (c.B.bs <= kSiteTable ? c.B.bs * 6 / E * sizeof(int) : 0);
    auto kern = restrict_tile_kernel<R, E, TI, TJ>;
    if (sm > 48 * 1024) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    kern<<<grid, 32 * warps, sm, st>>>(f.g, c.B, c.nv, P, (const cplx<R>*)r, (cplx<R>*)xc, nrhs, chunk, ring, act);
}
template <typename R, int E, int TJ>
static void launch_prolong(const FineOp& f, const Coarse& c, int nrhs, const cplx<R>* P, const void* xc, void* x,
                           cudaStream_t st, const int* act) {
    constexpr int per = (sizeof(R) == 8 ? 1 : 2) * kProlongT;   // pieces per CTA
    const int parts = (c.B.bs * 12 / E + per - 1) / per;
    const unsigned grid = (unsigned)c.B.nb * parts * ((nrhs + TJ - 1) / TJ);
    const size_t sm = sizeof(Piece<R, E>) * kAhead * per + 2 * (size_t)((c.nv + (c.nv & 1)) * TJ + 2) * sizeof(cplx<R>);
    prolong_tile_kernel<R, E, TJ><<<grid, kProlongT, sm, st>>>(f.g, c.B, c.nv, P, (const cplx<R>*)xc, (cplx<R>*)x, nrhs,
                                                               parts, act);
}

// FP32 tiles as wide as the right-hand sides fill, at most TJ.  Four wide while the
// warps of 16 right-hand sides (ceil(nv / 4) x 4) fit the 640 threads of that launch
// bound, nv <= 20; eight wide, with half the warps, beyond.
template <int E, int TJ>
static void restrict_width(const FineOp& f, const Coarse& c, int nrhs, const void* r, void* xc, cudaStream_t st,
                           const int* act) {
    if constexpr (TJ > 1)
        if (2 * nrhs <= TJ || (TJ == 8 && c.nv <= 20)) return restrict_width<E, TJ / 2>(f, c, nrhs, r, xc, st, act);
    launch_restrict<float, E, 4, TJ>(f, c, nrhs, std::min(nrhs, kTransferRhs<float>), c.P32, r, xc, st, act);
}
template <int E, int TJ>
static void prolong_width(const FineOp& f, const Coarse& c, int nrhs, const void* xc, void* x, cudaStream_t st,
                          const int* act) {
    if constexpr (TJ > 1)
        if (2 * nrhs <= TJ) return prolong_width<E, TJ / 2>(f, c, nrhs, xc, x, st, act);
    launch_prolong<float, E, TJ>(f, c, nrhs, c.P32, xc, x, st, act);
}
// FP64: fewer right-hand sides per CTA until two waves of CTAs are there, then the
// smallest tile whose warps fit its launch bound.  With 4 x 4 tiles and chunks of eight
// (restriction) or four right-hand sides and two pieces per thread (prolongation) five
// vectors and three right-hand sides took 140 us on 16 x 8^3 with 4^4 aggregates (one
// warp per vector before: 72) and 18 us on 12 x 6^3 with 3^4 (12); now 27 and 9.  16^4,
// 4^4 aggregates, nv 20, 8 right-hand sides: 943 and 845 us.
static void restrict_f64(const FineOp& f, const Coarse& c, int nrhs, const void* r, void* xc, cudaStream_t st,
                         const int* act) {
    int chunk = std::min(nrhs, kTransferRhs<double>);
    while (chunk > 1 && 2 * c.B.nb * ((nrhs + chunk - 1) / chunk) < 2 * coarse_gmres_grid()) chunk = (chunk + 1) / 2;
    const int nv = c.nv;
    if (nv * chunk <= 32) launch_restrict<double, 1, 1, 1>(f, c, nrhs, chunk, c.P64, r, xc, st, act);
    else if ((nv + 1) / 2 * chunk <= 32) launch_restrict<double, 1, 2, 1>(f, c, nrhs, chunk, c.P64, r, xc, st, act);
    else if ((nv + 3) / 4 * chunk <= 24) launch_restrict<double, 1, 4, 1>(f, c, nrhs, chunk, c.P64, r, xc, st, act);
    else launch_restrict<double, 1, 4, 2>(f, c, nrhs, chunk, c.P64, r, xc, st, act);
}

void mg_restrict(const FineOp& f, const Coarse& c, int prec, int nrhs, const void* r, void* xc, cudaStream_t st,
                 const int* act) {
    const double es = prec == QCD_FP64 ? 16.0 : 8.0;
    const double nfine = (double)f.g.V * 12;
    const int per = prec == QCD_FP64 ? kTransferRhs<double> : kTransferRhs<float>;
    KTimer kt(prec == QCD_FP64 ? "restrict_f64" : "restrict_f32",
              es * (nfine * c.nv * ((nrhs + per - 1) / per) + nrhs * (nfine + (double)c.gc.V * c.nc)),
              8.0 * nfine * c.nv * nrhs, st);
    if (prec == QCD_FP64) restrict_f64(f, c, nrhs, r, xc, st, act);
    else if ((uintptr_t)r & 15) restrict_width<1, 8>(f, c, nrhs, r, xc, st, act);
    else restrict_width<2, 8>(f, c, nrhs, r, xc, st, act);
}

void mg_prolong(const FineOp& f, const Coarse& c, int prec, int nrhs, const void* xc, void* x, cudaStream_t st,
                const int* act) {
    const double es = prec == QCD_FP64 ? 16.0 : 8.0;
    const double nfine = (double)f.g.V * 12;
    const int per = prec == QCD_FP64 ? kTransferRhs<double> : kTransferRhs<float>;
    KTimer kt(prec == QCD_FP64 ? "prolong_f64" : "prolong_f32",
              es * (nfine * c.nv * ((nrhs + per - 1) / per) + nrhs * (nfine + (double)c.gc.V * c.nc)),
              8.0 * nfine * c.nv * nrhs, st);
    if (prec == QCD_FP64 && nrhs % 2) launch_prolong<double, 1, 1>(f, c, nrhs, c.P64, xc, x, st, act);
    else if (prec == QCD_FP64) launch_prolong<double, 1, 2>(f, c, nrhs, c.P64, xc, x, st, act);
    else if ((uintptr_t)x & 15) prolong_width<1, 8>(f, c, nrhs, xc, x, st, act);
    else prolong_width<2, 8>(f, c, nrhs, xc, x, st, act);
}

void coarse_apply(const Coarse& c, int prec, int op, int nrhs, const void* x, void* y, const double* tau,
                  cudaStream_t st, bool tensor) {
    Shifts sh{};
    for (int j = 0; j < nrhs; ++j) sh.t[j] = tau ? tau[j] : 0.0;
    const double es = prec == QCD_FP64 ? 16.0 : 8.0;
    const bool tc = prec == QCD_FP32 && tensor && c.nc % 8 == 0 && c.nc <= 64;
    // staged kernel: FP32, 16-byte aligned vectors (faster than the general one at
    // every size measured, Nv 2 .. 24, 1 .. 20 right-hand sides, 16 to 4096 sites)
    const bool staged = prec == QCD_FP32 && !tc && c.nc <= 64 && ((uintptr_t)x & 15) == 0 &&
                      ((uintptr_t)c.A32 & 15) == 0;
    const int rchunk = tc ? kTcR : 16;
    KTimer kt(prec == QCD_FP64 ? "coarse_apply_f64"
                               : (tc ? "coarse_apply_tc" : (staged ? "coarse_apply_bulk" : "coarse_apply_f32")),
              es * ((double)c.gc.V * 9 * c.nc * c.nc * ((nrhs + rchunk - 1) / rchunk) +
                    2.0 * nrhs * c.gc.V * c.nc),
              8.0 * 9 * c.nc * c.nc * (double)c.gc.V * nrhs, st);
    if (staged) {
        const int rows = (c.nc + 15) / 16;
        const float2* xf = (const float2*)x;
        if (rows == 1) coarse_staged_rows<1>(c, op, nrhs, xf, (float2*)y, sh, st);
        else if (rows == 2) coarse_staged_rows<2>(c, op, nrhs, xf, (float2*)y, sh, st);
        else if (rows == 3) coarse_staged_rows<3>(c, op, nrhs, xf, (float2*)y, sh, st);
        else coarse_staged_rows<4>(c, op, nrhs, xf, (float2*)y, sh, st);
        return;
    }
    if (prec == QCD_FP32 && tensor && c.nc % 8 == 0 && c.nc <= 64) {
        const size_t sm = coarse_tc_smem(c.nc);
        if (sm + 1024 > 48 * 1024)
            cudaFuncSetAttribute(coarse_apply_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        const dim3 grid(c.gc.V, (nrhs + kTcR - 1) / kTcR);
        coarse_apply_tc_kernel<<<grid, 32 * (c.nc / 8), sm, st>>>(c.gc, c.nc, c.A32, (const float2*)x, (float2*)y,
                                                                  op, sh, nrhs);
        return;
    }
    // right-hand sides per CTA: a multiple of kCoarseRPT, at most kCoarseRC
    const int rc = std::min(kCoarseRC, (nrhs + kCoarseRPT - 1) / kCoarseRPT * kCoarseRPT);
    const dim3 grid(c.gc.V, (nrhs + rc - 1) / rc);
    const int threads = c.nc * (rc / kCoarseRPT);
    const size_t ebytes = prec == QCD_FP64 ? sizeof(double2) : sizeof(float2);
    const size_t sm = (size_t)9 * c.nc * rc * ebytes;
    if (prec == QCD_FP64) {
        if (sm + 1024 > 48 * 1024)
            cudaFuncSetAttribute(coarse_apply_mrhs_kernel<double2, double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sm);
        coarse_apply_mrhs_kernel<double2, double><<<grid, threads, sm, st>>>(c.gc, c.nc, c.A64, (const double2*)x,
                                                                            (double2*)y, op, sh, nrhs, rc);
    } else {
        if (sm + 1024 > 48 * 1024)
            cudaFuncSetAttribute(coarse_apply_mrhs_kernel<float2, float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sm);
        coarse_apply_mrhs_kernel<float2, float><<<grid, threads, sm, st>>>(c.gc, c.nc, c.A32, (const float2*)x,
                                                                          (float2*)y, op, sh, nrhs, rc);
    }
}

bool sap_forms_residual(const Blocking& B) { return B.b[0] == 2 && B.b[1] == 2 && B.b[2] == 2 && B.b[3] == 2; }

// Launch of sap_cube_kernel: rw right-hand sides (warps) share a CTA and its
// staged links, as few CTAs per block as hold at most four, evenly filled
// (5 right-hand sides: 3 + 2), fewer when the bases of many steps do not fit.
template <typename R, typename BT>
static void launch_cube(const FineOp& f, const SapPlan& sp, int colour, int op, int nrhs, const void* b, void* x,
                        const Shifts& sh, int iters, double tol, cudaStream_t st, const int* act) {
    int rw = (nrhs + 3) / 4;
    rw = (nrhs + rw - 1) / rw;
    while (rw > 1 && cube_layout<R, BT>(iters, rw).total > 226 * 1024) --rw;
    const size_t sm = cube_layout<R, BT>(iters, rw).total;
    if (sm + 1024 > 48 * 1024)
        cudaFuncSetAttribute(sap_cube_kernel<R, BT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    const dim3 grid(sp.ncol[colour], (nrhs + rw - 1) / rw);
    const bool dp = sizeof(R) == 8;
    sap_cube_kernel<R, BT><<<grid, 32 * rw, sm, st>>>(f.g, sp.B, dp ? (const cplx<R>*)f.U64 : (const cplx<R>*)f.U32,
                                                      dp ? (const R*)f.A64 : (const R*)f.A32,
                                                      sp.blocks_of_colour[colour], op, sh, (const cplx<R>*)b,
                                                      (cplx<R>*)x, iters, tol, act, nrhs);
}

bool sap_needs_scratch(const Blocking& B) { return B.bs != 16 && B.bs != 32; }

void sap_work_reset() {
    static const unsigned long long zero[2][64] = {};
    cudaMemcpyToSymbol(g_sap_work, zero, sizeof(zero));
}
void wait_probe(cudaStream_t st) {
    KTimer kt("wait_probe", 0.0, 0.0, st);
    wait_probe_kernel<<<1, 32, 0, st>>>(1ll << 21);
}

unsigned long long wait_timeouts_read() {
    unsigned long long h = 0;
    cudaMemcpyFromSymbol(&h, g_wait_timeouts, sizeof(h));
    return h;
}

void sap_work_read(double out[2]) {
    unsigned long long h[2][64];
    cudaMemcpyFromSymbol(h, g_sap_work, sizeof(h));
    out[0] = out[1] = 0.0;
    for (int i = 0; i < 64; ++i) {
        out[0] += (double)h[0][i];
        out[1] += (double)h[1][i];
    }
}

size_t sap_scratch_bytes(const SapPlan& sp, int prec, int nrhs, int iters) {
    if (!sap_needs_scratch(sp.B)) return 0;
    size_t per = (size_t)(iters + 1) * sp.B.bs * 12 * (prec == QCD_FP64 ? sizeof(double2) : sizeof(float2));
    int nmax = sp.ncol[0] > sp.ncol[1] ? sp.ncol[0] : sp.ncol[1];
    return per * nmax * nrhs;
}

void sap_blocks(const FineOp& f, const SapPlan& sp, int colour, int prec, int op, int nrhs, const void* r, void* x,
                const double* tau, int iters, double tol, void* scratch, cudaStream_t st, const int* act, bool half) {
    Shifts sh{};
    for (int j = 0; j < nrhs; ++j) sh.t[j] = tau ? tau[j] : 0.0;
    const int bs = sp.B.bs;
    const double rs = prec == QCD_FP64 ? 8.0 : 4.0;
    const double sites = (double)sp.ncol[colour] * bs;
    if (sap_forms_residual(sp.B)) {
        // b, x in and out, x of the other colour, links of both colours, clover
        KTimer kt(prec == QCD_FP64 ? "sap_block_f64" : (half ? "sap_block_f32h" : "sap_block_f32"),
                  rs * sites * (nrhs * 96.0 + 216.0), 1824.0 * sites * nrhs * (iters + 1), st);
        if (prec == QCD_FP64)
            launch_cube<double, double2>(f, sp, colour, op, nrhs, r, x, sh, iters, tol, st, act);
        else if (half)
            launch_cube<float, __half2>(f, sp, colour, op, nrhs, r, x, sh, iters, tol, st, act);
        else
            launch_cube<float, float2>(f, sp, colour, op, nrhs, r, x, sh, iters, tol, st, act);
        return;
    }
    KTimer kt(prec == QCD_FP64 ? "sap_block_f64" : (half && bs == 16 ? "sap_block_f32h" : "sap_block_f32"),
              rs * sites * (nrhs * 72.0 + 144.0),
              1824.0 * sites * nrhs * iters, st);
    if (bs == 16) {
        // one warp per block solve; with four or more right-hand sides four
        // of them share a CTA (and one staged copy of the block's links and
        // clover), so more block solves fit in shared memory per SM
        const int rw = nrhs >= 4 ? 4 : 1;
        dim3 grid(sp.ncol[colour], (nrhs + rw - 1) / rw);
        if (prec == QCD_FP64) {
            const size_t sm = chi_layout<double>(iters, sizeof(double2), rw).total;
            if (sm + 1024 > 48 * 1024)
                cudaFuncSetAttribute(sap_chi_kernel<double, double2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sm);
            sap_chi_kernel<double, double2><<<grid, 32 * rw, sm, st>>>(f.g, sp.B, f.U64, f.A64,
                sp.blocks_of_colour[colour], sp.ncol[colour], op, sh, (const double2*)r, (double2*)x, iters, tol,
                act, nrhs);
        } else if (half) {
            const size_t sm = chi_layout<float>(iters, sizeof(__half2), rw).total;
            if (sm + 1024 > 48 * 1024)
                cudaFuncSetAttribute(sap_chi_kernel<float, __half2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sm);
            sap_chi_kernel<float, __half2><<<grid, 32 * rw, sm, st>>>(f.g, sp.B, f.U32, f.A32,
                sp.blocks_of_colour[colour], sp.ncol[colour], op, sh, (const float2*)r, (float2*)x, iters, tol,
                act, nrhs);
        } else {
            const size_t sm = chi_layout<float>(iters, sizeof(float2), rw).total;
            if (sm + 1024 > 48 * 1024)
                cudaFuncSetAttribute(sap_chi_kernel<float, float2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sm);
            sap_chi_kernel<float, float2><<<grid, 32 * rw, sm, st>>>(f.g, sp.B, f.U32, f.A32,
                sp.blocks_of_colour[colour], sp.ncol[colour], op, sh, (const float2*)r, (float2*)x, iters, tol,
                act, nrhs);
        }
        return;
    }
    if (bs == 32) {
        // one 32-site block per single-warp CTA
        dim3 grid(sp.ncol[colour], nrhs);
        if (prec == QCD_FP64) {
            const size_t sm = sap_layout<double>(32, iters).total;
            if (sm + 1024 > 48 * 1024) cudaFuncSetAttribute(sap_warp_kernel<double, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
            sap_warp_kernel<double, 32><<<grid, 32, sm, st>>>(f.g, sp.B, f.U64, f.A64, sp.blocks_of_colour[colour],
                sp.ncol[colour], op, sh, (const double2*)r, (double2*)x, iters, tol, act);
        } else {
            const size_t sm = sap_layout<float>(32, iters).total;
            if (sm + 1024 > 48 * 1024) cudaFuncSetAttribute(sap_warp_kernel<float, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
            sap_warp_kernel<float, 32><<<grid, 32, sm, st>>>(f.g, sp.B, f.U32, f.A32, sp.blocks_of_colour[colour],
                sp.ncol[colour], op, sh, (const float2*)r, (float2*)x, iters, tol, act);
        }
        return;
    }
    // every other block size: one thread per block site, Krylov vectors in `scratch`
    dim3 grid(sp.ncol[colour], nrhs);
    size_t sm = sizeof(double2) * ((size_t)bs + (size_t)(iters + 1) * iters + (iters + 1) + 2 * iters) +
                sizeof(double) * iters + 4 * sizeof(int) +
                (size_t)bs * 12 * (prec == QCD_FP64 ? sizeof(double2) : sizeof(float2));
    if (prec == QCD_FP64) {
        if (sm + 1024 > 48 * 1024) cudaFuncSetAttribute(sap_block_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        sap_block_kernel<double><<<grid, bs, sm, st>>>(f.g, sp.B, f.U64, f.A64, sp.blocks_of_colour[colour], op, sh,
                                                       (const double2*)r, (double2*)x, iters, tol, (double2*)scratch, act);
    } else {
        if (sm + 1024 > 48 * 1024) cudaFuncSetAttribute(sap_block_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        sap_block_kernel<float><<<grid, bs, sm, st>>>(f.g, sp.B, f.U32, f.A32, sp.blocks_of_colour[colour], op, sh,
                                                      (const float2*)r, (float2*)x, iters, tol, (float2*)scratch, act);
    }
}

}  // namespace qcd
