// Host entry points over the host/device arithmetic of the library's headers.
#include "ffsum.cuh"

using namespace qcd;

extern "C" void host_cdot(const float* a, const float* b, int n, int terms, float* out) {
    for (int k = 0; k < n; ++k) {
        float re = 0.f, im = 0.f;
        for (int t = 0; t < terms; ++t) {
            const size_t e = 2 * ((size_t)k * terms + t);
            cdot(re, im, make_float2(a[e], a[e + 1]), make_float2(b[e], b[e + 1]));
        }
        out[2 * k] = re;
        out[2 * k + 1] = im;
    }
}

// n double-floats (h, l) summed as the Davidson kernels do: 32 lanes, 8 warps, CTAs.
// keep = 0 rounds every partial sum to a double-float between the stages.
extern "C" double host_stage_sum(const float* hl, int ctas, int keep) {
    auto stage = [&](const sum3_t& t) {
        if (keep) return t;
        const ffr s = two_sum(t.a, t.b), r = fast_two_sum(s.h, s.l + t.c);
        return sum3_t(r.h, r.l);
    };
    sum3_t total;
    for (int c = 0; c < ctas; ++c) {
        sum3_t cta;
        for (int w = 0; w < 8; ++w) {
            sum3_t warp;
            for (int l = 0; l < 32; ++l) {
                const float* p = hl + 2 * ((c * 8 + w) * 32 + l);
                warp.add(p[0], p[1]);
            }
            cta.add(stage(warp));
        }
        total.add(stage(cta));
    }
    return total.value();
}
