// Host entry points over the host/device arithmetic of the library's headers.
#include "common.cuh"

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
