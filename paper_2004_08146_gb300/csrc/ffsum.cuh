// Double-float sums shared by the Davidson kernels (host and device).
#pragma once

#include "common.cuh"

namespace qcd {

struct ffr {
    float h, l;
};

QCD_HD ffr two_sum(float a, float b) {
    const float s = a + b;
    const float bb = s - a;
    const float e = (a - (s - bb)) + (b - bb);
    return {s, e};
}
QCD_HD ffr fast_two_sum(float a, float b) {   // |a| >= |b| or a == 0
    const float s = a + b;
    return {s, b - (s - a)};
}
// Sum of many double-floats: three floats, each the exact rounding errors of the one
// before, so that the total is good to FP64 roundoff without the FP64 pipe (2
// additions per clock and SM).  All three go from stage to stage (lanes, warps, CTAs):
// two of them would round every partial sum to 2^-48.
struct sum3_t {
    float a, b, c;
    QCD_HD sum3_t(float a_ = 0.f, float b_ = 0.f, float c_ = 0.f) : a(a_), b(b_), c(c_) {}
    QCD_HD void add(float h, float l) {
        const ffr s = two_sum(a, h), t = two_sum(b, l), u = two_sum(t.h, s.l);
        a = s.h;
        b = u.h;
        c += t.l + u.l;
    }
    QCD_HD void add(const sum3_t& o) {
        add(o.a, o.b);
        c += o.c;
    }
    QCD_HD double value() const { return (double)a + ((double)b + (double)c); }
};

}  // namespace qcd
