// exact_meet.h -- the meet of FP32 boundaries without FP64 arithmetic.
#pragma once
#include <cmath>

#include <cuda_runtime.h>

#include "fp_internal.h"

namespace fpk {

// (rounded one by one: not to be fused)
#if defined(__CUDA_ARCH__)
FP_HD float fmul_rn(float a, float b) { return __fmul_rn(a, b); }
FP_HD float fadd_rn(float a, float b) { return __fadd_rn(a, b); }
FP_HD float fsub_rn(float a, float b) { return __fsub_rn(a, b); }
#else
FP_HD float fmul_rn(float a, float b) { volatile float r = a * b; return r; }
FP_HD float fadd_rn(float a, float b) { volatile float r = a + b; return r; }
FP_HD float fsub_rn(float a, float b) { volatile float r = a - b; return r; }
#endif

// A sum of floats in three words, each step exact to the last word's rounding (2^-72 of the sum).
struct Sum3 {
    float a = 0, b = 0, c = 0;
    FP_HD static float two(float &s, float x) {   // s <- s + x rounded; returns the rest, exactly
        const float t = fadd_rn(s, x), u = fsub_rn(t, s), r = fadd_rn(fsub_rn(s, fsub_rn(t, u)), fsub_rn(x, u));
        s = t;
        return r;
    }
    FP_HD void add(float x) { c += two(b, two(a, x)); }
    FP_HD void low(float x) { c += two(b, x); }   // |x| of the size of rounding errors
    FP_HD double value() const { return (double)a + ((double)b + (double)c); }
};

// Sums over a thread's terms t = L R: Re, Im, |t|, |t|^2.  FP32: Re and Im from exact products (a
// product and its rounding error), all four words of them summed, so that a term holds at least a
// double's bits; |t| and |t|^2, of which only the cancellation ratio and the error estimate are made,
// hold 2^-45 of a term that carries the boundaries' 2^-24.
template <typename C> struct ExactMeet;
template <> struct ExactMeet<double2> {
    double s[4] = {0, 0, 0, 0};
    FP_HD void add(double2 l, double2 r) {
        const double px = l.x * r.x - l.y * r.y, py = l.x * r.y + l.y * r.x, q = px * px + py * py;
        s[0] += px;
        s[1] += py;
        s[2] += sqrt(q);
        s[3] += q;
    }
    FP_HD double total(int c) const { return s[c]; }
};
template <> struct ExactMeet<float2> {
    Sum3 re, im, ab, sq;
    ExactMeet<double2> far;   // terms whose squares or rounding errors leave the range of float
    FP_HD void add(float2 l, float2 r) {
        // (fmul_rn: the products must not be fused into the sums)
        const float p1 = fmul_rn(l.x, r.x), p2 = fmul_rn(-l.y, r.y), p3 = fmul_rn(l.x, r.y), p4 = fmul_rn(l.y, r.x);
        const float m = fmaxf(fmaxf(fabsf(p1), fabsf(p2)), fmaxf(fabsf(p3), fabsf(p4)));
        if (!(m <= 0x1p60f && m >= 0x1p-46f)) {   // also NaN, and zero
            if (m != 0.f || !(l.x == 0.f && l.y == 0.f) || !(r.x == 0.f && r.y == 0.f))
                far.add(make_double2(l.x, l.y), make_double2(r.x, r.y));
            return;
        }
        const float e1 = fmaf(l.x, r.x, -p1), e2 = fmaf(-l.y, r.y, -p2), e3 = fmaf(l.x, r.y, -p3), e4 = fmaf(l.y, r.x, -p4);
        re.add(p1);
        re.add(p2);
        re.low(e1);
        re.low(e2);
        im.add(p3);
        im.add(p4);
        im.low(e3);
        im.low(e4);
        // |t|^2 and |t| to about 2^-45 of the term
        float x = p1, y = p3;
        const float xl = Sum3::two(x, p2) + (e1 + e2), yl = Sum3::two(y, p4) + (e3 + e4);
        const float qx = fmul_rn(x, x), qy = fmul_rn(y, y);
        float q = qx;
        const float ql = Sum3::two(q, qy) + (fmaf(x, x, -qx) + fmaf(y, y, -qy)) + 2.f * (x * xl + y * yl);
        sq.add(q);
        sq.low(ql);
        const float s = sqrtf(q);
        ab.add(s);
        if (s > 0.f) ab.low((fmaf(-s, s, q) + ql) * (0.5f / s));
    }
    FP_HD double total(int c) const {
        const Sum3 &v = c == 0 ? re : c == 1 ? im : c == 2 ? ab : sq;
        return v.value() + far.s[c];
    }
};

}  // namespace fpk
