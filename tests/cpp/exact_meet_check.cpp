// ExactMeet<float2> (exact_meet.h) on the host: Re and Im of a single term to a double's rounding, of
// sums to the rounding of the result, |t| and |t|^2 to 2^-44.
#include <cstdint>
#include <cstdio>

#include "exact_meet.h"

using namespace fpk;

static uint64_t state = 12345;
static uint32_t next() { return (uint32_t)((state = state * 6364136223846793005ull + 1442695040888963407ull) >> 33); }
static float rnd(int lo, int hi) {   // random sign and 24 bits, exponent in [lo, hi]
    const float m = 1.0f + (float)(next() & 0x7fffff) * 0x1.0p-23f;
    return std::ldexp(next() & 1 ? -m : m, lo + (int)(next() % (uint32_t)(hi - lo + 1)));
}

int main() {
    const long double u53 = std::ldexp(1.0L, -53);
    for (int part = 0; part < 4; ++part) {
        // single terms of like and of unlike magnitudes, long sums, single terms that leave the range of float
        // (those are summed in FP64, one rounding a term)
        const int terms = part == 2 ? 1 << 14 : 1, lo = part == 1 ? -12 : part == 3 ? -60 : -1, hi = part == 1 ? 12 : part == 3 ? 45 : 1;
        for (int rep = 0; rep < (part == 2 ? 20 : 100000); ++rep) {
            ExactMeet<float2> m;
            long double re = 0, im = 0, ab = 0, sq = 0, size = 0;
            for (int i = 0; i < terms; ++i) {
                const float2 l = make_float2(rnd(lo, hi), rnd(lo, hi)), r = make_float2(rnd(lo, hi), rnd(lo, hi));
                m.add(l, r);
                const long double x = (long double)((double)l.x * r.x) - (long double)((double)l.y * r.y);
                const long double y = (long double)((double)l.x * r.y) + (long double)((double)l.y * r.x);
                re += x;
                im += y;
                ab += std::sqrt(x * x + y * y);
                sq += x * x + y * y;
                size += std::fabs((long double)l.x * r.x) + std::fabs((long double)l.y * r.y);
            }
            // (long double holds 64 bits or more: 2^-62 of the terms over a long sum)
            const long double slack = size * std::ldexp(1.0L, -60), limit[2] = {std::fabs(re) * u53 + slack, std::fabs(im) * u53 + slack};
            if (std::fabs((long double)m.total(0) - re) > limit[0] || std::fabs((long double)m.total(1) - im) > limit[1] ||
                std::fabs((long double)m.total(2) - ab) > ab * std::ldexp(1.0L, -44) + slack ||
                std::fabs((long double)m.total(3) - sq) > sq * std::ldexp(1.0L, -43) + size * slack) {
                std::printf("part %d: %La %La, %La %La of %La\n", part, (long double)m.total(0), re, (long double)m.total(1), im, size);
                return 1;
            }
        }
    }
    std::puts("ok");
    return 0;
}
