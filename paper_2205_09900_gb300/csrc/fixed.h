// fixed.h -- FP64 boundary sweeps in 64-bit integers.  An FP64 instruction takes an SM
// quarter about 77 cycles per warp; a complex product below is 12 wide integer
// multiply-adds and some 20 additions and shifts on the integer pipes.
//
// Amplitudes are integers times 2^e with one e per thread's register block, coefficients
// (of magnitude at most 1) integers times 2^-61.  Both are split into balanced halves,
// x = 2^31 h + l with l in [-2^30, 2^30), so that the dropped product l l' is below half a
// unit of the result and, like the rounding of the shift, without a bias.  A block's
// largest amplitude is brought to 2^56 .. 2^57 before every exchange (fix_settle), which
// holds 2^-57 of it, against FP64's 2^-53 of each amplitude; an e per block needs no maximum
// over the boundary and keeps its bits where amplitudes spread over many octaves.  An amplitude
// more than 8 times below its block's largest so holds fewer bits than a double would give it; the error
// of a block as a vector, which is what a trace sees, stays below FP64's (rms 2^-54 of its norm an
// operation at most).  HEA traces
// at n = 9 and 50, L = 4..8, against extended precision: rms errors 1.2 to 5 times below those of
// FP64 arithmetic.
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

namespace fpk {
namespace {

constexpr int kFixCoef = 61;   // fraction bits of a coefficient
constexpr int kFixTop = 57;    // amplitudes are below 2^kFixTop before a product

__device__ __forceinline__ int2 fix_split(long long x) {   // (h, l)
    const int l = (int)((uint32_t)x << 1) >> 1;
    return make_int2((int)((x - l) >> 31), l);
}
// a coefficient as (re h, re l, im h, im l)
__device__ __forceinline__ int4 fix_coef(longlong2 q) {
    const int2 a = fix_split(q.x), b = fix_split(q.y);
    return make_int4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ longlong2 fix_join(int4 t) {
    return make_longlong2(((long long)t.x << 31) + t.y, ((long long)t.z << 31) + t.w);
}
// a double of magnitude at most 1 as such a coefficient's integer (no FP64 instruction)
__device__ __forceinline__ long long fix_unit(double t) {
    const long long b = __double_as_longlong(t);
    const int ex = (int)(b >> 52) & 0x7FF, sh = ex - (1023 + 52 - kFixCoef);   // sh <= 9
    const long long man = (b & 0xFFFFFFFFFFFFFll) | 0x10000000000000ll;
    const long long q = ex == 0 ? 0 : sh >= 0 ? man << sh : sh > -54 ? (man + (1ll << (-sh - 1))) >> -sh : 0;
    return b < 0 ? -q : q;
}
// sum of products v t of split amplitudes v = (2^31 a.x + a.y) + i (2^31 b.x + b.y)
struct FixSum {
    long long hr = 0, mr = 0, hi = 0, mi = 0;
    __device__ __forceinline__ void add(int2 a, int2 b, int4 t) {
        hr += (long long)a.x * t.x - (long long)b.x * t.z;
        mr += (long long)a.x * t.y + (long long)a.y * t.x - (long long)b.x * t.w - (long long)b.y * t.z;
        hi += (long long)a.x * t.z + (long long)b.x * t.x;
        mi += (long long)a.x * t.w + (long long)a.y * t.z + (long long)b.x * t.y + (long long)b.y * t.x;
    }
    __device__ __forceinline__ longlong2 value() const {
        constexpr int s = 62 - kFixCoef;
        return make_longlong2((hr << s) + ((mr + (1ll << (30 - s))) >> (31 - s)),
                              (hi << s) + ((mi + (1ll << (30 - s))) >> (31 - s)));
    }
};
__device__ __forceinline__ longlong2 cmul(longlong2 v, int4 t) {
    FixSum z;
    z.add(fix_split(v.x), fix_split(v.y), t);
    return z.value();
}
__device__ __forceinline__ void butterfly(longlong2 &a, longlong2 &b) {
    const longlong2 s = make_longlong2(a.x + b.x, a.y + b.y), d = make_longlong2(a.x - b.x, a.y - b.y);
    a = s;
    b = d;
}
// x / 2^r rounded, r <= 62
__device__ __forceinline__ long long fix_shr(long long x, int r) { return (x + ((1ll << r) >> 1)) >> r; }

constexpr int kFixZero = -(1 << 24);   // scale of a block of zeros

// bring a block's largest component to 2^(kFixTop - 1) .. 2^kFixTop (or 24 bits nearer)
template <int V>
__device__ __forceinline__ void fix_settle(longlong2 (&v)[V], int &e) {
    uint32_t m = 0;
#pragma unroll
    for (int i = 0; i < V; ++i) {
        const int x = (int)(v[i].x >> 32), y = (int)(v[i].y >> 32);
        m |= (uint32_t)(x ^ (x >> 31)) | (uint32_t)(y ^ (y >> 31));
    }
    if (m == 0) {
        unsigned long long any = 0;
#pragma unroll
        for (int i = 0; i < V; ++i) any |= (unsigned long long)v[i].x | (unsigned long long)v[i].y;
        if (any == 0) e = kFixZero;
    }
    const int sh = min(kFixTop - (64 - __clz((int)m)), 24);
    e -= sh;
    if (sh > 0) {
#pragma unroll
        for (int i = 0; i < V; ++i) v[i].x <<= sh, v[i].y <<= sh;
    } else if (sh < 0) {
#pragma unroll
        for (int i = 0; i < V; ++i) v[i].x = fix_shr(v[i].x, -sh), v[i].y = fix_shr(v[i].y, -sh);
    }
}
// amplitude v of scale e at the scale top >= e
__device__ __forceinline__ void fix_align(longlong2 &v, int e, int top) {
    const int r = min(top - e, 62);
    v.x = fix_shr(v.x, r);
    v.y = fix_shr(v.y, r);
}

}  // namespace
}  // namespace fpk
