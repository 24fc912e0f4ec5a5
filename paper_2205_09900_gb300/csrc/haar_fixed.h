// haar_fixed.h -- Haar gates in 64-bit fixed point: Box-Muller Gaussians and
// Gram-Schmidt columns on the integer pipe.
//
// GB300 issues 77 FP32 or integer operations in the time of one FP64 operation
// per lane.  Values are integers of up to 60 bits with the stated unit ("Q60": units
// of 2^-60); a product takes 30-bit halves, three 32 x 32 -> 64 multiply-adds (the
// product of the low halves, below the last place, is left out and its mean added
// where sums would collect it) and sums of products share their shifts.  The errors
// are a few 2^-58, where a double carries 2^-53: of a column of length 1, so that an entry
// below 2^-7 has fewer significant bits than a double, and an error still below the 2^-53 of
// its column that FP64 Gram-Schmidt or Householder leaves it.
//
// The same functions compile for the host (tests/cpp/haar_fixed_check.cpp measures
// their errors against extended precision).
#pragma once
#include <cmath>

#include "fp_internal.h"

#if defined(__CUDACC__)
#define FP_TABLE __device__ const __align__(16)
#else
#define FP_TABLE static const
#endif
#include "haar_tables.h"

namespace fpk {

FP_HD uint64_t umulhi(uint64_t a, uint64_t b) {
#if defined(__CUDA_ARCH__)
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
FP_HD int clz64(uint64_t x) {   // x != 0
#if defined(__CUDA_ARCH__)
    return __clzll((long long)x);
#else
    return __builtin_clzll(x);
#endif
}
FP_HD float rsqrt_seed(float x) {   // relative error below 2^-21
#if defined(__CUDA_ARCH__)
    return rsqrtf(x);
#else
    return 1.0f / std::sqrt(x);
#endif
}
FP_HD void table_pair(const int64_t *t, int k, int64_t &a, int64_t &b) {
#if defined(__CUDA_ARCH__)
    const longlong2 v = __ldg(reinterpret_cast<const longlong2 *>(t) + k);
    a = v.x;
    b = v.y;
#else
    a = t[2 * k];
    b = t[2 * k + 1];
#endif
}

struct Fx2 { int64_t x, y; };   // a complex fixed-point value
struct Half { int32_t h, l; };  // h 2^30 + l, 0 <= l < 2^30

FP_HD Half halves(int64_t a) { return {(int32_t)(a >> 30), (int32_t)a & 0x3FFFFFFF}; }   // |a| <= 2^60
FP_HD int64_t wide(int32_t a, int32_t b) { return (int64_t)a * b; }
// a b 2^-60 rounded (|a|, |b| <= 2^60)
FP_HD int64_t mul60(Half a, Half b) {
    return wide(a.h, b.h) + ((wide(a.h, b.l) + wide(a.l, b.h) + (1ll << 29)) >> 30);
}
FP_HD int32_t mulhi32(int32_t a, int32_t b) {
#if defined(__CUDA_ARCH__)
    return __mulhi(a, b);
#else
    return (int32_t)(((int64_t)a * b) >> 32);
#endif
}

FP_HD void table_halves(const int32_t *t, int k, Half &a, Half &b) {
#if defined(__CUDA_ARCH__)
    const int4 v = __ldg(reinterpret_cast<const int4 *>(t) + k);
    a = {v.x, v.y};
    b = {v.z, v.w};
#else
    a = {t[4 * k], t[4 * k + 1]};
    b = {t[4 * k + 2], t[4 * k + 3]};
#endif
}

constexpr uint64_t kLn2Q58 = 199786072581291495ull;        // ln 2 in 2^-58
constexpr int64_t kTwoPiQ57 = 905502432259640355ll;        // 2 pi in 2^-57
constexpr int64_t kOne60 = 1ll << 60;
FP_HD constexpr int64_t rec(int n, int q) { return ((1ll << q) + n / 2) / n; }   // 1/n in 2^-q

// 1/sqrt(a) for a in [2^62, 2^64) (units of 2^-64): the seed y0 in 2^-30 and
// e = 1 - a y0^2 in 2^-60, |e| < 2^-20, with
// 1/sqrt(a) = y0 (1 + e/2 + 3 e^2/8 + ...); returns the bracket minus 1 in 2^-80
FP_HD int64_t rsqrt_step(uint64_t a, uint32_t &y0) {
    const float f = (float)(uint32_t)(a >> 40) * 0x1.0p-24f;   // 24 bits: exact
    y0 = (uint32_t)(rsqrt_seed(f) * 0x1.0p30f);
    const int64_t e = (int64_t)((1ull << 60) - umulhi(a, (uint64_t)y0 * y0));
    const int64_t eh = e >> 10;
    return ((e >> 1) + ((3 * ((eh * eh) >> 40) + 5) >> 3)) << 20;   // (5/8: what the floors take, on average)
}

// cos and sin of 2 pi ph 2^-64 in Q60
FP_HD void cos_sin_fixed(uint64_t ph, Half &c, Half &d) {
    // the angle is k/512 + t turns, |t| <= 2^-10
    const uint64_t kk = (ph + (1ull << 54)) >> 55;
    const int64_t t = (int64_t)(ph - (kk << 55));
    Half ck, sk;
    table_halves(kCosSin, (int)(kk & 511), ck, sk);
    const Half x = halves(mul60(halves(t << 6), halves(kTwoPiQ57)));   // radians in Q67
    const int64_t x2 = mul60(x, x);                                    // Q74
    const Half x2h = halves(x2);
    const int64_t sv = kOne60 - (mul60(x2h, halves(rec(6, 60) - (wide(x2h.h, (int32_t)rec(120, 37)) >> 21))) >> 14);
    const int32_t cw = (int32_t)rec(24, 35) - (mulhi32(x2h.h, (int32_t)rec(720, 40)) >> 17);
    const Half cs = halves(kOne60 - (mul60(x2h, halves(rec(2, 60) - (wide(x2h.h, cw) >> 19))) >> 14));   // Q60
    const Half sn = halves(mul60(x, halves(sv)) >> 7);                                                   // Q60
    c = halves(wide(ck.h, cs.h) - wide(sk.h, sn.h) +
                          ((wide(ck.h, cs.l) + wide(ck.l, cs.h) - wide(sk.h, sn.l) - wide(sk.l, sn.h) + (1ll << 29)) >> 30));
    d = halves(wide(sk.h, cs.h) + wide(ck.h, sn.h) +
                          ((wide(sk.h, cs.l) + wide(sk.l, cs.h) + wide(ck.h, sn.l) + wide(ck.l, sn.h) + (1ll << 30)) >> 30));
}

// One complex Gaussian (E|Z|^2 = 1) from two Philox words, in units of 2^-57:
// Z = sqrt(-ln u1) e^{2 pi i u2}, u1 = ((xa >> 11) + 1) 2^-53, u2 = (xb >> 11) 2^-53
// (keying in fp.h).
FP_HD Fx2 gauss_fixed(uint64_t xa, uint64_t xb) {
    // L = -ln u1: u1 = z 2^-K with z in [3/4, 3/2) (units of 2^-63) and, with r the
    // tabulated value near 1/z, L = K ln 2 + ln r - log1p(z r - 1), |z r - 1| < 2^-9.5
    const uint64_t m = (xa >> 11) + 1;
    const int lz = clz64(m);                  // 10..63
    uint64_t z = (m << lz) >> 1;              // [1/2, 1) in 2^-63, u1 = z 2^(11 - lz)
    int K = lz - 11;
    if (z < (3ull << 61)) {
        z <<= 1;
        K += 1;
    }
    const int j = (int)((z - (3ull << 61) + (1ull << 53)) >> 54);
    int64_t rj, tj;
    table_pair(kRecLog, j, rj, tj);
    const uint64_t hi = umulhi(z, (uint64_t)rj), lo = z * (uint64_t)rj;
    const int64_t y = (int64_t)((hi - (1ull << 62)) << 10) | (int64_t)(lo >> 54);   // Q72
    // log1p(y) = y P, P = 1 - y/2 + y^2/3 - .. - y^5/6: each coefficient to the bits that
    // its power of y leaves it
    const int32_t y40 = (int32_t)(y >> 32);
    const Half yh = halves(y >> 2);           // Q70
    int32_t p = (int32_t)rec(5, 31) - (mulhi32(y40, (int32_t)rec(6, 31)) >> 8);       // Q31
    p = (int32_t)rec(4, 32) - (mulhi32(y40, p) >> 7);                                 // Q32
    int64_t P = rec(3, 60) - (wide(y40, p) >> 12);                                    // Q60
    P = rec(2, 60) - (mul60(yh, halves(P)) >> 10);
    P = kOne60 - (mul60(yh, halves(P)) >> 10);
    uint64_t L;
    int s;                                    // unit of L: 2^-s
    if (K == 0 && j == 128) {                 // r = 1: L = -y P keeps its relative accuracy as u1 -> 1
        const uint64_t d = (uint64_t)-y;      // z <= 1 here
        if (d == 0) return {0, 0};            // u1 = 1
        const int sh = clz64(d) - 1;
        L = umulhi(d << sh, (uint64_t)P << 3);
        s = 71 + sh;
    } else {
        L = (uint64_t)(tj - (mul60(yh, halves(P)) >> 8));   // Q62
        s = 62;
        if (K > 0) {
            L = (uint64_t)K * kLn2Q58 + (uint64_t)((int64_t)L >> 4);
            s = 58;
        }
    }
    // rad = sqrt(L): L = a 2^E, a in [1/4, 1) in 2^-64, E even
    const int lzl = clz64(L);
    uint64_t a = L << lzl;
    int E = 64 - lzl - s;
    if (E & 1) {
        a >>= 1;
        E += 1;
    }
    uint32_t y0;
    const int64_t c1 = rsqrt_step(a, y0);     // Q80
    int64_t rad = (int64_t)(((a >> 32) * y0 + (((uint64_t)(uint32_t)a * y0) >> 32)) >> 2);   // sqrt(a) (1 - c) in Q60
    rad += mul60(halves(rad), halves(c1)) >> 20;
    Half c, d;
    cos_sin_fixed(xb & ~0x7FFull, c, d);
    // E <= 6: |rad 2^(E/2)| <= 6.06
    const Half rh = halves(rad);
    const int64_t zr = mul60(rh, c), zi = mul60(rh, d);   // Q60
    const int half = 3 - E / 2;               // to units of 2^-57
    return {half < 64 ? zr >> half : 0, half < 64 ? zi >> half : 0};
}

// Pieces of the column steps, one entry at a time (a lane may hold one row):
// conj(q) v 2^-60 rounded, q in Q60
FP_HD Fx2 dot1_fixed(Fx2 q, Fx2 v) {
    constexpr int64_t r = 1ll << 29;          // rounds; a left-out product of low halves has mean 2^28
    const Half qx = halves(q.x), qy = halves(q.y), x = halves(v.x), y = halves(v.y);
    return {wide(qx.h, x.h) + wide(qy.h, y.h) +
                ((wide(qx.h, x.l) + wide(qx.l, x.h) + wide(qy.h, y.l) + wide(qy.l, y.h) + 2 * r) >> 30),
            wide(qx.h, y.h) - wide(qy.h, x.h) +
                ((wide(qx.h, y.l) + wide(qx.l, y.h) - wide(qy.h, x.l) - wide(qy.l, x.h) + r) >> 30)};
}
// v <- v - q h
FP_HD void sub1_fixed(Fx2 &v, Fx2 q, Half hr, Half hi) {
    constexpr int64_t r = 1ll << 29;
    const Half qx = halves(q.x), qy = halves(q.y);
    v.x -= wide(qx.h, hr.h) - wide(qy.h, hi.h) +
           ((wide(qx.h, hr.l) + wide(qx.l, hr.h) - wide(qy.h, hi.l) - wide(qy.l, hi.h) + r) >> 30);
    v.y -= wide(qx.h, hi.h) + wide(qy.h, hr.h) +
           ((wide(qx.h, hi.l) + wide(qx.l, hi.h) + wide(qy.h, hr.l) + wide(qy.l, hr.h) + 2 * r) >> 30);
}
FP_HD int lead1_fixed(Fx2 v) {
    return clz64((uint64_t)(v.x ^ (v.x >> 63)) | (uint64_t)(v.y ^ (v.y >> 63)) | 1);
}
FP_HD void shift1_fixed(Fx2 &v, int sh) {
    v.x = sh >= 0 ? (int64_t)((uint64_t)v.x << sh) : v.x >> -sh;
    v.y = sh >= 0 ? (int64_t)((uint64_t)v.y << sh) : v.y >> -sh;
}
// |v|^2 2^-60 of one entry.  The left-out squares of the low halves have mean 1/3 each and one sign: without
// them every column was too long, by 2^-55 of its length at D = 9, and a trace's error grew with its gates
// (Tr(U^dagger U) of qutrits at n = 50, l = 4: 2.7e-15, against 1.7e-15 in FP64).
FP_HD int64_t norm1_fixed(Fx2 v) {
    constexpr int64_t r = (1ll << 28) + (2ll << 29) / 3;   // rounds; twice the mean 2^29 / 3
    const Half x = halves(v.x), y = halves(v.y);
    return wide(x.h, x.h) + wide(y.h, y.h) + ((wide(x.h, x.l) + wide(y.h, y.l) + r) >> 29);
}
// 1/|v| from n2 = |v|^2 2^-60: v/|v| in Q60 is (v y 2^-60) 2^h (scale1_fixed)
FP_HD Half inv_norm_fixed(uint64_t n2, int &h) {
    const int lz = n2 ? clz64(n2) & ~1 : 2;
    const uint64_t a = n2 << lz;              // [2^62, 2^64)
    uint32_t y0 = 0;
    const int64_t c1 = a ? rsqrt_step(a, y0) : 0;
    int64_t y = (int64_t)((uint64_t)y0 << 29);   // 1/sqrt(a) in (1, 2], Q59
    y += (mul60(halves(y), halves(c1)) + (1ll << 19)) >> 20;
    // |v| = sqrt(a) 2^(62 - lz/2) with a read as a fraction: v/|v| 2^60 = v y 2^(lz/2 - 2), lz >= 2
    h = lz / 2 - 1;
    return halves(y);
}
FP_HD void scale1_fixed(Fx2 &v, Half y, int h) {
    v.x = (int64_t)((uint64_t)mul60(halves(v.x), y) << h);
    v.y = (int64_t)((uint64_t)mul60(halves(v.y), y) << h);
}

template <int D>
FP_HD int lead_fixed(const Fx2 (&v)[D]) {     // leading zero bits of the largest entry
    int l = 63;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        const int m = lead1_fixed(v[i]);
        l = m < l ? m : l;
    }
    return l;
}
template <int D>
FP_HD void shift_fixed(Fx2 (&v)[D], int sh) {
#pragma unroll
    for (int i = 0; i < D; ++i) shift1_fixed(v[i], sh);
}

// leading zeros before the norm: entries below 2^(64 - room), so that 2 D squares fit 63 bits
template <int D> constexpr int kUnitRoom = D <= 4 ? 5 : 6;
// v (any scale, D entries) becomes v/|v| in Q60; a zero vector stays zero
template <int D>
FP_HD void unit_fixed(Fx2 (&v)[D]) {
    shift_fixed<D>(v, lead_fixed<D>(v) - kUnitRoom<D>);
    int64_t n2 = 0;
#pragma unroll
    for (int i = 0; i < D; ++i) n2 += norm1_fixed(v[i]);
    int h;
    const Half y = inv_norm_fixed((uint64_t)n2, h);
#pragma unroll
    for (int i = 0; i < D; ++i) scale1_fixed(v[i], y, h);
}

constexpr int kRoom = 6;   // leading zeros of a vector to project: entries below 2^58

// v <- v - q <q, v>, q a unit vector in Q60, v in any unit with entries below 2^58.
template <int D>
FP_HD void project_fixed(const Fx2 (&q)[D], Fx2 (&v)[D]) {
    int64_t hr = 0, hi = 0;
    if (D <= 4) {   // one shift for the whole sum: the cross sums stay below sqrt(2 D) 2^60 + 2 D 2^58 < 2^63
        constexpr int64_t r = 1ll << 29;
        int64_t ac = r + D * r, bc = r;
#pragma unroll
        for (int i = 0; i < D; ++i) {
            const Half qx = halves(q[i].x), qy = halves(q[i].y), x = halves(v[i].x), y = halves(v[i].y);
            hr += wide(qx.h, x.h) + wide(qy.h, y.h);
            hi += wide(qx.h, y.h) - wide(qy.h, x.h);
            ac += wide(qx.h, x.l) + wide(qy.h, y.l) + wide(qx.l, x.h) + wide(qy.l, y.h);
            bc += wide(qx.h, y.l) - wide(qy.h, x.l) + wide(qx.l, y.h) - wide(qy.l, x.h);
        }
        hr += ac >> 30;
        hi += bc >> 30;
    } else {
#pragma unroll
        for (int i = 0; i < D; ++i) {
            const Fx2 t = dot1_fixed(q[i], v[i]);
            hr += t.x;
            hi += t.y;
        }
    }
    const Half a = halves(hr), b = halves(hi);
#pragma unroll
    for (int i = 0; i < D; ++i) sub1_fixed(v[i], q[i], a, b);
}

// A column that its projections shortened 2^kRedo-fold (16, or 4) or more keeps too few bits
// clear of their rounding: it is scaled up and projected once more.
template <int D> constexpr int kRedo = D <= 4 ? 4 : 2;

// the columns v[c] of a matrix become the columns of its unitary factor (R's
// diagonal positive), in Q60
template <int D>
FP_HD void gram_schmidt_fixed(Fx2 (&v)[D][D]) {
#pragma unroll
    for (int c = 0; c < D; ++c) {
        if (c) shift_fixed<D>(v[c], lead_fixed<D>(v[c]) - kRoom);   // entries below 2^58
#pragma unroll
        for (int k = 0; k < c; ++k) project_fixed<D>(v[k], v[c]);
        const int drop = c ? lead_fixed<D>(v[c]) - kRoom : 0;
        if (drop >= kRedo<D>) {
            shift_fixed<D>(v[c], drop);
#pragma unroll
            for (int k = 0; k < c; ++k) project_fixed<D>(v[k], v[c]);
        }
        unit_fixed<D>(v[c]);
    }
}

// x 2^-k as the nearest double or float (|x| < 2^63)
FP_HD double fx_to_double(int64_t x, int k) {
    const uint64_t s = (uint64_t)x >> 63;
    uint64_t a = s ? (uint64_t)-x : (uint64_t)x;
    if (a == 0) return 0.0;
    const int lz = clz64(a);
    a <<= lz;                                 // top bit set
    const uint64_t low = a & 0x7FF;
    uint64_t mant = a >> 11;                  // 53 bits
    mant += (low > 0x400 || (low == 0x400 && (mant & 1))) ? 1 : 0;
    const uint64_t bits = (s << 63) + ((uint64_t)(1023 + 63 - lz - k - 1) << 52) + mant;   // a carry moves the exponent
#if defined(__CUDA_ARCH__)
    return __longlong_as_double((long long)bits);
#else
    double d;
    __builtin_memcpy(&d, &bits, 8);
    return d;
#endif
}
FP_HD float fx_to_float(int64_t x, int k) {
    const uint64_t s = (uint64_t)x >> 63;
    uint64_t a = s ? (uint64_t)-x : (uint64_t)x;
    if (a == 0) return 0.0f;
    const int lz = clz64(a);
    a <<= lz;
    const uint32_t h = (uint32_t)(a >> 32) | ((uint32_t)a ? 1u : 0u);   // the rest as a sticky bit
    const uint32_t low = h & 0xFF;
    uint32_t mant = h >> 8;                   // 24 bits
    mant += (low > 0x80 || (low == 0x80 && (mant & 1))) ? 1 : 0;
    const uint32_t bits = (uint32_t)(s << 31) + ((uint32_t)(127 + 63 - lz - k - 1) << 23) + mant;
#if defined(__CUDA_ARCH__)
    return __uint_as_float(bits);
#else
    float f;
    __builtin_memcpy(&f, &bits, 4);
    return f;
#endif
}

}  // namespace fpk
