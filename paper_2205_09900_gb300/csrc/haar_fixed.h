// haar_fixed.h -- Haar gates in 64-bit fixed point: Box-Muller Gaussians and
// Gram-Schmidt columns on the integer pipe.
//
// GB300 issues 77 FP32 or integer operations in the time of one FP64 operation
// per lane, and a 64 x 64 -> high-64 product is about ten integer instructions:
// the same steps in fixed point take a seventh of the FP64 pipe's time and carry
// 59 to 62 significant bits where a double carries 53.  All values below are
// integers with the stated unit; products keep the high word, truncated.
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
FP_HD int64_t smulhi(int64_t a, int64_t b) {
#if defined(__CUDA_ARCH__)
    return __mul64hi(a, b);
#else
    return (int64_t)(((__int128)a * b) >> 64);
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

constexpr uint64_t kOne62 = 1ull << 62;
constexpr uint64_t kLn2Q58 = 199786072581291495ull;        // ln 2 in 2^-58
constexpr int64_t kTwoPiQ60 = 7244019458077122842ll;       // 2 pi in 2^-60
FP_HD constexpr int64_t rec62(int64_t n) { return (int64_t)((kOne62 + (uint64_t)n / 2) / (uint64_t)n); }   // 1/n in 2^-62

// 1/sqrt(a) for a in [2^62, 2^64) (units of 2^-64): the seed y0 in 2^-30 and
// e = 1 - a y0^2 in 2^-60, |e| < 2^-20, with
// 1/sqrt(a) = y0 (1 + e/2 + 3 e^2/8 + ...); returns the bracket minus 1 in 2^-80
FP_HD int64_t rsqrt_step(uint64_t a, uint32_t &y0) {
    const float f = (float)(uint32_t)(a >> 40) * 0x1.0p-24f;   // 24 bits: exact
    y0 = (uint32_t)(rsqrt_seed(f) * 0x1.0p30f);
    const int64_t e = (int64_t)((1ull << 60) - umulhi(a, (uint64_t)y0 * y0));
    const int64_t eh = e >> 10;
    return ((e >> 1) + ((3 * ((eh * eh) >> 40)) >> 3)) << 20;
}

// One complex Gaussian (E|Z|^2 = 1) from two Philox words, in units of 2^-59:
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
    const int64_t y = (int64_t)((hi - (1ull << 62)) << 10) | (int64_t)(lo >> 54);   // 2^-72
    const int64_t y64 = y >> 8;
    int64_t p = rec62(6);                     // log1p(y) = y P, P = 1 - y/2 + y^2/3 - .. - y^5/6
    p = rec62(5) - smulhi(y64, p);
    p = rec62(4) - smulhi(y64, p);
    p = rec62(3) - smulhi(y64, p);
    p = rec62(2) - smulhi(y64, p);
    p = (int64_t)kOne62 - smulhi(y64, p);
    uint64_t L;
    int s;                                    // unit of L: 2^-s
    if (K > 0) {
        L = (uint64_t)K * kLn2Q58 + (uint64_t)((tj - (smulhi(y, p) >> 8)) >> 4);
        s = 58;
    } else if (j != 128) {
        L = (uint64_t)(tj - (smulhi(y, p) >> 8));
        s = 62;
    } else {                                  // r = 1: L = -y P keeps its relative accuracy as u1 -> 1
        const uint64_t d = (uint64_t)-y;      // y <= 0 here when L matters; y > 0 cannot occur with K = 0, z <= 1
        if (d == 0) return {0, 0};            // u1 = 1
        const int sh = clz64(d) - 1;
        L = umulhi(d << sh, (uint64_t)p << 1);
        s = 71 + sh;
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
    const int64_t c1 = rsqrt_step(a, y0);     // 2^-80
    int64_t rad = (int64_t)umulhi(a, (uint64_t)y0 << 32);      // sqrt(a) (1 - c) in 2^-62
    rad += smulhi(rad, c1) >> 16;
    // cos, sin of 2 pi u2: u2 = k/512 + t, |t| <= 2^-10 turns
    const uint64_t ph = xb & ~0x7FFull;       // turns in 2^-64
    const uint64_t kk = (ph + (1ull << 54)) >> 55;
    const int64_t t = (int64_t)(ph - (kk << 55));
    int64_t ck, sk;
    table_pair(kCosSin, (int)(kk & 511), ck, sk);
    const int64_t x = smulhi(t << 8, kTwoPiQ60);   // radians in 2^-68
    const int64_t x2 = smulhi(x, x);               // 2^-72
    const int64_t sn = smulhi(x, (int64_t)kOne62 - (smulhi(x2, rec62(6) - (smulhi(x2, rec62(120)) >> 8)) >> 8)) >> 2;   // 2^-64
    const int64_t cs = (int64_t)kOne62 -
                       (smulhi(x2, rec62(2) - (smulhi(x2, rec62(24) - (smulhi(x2, rec62(720)) >> 8)) >> 8)) >> 8);      // 2^-62
    const int64_t c = smulhi(ck, cs) * 4 - (smulhi(sk, sn)), d = smulhi(sk, cs) * 4 + (smulhi(ck, sn));                 // 2^-62
    // E <= 6: |rad 2^(E/2)| <= 6.06
    const int half = E / 2 - 1;               // to units of 2^-59
    const int64_t zr = smulhi(rad, c), zi = smulhi(rad, d);    // 2^-60
    return half >= 0 ? Fx2{(int64_t)((uint64_t)zr << half), (int64_t)((uint64_t)zi << half)}
                     : Fx2{half > -64 ? zr >> -half : 0, half > -64 ? zi >> -half : 0};
}

// leading zero bits of the largest entry (63 for a zero vector)
template <int D>
FP_HD int lead_fixed(const Fx2 (&v)[D]) {
    uint64_t o = 1;
#pragma unroll
    for (int i = 0; i < D; ++i) o |= (uint64_t)(v[i].x ^ (v[i].x >> 63)) | (uint64_t)(v[i].y ^ (v[i].y >> 63));
    return clz64(o);
}
template <int D>
FP_HD void shift_fixed(Fx2 (&v)[D], int sh) {
#pragma unroll
    for (int i = 0; i < D; ++i) {
        v[i].x = sh >= 0 ? (int64_t)((uint64_t)v[i].x << sh) : v[i].x >> -sh;
        v[i].y = sh >= 0 ? (int64_t)((uint64_t)v[i].y << sh) : v[i].y >> -sh;
    }
}

// v (any scale, D entries) becomes v/|v| in units of 2^-62; a zero vector stays zero
template <int D>
FP_HD void unit_fixed(Fx2 (&v)[D]) {
    constexpr int room = D <= 4 ? 2 : 3;      // |entries| < 2^(64 - room): 2 D squares fit 64 bits
    shift_fixed<D>(v, lead_fixed<D>(v) - room);
    uint64_t n2 = 0;                          // |v|^2 2^-64
#pragma unroll
    for (int i = 0; i < D; ++i) n2 += (uint64_t)smulhi(v[i].x, v[i].x) + (uint64_t)smulhi(v[i].y, v[i].y);
    const int lz = n2 ? clz64(n2) & ~1 : 0;
    const uint64_t a = n2 << lz;              // [2^62, 2^64)
    uint32_t y0;
    const int64_t c1 = a ? rsqrt_step(a, y0) : (y0 = 0, 0);
    // 1/sqrt(a) in (1, 2], units of 2^-62 (2^-61 of room: values up to 2)
    int64_t y = (int64_t)((uint64_t)y0 << 31);
    y += smulhi(y, c1) >> 16;                 // 2^-61
    // |v| = sqrt(a) 2^(32 - lz/2) with a read as a fraction: v/|v| 2^62 = v y_real 2^(lz/2 - 2)
    const int h = lz / 2;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        v[i].x = (int64_t)((uint64_t)smulhi((int64_t)((uint64_t)v[i].x << 1), y) << h);
        v[i].y = (int64_t)((uint64_t)smulhi((int64_t)((uint64_t)v[i].y << 1), y) << h);
    }
}

// v <- v - q <q, v>, q a unit vector in 2^-62, v in any unit with |v| < 2^63
template <int D>
FP_HD void project_fixed(const Fx2 (&q)[D], Fx2 (&v)[D]) {
    int64_t hr = D, hi = 0;                   // <q, v> / 4 in v's unit; D: half of each truncated bit of 2 D terms
#pragma unroll
    for (int i = 0; i < D; ++i) {
        hr += smulhi(q[i].x, v[i].x) + smulhi(q[i].y, v[i].y);
        hi += smulhi(q[i].x, v[i].y) - smulhi(q[i].y, v[i].x);
    }
    hr *= 4;
    hi *= 4;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        v[i].x -= 4 * (smulhi(q[i].x, hr) - smulhi(q[i].y, hi));
        v[i].y -= 4 * (smulhi(q[i].x, hi) + smulhi(q[i].y, hr) + 1);
    }
}

// A column that its projections shortened 2^kRedo-fold (16, or 8) or more keeps too few bits
// clear of their rounding: it is scaled up and projected once more.
template <int D> constexpr int kRedo = D <= 9 ? 4 : 3;
// leading zeros that keep |v| below 2^63: entries below 2^(64 - room), 2 D of them
template <int D> constexpr int kRoom = D <= 4 ? 3 : 4;

// the columns v[c] of a matrix become the columns of its unitary factor (R's
// diagonal positive), in units of 2^-62
template <int D>
FP_HD void gram_schmidt_fixed(Fx2 (&v)[D][D]) {
#pragma unroll
    for (int c = 0; c < D; ++c) {
        if (c) shift_fixed<D>(v[c], lead_fixed<D>(v[c]) - kRoom<D>);   // |v| < 2^63
#pragma unroll
        for (int k = 0; k < c; ++k) project_fixed<D>(v[k], v[c]);
        const int drop = c ? lead_fixed<D>(v[c]) - kRoom<D> : 0;
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
