// Errors of the fixed-point Haar sampler (haar_fixed.h) against long double, and of a
// double-precision Householder factorisation of the same matrices beside it.
// Prints one line per quantity: name, largest error (and what it is compared with).
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "haar_fixed.h"

using namespace fpk;
typedef long double ld;
typedef std::complex<ld> lc;
typedef std::complex<double> dc;

static lc gauss_ld(uint64_t xa, uint64_t xb) {
    const ld u1 = ldexpl((ld)((xa >> 11) + 1), -53);
    const ld rad = sqrtl(-logl(u1));
    // the angle reduced exactly: u2 = k/8 + t, |t| <= 1/16
    const uint64_t u = xb >> 11;
    const uint64_t k = (u + (1ull << 49)) >> 50;
    const ld t = ldexpl((ld)(int64_t)(u - (k << 50)), -53) * 6.283185307179586476925286766559005768L;
    const ld h = 0.70710678118654752440084436210484903928L;
    const ld ck[8] = {1, h, 0, -h, -1, -h, 0, h}, sk[8] = {0, h, 1, h, 0, -h, -1, -h};
    const ld c = cosl(t), s = sinl(t);
    return {rad * (ck[k & 7] * c - sk[k & 7] * s), rad * (sk[k & 7] * c + ck[k & 7] * s)};
}

template <typename T>
static void qr_gs(const std::complex<T> *A, int d, std::complex<T> *Q) {   // Gram-Schmidt, twice
    for (int j = 0; j < d; ++j) {
        std::complex<T> v[16];
        for (int r = 0; r < d; ++r) v[r] = A[r * d + j];
        for (int pass = 0; pass < 2; ++pass)
            for (int k = 0; k < j; ++k) {
                std::complex<T> h = 0;
                for (int r = 0; r < d; ++r) h += std::conj(Q[r * d + k]) * v[r];
                for (int r = 0; r < d; ++r) v[r] -= Q[r * d + k] * h;
            }
        T n = 0;
        for (int r = 0; r < d; ++r) n += std::norm(v[r]);
        n = std::sqrt(n);
        for (int r = 0; r < d; ++r) Q[r * d + j] = v[r] / n;
    }
}

static void qr_householder(const dc *A0, int d, dc *Q) {   // double, R's diagonal made positive
    dc A[256];
    for (int i = 0; i < d * d; ++i) A[i] = A0[i], Q[i] = i / d == i % d ? 1.0 : 0.0;
    dc ph[16];
    for (int k = 0; k < d; ++k) {
        double n = 0;
        for (int r = k; r < d; ++r) n += std::norm(A[r * d + k]);
        n = std::sqrt(n);
        const double a0 = std::abs(A[k * d + k]);
        const dc p = a0 > 0 ? A[k * d + k] / a0 : dc(1, 0);
        ph[k] = k + 1 < d ? -p : p;
        if (k + 1 == d) break;
        dc v[16];
        for (int r = 0; r < d; ++r) v[r] = r < k ? 0 : A[r * d + k];
        v[k] += p * n;
        const double f = 1.0 / (n * (n + a0));
        for (int c = k; c < d; ++c) {
            dc s = 0;
            for (int r = k; r < d; ++r) s += std::conj(v[r]) * A[r * d + c];
            for (int r = k; r < d; ++r) A[r * d + c] -= v[r] * (f * s);
        }
        for (int r = 0; r < d; ++r) {
            dc s = 0;
            for (int j = k; j < d; ++j) s += Q[r * d + j] * v[j];
            for (int j = k; j < d; ++j) Q[r * d + j] -= f * s * std::conj(v[j]);
        }
    }
    for (int r = 0; r < d; ++r)
        for (int c = 0; c < d; ++c) Q[r * d + c] *= ph[c];
}

template <int D>
static void check_qr(std::mt19937_64 &g, int count) {
    ld worst = 0, worst_dbl = 0, orth = 0, orth_dbl = 0, sum = 0, sum_dbl = 0;
    for (int it = 0; it < count; ++it) {
        Fx2 v[D][D];   // v[c]: column c
        lc A[D * D], Q[D * D];
        dc Ad[D * D], Qd[D * D];
        for (int r = 0; r < D; ++r)
            for (int c = 0; c < D; ++c) {
                v[c][r] = gauss_fixed(g(), g());
                A[r * D + c] = {ldexpl((ld)v[c][r].x, -57), ldexpl((ld)v[c][r].y, -57)};
                Ad[r * D + c] = {(double)A[r * D + c].real(), (double)A[r * D + c].imag()};
            }
        gram_schmidt_fixed<D>(v);
        qr_gs<ld>(A, D, Q);
        qr_householder(Ad, D, Qd);
        ld e = 0, ed = 0;
        dc U[D * D];
        for (int r = 0; r < D; ++r)
            for (int c = 0; c < D; ++c) {
                U[r * D + c] = {fx_to_double(v[c][r].x, 60), fx_to_double(v[c][r].y, 60)};
                e += std::norm(lc(U[r * D + c]) - Q[r * D + c]);
                ed += std::norm(lc(Qd[r * D + c]) - Q[r * D + c]);
            }
        auto unitary = [&](const dc *M) {
            ld o = 0;
            for (int a = 0; a < D; ++a)
                for (int b = 0; b < D; ++b) {
                    lc s = 0;
                    for (int r = 0; r < D; ++r) s += std::conj(lc(M[r * D + a])) * lc(M[r * D + b]);
                    o += std::norm(s - (a == b ? (ld)1 : (ld)0));
                }
            return sqrtl(o);
        };
        const ld oh = unitary(U), od = unitary(Qd);
        e = sqrtl(e), ed = sqrtl(ed);
        worst = std::max(worst, e), worst_dbl = std::max(worst_dbl, ed);
        sum += e, sum_dbl += ed;
        orth = std::max(orth, oh), orth_dbl = std::max(orth_dbl, od);
    }
    printf("qr%d mean %.3Le householder %.3Le worst %.3Le householder %.3Le unitarity %.3Le householder %.3Le\n", D,
           sum / count, sum_dbl / count, worst, worst_dbl, orth, orth_dbl);
}

int main(int argc, char **argv) {
    const int count = argc > 1 ? atoi(argv[1]) : 200000;
    std::mt19937_64 g(12345);
    ld worst = 0;
    auto one = [&](uint64_t xa, uint64_t xb) {
        const Fx2 z = gauss_fixed(xa, xb);
        const lc w = gauss_ld(xa, xb);
        worst = std::max(worst, std::abs(lc(ldexpl((ld)z.x, -57), ldexpl((ld)z.y, -57)) - w));
    };
    for (int i = 0; i < count; ++i) one(g(), g());
    printf("gauss random %.3Le\n", worst);
    worst = 0;
    // u1 at every table edge and its neighbours, at powers of two and near 1; u2 at every table edge
    for (int j = 0; j <= 1024; ++j)
        for (int d = -3; d <= 3; ++d)
            for (int s = 0; s < 53; s += 4) {
                const uint64_t m = ((((uint64_t)j + 512) << 43) + (uint64_t)(int64_t)d) & ((1ull << 53) - 1);
                one((m >> s) << 11, g());
                one(g(), (m << 11));
            }
    for (int s = 0; s <= 52; ++s) {
        one(((1ull << 53) - (1ull << s)) << 11, g());
        one(((1ull << 53) - 1 - ((1ull << s) - 1) / 2) << 11, g());
        one((1ull << s) << 11, ~0ull);
    }
    one(0, 0);
    one(~0ull, 0);
    one(~0ull, ~0ull);
    printf("gauss edges %.3Le\n", worst);
    check_qr<4>(g, count / 4);
    check_qr<9>(g, count / 40);
    check_qr<16>(g, count / 100);
    worst = 0;
    for (int i = 0; i < count; ++i) {   // conversions: correctly rounded
        const int64_t x = (int64_t)g() >> (g() % 63);
        const ld want = ldexpl((ld)x, -62);
        worst = std::max(worst, fabsl((ld)fx_to_double(x, 62) - (ld)(double)want));
        worst = std::max(worst, fabsl((ld)fx_to_float(x, 62) - (ld)(float)want));
    }
    printf("conversions %.3Le\n", worst);
    return 0;
}
