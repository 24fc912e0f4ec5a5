// Columns of fixed-point Haar gates (haar_fixed.h) have length 1 on average: prints per dimension the
// mean and the rms of |column|^2 - 1, in units of 2^-60.
#include <cmath>
#include <cstdio>
#include <random>

#include "haar_fixed.h"

using namespace fpk;

template <int D>
static void lengths(int gates) {
    std::mt19937_64 g(7 + D);
    long double s = 0, s2 = 0;
    for (int it = 0; it < gates; ++it) {
        Fx2 v[D][D];
        for (int c = 0; c < D; ++c)
            for (int r = 0; r < D; ++r) {
                const uint64_t xa = g(), xb = g();
                v[c][r] = gauss_fixed(xa, xb);
            }
        gram_schmidt_fixed<D>(v);
        for (int c = 0; c < D; ++c) {
            long double q = -1;
            for (int r = 0; r < D; ++r) {
                const long double x = ldexpl((long double)v[c][r].x, -60), y = ldexpl((long double)v[c][r].y, -60);
                q += x * x + y * y;
            }
            q = ldexpl(q, 60);
            s += q;
            s2 += q * q;
        }
    }
    std::printf("%d %.4Lf %.4Lf\n", D, s / (gates * D), sqrtl(s2 / (gates * D)));
}

int main() {
    lengths<4>(100000);
    lengths<9>(20000);
    lengths<16>(5000);
    return 0;
}
