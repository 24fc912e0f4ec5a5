// Windows of the spiral sweep (spiral_windows): the maps of a window act on consecutive
// bits of its walk, and the groups that a window leaves out (SpiralWin::half) hold zeros
// only.  Random complex coefficients, state in its CTA parts as the kernel addresses it.
//   spiral_walk_check n L R split
#include "planner.h"
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
using namespace fpk;
typedef std::complex<double> cd;
static int fail(const char *what) { printf("FAIL %s\n", what); return 1; }
int main(int argc, char **argv) {
    if (argc < 5) return fail("usage");
    const int n = atoi(argv[1]), L = atoi(argv[2]), R = atoi(argv[3]), split = atoi(argv[4]);
    const auto U = layout_hea_pauli(n, L, false);
    const SpiralPlan P = make_spiral_plan(n, U, U, RAW_PAULI);
    if (!P.ok) return fail("plan");
    const int B = P.bits;
    std::vector<SpiralWin> wins;
    std::vector<uint8_t> ij;
    int h[2];
    spiral_windows(P, R, split, wins, ij, h);
    std::mt19937_64 rng(5);
    std::normal_distribution<double> N01;
    std::vector<cd> st((size_t)1 << B);
    for (size_t x = 0; x < st.size(); ++x) st[x] = ((x >> (B - 1) ^ x >> P.first_bit) & 1) ? 0.0 : 1.0;
    const uint32_t G = 1u << (B - R - split);
    int halves = 0;
    for (const SpiralWin &w : wins) {
        unsigned perm = 0;
        for (int k = 0; k < w.nb; ++k) perm |= 1u << w.walk[k];
        if (perm != (1u << w.nb) - 1u || w.n_maps > w.nb - 1) return fail("walk");
        for (int k = 0; k < w.n_maps; ++k)
            if (P.maps[w.first + k].a != w.bits[w.walk[k]] || P.maps[w.first + k].b != w.bits[w.walk[k + 1]]) return fail("map off its walk");
        halves += w.half;
        for (int r = 0; w.half && r < (1 << split); ++r)
            for (uint32_t t = G / 2; t < G; ++t)
                for (uint32_t i = 0; i < 1u << R; ++i) {
                    uint32_t x = 0;
                    for (int j = 0; j < w.n_pos; ++j) x |= ((r * G + t) >> j & 1u) << w.pos[j];
                    for (int k = 0; k < R; ++k) x |= (i >> k & 1u) << w.bits[k];
                    if (st[x] != 0.0) return fail("a left-out amplitude is not zero");
                }
        for (int m = w.first; m < w.first + w.n_maps; ++m) {   // the map's zero pattern, random values
            const SpiralMap &mp = P.maps[m];
            cd T[4][4];
            double mean = 0;
            for (int o = 0; o < 4; ++o)
                for (int f = 0; f < 4; ++f) {
                    const int oa = o & 1, ob = o >> 1, ia = f & 1, ib = f >> 1;
                    bool on = true;
                    switch (mp.type) {
                        case SP_DIAG_BA: on = o == f; break;
                        case SP_START: on = oa == ob; break;
                        case SP_MID_AUX: on = ob == ib; break;
                        case SP_RL: on = oa == ia; break;
                        case SP_MID_RR: on = ib == 0; break;
                        case SP_RR: on = oa == ia && ib == 0; break;
                        case SP_LL: on = oa == 0; break;
                        case SP_LL_AUX: on = oa == 0 && ob == ib; break;
                        default: break;
                    }
                    T[o][f] = on ? cd(N01(rng), N01(rng)) : cd(0);
                }
            for (size_t x = 0; x < st.size(); ++x) {
                if (x >> mp.a & 1 || x >> mp.b & 1) continue;
                cd y[4];
                for (int o = 0; o < 4; ++o) {
                    y[o] = 0;
                    for (int f = 0; f < 4; ++f) y[o] += T[o][f] * st[x | (size_t)(f & 1) << mp.a | (size_t)(f >> 1) << mp.b];
                }
                for (int o = 0; o < 4; ++o) { st[x | (size_t)(o & 1) << mp.a | (size_t)(o >> 1) << mp.b] = y[o]; mean += std::abs(y[o]); }
            }
            for (cd &v : st) v *= (double)st.size() / mean;
        }
    }
    printf("ok windows %zu halves %d\n", wins.size(), halves);
    return 0;
}
