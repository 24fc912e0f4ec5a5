// Brickwork and HEA tile schedules (make_brick_plan): every gate once, in an order that
// respects the layers, its two bits inside the pass's arc and the window; and, for
// 12-bit tiles with 5-bit windows, the exchange maps of the tensor-memory form with
// ascending rows (make_tc_windows without rotations): bijections on the 4096 slots, the
// 16 storing and the 16 loading lanes of a half-warp on 16 distinct bank pairs each, and
// the per-thread tables equal to the maps.
//   brick_schedule_check n l tile_bits low_bits win_bits kind
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "brick.h"

using namespace fpk;

static int fail(const char *what) {
    printf("FAIL %s\n", what);
    return 1;
}

int main(int argc, char **argv) {
    if (argc < 7) return fail("usage");
    const int n = atoi(argv[1]), l = atoi(argv[2]), K = atoi(argv[3]), low = atoi(argv[4]), R = atoi(argv[5]), kind = atoi(argv[6]);
    const BrickHostPlan P = make_brick_plan(n, l, K, low, R, kind);
    const BrickDev &d = P.dev;
    int windows = 0;
    for (int side = 0; side < 2; ++side) {
        const int N = d.N, L = d.n_layers[side], m = d.m;
        std::vector<int> height(N, 0);
        std::vector<char> seen((size_t)L * m, 0);
        for (int p = 0; p < d.n_passes[side]; ++p) {
            const BrickPass &ps = P.passes[d.pass_off[side] + p];
            std::vector<int> phys;
            for (int b = 0; b < N; ++b)
                if (ps.smask >> b & 1) phys.push_back(b);
            if ((int)phys.size() != K) return fail("tile bits");
            std::vector<char> used(ps.n_gates, 0);
            for (int w = 0; w < ps.n_rp; ++w) {
                const RegPass &rp = P.rpasses[ps.rp_off + w];
                for (int k = 1; k < rp.r; ++k) {
                    if ((phys[rp.win[k - 1]] + 1) % N != phys[rp.win[k]]) return fail("window bits not consecutive");
                    if (rp.srt[k - 1] >= rp.srt[k]) return fail("sorted window bits");
                }
                for (int g = 0; g < rp.n_gates; ++g) {
                    const RegGate &rg = P.rgates[rp.gate_off + g];
                    const BrickGate &bg = P.gates[ps.gate_off + rg.slot];
                    if (rg.slot >= ps.n_gates || used[rg.slot]++) return fail("gate slot");
                    const int a = phys[bg.a], b = phys[bg.b], t = bg.layer;
                    if (rp.win[rg.type] != bg.a || rp.win[rg.type + 1] != bg.b) return fail("gate outside its window");
                    if (a != 2 * bg.j + layer_parity(d, side, t) || b != (a + 1) % N) return fail("gate bits");
                    if (height[a] != t || height[b] != t) return fail("gate before its predecessors");
                    height[a] = height[b] = t + 1;
                    if (seen[(size_t)t * m + bg.j]++) return fail("gate twice");
                }
                ++windows;
            }
            for (int g = 0; g < ps.n_gates; ++g)
                if (!used[g]) return fail("unused gate");
        }
        for (char s : seen)
            if (!s) return fail("missing gate");
    }
    if (K == kTcTile && R == kMaxWin) {
        const std::vector<TcWin> W = make_tc_windows(P, false);
        const std::vector<TcXa> X = make_tc_xaddr(P, W);
        for (const BrickPass &ps : P.passes)
            for (int w = 0; w < ps.n_rp; ++w) {
                const TcWin &t = W[ps.rp_off + w];
                auto addr = [&](uint32_t i) {
                    uint32_t a = 0;
                    for (int b = 0; b < kTcTile; ++b)
                        if (i >> b & 1) a ^= t.xcb[b];
                    return a;
                };
                std::vector<char> hit(4096, 0);
                for (uint32_t i = 0; i < 4096; ++i) {
                    const uint32_t a = addr(i);
                    if (a % 8 || a >= 32768 || hit[a / 8]++) return fail("exchange map not a bijection");
                }
                const uint8_t load0[4] = {0, 1, 2, 3};
                for (int s = 0; s < 2; ++s) {   // storing lanes (the previous window's rows), loading lanes
                    const uint8_t *r = s ? t.row : w ? W[ps.rp_off + w - 1].row : load0;
                    unsigned banks = 0;
                    for (int lane = 0; lane < 16; ++lane) {
                        uint32_t i = 0;
                        for (int k = 0; k < 4; ++k)
                            if (lane >> k & 1) i |= 1u << r[k];
                        banks |= 1u << ((addr(i) >> 3) & 15u);
                    }
                    if (banks != 0xFFFFu) return fail("bank pairs");
                }
                for (int warp = 0; warp < 8; ++warp)
                    for (int lane = 0; lane < 32; ++lane)
                        for (int u = 0; u < 16; ++u) {
                            const int row = 32 * (warp & 3) + lane, col = 16 * (warp >> 2) + u;
                            uint32_t i = 0;
                            for (int k = 0; k < kTcRows; ++k)
                                if (row >> k & 1) i |= 1u << t.row[k];
                            for (int k = 0; k < kMaxWin; ++k)
                                if (col >> k & 1) i |= 1u << t.win[k];
                            const TcXa &x = X[ps.rp_off + w];
                            uint32_t a = x.ld_lane[lane] ^ x.ld_warp[warp];
                            for (int k = 0; k < 4; ++k)
                                if (u >> k & 1) a ^= x.ld_c[k];
                            if (a != addr(i)) return fail("address tables");
                        }
            }
    }
    printf("ok windows %d passes %d gates %zu\n", windows, d.n_passes[0] + d.n_passes[1], P.gates.size());
    return 0;
}
