// kernels_hea.cu -- boundary sweep of the hardware-efficient ansatz (RY RZ
// rotations and CZ ladders) for boundaries of N = 2L - 2 <= 14 bits.
//
// Absorbing a qubit (brick.h) multiplies the boundary by the qubit's rotation
// factors, a product of N functions of two ring-adjacent bits (slot s: bits s-1
// and s), and then crosses the CZ ladder, a Hadamard on every bit.  As 4x4 maps
// that is 4 N complex multiply-adds per amplitude; here it is N complex
// additions and one complex product per register window:
//   * a thread holds 2^R amplitudes of a window of R consecutive bits; the
//     factors that touch the window's bits come from one table per window,
//     indexed by the window's bits and the one or two ring neighbours outside
//     it, built once per qubit from the N 2x2 matrices;
//   * the Hadamards are butterflies on registers;
//   * windows change through one exchange in shared memory, and a qubit's windows
//     run in the opposite order of the previous qubit's, so that N = 14 takes two
//     exchanges per qubit; every exchange then stores where the same thread last
//     read, which leaves one barrier per exchange, and that between the two lowest
//     windows stays inside a warp.
// Two side sweeps (left half kept in `lscr`), then the FP64 meet.  A boundary
// belongs to T = 2^(N-R) threads: a few per warp for the small ones, 512 threads
// at N = 14 (128 KB of shared memory in FP32; FP64 splits the highest bit over a
// 2-CTA cluster, whose Hadamard reads the partner's amplitudes).
//
// Bound: FP32 adds and FMAs (5,100 clocks per qubit at N = 14) beside the
// exchange's shared-memory traffic (two 8-byte accesses per amplitude and
// exchange, with the table reads 5,600).  FP64 (N >= 6) computes in 64-bit integers
// (fixed.h): bound by the integer pipes instead of the FP64 pipe.  Measured per pair
// at n = 50 on a GB300, against dense 4x4 maps on the same boundary: L = 8 FP32
// 1.6 us against 11.0 (tensor-core tile passes), L = 7 0.31 against 5.6, L = 6
// 0.07 against 1.5 (one map per shared-memory pass); L = 8 FP64, 214 pairs, 76 us in FP64
// arithmetic against 320 (FMA tile passes).  100,000 pairs, L = 1..8, of which about 700 go
// through FP64: 61.5 ms with FP64 arithmetic, 46.7 with integers, 42.7 with the slots
// sampled in fixed point too, 42.2 with a lane per amplitude at 2 and 4 bits in FP64.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "brick.h"
#include "fixed.h"
#include "kernels.h"
#include "meet.h"

namespace cg = cooperative_groups;

namespace fpk {
namespace {

template <typename C, int N> struct HeaShape;   // window bits, cluster bits
template <> struct HeaShape<float2, 6> { static constexpr int R = 3, CLB = 0; };
template <> struct HeaShape<float2, 8> { static constexpr int R = 4, CLB = 0; };
template <> struct HeaShape<float2, 10> { static constexpr int R = 5, CLB = 0; };
template <> struct HeaShape<float2, 12> { static constexpr int R = 5, CLB = 0; };
template <> struct HeaShape<float2, 14> { static constexpr int R = 5, CLB = 0; };
template <> struct HeaShape<longlong2, 6> { static constexpr int R = 3, CLB = 0; };
template <> struct HeaShape<longlong2, 8> { static constexpr int R = 4, CLB = 0; };
template <> struct HeaShape<longlong2, 10> { static constexpr int R = 4, CLB = 0; };
template <> struct HeaShape<longlong2, 12> { static constexpr int R = 4, CLB = 0; };
template <> struct HeaShape<longlong2, 14> { static constexpr int R = 4, CLB = 1; };

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
// (a, b) <- (a + b, a - b); FP32 as packed pairs
__device__ __forceinline__ void butterfly(float2 &a, float2 &b) {
    float2 s, d;
    asm("{\n\t.reg .b64 ra, rb, rm, rs, rd;\n\t"
        "mov.b64 ra, {%4, %5};\n\tmov.b64 rb, {%6, %7};\n\tmov.b64 rm, {%8, %8};\n\t"
        "add.rn.f32x2 rs, ra, rb;\n\tfma.rn.f32x2 rd, rb, rm, ra;\n\t"
        "mov.b64 {%0, %1}, rs;\n\tmov.b64 {%2, %3}, rd;\n\t}"
        : "=f"(s.x), "=f"(s.y), "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(-1.0f));
    a = s;
    b = d;
}
__device__ __forceinline__ void butterfly(double2 &a, double2 &b) {
    const double2 s = make_double2(a.x + b.x, a.y + b.y), d = make_double2(a.x - b.x, a.y - b.y);
    a = s;
    b = d;
}

// What a boundary of C needs: its coefficients, and its left half's amplitudes for the meet.
template <typename C> struct HeaNum { using Coef = C; using Out = C; };
template <> struct HeaNum<longlong2> { using Coef = int4; using Out = double2; };   // FP64 (fixed.h)

// Geometry of the sweep, all compile-time.  Window w holds local bits
// [lo(w), lo(w) + R) in registers and applies the Hadamards of bits
// [h0(w), h1(w)); the last window may overlap the one before.
template <int N, int R, int CLB>
struct Hea {
    static constexpr int NL = N - CLB, T = 1 << (NL - R), NW = (NL + R - 1) / R;
    static constexpr int kCta = T >= 32 ? (T == 32 ? 128 : T) : 128, GP = kCta / T;
    static constexpr int kStride = (1 << NL) + (T < 16 ? 8 : 0);   // group stride of the exchange buffer
    __host__ __device__ static constexpr int lo(int w) { return w * R < NL - R ? w * R : NL - R; }
    __host__ __device__ static constexpr int h0(int w) { return w * R; }
    __host__ __device__ static constexpr int h1(int w) { return (w + 1) * R < NL ? (w + 1) * R : NL; }
    // The slots that window w applies in a pass of the given direction: those that
    // touch its Hadamard bits and no bit of an earlier window.  Slot of chain bit j
    // (j >= 1) joins chain bits j-1 and j; the chain is bits first, first+1, .. mod N.
    __host__ __device__ static constexpr int first(int w, bool fwd) {
        return fwd ? (w == 0 ? N - 1 : h0(w)) : (w == 0 ? 0 : h0(w) - 1);
    }
    __host__ __device__ static constexpr int len(int w, bool fwd) {   // chain bits
        if (fwd) {
            const int last = w == NW - 1 ? (CLB ? NL : NL - 1) : h1(w);   // last chain bit
            return w == 0 ? last + 2 : last - h0(w) + 1;
        }
        if (w == NW - 1) return N - (h0(w) - 1) + 1;   // up to bit N-1, then bit 0
        return w == 0 ? h1(0) : h1(w) - (h0(w) - 1);
    }
    __host__ __device__ static constexpr int bit(int w, bool fwd, int j) { return (first(w, fwd) + j) % N; }
    __host__ __device__ static constexpr bool in_reg(int w, int b) { return b >= lo(w) && b < lo(w) + R; }
    // table index position of chain bit j: the register bits first
    __host__ __device__ static constexpr int regs(int w, bool fwd) {
        int c = 0;
        for (int j = 0; j < len(w, fwd); ++j) c += in_reg(w, bit(w, fwd, j)) ? 1 : 0;
        return c;
    }
    __host__ __device__ static constexpr int pos(int w, bool fwd, int j) {
        int r = 0, o = regs(w, fwd);
        for (int k = 0; k < j; ++k) (in_reg(w, bit(w, fwd, k)) ? r : o) += 1;
        return in_reg(w, bit(w, fwd, j)) ? r : o;
    }
    __host__ __device__ static constexpr int shift(int w, bool fwd) {   // register bit of the first register chain bit
        for (int j = 0; j < len(w, fwd); ++j)
            if (in_reg(w, bit(w, fwd, j))) return bit(w, fwd, j) - lo(w);
        return 0;
    }
    __host__ __device__ static constexpr int size(int w, bool fwd) { return len(w, fwd) < 2 ? 0 : 1 << len(w, fwd); }
    __host__ __device__ static constexpr int off(int w, bool fwd) {
        int o = 0;
        for (int k = 0; k < w; ++k) o += size(k, fwd);
        return o;
    }
    // the exchange between two windows stays inside a warp when both give the thread
    // bits above the lanes to the same bits
    __host__ __device__ static constexpr int ybit(int w, int j) { return j < lo(w) ? j : j + R; }
    __host__ __device__ static constexpr bool in_warp(int a, int b) {
        for (int j = 5; j < NL - R; ++j)
            if (ybit(a, j) != ybit(b, j)) return false;
        return true;
    }
    // the step of a pass whose exchange holds the group's barrier (the first that leaves the warp)
    __host__ __device__ static constexpr int meet_step(bool fwd) {
        for (int s = 0; s < NW - 1; ++s)
            if (!in_warp(fwd ? s : NW - 1 - s, fwd ? s + 1 : NW - 2 - s)) return s;
        return 0;
    }
    static constexpr int kTab = off(NW, true) > off(NW, false) ? off(NW, true) : off(NW, false);
    template <typename C>
    static constexpr size_t smem() {
        return ((size_t)GP * kStride + (size_t)GP * 3 * kTab + (size_t)GP * 2 * 4 * N) * sizeof(C);
    }
};

// Shared-memory slot of local amplitude y: its low bits XORed with the bits above
// the first window, so that the lanes of every window hit distinct banks (linear:
// the slot of disjoint bit groups is the XOR of their slots).
template <typename C, int R>
__host__ __device__ constexpr uint32_t hslot(uint32_t y) { return y ^ ((y >> R) & (sizeof(C) == 8 ? 15u : 7u)); }

template <typename C, int N, int R, int CLB>
__global__ void __launch_bounds__((Hea<N, R, CLB>::kCta), (512 / Hea<N, R, CLB>::kCta))   // at most 128 registers
    hea_sweep_kernel(int n, int cut, const PairInfo *__restrict__ pairs, int npairs,
                     const typename HeaNum<C>::Coef *__restrict__ slots, typename HeaNum<C>::Out *__restrict__ lscr,
                     double err_scale, double *__restrict__ tr, double *__restrict__ kappa,
                     double *__restrict__ err) {
    using H = Hea<N, R, CLB>;
    using Coef = typename HeaNum<C>::Coef;
    using Out = typename HeaNum<C>::Out;
    constexpr bool fix = std::is_same<C, longlong2>::value;
    static_assert(sizeof(Coef) == sizeof(C), "the shared-memory layout");
    constexpr int T = H::T, NW = H::NW, V = 1 << R, NL = H::NL;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int grp = threadIdx.x / T, t = threadIdx.x % T;
    const uint32_t rank = CLB ? blockIdx.x & 1u : 0u;
    const int pw = (int)(CLB ? blockIdx.x >> 1 : blockIdx.x) * H::GP + grp;
    const int p = pw < npairs ? pw : npairs - 1;   // spare groups repeat the last pair and write nothing
    C *buf = (C *)smem_raw + (size_t)grp * H::kStride;
    Coef *tabs = (Coef *)smem_raw + (size_t)H::GP * H::kStride + (size_t)grp * 3 * H::kTab;
    Coef *sl = (Coef *)smem_raw + (size_t)H::GP * (H::kStride + 3 * H::kTab) + (size_t)grp * 8 * N;
    const Coef *gs = slots + (size_t)p * n * N * 4;
    auto sync = [] {
        if constexpr (T <= 32) __syncwarp();
        else __syncthreads();
    };
    auto qubit = [&](int k) { return k < cut ? k : n - 1 - (k - cut); };
    auto forward = [&](int k) { return k < cut ? (k & 1) == 0 : (((cut - 1) ^ (n - 1 - k)) & 1) == 0; };
    auto load_slots = [&](int k) {   // pass k's N 2x2 matrices, 16 bytes per copy
        constexpr int per = 16 / (int)sizeof(C);
        if (k < n)
            for (int i = t; i < 4 * N / per; i += T)
                cp_async<16>(sl + (k & 1) * 4 * N + i * per, gs + (size_t)qubit(k) * N * 4 + i * per);
    };
    // value of chain bit b of this thread in window w (b outside the registers)
    auto outside = [&](auto wc, int b) -> uint32_t {
        constexpr int w = decltype(wc)::value;
        if (CLB && b == N - 1) return rank;
        return b < H::lo(w) ? ((uint32_t)t >> b) & 1u : ((uint32_t)t >> (b - R)) & 1u;
    };
    auto build_dir = [&](auto fc, const Coef *s, Coef *tab) {
        constexpr bool fwd = decltype(fc)::value;
        static_for<NW>([&](auto wc) {
            constexpr int w = decltype(wc)::value;
            for (int e = t; e < H::size(w, fwd); e += T) {
                C f;
                uint32_t prev = ((uint32_t)e >> H::pos(w, fwd, 0)) & 1u;
                static_for<H::len(w, fwd) - 1>([&](auto jc) {
                    constexpr int j = decltype(jc)::value + 1;
                    const uint32_t cur = ((uint32_t)e >> H::pos(w, fwd, j)) & 1u;
                    const Coef m = s[4 * H::bit(w, fwd, j) + 2 * cur + prev];
                    if constexpr (j > 1) f = cmul(f, m);
                    else if constexpr (fix) f = fix_join(m);
                    else f = m;
                    prev = cur;
                });
                if constexpr (fix) tab[H::off(w, fwd) + e] = fix_coef(f);
                else tab[H::off(w, fwd) + e] = f;
            }
        });
    };
    auto build = [&](int k) {
        if (forward(k)) build_dir(std::true_type{}, sl + (k & 1) * 4 * N, tabs + (k % 3) * H::kTab);
        else build_dir(std::false_type{}, sl + (k & 1) * 4 * N, tabs + (k % 3) * H::kTab);
    };
    C v[V];
    int scale = 0;   // fixed point: amplitudes are v 2^scale
    auto ones = [&] {
        if constexpr (fix) scale = 1 - kFixTop;
#pragma unroll
        for (int i = 0; i < V; ++i) {
            if constexpr (fix) v[i].x = 1ll << (kFixTop - 1);
            else v[i].x = 1;
            v[i].y = 0;
        }
    };
    // Fixed point: every thread's block has its own scale, published beside the amplitudes.  A
    // window's product and R Hadamards grow a component at most 16 sqrt(2) times and the CTAs'
    // Hadamard doubles it, to below 2^63.  Four copies: between two writes of one copy
    // lies an exchange with a barrier of the whole group (at most two in a row are a warp's).
    __shared__ int scale_sh[fix ? 4 * H::kCta : 1];
    [[maybe_unused]] int turn = 0;
    auto scales = [&] { return scale_sh + (4 * grp + (turn & 3)) * T; };
    // for the meet
    auto result = [&](const C &a) -> Out {
        if constexpr (fix) {
            const double f = ldexp(1.0, scale);
            return make_double2((double)a.x * f, (double)a.y * f);
        } else {
            return a;
        }
    };
    // window w's factors, then its Hadamards
    auto window = [&](auto wc, auto fc, const Coef *tab, bool ladder) {
        constexpr int w = decltype(wc)::value;
        constexpr bool fwd = decltype(fc)::value;
        if constexpr (H::size(w, fwd) > 0) {
            uint32_t o = H::off(w, fwd);
            static_for<H::len(w, fwd)>([&](auto jc) {
                constexpr int j = decltype(jc)::value, b = H::bit(w, fwd, j);
                if constexpr (!H::in_reg(w, b)) o += outside(wc, b) << H::pos(w, fwd, j);
            });
            constexpr int sh = H::shift(w, fwd), nr = H::regs(w, fwd);
#pragma unroll
            for (int i = 0; i < V; ++i) v[i] = cmul(v[i], tab[o + ((i >> sh) & ((1 << nr) - 1))]);
        }
        if (ladder) {
#pragma unroll
            for (int b = H::h0(w) - H::lo(w); b < H::h1(w) - H::lo(w); ++b)
#pragma unroll
                for (int i = 0; i < V; ++i)
                    if (!(i & (1 << b))) butterfly(v[i], v[i | (1 << b)]);
        }
    };
    auto base = [&](auto wc) {   // slot of the thread's register 0 in window w
        constexpr int l = H::lo(decltype(wc)::value);
        return hslot<C, R>(((uint32_t)t & ((1u << l) - 1u)) | (((uint32_t)t >> l) << (l + R)));
    };
    auto pass_dir = [&](auto fc, int k, bool ladder) {
        constexpr bool fwd = decltype(fc)::value;
        const Coef *tab = tabs + (k % 3) * H::kTab;
        static_for<NW>([&](auto kc) {
            constexpr int step = decltype(kc)::value, w = fwd ? step : NW - 1 - step;
            using WC = std::integral_constant<int, w>;
            window(WC{}, fc, tab, ladder);
            if constexpr (CLB > 0 && w == NW - 1) {
                if (ladder) {   // the Hadamard of the bit that numbers the CTAs
                    const uint32_t a0 = base(WC{});
#pragma unroll
                    for (int i = 0; i < V; ++i) buf[a0 ^ hslot<C, R>((uint32_t)i << H::lo(w))] = v[i];
                    if constexpr (fix) scales()[t] = scale;
                    cg::this_cluster().sync();
                    const C *other = cg::this_cluster().map_shared_rank(buf, rank ^ 1u);
                    [[maybe_unused]] int so = 0, top = 0;
                    if constexpr (fix) {
                        so = cg::this_cluster().map_shared_rank(scales(), rank ^ 1u)[t];
                        top = max(scale, so);
                        ++turn;
                    }
#pragma unroll
                    for (int i = 0; i < V; ++i) {
                        C u = other[a0 ^ hslot<C, R>((uint32_t)i << H::lo(w))];
                        if constexpr (fix) {
                            fix_align(u, so, top);
                            fix_align(v[i], scale, top);
                        }
                        v[i].x = rank ? u.x - v[i].x : v[i].x + u.x;
                        v[i].y = rank ? u.y - v[i].y : v[i].y + u.y;
                    }
                    if constexpr (fix) scale = top;
                    cg::this_cluster().sync();   // read before either side writes again
                }
            }
            if constexpr (step < NW - 1) {
                constexpr int wn = fwd ? w + 1 : w - 1;
                const uint32_t a0 = base(WC{}), a1 = base(std::integral_constant<int, wn>{});
                if constexpr (fix) {
                    fix_settle(v, scale);
                    scales()[t] = scale;
                }
#pragma unroll
                for (int i = 0; i < V; ++i) buf[a0 ^ hslot<C, R>((uint32_t)i << H::lo(w))] = v[i];
                // tables k+1 (over those of pass k-2, which everyone has left) and the
                // matrices of pass k+2 are in place after the pass's group barrier
                if constexpr (step == H::meet_step(fwd)) {
                    if (k + 1 < n) build(k + 1);
                    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
                }
                if constexpr (H::in_warp(w, wn)) __syncwarp();
                else __syncthreads();
#pragma unroll
                for (int i = 0; i < V; ++i) v[i] = buf[a1 ^ hslot<C, R>((uint32_t)i << H::lo(wn))];
                if constexpr (fix) {
                    // the thread that had register i's amplitude in window w
                    auto had = [](uint32_t y) { return (y & ((1u << H::lo(w)) - 1u)) | ((y >> (H::lo(w) + R)) << H::lo(w)); };
                    const int *e = scales() + had(((uint32_t)t & ((1u << H::lo(wn)) - 1u)) | (((uint32_t)t >> H::lo(wn)) << (H::lo(wn) + R)));
                    int top = e[0];
#pragma unroll
                    for (int i = 1; i < V; ++i) top = max(top, e[had((uint32_t)i << H::lo(wn))]);
#pragma unroll
                    for (int i = 0; i < V; ++i) fix_align(v[i], e[had((uint32_t)i << H::lo(wn))], top);
                    scale = top;
                    ++turn;
                }
            }
        });
    };
    auto commit = [] { asm volatile("cp.async.commit_group;\n" ::: "memory"); };
    load_slots(0);
    commit();
    load_slots(1);
    commit();
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    sync();
    build(0);
    sync();
    ones();
    Out *lp = lscr + (((size_t)pw << N) | ((size_t)rank << NL));
    for (int k = 0; k < n; ++k) {
        load_slots(k + 2);   // over pass k's matrices, whose tables are built
        commit();
        if (forward(k)) pass_dir(std::true_type{}, k, k + 1 < n);
        else pass_dir(std::false_type{}, k, k + 1 < n);
        if (k == cut - 1) {   // the left half is done; both halves end in the same window
            if (pw < npairs)
#pragma unroll
                for (int i = 0; i < V; ++i) lp[(size_t)i * T + t] = result(v[i]);
            ones();
            sync();   // the next pass may start in another window than this one ended in
        } else if (k + 1 < n) {   // the next pass goes on in the same window
            if constexpr (fix) fix_settle(v, scale);
        }
    }
    MeetAcc<Out> acc;
    if (pw < npairs) {
#pragma unroll
        for (int i = 0; i < V; ++i) {
            acc.add(lp[(size_t)i * T + t], result(v[i]));
            if ((i & 7) == 7) acc.flush();
        }
        acc.flush();
    }
    double s[4] = {acc.sr, acc.si, (double)acc.sa, (double)acc.s2};
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int d = (T < 32 ? T : 32) / 2; d > 0; d >>= 1) s[c] += __shfl_xor_sync(0xffffffffu, s[c], d);
    if constexpr (T > 32) {
        __shared__ double red[4][T / 32];
        __shared__ double part[4];
        if ((t & 31) == 0)
            for (int c = 0; c < 4; ++c) red[c][t >> 5] = s[c];
        __syncthreads();
        if (t == 0)
            for (int c = 0; c < 4; ++c) {
                s[c] = 0;
                for (int w = 0; w < T / 32; ++w) s[c] += red[c][w];
            }
        if constexpr (CLB > 0) {
            if (rank == 1 && t == 0) {
                double *p0 = cg::this_cluster().map_shared_rank(part, 0);
                for (int c = 0; c < 4; ++c) p0[c] = s[c];
            }
            cg::this_cluster().sync();
            if (t == 0)
                for (int c = 0; c < 4; ++c) s[c] += part[c];
        }
    }
    if (t == 0 && rank == 0 && pw < npairs) write_meet(pairs[pw], s, err_scale, tr, kappa, err);
}

// Boundaries of 2 and 4 bits in FP64: a lane per amplitude, the Hadamards by shuffles.  An FP64
// instruction takes an SM quarter about 77 cycles per warp whatever its lanes do, so this takes as many
// of them per pair as a thread per pair and 2^N times fewer one after another: one pair of n = 50, L = 3
// 95 us with its call against 669 with a thread per pair (548 as dense maps on a warp).
template <int N>
__global__ void __launch_bounds__(128) hea_lane_kernel(int n, int cut, const PairInfo *__restrict__ pairs, int npairs,
                                                       const double2 *__restrict__ slots, double err_scale,
                                                       double *__restrict__ tr, double *__restrict__ kappa,
                                                       double *__restrict__ err) {
    constexpr int V = 1 << N;
    const int id = blockIdx.x * blockDim.x + threadIdx.x, pw = id / V, i = id % V;
    const int p = pw < npairs ? pw : npairs - 1;   // spare lanes repeat the last pair and write nothing
    const double2 *gs = slots + (size_t)p * n * N * 4;
    auto load = [&](int k, double2 (&m)[N]) {
        const int q = k < cut ? k : n - 1 - (k - cut);
#pragma unroll
        for (int s = 0; s < N; ++s) m[s] = gs[((size_t)q * N + s) * 4 + 2 * ((i >> s) & 1) + ((i >> ((s + N - 1) % N)) & 1)];
    };
    double2 v = make_double2(1, 0), left = v, next[N];
    load(0, next);
    for (int k = 0; k < n; ++k) {
        double2 m[N];
#pragma unroll
        for (int s = 0; s < N; ++s) m[s] = next[s];
        if (k + 1 < n) load(k + 1, next);   // arrives while this qubit computes
#pragma unroll
        for (int s = 0; s < N; ++s) v = cmul(v, m[s]);
        if (k + 1 < n) {
#pragma unroll
            for (int b = 0; b < N; ++b) {
                const double2 u = make_double2(__shfl_xor_sync(0xffffffffu, v.x, 1 << b), __shfl_xor_sync(0xffffffffu, v.y, 1 << b));
                const double sign = (i >> b) & 1 ? -1.0 : 1.0;
                v = make_double2(fma(sign, v.x, u.x), fma(sign, v.y, u.y));   // (exact products)
            }
        }
        if (k == cut - 1) {
            left = v;
            v = make_double2(1, 0);
        }
    }
    MeetAcc<double2> acc;
    acc.add(left, v);
    double s[4] = {acc.sr, acc.si, acc.sa, acc.s2};
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int d = V / 2; d > 0; d >>= 1) s[c] += __shfl_xor_sync(0xffffffffu, s[c], d);
    if (i == 0 && pw < npairs) write_meet(pairs[pw], s, err_scale, tr, kappa, err);
}

// The same in FP32: a thread per pair, the whole boundary in registers,
// every slot applied by itself.
template <int N>
__global__ void __launch_bounds__(128) hea_thread_kernel(int n, int cut, const PairInfo *__restrict__ pairs, int npairs,
                                                         const float2 *__restrict__ slots, double err_scale,
                                                         double *__restrict__ tr, double *__restrict__ kappa,
                                                         double *__restrict__ err) {
    constexpr int V = 1 << N;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= npairs) return;
    const float2 *gs = slots + (size_t)p * n * N * 4;
    float2 v[V], left[V];
#pragma unroll
    for (int i = 0; i < V; ++i) v[i].x = 1, v[i].y = 0;
    for (int k = 0; k < n; ++k) {
        const int q = k < cut ? k : n - 1 - (k - cut);
#pragma unroll
        for (int s = 0; s < N; ++s) {
            float2 m[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) m[e] = gs[((size_t)q * N + s) * 4 + e];
#pragma unroll
            for (int i = 0; i < V; ++i) v[i] = cmul(v[i], m[2 * ((i >> s) & 1) + ((i >> ((s + N - 1) % N)) & 1)]);
        }
        if (k + 1 < n) {
#pragma unroll
            for (int b = 0; b < N; ++b)
#pragma unroll
                for (int i = 0; i < V; ++i)
                    if (!(i & (1 << b))) butterfly(v[i], v[i | (1 << b)]);
        }
        if (k == cut - 1) {
#pragma unroll
            for (int i = 0; i < V; ++i) {
                left[i] = v[i];
                v[i].x = 1;
                v[i].y = 0;
            }
        }
    }
    MeetAcc<float2> acc;
#pragma unroll
    for (int i = 0; i < V; ++i) {
        acc.add(left[i], v[i]);
        if ((i & 7) == 7) acc.flush();
    }
    acc.flush();
    const double s[4] = {acc.sr, acc.si, (double)acc.sa, (double)acc.s2};
    write_meet(pairs[p], s, err_scale, tr, kappa, err);
}

template <typename C, int N>
cudaError_t run_few_bits(const BrickDev &d, const PairInfo *pairs, int npairs, const C *slots, double err_scale, double *tr,
                         double *kappa, double *err, cudaStream_t st) {
    if constexpr (std::is_same<C, double2>::value) {
        constexpr int per = 128 >> N;   // pairs per CTA
        hea_lane_kernel<N><<<(npairs + per - 1) / per, 128, 0, st>>>(d.n, d.cut, pairs, npairs, slots, err_scale, tr, kappa, err);
    } else {
        hea_thread_kernel<N><<<(npairs + 127) / 128, 128, 0, st>>>(d.n, d.cut, pairs, npairs, slots, err_scale, tr, kappa, err);
    }
    return cudaGetLastError();
}

template <typename C, int N>
cudaError_t run_sweep(const BrickDev &d, const PairInfo *pairs, int npairs, const typename HeaNum<C>::Coef *slots,
                      typename HeaNum<C>::Out *lscr, double err_scale,
                      double *tr, double *kappa, double *err, cudaStream_t st) {
    constexpr int R = HeaShape<C, N>::R, CLB = HeaShape<C, N>::CLB;
    using H = Hea<N, R, CLB>;
    auto k = hea_sweep_kernel<C, N, R, CLB>;
    const size_t smem = H::template smem<C>();
    cudaError_t e = allow_smem(k, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    cfg.gridDim = dim3((unsigned)((npairs + H::GP - 1) / H::GP) << CLB);
    cfg.blockDim = dim3(H::kCta);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1 << CLB;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = CLB ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, d.n, d.cut, pairs, npairs, slots, lscr, err_scale, tr, kappa, err);
}

// C: FP32, or FP64 up to 4 bits; W: what the wider sweeps compute in
template <typename C, typename W>
cudaError_t launch_t(const BrickDev &d, const PairInfo *pairs, int npairs, const void *slots, void *lscr, double err_scale,
                     double *tr, double *kappa, double *err, cudaStream_t st) {
    const C *ts = (const C *)slots;
    const auto *ws = (const typename HeaNum<W>::Coef *)slots;
    auto *ls = (typename HeaNum<W>::Out *)lscr;
    switch (d.N) {
        case 2: return run_few_bits<C, 2>(d, pairs, npairs, ts, err_scale, tr, kappa, err, st);
        case 4: return run_few_bits<C, 4>(d, pairs, npairs, ts, err_scale, tr, kappa, err, st);
        case 6: return run_sweep<W, 6>(d, pairs, npairs, ws, ls, err_scale, tr, kappa, err, st);
        case 8: return run_sweep<W, 8>(d, pairs, npairs, ws, ls, err_scale, tr, kappa, err, st);
        case 10: return run_sweep<W, 10>(d, pairs, npairs, ws, ls, err_scale, tr, kappa, err, st);
        case 12: return run_sweep<W, 12>(d, pairs, npairs, ws, ls, err_scale, tr, kappa, err, st);
        case 14: return run_sweep<W, 14>(d, pairs, npairs, ws, ls, err_scale, tr, kappa, err, st);
        default: return cudaErrorInvalidValue;
    }
}

template <typename C, int N>
void shape_t(int *win_bits, int *threads) {
    using H = Hea<N, HeaShape<C, N>::R, HeaShape<C, N>::CLB>;
    *win_bits = HeaShape<C, N>::R;
    *threads = H::kCta;
}

}  // namespace

bool hea_shape(int N, bool fp32, int *win_bits, int *threads) {
    switch (N) {
        case 2: case 4: *win_bits = N; *threads = 128; return true;
        case 6: fp32 ? shape_t<float2, 6>(win_bits, threads) : shape_t<longlong2, 6>(win_bits, threads); return true;
        case 8: fp32 ? shape_t<float2, 8>(win_bits, threads) : shape_t<longlong2, 8>(win_bits, threads); return true;
        case 10: fp32 ? shape_t<float2, 10>(win_bits, threads) : shape_t<longlong2, 10>(win_bits, threads); return true;
        case 12: fp32 ? shape_t<float2, 12>(win_bits, threads) : shape_t<longlong2, 12>(win_bits, threads); return true;
        case 14: fp32 ? shape_t<float2, 14>(win_bits, threads) : shape_t<longlong2, 14>(win_bits, threads); return true;
        default: return false;
    }
}

cudaError_t launch_hea_sweep(const BrickDev &d, const PairInfo *pairs, int npairs, const void *slots, void *states,
                             bool fp32, double err_scale, double *tr, double *kappa, double *err, cudaStream_t st) {
    if (npairs <= 0) return cudaSuccess;
    return fp32 ? launch_t<float2, float2>(d, pairs, npairs, slots, states, err_scale, tr, kappa, err, st)
                : launch_t<double2, longlong2>(d, pairs, npairs, slots, states, err_scale, tr, kappa, err, st);
}

}  // namespace fpk
