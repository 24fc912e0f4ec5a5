// kernels_spiral.cu -- spiral sweep of the paper's hardware-efficient ansatz.
//
// The planner (make_spiral_plan) turns Tr(U^dagger V) of an ensemble whose
// wires are rings of segments, each tapped by one CZ, into a sequence of
// in-place 4x4 maps on a state of 2^bits amplitudes (one bit per CZ of a bond
// plus an auxiliary bit).  Per pair:
//   spiral_maps_kernel   the coefficients of every map from the pair's merged
//                        1-qubit operators (FP64 products, stored in C; FP32 as
//                        broadcast pairs for packed FMAs);
//   spiral_win_kernel    register windows: consecutive maps that walk at most R
//                        state bits run on 2^R amplitudes per thread in
//                        registers, one barrier per window.  The state sits
//                        in shared memory (swizzled), in one CTA or split
//                        over a cluster of 2 to 16 CTAs (distributed shared memory);
//   spiral_sweep_kernel  one map per pass (small states, or states too large
//                        for four CTAs: a per-pair global slice).
// Both sweeps start from delta(aux, first bit) and end with the FP64 sum of
// the state = Tr, its cancellation ratio and rounding-error estimate.
//
// Arithmetic bounds the windows (the FMA pipe in FP32, the FP64 pipe at 1/77 of
// its rate in FP64), so a map is applied by its type, not as 16 entries: the
// coupling H as two additions, then 2 products per output (SP_MID, the bulk) or
// 1, in place of 4 products (SP_MID: 20 packed operations instead of 32, RL, LL
// 12, DIAG 8).  And no window touches a freed bit's zero half (SpiralWin::half).
// n = 50, about 2,000 pairs per depth: FP32 L = 8 (two CTAs) 36.8 ms instead of 47, L = 7 (one
// CTA) 4.5 ms instead of 7.0; FP64 with few pairs (four CTAs) 20.9 ms instead of 44.  The two-CTA
// form is held back by its cross windows and barriers (30 % of the issue slots, 16 warps).
// FP64 L = 8, 4 pairs: 16 CTAs each 4.7 ms, 4 CTAs each 13.9.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>

#include "kernels.h"

namespace cg = cooperative_groups;

namespace fpk {
namespace {

template <int X> constexpr int kLog2 = 1 + kLog2<X / 2>;
template <> constexpr int kLog2<1> = 0;

__device__ __forceinline__ uint32_t ins0s(uint32_t x, int p) {   // insert a zero bit at position p
    return (x & ((1u << p) - 1u)) | ((x >> p) << (p + 1));
}

// Shared-memory slot of local amplitude y: y ^ fold4(y >> 4).  Linear over
// XOR, so the slot of a sum of disjoint bit groups is the XOR of their slots.
__device__ __forceinline__ uint32_t swz(uint32_t y) {
    const uint32_t q = y >> 4;
    return y ^ ((q ^ (q >> 4) ^ (q >> 8) ^ (q >> 12)) & 15u);
}

template <typename C> __device__ __forceinline__ C mk(double re, double im);
template <> __device__ __forceinline__ double2 mk<double2>(double re, double im) { return make_double2(re, im); }
template <> __device__ __forceinline__ float2 mk<float2>(double re, double im) { return make_float2((float)re, (float)im); }

__device__ __forceinline__ double2 zm(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// Coefficients of a stored map: 8 (entry 4 ia + 2 ob + oa of the types with two 1-qubit
// operators) or 4 (entry 2 ob + ia), see spiral_maps_kernel.  FP64 keeps them as they are;
// FP32 keeps a coefficient t as the pairs (tr, tr) and (-ti, ti), so that acc += t x is
// two packed FMAs: (tr, tr) * (xr, xi) + (-ti, ti) * (xi, xr).
constexpr int kCoefs = 8;
template <typename C> struct MapW { static constexpr int w = kCoefs; };
template <> struct MapW<float2> { static constexpr int w = 2 * kCoefs; };

__device__ __forceinline__ void put_entry(double2 *dst, int e, double2 t) { dst[e] = t; }
__device__ __forceinline__ void put_entry(float2 *dst, int e, double2 t) {   // one 16-byte store
    *reinterpret_cast<float4 *>(dst + 2 * e) = make_float4((float)t.x, (float)t.x, (float)-t.y, (float)t.y);
}

// One thread per coefficient, so the 8 threads of a map store its record contiguously.
//   SP_MID, SP_MID_AUX, SP_MID_RR: F[o_a][i_a] G[o_b][o_a] at 4 i_a + 2 o_b + o_a
//   the others (but SP_START):     G[o_b][i_a] at 2 o_b + i_a
template <typename C>
__global__ void spiral_maps_kernel(const PairInfo *__restrict__ pairs, int npairs, const SpiralMap *__restrict__ sm,
                                   int nmaps, const double2 *__restrict__ merged, C *__restrict__ maps) {
    const int gid = blockIdx.x * blockDim.x + threadIdx.x;
    const int m = gid / kCoefs, e = gid % kCoefs;
    if (m >= nmaps) return;
    const SpiralMap s = sm[m];
    if (s.type == SP_START || (s.f < 0 && e >= 4)) return;
    for (int p = blockIdx.y; p < npairs; p += gridDim.y) {   // grid.y is capped at 65535
        const int64_t mo = pairs[p].merged_off;
        auto mat = [&](int k, int r, int c) { return merged[(mo + k) * 16 + 2 * r + c]; };
        const int a = e & 1, ob = (e >> 1) & 1;
        double2 v = mat(s.g, ob, a);
        if (s.f >= 0) v = zm(mat(s.f, a, e >> 2), v);
        put_entry(maps + ((size_t)p * nmaps + m) * MapW<C>::w, e, v);
    }
}

__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {   // a * b + c, lane-wise
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
        "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
__device__ __forceinline__ float2 fmul2(float2 a, float2 b) {
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "mul.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 fadd2(float2 a, float2 b) {
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}

// complex sum, difference and t0 x0 (+ t1 x1) for a stored coefficient t
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return fadd2(a, b); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return ffma2(b, make_float2(-1.f, -1.f), a); }   // exact product
struct Coef64 { double2 t; };
struct Coef32 { float2 r, i; };
__device__ __forceinline__ Coef64 coef(const double2 *T, int e) { return {T[e]}; }
__device__ __forceinline__ Coef32 coef(const float2 *T, int e) {
    const float4 q = *reinterpret_cast<const float4 *>(T + 2 * e);
    return {make_float2(q.x, q.y), make_float2(q.z, q.w)};
}
__device__ __forceinline__ double2 cmul(const Coef64 &c, double2 x) {
    return make_double2(fma(-c.t.y, x.y, c.t.x * x.x), fma(c.t.y, x.x, c.t.x * x.y));
}
__device__ __forceinline__ double2 cmac(const Coef64 &c, double2 x, double2 acc) {
    acc.x = fma(c.t.x, x.x, acc.x);
    acc.x = fma(-c.t.y, x.y, acc.x);
    acc.y = fma(c.t.x, x.y, acc.y);
    acc.y = fma(c.t.y, x.x, acc.y);
    return acc;
}
__device__ __forceinline__ float2 cmul(const Coef32 &c, float2 x) {
    return ffma2(c.i, make_float2(x.y, x.x), fmul2(c.r, x));
}
__device__ __forceinline__ float2 cmac(const Coef32 &c, float2 x, float2 acc) {
    return ffma2(c.i, make_float2(x.y, x.x), ffma2(c.r, x, acc));
}

// A map of SpiralType on the quads x[i_a][i_b] of a register block (or of one quad): first
// PRE, what becomes of the input of bit b: 0 nothing, 1 the coupling H, 2 only i_b = 0 (a
// freed bit); then CORE for each output bit o_b: 0 F and G (8 coefficients), 1 G with the
// bit a kept (4), 2 G with i_a summed and the output bit a zero (4), 3 the start (a = b,
// old a summed).  All quads pass one stage before the next, in place, so that the
// coefficients of one o_b are live at a time: with all 8 a window of 32 amplitudes spills.
template <typename C, int PRE, int CORE>
struct TypedMap {
    const C *T;
    template <int N, int A, int B>
    __device__ __forceinline__ void apply(C (&v)[N]) const {
        if constexpr (PRE != 0) {
#pragma unroll
            for (int x = 0; x < N; ++x) {
                if (x & B) continue;
                const C x0 = v[x], x1 = v[x | B];
                if constexpr (PRE == 1) v[x] = cadd(x0, x1);
                v[x | B] = PRE == 1 ? csub(x0, x1) : x0;
            }
        }
#pragma unroll
        for (int ob = 0; ob < 2; ++ob) {
            using K = decltype(coef(T, 0));
            if constexpr (CORE == 3) {
#pragma unroll
                for (int x = 0; x < N; ++x) {
                    if ((x & A) || ((x & B) != 0) != (ob != 0)) continue;
                    const C y = cadd(v[x], v[x | A]);
                    v[x] = ob == 0 ? y : mk<C>(0.0, 0.0);
                    v[x | A] = ob == 0 ? mk<C>(0.0, 0.0) : y;
                }
            } else {
                const K t00 = coef(T, 2 * ob), t01 = coef(T, 2 * ob + 1);
                K t10 = t00, t11 = t00;
                if constexpr (CORE == 0) { t10 = coef(T, 4 + 2 * ob); t11 = coef(T, 4 + 2 * ob + 1); }
#pragma unroll
                for (int x = 0; x < N; ++x) {
                    if ((x & A) || ((x & B) != 0) != (ob != 0)) continue;
                    const C u0 = v[x], u1 = v[x | A];
                    if constexpr (CORE == 0) {
                        v[x] = cmac(t10, u1, cmul(t00, u0));
                        v[x | A] = cmac(t11, u1, cmul(t01, u0));
                    } else if constexpr (CORE == 1) {
                        v[x] = cmul(t00, u0);
                        v[x | A] = cmul(t01, u1);
                    } else {
                        v[x] = cmac(t01, u1, cmul(t00, u0));
                        v[x | A] = mk<C>(0.0, 0.0);
                    }
                }
            }
        }
    }
};

// f(the map of this type)
template <typename C, typename F>
__device__ __forceinline__ void with_map(int type, const C *__restrict__ T, F f) {
    switch (type) {
        case SP_MID: f(TypedMap<C, 1, 0>{T}); break;
        case SP_DIAG_BA: f(TypedMap<C, 0, 1>{T}); break;
        case SP_START: f(TypedMap<C, 1, 3>{T}); break;
        case SP_MID_AUX: f(TypedMap<C, 0, 0>{T}); break;
        case SP_RL: f(TypedMap<C, 1, 1>{T}); break;
        case SP_MID_RR: f(TypedMap<C, 2, 0>{T}); break;
        case SP_RR: f(TypedMap<C, 2, 1>{T}); break;
        case SP_LL: f(TypedMap<C, 1, 2>{T}); break;
        default: f(TypedMap<C, 0, 2>{T}); break;   // SP_LL_AUX
    }
}

__device__ __forceinline__ void cp_async16(void *smem_dst, const void *gmem_src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

__device__ __forceinline__ double wsum_s(double v) {
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
    return v;
}

// Block sums of (Re, Im, |t|, |t|^2) over the amplitudes this CTA holds; the
// totals land in thread 0.
template <typename C>
__device__ __forceinline__ void block_sums(const C *st, uint32_t S, double (&red)[4][16], double (&out)[4]) {
    double sr = 0, si = 0, sa = 0, s2 = 0;
    for (uint32_t x = threadIdx.x; x < S; x += blockDim.x) {
        const double re = (double)st[x].x, im = (double)st[x].y, q = re * re + im * im;
        sr += re; si += im; sa += sqrt(q); s2 += q;
    }
    sr = wsum_s(sr); si = wsum_s(si); sa = wsum_s(sa); s2 = wsum_s(s2);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) { red[0][wid] = sr; red[1][wid] = si; red[2][wid] = sa; red[3][wid] = s2; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int c = 0; c < 4; ++c) {
            out[c] = 0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) out[c] += red[c][w];
        }
    }
}

__device__ __forceinline__ void write_result(const PairInfo &pi, const double (&s)[4], double err_scale, double *tr,
                                             double *kappa, double *err) {
    tr[2 * pi.out] = s[0];
    tr[2 * pi.out + 1] = s[1];
    const double mag = sqrt(s[0] * s[0] + s[1] * s[1]);
    if (kappa) kappa[pi.out] = mag > 0 ? s[2] / mag : __longlong_as_double(0x7ff0000000000000LL);
    if (err) err[pi.out] = err_scale * (sqrt(s[3]) + mag);
}

template <typename C, bool SMEM>
__global__ void __launch_bounds__(512) spiral_sweep_kernel(const PairInfo *__restrict__ pairs, const SpiralMap *__restrict__ sm,
                                                           int nmaps, int bits, int first_bit,
                                                           const C *__restrict__ maps, C *__restrict__ scratch,
                                                           double err_scale, double *__restrict__ tr,
                                                           double *__restrict__ kappa, double *__restrict__ err) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[4][16];
    const uint32_t S = 1u << bits;
    C *st = SMEM ? (C *)smem_raw : scratch + (size_t)blockIdx.x * S;
    const int aux = bits - 1;
    for (uint32_t x = threadIdx.x; x < S; x += blockDim.x)
        st[x] = mk<C>((((x >> aux) ^ (x >> first_bit)) & 1u) ? 0.0 : 1.0, 0.0);
    __syncthreads();
    const C *mp = maps + (size_t)blockIdx.x * nmaps * MapW<C>::w;
    for (int k = 0; k < nmaps; ++k) {
        const SpiralMap s = sm[k];
        const C *T = mp + (size_t)k * MapW<C>::w;
        const int lo = s.a < s.b ? s.a : s.b, hi = s.a < s.b ? s.b : s.a;
        const uint32_t ia = 1u << s.a, ib = 1u << s.b;
        with_map<C>(s.type, T, [&](const auto &map) {
            for (uint32_t q = threadIdx.x; q < (S >> 2); q += blockDim.x) {
                const uint32_t i0 = ins0s(ins0s(q, lo), hi);
                C v[4] = {st[i0], st[i0 | ia], st[i0 | ib], st[i0 | ia | ib]};
                map.template apply<4, 1, 2>(v);
                st[i0] = v[0];
                st[i0 | ia] = v[1];
                st[i0 | ib] = v[2];
                st[i0 | ia | ib] = v[3];
            }
        });
        __syncthreads();
    }
    double s[4];
    block_sums<C>(st, S, red, s);
    if (threadIdx.x == 0) write_result(pairs[blockIdx.x], s, err_scale, tr, kappa, err);
}

// The window's maps: map k acts on its walk's bits k and k + 1.
template <typename C, int R, int K = 0>
__device__ __forceinline__ void win_maps(int n_maps, const SpiralMap *__restrict__ sm, C (&v)[1 << R], const C *T) {
    if constexpr (K + 1 < R) {
        if (K >= n_maps) return;
        with_map<C>(sm[K].type, T + K * MapW<C>::w, [&](const auto &map) { map.template apply<(1 << R), 1 << K, 2 << K>(v); });
        win_maps<C, R, K + 1>(n_maps, sm, v, T);
    }
}

// Distributed shared memory through 32-bit shared::cluster addresses.
__device__ __forceinline__ uint32_t cluster_addr(const void *p, uint32_t rank) {
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ float2 dsm_ld(uint32_t a, float2) {
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ double2 dsm_ld(uint32_t a, double2) {
    double2 v;
    asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void dsm_st(uint32_t a, float2 v) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void dsm_st(uint32_t a, double2 v) {
    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(v.x), "d"(v.y) : "memory");
}

template <int CL>
__device__ __forceinline__ void win_sync(bool cluster_wide) {
    if constexpr (CL > 1) {
        if (cluster_wide) { cg::this_cluster().sync(); return; }
    }
    __syncthreads();
}

// Address of rank r's part in the cluster window: kept for up to 4 ranks, else computed.
template <int CL> struct CtaParts {
    static constexpr int n = CL <= 4 ? CL : 1;
    uint32_t ac[n];
    __device__ __forceinline__ explicit CtaParts(const void *st) {
#pragma unroll
        for (int r = 0; r < n; ++r) ac[r] = CL == 1 ? 0u : CL <= 4 ? cluster_addr(st, r) : (uint32_t)__cvta_generic_to_shared(st);
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t r) const {
        if constexpr (CL == 1) return ac[0];
        else if constexpr (CL == 2) return r ? ac[1] : ac[0];
        else if constexpr (CL == 4) return (r & 2) ? ((r & 1) ? ac[3] : ac[2]) : ((r & 1) ? ac[1] : ac[0]);
        else {
            uint32_t a;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(ac[0]), "r"(r));
            return a;
        }
    }
};

// Register windows over a state held in the shared memory of CL = 1, 2, 4, 8 or 16
// CTAs (one pair per CTA or per cluster).  With CL > 1 the cluster bits h of an
// amplitude give its CTA rank; a window holding one of them
// ("cross" window) reads and writes other CTAs' parts through distributed
// shared memory and is fenced by cluster barriers; the other windows stay in
// their own CTA.  Addressing: SpiralWin.  8 and 16 CTAs serve FP64 batches of a few pairs
// (spiral_variant in api.cu chooses): an FP64 instruction occupies its SM quarter for about 77 cycles, so a
// pair is as fast as the number of quarters that share it.
// Threads per CTA: the FP32 two-CTA form runs one CTA per SM (its half of the
// state fills the shared memory), so it takes as many warps as its registers allow.
template <typename C, int CL> struct WinThreads { static constexpr int n = 256; };
template <> struct WinThreads<float2, 2> { static constexpr int n = 512; };

template <typename C, int R, int CL>
__global__ void __launch_bounds__(WinThreads<C, CL>::n, sizeof(C) == 8 ? 512 / WinThreads<C, CL>::n : 1)
    spiral_win_kernel(const PairInfo *__restrict__ pairs, const SpiralWin *__restrict__ wins, int nwins,
                                                         const SpiralMap *__restrict__ sm, int nmaps, int bits,
                                                         int first_bit, SpiralCut cut, const C *__restrict__ maps,
                                                         double err_scale, double *__restrict__ tr,
                                                         double *__restrict__ kappa, double *__restrict__ err) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[4][16];
    __shared__ double part[CL][4];   // CL > 1: ranks 1.. write their sums into rank 0
    constexpr int c = kLog2<CL>;
    constexpr int MB = kSpiralWinMaxMaps * MapW<C>::w;   // elements of one staged window of coefficients
    C *st = (C *)smem_raw;
    const uint32_t SL = 1u << (bits - c);
    C *mbuf = st + SL;   // two windows of maps: this one and the next (cp.async)
    uint32_t rank = 0;
    const CtaParts<CL> cta(st);
    double *part0 = &part[0][0];
    if constexpr (CL > 1) {
        cg::cluster_group cl = cg::this_cluster();
        rank = cl.block_rank();
        part0 = cl.map_shared_rank(&part[0][0], 0);
    }
    const int aux = bits - 1;
    for (uint32_t y = threadIdx.x; y < SL; y += blockDim.x) {
        uint32_t x = y;
#pragma unroll
        for (int q = 0; q < c; ++q) x = ins0s(x, cut.h[q]) | (((rank >> q) & 1u) << cut.h[q]);
        st[swz(y)] = mk<C>((((x >> aux) ^ (x >> first_bit)) & 1u) ? 0.0 : 1.0, 0.0);
    }
    const C *mp = maps + (size_t)(blockIdx.x / CL) * nmaps * MapW<C>::w;
    // 16-byte chunks of window v's maps into buffer v & 1
    auto stage = [&](int v) {
        const int chunks = wins[v].n_maps * (int)(MapW<C>::w * sizeof(C) / 16);
        const unsigned char *src = (const unsigned char *)(mp + (size_t)wins[v].first * MapW<C>::w);
        unsigned char *dst = (unsigned char *)(mbuf + (v & 1) * MB);
        for (int q = threadIdx.x; q < chunks; q += blockDim.x) cp_async16(dst + 16 * q, src + 16 * q);
    };
    if (nwins > 0) stage(0);
    cp_async_wait_all();
    win_sync<CL>(true);   // with CL > 1 also: every part exists before any remote access
    const uint32_t G = 1u << (bits - R - c);   // groups this CTA handles per window
    for (int w = 0; w < nwins; ++w) {
        const SpiralWin *W = wins + w;   // uniform reads (read-only path)
        const int n_pos = W->n_pos, first = W->first, n_maps = W->n_maps;
        const bool cross = CL > 1 && W->cross;
        if (w + 1 < nwins) stage(w + 1);   // lands while this window computes
        const C *mw = mbuf + (w & 1) * MB;
        const uint32_t Gw = G >> W->half;   // without the groups of a freed bit's zero half
        for (uint32_t t = threadIdx.x; t < Gw; t += blockDim.x) {
            const uint32_t tt = rank * G + t;
            uint32_t base = 0;
            for (int j = 0; j < n_pos; ++j) base ^= ((tt >> j) & 1u) ? W->gx[j] : 0u;
            C v[1 << R];
            uint32_t vx[R];
#pragma unroll
            for (int k = 0; k < R; ++k) vx[k] = W->vx[k];
            auto at = [&](int i) {
                uint32_t a = base;
#pragma unroll
                for (int k = 0; k < R; ++k) if ((i >> k) & 1) a ^= vx[k];
                return a;
            };
            auto remote = [&](uint32_t a) { return cta(a >> 16) + (a & 0xffffu) * (uint32_t)sizeof(C); };
            if (!cross) {   // rank bits are its own
#pragma unroll
                for (int i = 0; i < (1 << R); ++i) v[i] = st[at(i) & 0xffffu];
            } else {
#pragma unroll
                for (int i = 0; i < (1 << R); ++i) v[i] = dsm_ld(remote(at(i)), C());
            }
            win_maps<C, R>(n_maps, sm + first, v, mw);
            // the store addresses are rebuilt (not kept live across the maps)
            asm volatile("" : "+r"(base), "+l"(W));
#pragma unroll
            for (int k = 0; k < R; ++k) vx[k] = W->vx[k];
            if (!cross) {
#pragma unroll
                for (int i = 0; i < (1 << R); ++i) st[at(i) & 0xffffu] = v[i];
            } else {
#pragma unroll
                for (int i = 0; i < (1 << R); ++i) dsm_st(remote(at(i)), v[i]);
            }
        }
        const bool next_cross = CL > 1 && w + 1 < nwins && wins[w + 1].cross;
        cp_async_wait_all();   // the next window's maps are in place before the barrier
        win_sync<CL>(cross || next_cross);
    }
    double s[4];
    block_sums<C>(st, SL, red, s);
    if constexpr (CL > 1) {
        if (rank > 0 && threadIdx.x == 0)
            for (int k = 0; k < 4; ++k) part0[(rank - 1) * 4 + k] = s[k];
        cg::this_cluster().sync();   // every rank's sums are in rank 0; ranks > 0 may exit after this
        if (rank == 0 && threadIdx.x == 0) {
            for (int r = 1; r < CL; ++r)
                for (int k = 0; k < 4; ++k) s[k] += part[r - 1][k];
            write_result(pairs[blockIdx.x / CL], s, err_scale, tr, kappa, err);
        }
    } else {
        if (threadIdx.x == 0) write_result(pairs[blockIdx.x], s, err_scale, tr, kappa, err);
    }
}

template <typename C, int R, int CL>
cudaLaunchConfig_t win_config(int npairs, int bits, cudaLaunchAttribute *attr, cudaStream_t st) {
    constexpr int c = kLog2<CL>;
    const uint32_t G = 1u << (bits - R - c);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(npairs * CL));
    cfg.blockDim = dim3((unsigned)std::min<uint32_t>(WinThreads<C, CL>::n, std::max<uint32_t>(32u, G)));
    cfg.dynamicSmemBytes = (((size_t)1 << (bits - c)) + 2 * kSpiralWinMaxMaps * MapW<C>::w) * sizeof(C);
    cfg.stream = st;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = CL;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

template <typename C, int R, int CL>
cudaError_t win_prepare() {
    auto k = spiral_win_kernel<C, R, CL>;
    cudaError_t e = allow_smem(k, kSpiralSmemMax + 2 * kSpiralWinMaxMaps * MapW<C>::w * sizeof(C));   // a CTA's part, two windows' maps
    if (e == cudaSuccess && CL > 8) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

// clusters of this form that the device holds at a time (0: it cannot run them)
template <int CL>
int resident_fp64(int bits) {
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = win_config<double2, 4, CL>(1, bits, attr, nullptr);
    int n = 0;
    if (win_prepare<double2, 4, CL>() != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, spiral_win_kernel<double2, 4, CL>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

template <typename C, int R, int CL>
cudaError_t win_t(const PairInfo *pairs, int npairs, const SpiralWin *wins, int nwins, const SpiralMap *sm, int nmaps,
                  int bits, int first_bit, const SpiralCut &cut, const void *maps, double err_scale, double *tr, double *kappa,
                  double *err, cudaStream_t st) {
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = win_config<C, R, CL>(npairs, bits, attr, st);
    cudaError_t e = win_prepare<C, R, CL>();
    if (e != cudaSuccess) return e;
    return cudaLaunchKernelEx(&cfg, spiral_win_kernel<C, R, CL>, pairs, wins, nwins, sm, nmaps, bits, first_bit, cut,
                              (const C *)maps, err_scale, tr, kappa, err);
}

template <typename C>
cudaError_t sweep_t(const PairInfo *pairs, int npairs, const SpiralMap *sm, int nmaps, int bits, int first_bit,
                    const void *maps, void *scratch, double err_scale, double *tr, double *kappa, double *err,
                    cudaStream_t st) {
    const size_t bytes = ((size_t)1 << bits) * sizeof(C);
    const int threads = bits >= 11 ? 512 : (bits >= 9 ? 128 : 32);
    if (bytes <= kSpiralSmemMax) {
        auto k = spiral_sweep_kernel<C, true>;
        cudaError_t e = allow_smem(k, kSpiralSmemMax);
        if (e != cudaSuccess) return e;
        k<<<npairs, threads, bytes, st>>>(pairs, sm, nmaps, bits, first_bit, (const C *)maps, nullptr, err_scale, tr,
                                          kappa, err);
    } else {
        spiral_sweep_kernel<C, false><<<npairs, threads, 0, st>>>(pairs, sm, nmaps, bits, first_bit, (const C *)maps,
                                                                 (C *)scratch, err_scale, tr, kappa, err);
    }
    return cudaGetLastError();
}

}  // namespace

size_t spiral_map_elems(bool fp32) { return fp32 ? MapW<float2>::w : MapW<double2>::w; }

SpiralConfig spiral_config(int bits, bool fp32, int min_split) {
    SpiralConfig c;
    const size_t bytes = ((size_t)1 << bits) * (fp32 ? sizeof(float2) : sizeof(double2));
    c.split = bytes <= kSpiralSmemMax ? 0 : bytes <= 2 * kSpiralSmemMax ? 1 : bytes <= 4 * kSpiralSmemMax ? 2 : -1;
    if (const char *ev = std::getenv("FP_SPIRAL_SPLIT")) min_split = std::max(min_split, std::atoi(ev));   // tuning
    if (c.split >= 0) c.split = std::max(c.split, std::min(min_split, fp32 ? 2 : kSpiralMaxSplit));
    // measured on GB300 (n = 50, depths 5..8): 5-bit windows from 2^13 FP32
    // amplitudes up, else 4
    c.R = fp32 && bits >= 13 ? 5 : 4;
    if (const char *ev = std::getenv("FP_SPIRAL_WIN")) c.R = std::atoi(ev);   // tuning override: 0, 4 or 5
    if (c.R != 0 && c.R != 4 && !(c.R == 5 && fp32)) c.R = 4;
    // windows need 16 lane groups per CTA and a state in (distributed) shared memory
    if (c.split < 0 || bits - c.R - c.split < 4 || bits - c.R > kSpiralMaxPos) c.R = 0;
    if (c.R == 0) c.split = 0;
    c.scratch_elems = (c.R == 0 && bytes > kSpiralSmemMax) ? ((size_t)1 << bits) : 0;
    return c;
}

int spiral_resident(int bits, const SpiralConfig &cfg) {
    if (cfg.R != 4) return 0;
    switch (cfg.split) {
        case 0: return resident_fp64<1>(bits);
        case 1: return resident_fp64<2>(bits);
        case 2: return resident_fp64<4>(bits);
        case 3: return resident_fp64<8>(bits);
        default: return resident_fp64<16>(bits);
    }
}

double spiral_wave_us(int bits, int split) {
    const int w = bits - 4 - 5 - split;   // log2 of a CTA's warps of groups
    return 14.8 * (w > 2 ? 1 << (w - 2) : 1) + (split ? 2.5 : 0.7);
}

cudaError_t launch_spiral(const PairInfo *pairs, int npairs, const SpiralMap *sm, int nmaps, int bits, int first_bit,
                          const SpiralConfig &cfg, const SpiralWin *wins, int nwins, const SpiralCut &cut,
                          const double2 *merged, void *maps, void *scratch, bool fp32, double err_scale, double *tr,
                          double *kappa, double *err, cudaStream_t st) {
    if (npairs <= 0) return cudaSuccess;
    dim3 gm((kCoefs * nmaps + 255) / 256, std::min(npairs, 65535));
    if (fp32) spiral_maps_kernel<float2><<<gm, 256, 0, st>>>(pairs, npairs, sm, nmaps, merged, (float2 *)maps);
    else spiral_maps_kernel<double2><<<gm, 256, 0, st>>>(pairs, npairs, sm, nmaps, merged, (double2 *)maps);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (wins && cfg.R > 0) {
#define FP_SPIRAL_WIN_CASE(C, R, CL)                                                                               \
    return win_t<C, R, CL>(pairs, npairs, wins, nwins, sm, nmaps, bits, first_bit, cut, maps, err_scale, tr, kappa, \
                           err, st)
        const int CL = 1 << cfg.split;
        if (!fp32) {
            if (cfg.R != 4) return cudaErrorInvalidValue;
            if (CL == 1) FP_SPIRAL_WIN_CASE(double2, 4, 1);
            if (CL == 2) FP_SPIRAL_WIN_CASE(double2, 4, 2);
            if (CL == 4) FP_SPIRAL_WIN_CASE(double2, 4, 4);
            if (CL == 8) FP_SPIRAL_WIN_CASE(double2, 4, 8);
            if (CL == 16) FP_SPIRAL_WIN_CASE(double2, 4, 16);
        } else if (cfg.R == 4) {
            if (CL == 1) FP_SPIRAL_WIN_CASE(float2, 4, 1);
            if (CL == 2) FP_SPIRAL_WIN_CASE(float2, 4, 2);
            if (CL == 4) FP_SPIRAL_WIN_CASE(float2, 4, 4);
        } else if (cfg.R == 5) {
            if (CL == 1) FP_SPIRAL_WIN_CASE(float2, 5, 1);
            if (CL == 2) FP_SPIRAL_WIN_CASE(float2, 5, 2);
            if (CL == 4) FP_SPIRAL_WIN_CASE(float2, 5, 4);
        }
#undef FP_SPIRAL_WIN_CASE
        return cudaErrorInvalidValue;
    }
    return fp32 ? sweep_t<float2>(pairs, npairs, sm, nmaps, bits, first_bit, maps, scratch, err_scale, tr, kappa, err, st)
                : sweep_t<double2>(pairs, npairs, sm, nmaps, bits, first_bit, maps, scratch, err_scale, tr, kappa, err, st);
}

}  // namespace fpk
