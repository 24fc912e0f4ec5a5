// kernels_qudit.cu -- brickwork circuits of qudits (local dimension q = 3, 4):
// the dual-circuit sweep of the qubit path (brick.h) with q-ary segment
// variables.  The paper states its method for general local dimension (Sec.
// "Frame potential", and the qudit paragraph of Sec. "Algorithm description");
// its generalised-Hadamard formula serves only the ancilla form, which this
// direct trace contraction does not use.
//
// K1q  qudit_haar_maps: Haar U(q^2) gates in 64-bit fixed point (haar_fixed.h) and, in
//                     the same kernel, the q^2 x q^2 maps the sweep applies: Gaussian
//                     draws by all threads, Gram-Schmidt with a lane per row (3 or 2
//                     gates a warp, sums over the rows by shuffles), the maps entry by
//                     entry.  Bound: the integer pipe.  With FP64 Householder QR by a
//                     thread per gate (its 9 x 9 arrays in local memory) and a separate
//                     map kernel 500 pairs of l = 2 at n = 50, q = 3, nearly all of it
//                     this kernel, took 2.5 ms; they take 0.46.
// K3q  qudit_sweep:   one CTA per pair: the boundary over the 2m segment digits
//                     of one qudit (q^{2m} amplitudes, in shared memory when it
//                     fits, else in a per-pair global slot), both chain halves,
//                     then the FP64 meet with the cancellation ratio and the
//                     error estimate.
#include <cuda_runtime.h>

#include <algorithm>

#include "haar_items.h"
#include "kernels.h"
#include "meet.h"

namespace fpk {
namespace {

constexpr size_t kQuditSmem = 200 * 1024;   // shared memory of a boundary's two copies

// A stored map entry: FP64 the complex entry; FP32 the pairs (re, re), (-im, im), so that a
// complex multiply-add is two packed FMAs on (x.re, x.im) and (x.im, x.re).
struct alignas(16) Pair2 { float2 r, i; };
template <typename C> struct Entry;
template <> struct Entry<float2> { using T = Pair2; };
template <> struct Entry<double2> { using T = double2; };
template <typename C> using EntryT = typename Entry<C>::T;
__device__ __forceinline__ void put_entry(double2 *out, Fx2 z) { *out = fx_out<double2>(z, 60); }
__device__ __forceinline__ void put_entry(Pair2 *out, Fx2 z) {
    const float2 v = fx_out<float2>(z, 60);
    *out = {make_float2(v.x, v.x), make_float2(-v.y, v.y)};
}

template <int Q> constexpr int kGates = 4 * (32 / (Q * Q));   // gates per CTA: 12 (q = 3), 8 (q = 4)

template <int Q, typename C>
__global__ void __launch_bounds__(128) qudit_haar_maps_kernel(BrickDev d, uint64_t seed, int self_pair, Items it,
                                                              const PairInfo *__restrict__ pairs,
                                                              EntryT<C> *__restrict__ maps) {
    constexpr int D = Q * Q, G = kGates<Q>, GW = 32 / D, NB = (D * D + 1) / 2;
    constexpr int RS = D | 1;   // row stride: odd, so that the rows of a column lie in different banks
    __shared__ Fx2 sm[G][D * RS];
    __shared__ GateOf gate[G];
    __shared__ uint8_t on[G];
    const int64_t first = (int64_t)blockIdx.x * G;
    if (threadIdx.x < G) on[threadIdx.x] = gate_of(d, it, first + threadIdx.x, gate[threadIdx.x]) ? 1 : 0;
    __syncthreads();
    for (int i = threadIdx.x; i < G * NB; i += 128) {
        const int g = i / NB, j = i - g * NB;
        if (!on[g]) continue;
        const GateOf &o = gate[g];
        const U64x4 x = philox(seed, (uint64_t)j, (uint64_t)o.g, pairs[o.pair].pair, (uint64_t)(self_pair ? 0 : o.w));
#pragma unroll 1
        for (int h = 0; h < 2; ++h)
            if (const int e = 2 * j + h; e < D * D)
                sm[g][e / D * RS + e % D] = gauss_fixed(h ? x.x[2] : x.x[0], h ? x.x[3] : x.x[1]);
    }
    __syncthreads();
    {
        // lane = (gate of the warp, row); spare lanes repeat row 0 of the warp's first gate and
        // write nothing.  Every lane runs every step, so the shuffles are warp-wide.
        const int lane = threadIdx.x & 31;
        const bool act = lane < GW * D;
        const int gw = act ? lane / D : 0, r = act ? lane - gw * D : 0, g = (threadIdx.x >> 5) * GW + gw;
        auto src = [&](int k) { return act ? gw * D + (r + k) % D : lane; };
        const int s1 = src(1), s2 = src(2), s3 = src(3), s6 = src(6);
        // over the rows of a gate: threes of threes (D = 9) or halves (D = 16)
        auto rows = [&](auto x, auto op) {
            if constexpr (D == 9) {
                x = op(op(x, __shfl_sync(0xffffffffu, x, s3)), __shfl_sync(0xffffffffu, x, s6));
                return op(op(x, __shfl_sync(0xffffffffu, x, s1)), __shfl_sync(0xffffffffu, x, s2));
            } else {
#pragma unroll
                for (int k = 8; k > 0; k >>= 1) x = op(x, __shfl_xor_sync(0xffffffffu, x, k));
                return x;
            }
        };
        auto sum = [&](int64_t x) {
            return (int64_t)rows((long long)x, [](long long a, long long b) { return a + b; });
        };
        auto lead = [&](Fx2 v) { return rows(lead1_fixed(v), [](int a, int b) { return min(a, b); }); };
#pragma unroll 1
        for (int c = 0; c < D; ++c) {
            Fx2 v = sm[g][r * RS + c];
            if (c) {
                auto project = [&](Fx2 u) {
#pragma unroll 1
                    for (int k = 0; k < c; ++k) {
                        const Fx2 q = sm[g][r * RS + k], t = dot1_fixed(q, u);
                        sub1_fixed(u, q, halves(sum(t.x)), halves(sum(t.y)));
                    }
                    return u;
                };
                shift1_fixed(v, lead(v) - kRoom);
                v = project(v);
                // a second time where this gate needs it; the warp's other gates go along and keep
                // what they had, so that a gate is the same wherever in a batch it is made
                const int drop = lead(v) - kRoom;
                const bool again = act && on[g] && drop >= kRedo<D>;
                if (__any_sync(0xffffffffu, again)) {
                    Fx2 u = v;
                    shift1_fixed(u, drop);
                    u = project(u);
                    if (again) v = u;
                }
            }
            shift1_fixed(v, lead(v) - kUnitRoom<D>);
            int h;
            const Half y = inv_norm_fixed((uint64_t)sum(norm1_fixed(v)), h);
            scale1_fixed(v, y, h);
            if (act) sm[g][r * RS + c] = v;
            __syncwarp();
        }
    }
    __syncthreads();
    // maps, coalesced: entry e = row D + column; index e = w_tau + q w_tau+1 of the qudit's
    // segments, rows the neighbour's (x) in a left map, columns in a right one
    const bool outer = first >= it.inner;
    for (int i = threadIdx.x; i < (outer ? G / 2 : G) * D * D; i += 128) {
        const int p = i / (D * D), e = i - p * D * D, g = outer ? 2 * p : p;
        if (!on[g]) continue;
        const GateOf &o = gate[g];
        const bool left = o.b < d.cut;
        const int ex = left ? e / D : e % D, ey = left ? e % D : e / D;
        const int r = (ey / Q) * Q + ex / Q, c = (ey % Q) * Q + ex % Q;   // gate row (after), column (before): q y + x
        Fx2 z;
        if (!outer) {
            z = o.w ? sm[g][r * RS + c] : sm[g][c * RS + r];
            if (!o.w) z.y = -z.y;
        } else {   // U_l^dagger V_l, or V_1 U_1^dagger
            const bool mid = o.tl == d.l;
            z = {0, 0};
#pragma unroll 1
            for (int k = 0; k < D; ++k) {
                const Fx2 t = dot1_fixed(sm[g][mid ? k * RS + r : c * RS + k], sm[g + 1][mid ? k * RS + c : r * RS + k]);
                z.x += t.x;
                z.y += t.y;
            }
        }
        put_entry(&maps[((size_t)o.pair * maps_per_pair(d) + map_of(d, o)) * D * D + e], z);
    }
}

// acc + t x; the FP32 form takes x and its swapped copy xs
__device__ __forceinline__ double2 cfmaq(double2 t, double2 x, double2, double2 acc) {
    acc.x = fma(t.x, x.x, acc.x);
    acc.x = fma(-t.y, x.y, acc.x);
    acc.y = fma(t.x, x.y, acc.y);
    acc.y = fma(t.y, x.x, acc.y);
    return acc;
}
__device__ __forceinline__ float2 cfmaq(const Pair2 &t, float2 x, float2 xs, float2 acc) {
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rc, rd, re;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
        "mov.b64 rd, {%8, %9};\n\tmov.b64 re, {%10, %11};\n\t"
        "fma.rn.f32x2 re, ra, rc, re;\n\tfma.rn.f32x2 re, rb, rd, re;\n\tmov.b64 {%0, %1}, re;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(t.r.x), "f"(t.r.y), "f"(t.i.x), "f"(t.i.y), "f"(x.x), "f"(x.y), "f"(xs.x), "f"(xs.y), "f"(acc.x), "f"(acc.y));
    return d;
}
template <typename C> __device__ __forceinline__ C swapped(C x) {
    C s;
    s.x = x.y;
    s.y = x.x;
    return s;
}

__device__ __forceinline__ double qsum(double v) {
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
    return v;
}

// Results of a pair from the thread sums of its meet (all threads of the CTA).
__device__ __forceinline__ void qudit_results(double sr, double si, double sa, double s2, const PairInfo &pi,
                                              double err_scale, double *tr, double *kappa, double *err) {
    __shared__ double red[4][8];
    sr = qsum(sr); si = qsum(si); sa = qsum(sa); s2 = qsum(s2);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) { red[0][wid] = sr; red[1][wid] = si; red[2][wid] = sa; red[3][wid] = s2; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double s[4] = {0, 0, 0, 0};
        for (int c = 0; c < 4; ++c)
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s[c] += red[c][w];
        write_meet(pi, s, err_scale, tr, kappa, err);
    }
}

template <typename C>
__device__ __forceinline__ void meet_term(C l, C r, double &sr, double &si, double &sa, double &s2) {
    const double px = (double)l.x * r.x - (double)l.y * r.y, py = (double)l.x * r.y + (double)l.y * r.x;
    sr += px;
    si += py;
    sa += sqrt(px * px + py * py);
    s2 += px * px + py * py;
}

// Boundaries that fit shared memory twice (q^N <= 200 KB / 2): one CTA per pair, every map
// read from one copy and written to the other, so that one barrier per map suffices.  A
// work item is a group of q^2 amplitudes and q of its outputs (a boundary of 9^3 would keep
// 81 of 256 threads busy with a group each), or, for BIG boundaries, two groups and all
// their outputs, which reads every map entry from shared memory once for two products.
// The next map arrives by cp.async meanwhile.  The left half waits in `lscr`.
// Bound: FP32 issue.  500 pairs at n = 50, q = 3, FP32, sampler and maps included: l = 5 2.8 ms
// against 8.0, l = 4 1.0 against 5.0 (a group per thread in place, two barriers per map).
template <int Q, typename C, bool BIG>
__global__ void __launch_bounds__(256) qudit_smem_kernel(BrickDev d, const PairInfo *__restrict__ pairs,
                                                         const EntryT<C> *__restrict__ maps, C *__restrict__ lscr,
                                                         double err_scale, double *__restrict__ tr,
                                                         double *__restrict__ kappa, double *__restrict__ err) {
    constexpr int D = Q * Q, GI = BIG ? 2 : 1, OI = BIG ? Q : 1;   // groups and output rows of an item
    extern __shared__ __align__(16) unsigned char qsm[];
    __shared__ __align__(16) EntryT<C> T[2][D * D];
    const int p = blockIdx.x, N = d.N;
    uint32_t S = 1;
    for (int i = 0; i < N; ++i) S *= Q;
    C *A = (C *)qsm, *B = A + S;
    const EntryT<C> *mp = maps + (size_t)p * maps_per_pair(d) * D * D;
    const int nmaps = maps_per_pair(d);   // side 0's maps, then side 1's, in sweep order
    auto stage = [&](int k) {
        if (k < nmaps)
            for (int i = threadIdx.x; i < D * D; i += blockDim.x) cp_async<16>(&T[k & 1][i], &mp[(size_t)k * D * D + i]);
    };
    stage(0);
    int k = 0;
    for (int side = 0; side < 2; ++side) {
        const int par = d.delta_par[side];
        for (uint32_t w = threadIdx.x; w < S; w += blockDim.x) {
            bool ok = true;
            uint32_t x = w, prev = 0, w0 = 0;
            for (int t = 0; t < N; ++t) {   // digits t and t+1 (mod N) equal for t of parity par
                const uint32_t dig = x % Q;
                x /= Q;
                if (t == 0) w0 = dig;
                else if (((t - 1) & 1) == par) ok = ok && dig == prev;
                prev = dig;
            }
            if (((N - 1) & 1) == par) ok = ok && prev == w0;
            C v;
            v.x = ok ? 1 : 0;
            v.y = 0;
            A[w] = v;
        }
        for (int t = 0; t < d.n_layers[side]; ++t) {
            const int par_t = layer_parity(d, side, t);
            for (int j = 0; j < d.m; ++j, ++k) {
                cp_async_wait_all();
                __syncthreads();   // this map and the state are in place; the other buffers are free
                stage(k + 1);
                const EntryT<C> *Tk = T[k & 1];
                const int pa = 2 * j + par_t, pb = (pa + 1) % N;
                uint32_t sa = 1, sb = 1;   // powers of q
                for (int i = 0; i < pa; ++i) sa *= Q;
                for (int i = 0; i < pb; ++i) sb *= Q;
                const uint32_t plo = pa < pb ? sa : sb, phi = pa < pb ? sb : sa;
                const uint32_t ng = S / D, half = BIG ? (ng + 1) / 2 : ng;
                for (uint32_t item = threadIdx.x; item < half * (BIG ? 1 : Q); item += blockDim.x) {
                    const uint32_t og0 = item / half, g0 = item - og0 * half;
                    uint32_t base[GI];
                    C x[GI][D], xs[GI][D];
#pragma unroll
                    for (int u = 0; u < GI; ++u) {
                        const uint32_t g = u == 0 || g0 + half < ng ? g0 + u * half : g0;   // (odd count: the middle one twice)
                        const uint32_t r1 = g / plo, x1 = g + r1 * plo * (Q - 1);           // zero digits at the two positions
                        const uint32_t r2 = x1 / phi;
                        base[u] = x1 + r2 * phi * (Q - 1);
#pragma unroll
                        for (int e = 0; e < D; ++e) x[u][e] = A[base[u] + (e % Q) * sa + (e / Q) * sb], xs[u][e] = swapped(x[u][e]);
                    }
#pragma unroll 1
                    for (int oi = 0; oi < OI; ++oi) {
                        const uint32_t og = BIG ? (uint32_t)oi : og0;
                        C acc[GI][Q];
#pragma unroll
                        for (int u = 0; u < GI; ++u)
#pragma unroll
                            for (int o = 0; o < Q; ++o) acc[u][o].x = 0, acc[u][o].y = 0;
                        const EntryT<C> *row = Tk + og * Q * D;
#pragma unroll
                        for (int e = 0; e < D; ++e)
#pragma unroll
                            for (int o = 0; o < Q; ++o) {
                                const EntryT<C> tv = row[o * D + e];
#pragma unroll
                                for (int u = 0; u < GI; ++u) acc[u][o] = cfmaq(tv, x[u][e], xs[u][e], acc[u][o]);
                            }
#pragma unroll
                        for (int u = 0; u < GI; ++u)
#pragma unroll
                            for (int o = 0; o < Q; ++o) B[base[u] + o * sa + og * sb] = acc[u][o];   // output og q + o
                    }
                }
                C *tmp = A;
                A = B;
                B = tmp;
            }
        }
        __syncthreads();
        if (side == 0)
            for (uint32_t w = threadIdx.x; w < S; w += blockDim.x) lscr[(size_t)p * S + w] = A[w];
        // (each thread reads back what it wrote, and rewrites A only where it has read it)
    }
    double sr = 0, si = 0, sa = 0, s2 = 0;
    for (uint32_t w = threadIdx.x; w < S; w += blockDim.x) meet_term(lscr[(size_t)p * S + w], A[w], sr, si, sa, s2);
    qudit_results(sr, si, sa, s2, pairs[p], err_scale, tr, kappa, err);
}

// Larger boundaries: one CTA per pair, the state and the left boundary in the pair's
// global slot.  Maps are applied one at a time, in place:
// every thread takes groups of q^2 amplitudes that differ only in digits
// (tau, tau+1 mod N), one barrier per map.
template <int Q, typename C>
__global__ void __launch_bounds__(256) qudit_sweep_kernel(BrickDev d, const PairInfo *__restrict__ pairs,
                                                           const EntryT<C> *__restrict__ maps, C *__restrict__ gstate,
                                                           double err_scale, double *__restrict__ tr,
                                                           double *__restrict__ kappa, double *__restrict__ err) {
    constexpr int D = Q * Q;
    __shared__ EntryT<C> T[D * D];
    const int p = blockIdx.x, N = d.N;
    uint32_t S = 1;
    for (int i = 0; i < N; ++i) S *= Q;
    C *st = gstate + (size_t)p * 2 * S;
    C *lb = st + S;
    const EntryT<C> *mp = maps + (size_t)p * maps_per_pair(d) * D * D;
    uint32_t pw[32];
    pw[0] = 1;
    for (int i = 1; i <= N; ++i) pw[i] = pw[i - 1] * Q;
    for (int side = 0; side < 2; ++side) {
        // chain end: prod over tau of parity delta_par[side] of delta(w_tau, w_tau+1 mod N)
        const int par = d.delta_par[side];
        for (uint32_t w = threadIdx.x; w < S; w += blockDim.x) {
            bool ok = true;
            for (int tau = par; tau < N; tau += 2) {
                const uint32_t a = (w / pw[tau]) % Q, b = (w / pw[(tau + 1) % N]) % Q;
                ok = ok && a == b;
            }
            C v;
            v.x = ok ? 1 : 0;
            v.y = 0;
            st[w] = v;
        }
        __syncthreads();
        for (int t = 0; t < d.n_layers[side]; ++t) {
            const int par_t = layer_parity(d, side, t);
            for (int j = 0; j < d.m; ++j) {
                const EntryT<C> *src = mp + (size_t)map_index(d, side, t, j) * D * D;
                for (int i = threadIdx.x; i < D * D; i += blockDim.x) T[i] = src[i];
                __syncthreads();
                const int pa = 2 * j + par_t, pb = (pa + 1) % N;
                const uint32_t sa = pw[pa], sb = pw[pb];
                const int lo = pa < pb ? pa : pb, hi = pa < pb ? pb : pa;
                for (uint32_t gq = threadIdx.x; gq < S / D; gq += blockDim.x) {
                    // insert zero digits at positions lo and hi
                    const uint32_t a1 = gq % pw[lo], r1 = gq / pw[lo];
                    const uint32_t x1 = a1 + r1 * pw[lo + 1];
                    const uint32_t a2 = x1 % pw[hi], r2 = x1 / pw[hi];
                    const uint32_t base = a2 + r2 * pw[hi + 1];
                    C x[D];
#pragma unroll
                    for (int e = 0; e < D; ++e) x[e] = st[base + (e % Q) * sa + (e / Q) * sb];
                    // q outputs at a time: with all q^2 in flight the FP64 and q = 4 forms spilled
#pragma unroll 1
                    for (int og = 0; og < Q; ++og) {
                        C acc[Q];
#pragma unroll
                        for (int o = 0; o < Q; ++o) acc[o].x = 0, acc[o].y = 0;
#pragma unroll
                        for (int e = 0; e < D; ++e)
#pragma unroll
                            for (int o = 0; o < Q; ++o) acc[o] = cfmaq(T[(og * Q + o) * D + e], x[e], swapped(x[e]), acc[o]);
#pragma unroll
                        for (int o = 0; o < Q; ++o) st[base + o * sa + og * sb] = acc[o];
                    }
                }
                __syncthreads();
            }
        }
        if (side == 0) {
            for (uint32_t w = threadIdx.x; w < S; w += blockDim.x) lb[w] = st[w];
            __syncthreads();
        }
    }
    double sr = 0, si = 0, sa = 0, s2 = 0;
    for (uint32_t w = threadIdx.x; w < S; w += blockDim.x) meet_term(lb[w], st[w], sr, si, sa, s2);
    qudit_results(sr, si, sa, s2, pairs[p], err_scale, tr, kappa, err);
}

template <int Q, typename C>
cudaError_t run_qc(const BrickDev &d, uint64_t seed, const PairInfo *pairs, int npairs, int self_pair, void *ws,
                   double err_scale, double *tr, double *kappa, double *err, cudaStream_t st) {
    constexpr int D = Q * Q;
    size_t S = 1;
    for (int i = 0; i < d.N; ++i) S *= Q;
    EntryT<C> *maps = (EntryT<C> *)ws;
    C *state = (C *)(maps + (size_t)npairs * maps_per_pair(d) * D * D);
    const Items it = make_items(d, npairs, kGates<Q>);
    const unsigned grid = (unsigned)((it.inner + it.outer_count + kGates<Q> - 1) / kGates<Q>);
    qudit_haar_maps_kernel<Q, C><<<grid, 128, 0, st>>>(d, seed, self_pair, it, pairs, maps);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const size_t smem = 2 * S * sizeof(C);
    if (smem <= kQuditSmem) {
        // two groups a thread from 512 groups up (q = 3, l = 5), where they still fill 192 threads twice
        const bool big = S / D >= 512;
        auto kern = big ? qudit_smem_kernel<Q, C, true> : qudit_smem_kernel<Q, C, false>;
        if ((e = allow_smem(kern, kQuditSmem)) != cudaSuccess) return e;
        const int threads = big ? 192 : std::min(256, ((int)(S / Q) + 31) / 32 * 32);
        kern<<<npairs, threads, smem, st>>>(d, pairs, maps, state, err_scale, tr, kappa, err);
    } else {
        qudit_sweep_kernel<Q, C><<<npairs, 256, 0, st>>>(d, pairs, maps, state, err_scale, tr, kappa, err);
    }
    return cudaGetLastError();
}

}  // namespace

size_t qudit_workspace_per_pair(int q, const BrickDev &d, bool fp32) {
    const size_t D = (size_t)q * q, celem = fp32 ? sizeof(float2) : sizeof(double2);
    size_t S = 1;
    for (int i = 0; i < d.N; ++i) S *= (size_t)q;
    return (size_t)maps_per_pair(d) * D * D * 16 + (2 * S * celem <= kQuditSmem ? S : 2 * S) * celem;
}

cudaError_t launch_qudit(int q, const BrickDev &d, uint64_t seed, const PairInfo *pairs, int npairs, int self_pair,
                         bool fp32, void *ws, double err_scale, double *tr, double *kappa, double *err,
                         cudaStream_t st) {
    if (npairs <= 0) return cudaSuccess;
    switch (q) {
        case 3: return fp32 ? run_qc<3, float2>(d, seed, pairs, npairs, self_pair, ws, err_scale, tr, kappa, err, st)
                            : run_qc<3, double2>(d, seed, pairs, npairs, self_pair, ws, err_scale, tr, kappa, err, st);
        case 4: return fp32 ? run_qc<4, float2>(d, seed, pairs, npairs, self_pair, ws, err_scale, tr, kappa, err, st)
                            : run_qc<4, double2>(d, seed, pairs, npairs, self_pair, ws, err_scale, tr, kappa, err, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace fpk
