// kernels_haar.cu -- Haar U(4) gates (K1) in 64-bit fixed point (haar_fixed.h),
// and, for brickwork, the 4x4 maps of the boundary sweep (K2b) made from them in
// the same kernel.
//
// A CTA makes G gates in three phases over shared memory: the Gaussian draws (8
// Philox blocks per gate, spread over all threads), Gram-Schmidt (one thread per
// gate, its columns in its own slice), and the output: the gate as 16 doubles
// pairs (raw records), or its realigned map (brick.h) rounded once to the sweep's
// precision.  Every brickwork gate enters exactly one map; those of the first and
// the last layer enter as products of a U and a V gate, which sit on neighbouring
// threads.  Nothing but the maps goes to global memory.
//
// Bound: the integer pipe (about 17,000 instructions a gate, the 32 x 32 -> 64 products above all).  The FP64 form (Box-Muller
// and Householder QR on the FP64 pipe, maps by a third kernel) took 19.6 ms for
// 5.0 million gates (n = 51, l = 5, 20,001 pairs); this takes 3.4 ms.
#include <cuda_runtime.h>

#include "brick.h"
#include "haar_items.h"
#include "kernels.h"

namespace fpk {
namespace {

constexpr int TH = 128;

// phase 1: the Gaussian entries 2j, 2j+1 (row-major) of a gate from Philox block j
template <int G>
__device__ __forceinline__ void gauss_block(uint64_t seed, uint64_t pair, int stream, int g, int j, Fx2 *sm, int slot) {
    const U64x4 x = philox(seed, (uint64_t)j, (uint64_t)g, pair, (uint64_t)stream);
#pragma unroll 1   // one copy of the code: it is 400 instructions long
    for (int h = 0; h < 2; ++h) sm[(2 * j + h) * G + slot] = gauss_fixed(h ? x.x[2] : x.x[0], h ? x.x[3] : x.x[1]);
}

// phase 2: Gram-Schmidt on the gate in slice `slot`; entry k of the matrix at
// sm[k G + slot] (gram_schmidt_fixed, with the columns in shared memory so that one
// copy of each step serves all columns)
template <int G>
__device__ __forceinline__ void columns(Fx2 *sm, int slot) {
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {
        Fx2 v[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) v[r] = sm[(4 * r + c) * G + slot];
        if (c) {
            shift_fixed<4>(v, lead_fixed<4>(v) - kRoom);
            for (int pass = 0; pass < 2; ++pass) {
#pragma unroll 1
                for (int k = 0; k < c; ++k) {
                    Fx2 q[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) q[r] = sm[(4 * r + k) * G + slot];
                    project_fixed<4>(q, v);
                }
                const int drop = lead_fixed<4>(v) - kRoom;
                if (drop < kRedo<4>) break;
                if (pass == 0) shift_fixed<4>(v, drop);
            }
        }
        unit_fixed<4>(v);
#pragma unroll
        for (int r = 0; r < 4; ++r) sm[(4 * r + c) * G + slot] = v[r];
    }
}

// raw records: gate g of circuit w of pair p at raw[(raw_off + w n_raw + g) 16]
template <int G>
__global__ void __launch_bounds__(TH) haar_raw_kernel(SampleParams sp, const PairInfo *__restrict__ pairs,
                                                      double2 *__restrict__ raw) {
    __shared__ Fx2 sm[16 * G];
    const PairInfo pi = pairs[blockIdx.y];
    const int first = blockIdx.x * G, n = 2 * pi.n_raw - first;
    if (n <= 0) return;
    for (int i = threadIdx.x; i < 8 * G; i += TH) {
        const int slot = i % G, idx = first + slot;
        if (slot >= n) continue;
        const int w = idx / pi.n_raw;
        gauss_block<G>(sp.seed, pi.pair, sp.self_pair ? 0 : w, idx - w * pi.n_raw, i / G, sm, slot);
    }
    __syncthreads();
    const int slot = threadIdx.x;
    if (slot >= G || slot >= n) return;
    columns<G>(sm, slot);
    double2 *out = raw + (pi.raw_off + first + slot) * 16;
#pragma unroll 4
    for (int e = 0; e < 16; ++e) {
        const Fx2 z = sm[e * G + slot];
        out[e] = make_double2(fx_to_double(z.x, 60), fx_to_double(z.y, 60));
    }
}

template <typename C, int G>
__global__ void __launch_bounds__(TH) brick_haar_maps_kernel(BrickDev d, SampleParams sp, Items it,
                                                             const PairInfo *__restrict__ pairs, C *__restrict__ maps) {
    __shared__ Fx2 sm[16 * G];
    const int64_t first = (int64_t)blockIdx.x * G;
    for (int i = threadIdx.x; i < 8 * G; i += TH) {
        const int slot = i % G;
        GateOf o;
        if (gate_of(d, it, first + slot, o))
            gauss_block<G>(sp.seed, pairs[o.pair].pair, sp.self_pair ? 0 : o.w, o.g, i / G, sm, slot);
    }
    __syncthreads();
    const int slot = threadIdx.x;
    if (slot >= G) return;
    GateOf o;
    const bool on = gate_of(d, it, first + slot, o);
    if (on) columns<G>(sm, slot);
    __syncwarp();
    if (!on) return;
    const bool outer = first >= it.inner;
    const bool left = o.b < d.cut;
    C *out = maps + ((size_t)o.pair * maps_per_pair(d) + map_of(d, o)) * 16;
    // entry (r, c) of the gate at r = 2 y' + x', c = 2 y + x (x: qubit b+1, primes: after the
    // gate) goes to row x + 2 x', column y + 2 y' of a left map, transposed in a right one
    auto put = [&](int r, int c, C z) {
        const int ex = (c & 1) + 2 * (r & 1), ey = (c >> 1) + 2 * (r >> 1);
        out[left ? 4 * ex + ey : 4 * ey + ex] = z;
    };
    if (!outer) {   // V's gate, or U's conjugate transpose
#pragma unroll 4
        for (int e = 0; e < 16; ++e) {
            Fx2 z = sm[e * G + slot];
            const int r = e >> 2, c = e & 3;
            if (!o.w) z.y = -z.y;
            put(o.w ? r : c, o.w ? c : r, fx_out<C>(z, 60));
        }
        return;
    }
    // U_l^dagger V_l, or V_1 U_1^dagger: the two threads of a place make two rows each
    const int us = slot & ~1, vs = slot | 1;
    const bool mid = o.tl == d.l;
#pragma unroll 1
    for (int h = 0; h < 8; ++h) {
        const int r = 2 * o.w + (h >> 2), c = h & 3;
        Fx2 z = {0, 0};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const Fx2 t = dot1_fixed(sm[(mid ? 4 * k + r : 4 * c + k) * G + us], sm[(mid ? 4 * k + c : 4 * r + k) * G + vs]);
            z.x += t.x;
            z.y += t.y;
        }
        put(r, c, fx_out<C>(z, 60));
    }
}

template <typename C>
cudaError_t maps_t(const BrickDev &d, const SampleParams &sp, const PairInfo *pairs, int npairs, C *maps,
                   cudaStream_t st) {
    // few gates: 32 per CTA, whose draws all 128 threads share (a batch that fits the SMs
    // several times over has work enough with one thread per gate throughout)
    const bool small = brick_gates(d, npairs) <= 152 * 4 * 128;
    const int G = small ? 32 : TH;
    const Items it = make_items(d, npairs, G);
    const unsigned grid = (unsigned)((it.inner + it.outer_count + G - 1) / G);
    if (small) brick_haar_maps_kernel<C, 32><<<grid, TH, 0, st>>>(d, sp, it, pairs, maps);
    else brick_haar_maps_kernel<C, TH><<<grid, TH, 0, st>>>(d, sp, it, pairs, maps);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_haar_raw(const SampleParams &sp, const PairInfo *pairs, int npairs, int max_raw, double2 *raw,
                            cudaStream_t st) {
    if (npairs <= 0 || max_raw <= 0) return cudaSuccess;
    if ((int64_t)npairs * 2 * max_raw <= 152 * 4 * 128)
        haar_raw_kernel<32><<<dim3((2 * max_raw + 31) / 32, npairs), TH, 0, st>>>(sp, pairs, raw);
    else
        haar_raw_kernel<TH><<<dim3((2 * max_raw + TH - 1) / TH, npairs), TH, 0, st>>>(sp, pairs, raw);
    return cudaGetLastError();
}

cudaError_t launch_brick_haar_maps(const BrickDev &d, const SampleParams &sp, const PairInfo *pairs, int npairs,
                                   void *maps, bool fp32, cudaStream_t st) {
    if (npairs <= 0) return cudaSuccess;
    return fp32 ? maps_t<float2>(d, sp, pairs, npairs, (float2 *)maps, st)
                : maps_t<double2>(d, sp, pairs, npairs, (double2 *)maps, st);
}

}  // namespace fpk
