// haar_items.h -- the gates of a batch of brickwork pairs as work items of the kernels
// that sample Haar gates and write the boundary sweep's maps (kernels_haar.cu,
// kernels_qudit.cu).
#pragma once
#include <cuda_runtime.h>

#include "brick.h"
#include "haar_fixed.h"

namespace fpk {
namespace {

template <typename C> __device__ __forceinline__ C fx_out(Fx2 z, int k);
template <> __device__ __forceinline__ float2 fx_out<float2>(Fx2 z, int k) {
    return make_float2(fx_to_float(z.x, k), fx_to_float(z.y, k));
}
template <> __device__ __forceinline__ double2 fx_out<double2>(Fx2 z, int k) {
    return make_double2(fx_to_double(z.x, k), fx_to_double(z.y, k));
}

// One gate of a brickwork pair: gate g of circuit w (0 = U, 1 = V), in circuit layer
// tl (1-based) on bond b.
struct GateOf { int pair, w, g, tl, b; };

// Items: first the gates of the inner layers 2..l-1 (V's and U's, item = (pair, w, gate)),
// then, from item `inner` (a multiple of G) on, those of layers 1 and l, the U and the V
// gate of one place next to each other.  Blocks never mix the two kinds.
struct Items { int64_t inner_count, inner, outer_count; int nmid, nout, c0, c1, gl; };

__device__ __forceinline__ bool gate_of(const BrickDev &d, const Items &it, int64_t i, GateOf &o) {
    if (i < it.inner) {
        if (i >= it.inner_count) return false;
        const int per = 2 * it.nmid;
        o.pair = (int)(i / per);
        const int r = (int)(i - (int64_t)o.pair * per);
        o.w = r / it.nmid;
        const int k = r - o.w * it.nmid, two = it.c0 + it.c1, lay = k / two, rem = k - lay * two;
        const bool odd = rem >= it.c1;   // layer 2 (c1 gates), 3 (c0 gates), 4, ..
        o.g = it.c0 + k;
        o.tl = 2 + 2 * lay + (odd ? 1 : 0);
        o.b = 2 * (odd ? rem - it.c1 : rem) + (o.tl - 1) % 2;
        return true;
    }
    i -= it.inner;
    if (i >= it.outer_count) return false;
    const int per = 2 * it.nout;
    o.pair = (int)(i / per);
    const int r = (int)(i - (int64_t)o.pair * per), k = r >> 1;
    o.w = r & 1;
    const bool last = k >= it.c0;
    o.tl = last ? d.l : 1;
    o.g = last ? it.gl + k - it.c0 : k;
    o.b = 2 * (last ? k - it.c0 : k) + (o.tl - 1) % 2;
    return true;
}

inline int64_t brick_gates(const BrickDev &d, int npairs) {
    return (int64_t)npairs * 2 * ((d.l + 1) / 2 * (d.n / 2) + d.l / 2 * ((d.n - 1) / 2));
}

inline Items make_items(const BrickDev &d, int npairs, int G) {
    Items it;
    it.c0 = d.n / 2;
    it.c1 = (d.n - 1) / 2;
    const int cl = d.l % 2 ? it.c0 : it.c1;
    it.gl = (d.l / 2) * it.c0 + ((d.l - 1) / 2) * it.c1;   // gates before layer l
    it.nmid = it.gl - it.c0;
    it.nout = it.c0 + cl;
    it.inner_count = (int64_t)npairs * 2 * it.nmid;
    it.outer_count = (int64_t)npairs * 2 * it.nout;
    it.inner = (it.inner_count + G - 1) / G * G;
    return it;
}

// position of the merged gate of circuit layer tl, circuit w on the cycle of 2(l-1) (brick.h)
__device__ __forceinline__ int cycle_pos(const BrickDev &d, const GateOf &o) {
    return o.tl == 1 ? 2 * d.l - 3 : o.tl == d.l ? d.l - 2 : o.w ? o.tl - 2 : 2 * d.l - 2 - o.tl;
}
// index of its map
__device__ __forceinline__ int map_of(const BrickDev &d, const GateOf &o) {
    const int j = (cycle_pos(d, o) - (o.b + 1) % 2) / 2;
    return o.b < d.cut ? map_index(d, 0, o.b, j) : map_index(d, 1, d.n - 2 - o.b, j);
}

}  // namespace
}  // namespace fpk
