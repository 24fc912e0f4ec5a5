// meet.h -- device helpers shared by the boundary sweeps: the accumulators of
// the final dot product, its results, cp.async copies, compile-time loops.
#pragma once
#include <cstdint>
#include <type_traits>
#include <utility>

#include <cuda_runtime.h>

#include "fp_internal.h"

namespace fpk {
namespace {

// f(integral_constant<int, 0>), .., f(integral_constant<int, N-1>)
template <int N, typename F, int... I>
__device__ __forceinline__ void static_for_impl(F &&f, std::integer_sequence<int, I...>) {
    (f(std::integral_constant<int, I>{}), ...);
}
template <int N, typename F>
__device__ __forceinline__ void static_for(F &&f) {
    static_for_impl<N>(f, std::make_integer_sequence<int, N>{});
}

// Accumulators of the meet: the trace sum in FP64; the |t| and |t|^2 sums
// (cancellation ratio, error estimate) in the boundary precision per thread,
// combined in FP64 across threads.  A term t = L_j R_j is formed in the
// boundary's own precision (one rounding of values that carry FP32 rounding
// already); FP64 conversions and square roots are costly on this part.
template <typename C> struct MeetAcc;
template <> struct MeetAcc<float2> {
    double sr = 0, si = 0;
    float sa = 0, s2 = 0;
    float fr = 0, fi = 0;   // the current run of products, folded into sr, si by flush
    __device__ __forceinline__ void add(float2 l, float2 r) {
        const float px = fmaf(l.x, r.x, -l.y * r.y), py = fmaf(l.x, r.y, l.y * r.x);
        const float q = fmaf(px, px, py * py);
        fr += px;
        fi += py;
        sa += sqrtf(q);
        s2 += q;
    }
    __device__ __forceinline__ void flush() {
        sr += (double)fr;
        si += (double)fi;
        fr = fi = 0;
    }
};
template <> struct MeetAcc<double2> {
    double sr = 0, si = 0, sa = 0, s2 = 0;
    __device__ __forceinline__ void add(double2 l, double2 r) {
        const double px = l.x * r.x - l.y * r.y, py = l.x * r.y + l.y * r.x;
        const double q = px * px + py * py;
        sr += px; si += py; sa += sqrt(q); s2 += q;
    }
    __device__ __forceinline__ void flush() {}
};

__device__ __forceinline__ double wsum(double v) {
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
    return v;
}

// Asynchronous global -> shared copies (cp.async): every element of a tile
// is requested before any is waited for, so a tile load costs about one
// memory latency instead of one per few elements.
template <int BYTES>
__device__ __forceinline__ void cp_async(void *smem_dst, const void *gmem_src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_dst);
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gmem_src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(d), "l"(gmem_src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// trace, cancellation ratio and error estimate from the sums (Re, Im, |t|, |t|^2)
__device__ __forceinline__ void write_meet(const PairInfo &pi, const double (&s)[4], double err_scale,
                                           double *__restrict__ tr, double *__restrict__ kappa,
                                           double *__restrict__ err) {
    tr[2 * pi.out] = s[0];
    tr[2 * pi.out + 1] = s[1];
    const double mag = sqrt(s[0] * s[0] + s[1] * s[1]);
    if (kappa) kappa[pi.out] = mag > 0 ? s[2] / mag : __longlong_as_double(0x7ff0000000000000LL);
    if (err) err[pi.out] = err_scale * (sqrt(s[3]) + mag);
}

}  // namespace
}  // namespace fpk
