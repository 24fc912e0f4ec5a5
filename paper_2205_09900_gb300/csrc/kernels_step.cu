// kernels_step.cu -- lock-step boundary sweep of local-circuit pairs with large
// boundaries (2^14 amplitudes and more).
//
// Every pair has its own topology and its own sequence of operations.  Step k of a
// batch applies operation k of both sides of every pair in one launch: a work list
// (StepItem, built by the host) gives each CTA a range of one operation's outputs, so
// that all SMs share every boundary, the largest one included, and the launch is the
// barrier.  (The ticket-queue sweep of kernels_sweep.cu gives a pair to one cluster of
// 16 CTAs: a boundary of 2^24 amplitudes then streams through a tenth of the chip, and
// a batch lasts as long as its largest pairs.)  Operations that keep the boundary's
// shape (two summed, two new variables in their places: two thirds of the work) run in
// place.  Bound: HBM (the boundaries of a batch exceed L2), one read and one write of
// the boundary per operation.
//
// The meet (exact_meet.h) takes FP32 operations whose products and sums of Re and Im are
// exact to more bits than a double's: in FP64, 35 operations per term on a pipe 77 times
// slower, it took longer than the sweep.
// 4,000 pairs at n = 20, T = 20..100 (1,792 of them here): 17 ms of sweeps and meet against 93.
#include <cuda_runtime.h>

#include <algorithm>

#include "kernels.h"
#include "exact_meet.h"
#include "meet.h"

namespace fpk {
namespace {

__device__ __forceinline__ uint32_t ins_bit(uint32_t x, int p, uint32_t v) {
    return (x & ((1u << p) - 1u)) | (v << p) | ((x >> p) << (p + 1));
}
template <typename C>
__device__ __forceinline__ C cmadd(C a, C b, C acc) {   // acc + a*b
    acc.x = fma(a.x, b.x, acc.x);
    acc.x = fma(-a.y, b.y, acc.x);
    acc.y = fma(a.x, b.y, acc.y);
    acc.y = fma(a.y, b.x, acc.y);
    return acc;
}

// two summed, two new variables in place at bits p0 < p1: quads [u0, u1)
__device__ __forceinline__ void quad4(const float2 (&t)[16], const float2 (&a)[4], float2 (&y)[4]) {
#pragma unroll
    for (int o = 0; o < 4; ++o) {
        y[o] = make_float2(0.f, 0.f);
#pragma unroll
        for (int b = 0; b < 4; ++b) y[o] = cmadd(t[b | (o << 2)], a[b], y[o]);
    }
}
__device__ __forceinline__ void quad4(const double2 (&t)[16], const double2 (&a)[4], double2 (&y)[4]) {
#pragma unroll
    for (int o = 0; o < 4; ++o) {
        y[o] = make_double2(0, 0);
#pragma unroll
        for (int b = 0; b < 4; ++b) y[o] = cmadd(t[b | (o << 2)], a[b], y[o]);
    }
}
__device__ __forceinline__ void in_place(const float2 (&t)[16], float2 *s, int p0, int p1, uint32_t u0, uint32_t u1) {
    if (p0 == 0) {   // the two amplitudes of bit p0 are one 16-byte word
        for (uint32_t q = u0 + threadIdx.x; q < u1; q += blockDim.x) {
            float4 *w0 = reinterpret_cast<float4 *>(s + ins_bit(q << 1, p1, 0)), *w1 = w0 + (1u << (p1 - 1));
            const float4 lo = *w0, hi = *w1;
            const float2 a[4] = {make_float2(lo.x, lo.y), make_float2(lo.z, lo.w), make_float2(hi.x, hi.y),
                                 make_float2(hi.z, hi.w)};
            float2 y[4];
            quad4(t, a, y);
            *w0 = make_float4(y[0].x, y[0].y, y[1].x, y[1].y);
            *w1 = make_float4(y[2].x, y[2].y, y[3].x, y[3].y);
        }
        return;
    }
    // two neighbouring quads (bit 0 is in neither place) share 16-byte words
    for (uint32_t q = u0 + 2 * threadIdx.x; q < u1; q += 2 * blockDim.x) {
        const uint32_t i = ins_bit(ins_bit(q, p0, 0), p1, 0);
        float4 *w[4], v[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            w[b] = reinterpret_cast<float4 *>(s + (i | ((b & 1) << p0) | ((b >> 1) << p1)));
            v[b] = *w[b];
        }
        const float2 a0[4] = {make_float2(v[0].x, v[0].y), make_float2(v[1].x, v[1].y), make_float2(v[2].x, v[2].y),
                              make_float2(v[3].x, v[3].y)};
        const float2 a1[4] = {make_float2(v[0].z, v[0].w), make_float2(v[1].z, v[1].w), make_float2(v[2].z, v[2].w),
                              make_float2(v[3].z, v[3].w)};
        float2 y0[4], y1[4];
        quad4(t, a0, y0);
        quad4(t, a1, y1);
#pragma unroll
        for (int b = 0; b < 4; ++b) *w[b] = make_float4(y0[b].x, y0[b].y, y1[b].x, y1[b].y);
    }
}
__device__ __forceinline__ void in_place(const double2 (&t)[16], double2 *s, int p0, int p1, uint32_t u0, uint32_t u1) {
    for (uint32_t q = u0 + threadIdx.x; q < u1; q += blockDim.x) {
        const uint32_t i = ins_bit(ins_bit(q, p0, 0), p1, 0);
        double2 a[4], y[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) a[b] = s[i | ((b & 1) << p0) | ((b >> 1) << p1)];
        quad4(t, a, y);
#pragma unroll
        for (int b = 0; b < 4; ++b) s[i | ((b & 1) << p0) | ((b >> 1) << p1)] = y[b];
    }
}

// NC summed and NN new variables, none kept, the new ones on top of the others: units are
// the values of the variables that stay
template <typename C, int NC, int NN>
__device__ __forceinline__ void reshape(const DevOp &op, const C *T, const C *__restrict__ in, C *__restrict__ out,
                                        uint32_t u0, uint32_t u1) {
    C t[1 << (NC + NN)];
#pragma unroll
    for (int e = 0; e < (1 << (NC + NN)); ++e) t[e] = T[e];
    const int top = op.b_in - NC;
    for (uint32_t r = u0 + threadIdx.x; r < u1; r += blockDim.x) {
        C x[1 << NC];
#pragma unroll
        for (int cv = 0; cv < (1 << NC); ++cv) {
            uint32_t i = r;
#pragma unroll
            for (int z = 0; z < NC; ++z) i = ins_bit(i, op.cons_pos[z], (cv >> z) & 1);
            x[cv] = in[i];
        }
#pragma unroll
        for (int nv = 0; nv < (1 << NN); ++nv) {
            C acc;
            acc.x = 0;
            acc.y = 0;
#pragma unroll
            for (int cv = 0; cv < (1 << NC); ++cv) acc = cmadd(t[cv | (nv << NC)], x[cv], acc);
            out[r | ((uint32_t)nv << top)] = acc;
        }
    }
}

template <typename C>
__global__ void __launch_bounds__(256) step_kernel(const StepItem *__restrict__ items, const uint32_t *__restrict__ which,
                                                   const DevOp *__restrict__ ops, const C *__restrict__ tables,
                                                   C *__restrict__ ws) {
    const StepItem it = items[which[blockIdx.x]];
    const DevOp op = ops[it.op];
    const uint32_t u0 = (blockIdx.x - it.first) << it.log_units, u1 = min(u0 + (1u << it.log_units), it.units);
    const C *T = tables + it.table * 16, *in = ws + it.in;
    C *out = ws + it.out;
    switch (it.form) {
        case STEP_IN_PLACE: {
            C t[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) t[e] = T[e];
            in_place(t, out, op.cons_pos[0], op.cons_pos[1], u0, u1);
            return;
        }
        case STEP_1_3: reshape<C, 1, 3>(op, T, in, out, u0, u1); return;
        case STEP_3_1: reshape<C, 3, 1>(op, T, in, out, u0, u1); return;
        case STEP_0_4: reshape<C, 0, 4>(op, T, in, out, u0, u1); return;
        case STEP_4_0: reshape<C, 4, 0>(op, T, in, out, u0, u1); return;
        default: break;
    }
    // any other operation: units are its outputs
    const int nc = op.nc, nk = op.nk, nn = op.nn;
    for (uint32_t o = u0 + threadIdx.x; o < u1; o += blockDim.x) {
        uint32_t nv = 0, kv = 0, r = o;
        for (int z = 0; z < nn; ++z) nv |= ((o >> op.new_pos[z]) & 1u) << z;
        for (int z = 0; z < nk; ++z) kv |= ((o >> op.keep_pos[z]) & 1u) << z;
        for (int z = nn - 1; z >= 0; --z) r = (r & ((1u << op.new_pos[z]) - 1u)) | ((r >> (op.new_pos[z] + 1)) << op.new_pos[z]);
        const uint32_t tb = (kv << nc) | (nv << (nc + nk));
        C acc;
        acc.x = 0;
        acc.y = 0;
        for (uint32_t cv = 0; cv < (1u << nc); ++cv) {
            uint32_t i = r;
            for (int z = 0; z < nc; ++z) i = ins_bit(i, op.cons_pos[z], (cv >> z) & 1u);
            acc = cmadd(T[cv | tb], in[i], acc);
        }
        out[o] = acc;
    }
}

template <typename C>
__global__ void step_init_kernel(const StepPair *__restrict__ sp, int npairs, C *__restrict__ ws) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 2 * npairs) return;
    C one;
    one.x = 1;
    one.y = 0;
    ws[sp[i >> 1].base[i & 1]] = one;
}

struct Sums { double v[4]; };

// Meet: a CTA sums one chunk of a pair's final boundary; the right one is read through the
// permutation of its bits.
template <typename C>
__global__ void __launch_bounds__(256) step_meet_kernel(const StepPair *__restrict__ sp, const uint32_t *__restrict__ which,
                                                        const PairInfo *__restrict__ pairs,
                                                        const DevPlan *__restrict__ plans, const C *__restrict__ ws,
                                                        Sums *__restrict__ part) {
    __shared__ uint32_t lut[2][128];
    __shared__ double red[4][8];
    const StepPair s = sp[which[blockIdx.x]];
    const DevPlan &pl = plans[pairs[which[blockIdx.x]].plan];
    const int bits = pl.bits_final;
    const uint32_t base = (blockIdx.x - s.first) << kMeetChunk;
    for (int i = threadIdx.x; i < 256; i += 256) {
        const int h = i >> 7;
        uint32_t o = 0;
        for (int k = 0; k < 7; ++k)
            if (7 * h + k < bits) o |= ((i >> k) & 1u) << pl.dot_perm[7 * h + k];
        lut[h][i & 127] = o;
    }
    uint32_t rbase = 0;
    for (int k = kMeetChunk; k < bits; ++k) rbase |= ((base >> k) & 1u) << pl.dot_perm[k];
    __syncthreads();
    const C *L = ws + s.final[0], *R = ws + s.final[1];
    const uint32_t n = min(1u << kMeetChunk, (1u << bits) - base);
    ExactMeet<C> acc;
    for (uint32_t i = threadIdx.x; i < n; i += 256) acc.add(L[base + i], R[rbase | lut[0][i & 127] | lut[1][i >> 7]]);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        double v = acc.total(c);
        for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
        if (lane == 0) red[c][wid] = v;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double t[4] = {0, 0, 0, 0};
        for (int c = 0; c < 4; ++c)
            for (int w = 0; w < 8; ++w) t[c] += red[c][w];
        part[blockIdx.x] = {{t[0], t[1], t[2], t[3]}};
    }
}

__global__ void step_results_kernel(const StepPair *__restrict__ sp, int npairs, const PairInfo *__restrict__ pairs,
                                    const DevPlan *__restrict__ plans, const Sums *__restrict__ part,
                                    double err_unit, double *__restrict__ tr, double *__restrict__ kappa,
                                    double *__restrict__ err) {
    const int i = blockIdx.x;   // one warp per pair: chunks in a fixed order
    const PairInfo pi = pairs[i];
    const DevPlan &pl = plans[pi.plan];
    const uint32_t chunks = pl.bits_final > kMeetChunk ? 1u << (pl.bits_final - kMeetChunk) : 1u;
    double s[4] = {0, 0, 0, 0};
    for (uint32_t c = threadIdx.x; c < chunks; c += 32) {
        const Sums p = part[sp[i].first + c];
        for (int j = 0; j < 4; ++j) s[j] += p.v[j];
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
        for (int d = 16; d > 0; d >>= 1) s[c] += __shfl_xor_sync(0xffffffffu, s[c], d);
    if (threadIdx.x != 0) return;
    const double mag = sqrt(s[0] * s[0] + s[1] * s[1]);
    if (err) err[pi.out] = err_unit * pl.sqrt_ops * pl.prefactor * (sqrt(s[3]) + mag);
    tr[2 * pi.out] = pl.prefactor * s[0];
    tr[2 * pi.out + 1] = pl.prefactor * s[1];
    if (kappa) kappa[pi.out] = mag > 0 ? s[2] / mag : __longlong_as_double(0x7ff0000000000000LL);
}

template <typename C>
cudaError_t steps_t(const StepBatch &b, const PairInfo *pairs, int npairs, const DevPlan *plans, const DevOp *ops,
                    const void *tables, void *ws, double err_unit, double *tr, double *kappa, double *err,
                    cudaStream_t st) {
    step_init_kernel<C><<<(2 * npairs + 127) / 128, 128, 0, st>>>(b.pairs, npairs, (C *)ws);
    cudaError_t e = cudaGetLastError();
    for (size_t k = 0; k + 1 < b.step_first.size() && e == cudaSuccess; ++k) {
        const uint32_t grid = b.step_first[k + 1] - b.step_first[k];
        if (grid == 0) continue;
        step_kernel<C><<<grid, 256, 0, st>>>(b.items, b.which + b.step_first[k], ops, (const C *)tables, (C *)ws);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return e;
    step_meet_kernel<C><<<b.meet_blocks, 256, 0, st>>>(b.pairs, b.meet_which, pairs, plans, (const C *)ws, (Sums *)b.partials);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    step_results_kernel<<<npairs, 32, 0, st>>>(b.pairs, npairs, pairs, plans, (const Sums *)b.partials, err_unit, tr,
                                               kappa, err);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_steps(const StepBatch &b, const PairInfo *pairs, int npairs, const DevPlan *plans, const DevOp *ops,
                         const void *tables, bool fp32, void *ws, double err_unit, double *tr, double *kappa, double *err,
                         cudaStream_t st) {
    if (npairs <= 0) return cudaSuccess;
    return fp32 ? steps_t<float2>(b, pairs, npairs, plans, ops, tables, ws, err_unit, tr, kappa, err, st)
                : steps_t<double2>(b, pairs, npairs, plans, ops, tables, ws, err_unit, tr, kappa, err, st);
}

}  // namespace fpk
