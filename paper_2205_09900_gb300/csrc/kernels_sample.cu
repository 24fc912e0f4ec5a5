// kernels_sample.cu -- sampler of the gates that are not Haar (K1; Haar gates:
// kernels_haar.cu), gate merging and op-table builder (K2).
#include <cuda_runtime.h>

#include <type_traits>

#include "fixed.h"
#include "haar_fixed.h"
#include "kernels.h"

namespace fpk {
namespace {

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }

__global__ void sample_kernel(SampleParams sp, const PairInfo *__restrict__ pairs, double2 *__restrict__ raw) {
    const PairInfo pi = pairs[blockIdx.y];
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= 2 * pi.n_raw) return;
    int w = idx / pi.n_raw, g = idx % pi.n_raw;
    int wr = sp.self_pair ? 0 : w;
    double2 *out = raw + (pi.raw_off + idx) * 16;
    if (sp.raw_kind == RAW_DIAG4) {
        U64x4 x = philox(sp.seed, 0, (uint64_t)g, pi.pair, (uint64_t)wr);
#pragma unroll
        for (int k = 0; k < 16; ++k) out[k] = make_double2(0, 0);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            double s, c;
            sincospi(2.0 * ((double)(x.x[k] >> 11) * 0x1.0p-53), &s, &c);
            out[5 * k] = make_double2(c, s);
        }
    } else if (sp.raw_kind == RAW_PAULI) {
        // the paper's HEA (Fig. 2c): H, the RY(pi/4) wall, Pauli rotations
#pragma unroll
        for (int k = 0; k < 16; ++k) out[k] = make_double2(0, 0);
        if (g == 0) {
            const double h = 0.70710678118654752440;
            out[0] = make_double2(h, 0); out[1] = make_double2(h, 0);
            out[2] = make_double2(h, 0); out[3] = make_double2(-h, 0);
        } else if (g <= sp.n) {
            // RY(pi/4) = [[c, -s], [s, c]], c = cos(pi/8), s = sin(pi/8)
            double s, c;
            sincospi(0.125, &s, &c);
            out[0] = make_double2(c, 0); out[1] = make_double2(-s, 0);
            out[2] = make_double2(s, 0); out[3] = make_double2(c, 0);
        } else {
            const int r = g - 1 - sp.n, t = r / sp.n, q = r % sp.n;
            U64x4 x = philox(sp.seed, (uint64_t)t, (uint64_t)q, pi.pair, (uint64_t)wr);
            const double th = (double)(x.x[0] >> 11) * 0x1.0p-53;   // theta in turns of 2 pi
            const uint32_t axis = pick(x.x[1], 3u);
            double s, c;
            sincospi(th, &s, &c);                // sin, cos of theta/2
            // exp(-i theta P/2) = c I - i s P
            if (axis == 0) {        // X
                out[0] = make_double2(c, 0); out[1] = make_double2(0, -s);
                out[2] = make_double2(0, -s); out[3] = make_double2(c, 0);
            } else if (axis == 1) { // Y
                out[0] = make_double2(c, 0); out[1] = make_double2(-s, 0);
                out[2] = make_double2(s, 0); out[3] = make_double2(c, 0);
            } else {                // Z
                out[0] = make_double2(c, -s); out[3] = make_double2(c, s);
            }
        }
    } else {   // RAW_ROT2: HEA rotation RY(theta) RZ(phi), raw index g = t*n + q
        int t = g / sp.n, q = g % sp.n;
        U64x4 x = philox(sp.seed, (uint64_t)t, (uint64_t)q, pi.pair, (uint64_t)wr);
        double th = (double)(x.x[0] >> 11) * 0x1.0p-53;   // in turns of 2 pi
        double ph = (double)(x.x[1] >> 11) * 0x1.0p-53;
        double sth, cth, sph, cph;
        sincospi(th, &sth, &cth);            // sin, cos of theta/2 = pi * th
        sincospi(ph, &sph, &cph);            // sin, cos of phi/2
        double2 em = make_double2(cph, -sph), ep = make_double2(cph, sph);
#pragma unroll
        for (int k = 4; k < 16; ++k) out[k] = make_double2(0, 0);
        out[0] = make_double2(cth * em.x, cth * em.y);
        out[1] = make_double2(-sth * ep.x, -sth * ep.y);
        out[2] = make_double2(sth * em.x, sth * em.y);
        out[3] = make_double2(cth * ep.x, cth * ep.y);
    }
}

// The 2x2 factors of the HEA boundary sweep (kernels_hea.cu), sampled and merged in
// one pass: slot s of qubit q (brick.h), entry 2 y_s + y_{s-1}, at
// slots[((p n + q) N + s) 4].  One thread per slot, the lanes of a warp over the
// qubits of one slot (with the slots over the lanes every warp would run all three
// branches: 3.9 ms against 1.4 ms for 12,500 pairs at n = 50, L = 8); only the two
// merged slots sample both circuits.  Angles and products in fixed point (haar_fixed.h): for
// 100,000 pairs of L = 2..8 3.2 ms instead of 7.0 with tabulated FP64 sines, and errors of a few
// 2^-58 instead of 2^-52.
__device__ __forceinline__ void hea_rotation(uint64_t seed, uint64_t pair, int w, int t, int q, Fx2 (&m)[4]) {
    const U64x4 x = philox(seed, (uint64_t)t, (uint64_t)q, pair, (uint64_t)w);
    Half cth, sth, cph, sph;   // of theta/2 and phi/2: (x >> 11) 2^-54 turns
    cos_sin_fixed((x.x[0] >> 11) << 10, cth, sth);
    cos_sin_fixed((x.x[1] >> 11) << 10, cph, sph);
    const int64_t a = mul60(cth, cph), b = mul60(cth, sph), c = mul60(sth, cph), d = mul60(sth, sph);
    m[0] = {a, -b};
    m[1] = {-c, -d};
    m[2] = {c, -d};
    m[3] = {a, b};
}

// acc + conj(a) b
__device__ __forceinline__ Fx2 cmac_fixed(Fx2 a, Fx2 b, Fx2 acc) {
    const Half ax = halves(a.x), ay = halves(a.y), bx = halves(b.x), by = halves(b.y);
    acc.x += mul60(ax, bx) + mul60(ay, by);
    acc.y += mul60(ax, by) - mul60(ay, bx);
    return acc;
}

__device__ __forceinline__ void put_slot(float2 &o, Fx2 v) { o = make_float2(fx_to_float(v.x, 60), fx_to_float(v.y, 60)); }
__device__ __forceinline__ void put_slot(double2 &o, Fx2 v) { o = make_double2(fx_to_double(v.x, 60), fx_to_double(v.y, 60)); }
__device__ __forceinline__ void put_slot(int4 &o, Fx2 v) {
    o = fix_coef(make_longlong2(v.x << (kFixCoef - 60), v.y << (kFixCoef - 60)));
}

template <typename C>
__global__ void __launch_bounds__(128) hea_slots_kernel(SampleParams sp, const PairInfo *__restrict__ pairs, int npairs,
                                                        int L, C *__restrict__ slots) {
    const int N = 2 * L - 2, per = sp.n * N;
    const int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (id >= (int64_t)npairs * per) return;
    const int p = (int)(id / per), r = (int)(id - (int64_t)p * per), s = r / sp.n, q = r - s * sp.n;
    const uint64_t pair = pairs[p].pair;
    const int wv = sp.self_pair ? 0 : 1;
    Fx2 R[4];
    if (s == 0 || s == L - 1) {   // R_1^V R_1^U^dagger; R_L^U^dagger R_L^V
        Fx2 A[4], B[4];
        hea_rotation(sp.seed, pair, 0, s, q, A);
        hea_rotation(sp.seed, pair, wv, s, q, B);
#pragma unroll
        for (int r2 = 0; r2 < 2; ++r2)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                Fx2 acc{0, 0};
#pragma unroll
                for (int k = 0; k < 2; ++k)
                    acc = s == 0 ? cmac_fixed(A[2 * c + k], B[2 * r2 + k], acc) : cmac_fixed(A[2 * k + r2], B[2 * k + c], acc);
                R[2 * r2 + c] = acc;
            }
    } else if (s < L - 1) {
        hea_rotation(sp.seed, pair, wv, s, q, R);
    } else {
        Fx2 A[4];
        hea_rotation(sp.seed, pair, 0, 2 * L - 2 - s, q, A);
#pragma unroll
        for (int e = 0; e < 4; ++e) R[e] = {A[2 * (e & 1) + (e >> 1)].x, -A[2 * (e & 1) + (e >> 1)].y};
    }
    C *out = slots + ((int64_t)p * per + q * N + s) * 4;
#pragma unroll
    for (int e = 0; e < 4; ++e) put_slot(out[e], R[e]);
}

__global__ void merge_kernel(const PairInfo *__restrict__ pairs, const DevPlan *__restrict__ plans,
                             const MergeItem *__restrict__ items, const MergeRef *__restrict__ refs,
                             const double2 *__restrict__ raw, double2 *__restrict__ merged) {
    const PairInfo pi = pairs[blockIdx.y];
    const DevPlan &pl = plans[pi.plan];
    int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= pl.n_merged) return;
    MergeItem it = items[pl.merge_off + m];
    double2 M[16];
    int dim = refs[pl.ref_off + it.first].dim;
#pragma unroll
    for (int k = 0; k < 16; ++k) M[k] = make_double2(0, 0);
    for (int r = 0; r < dim; ++r) M[r * dim + r] = make_double2(1, 0);
    for (int c = 0; c < it.count; ++c) {
        MergeRef rf = refs[pl.ref_off + it.first + c];
        const double2 *A = raw + (pi.raw_off + (int64_t)rf.which * pi.n_raw + rf.gate) * 16;
        double2 G[16], N[16];
        for (int r = 0; r < dim; ++r)
            for (int s = 0; s < dim; ++s)
                G[r * dim + s] = rf.dagger ? cconj(A[s * dim + r]) : A[r * dim + s];
        for (int r = 0; r < dim; ++r)
            for (int s = 0; s < dim; ++s) {
                double2 acc = make_double2(0, 0);
                for (int k = 0; k < dim; ++k) {
                    double2 t = cmul(G[r * dim + k], M[k * dim + s]);
                    acc.x += t.x; acc.y += t.y;
                }
                N[r * dim + s] = acc;
            }
        for (int k = 0; k < dim * dim; ++k) M[k] = N[k];
    }
    double2 *out = merged + (pi.merged_off + m) * 16;
#pragma unroll
    for (int k = 0; k < 16; ++k) out[k] = M[k];
}

template <typename C>
__device__ __forceinline__ C to_c(double re, double im);
template <>
__device__ __forceinline__ double2 to_c<double2>(double re, double im) { return make_double2(re, im); }
template <>
__device__ __forceinline__ float2 to_c<float2>(double re, double im) { return make_float2((float)re, (float)im); }

template <typename C>
__global__ void table_kernel(const PairInfo *__restrict__ pairs, const DevPlan *__restrict__ plans,
                             const DevRecipe *__restrict__ recipes, const double2 *__restrict__ merged,
                             C *__restrict__ tables) {
    const PairInfo pi = pairs[blockIdx.y];
    const DevPlan &pl = plans[pi.plan];
    int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= pl.n_left + pl.n_right) return;
    const DevRecipe &r = recipes[pl.rec_off + o];
    C *out = tables + (pi.table_off + o) * 16;
    const double2 *M = r.merged >= 0 ? merged + (pi.merged_off + r.merged) * 16 : nullptr;
    for (int e = 0; e < 16; ++e) {
        double re = 0, im = 0;
        if (e < r.nent) {
            if (M) {
                for (int s = 0; s < 4; ++s) {
                    const int k = r.src[e][s];
                    if (k < 0) continue;
                    const double2 m = M[k & 15];
                    re += k & 64 ? -m.x : m.x;
                    im += k & 64 ? -m.y : m.y;
                }
            } else {
                re = r.src[e][0];
            }
        }
        out[e] = to_c<C>(re, im);
    }
}

}  // namespace

cudaError_t launch_sample(const SampleParams &sp, const PairInfo *pairs, int npairs, int max_raw,
                          double2 *raw, cudaStream_t st) {
    if (npairs <= 0) return cudaSuccess;
    if (sp.raw_kind == RAW_HAAR4) return launch_haar_raw(sp, pairs, npairs, max_raw, raw, st);   // kernels_haar.cu
    dim3 grid((2 * max_raw + 127) / 128, npairs);
    sample_kernel<<<grid, 128, 0, st>>>(sp, pairs, raw);
    return cudaGetLastError();
}

cudaError_t launch_hea_slots(const SampleParams &sp, const PairInfo *pairs, int npairs, int L, void *slots, bool fp32,
                             cudaStream_t st) {
    if (npairs <= 0) return cudaSuccess;
    const int64_t total = (int64_t)npairs * sp.n * (2 * L - 2);
    const unsigned grid = (unsigned)((total + 127) / 128);
    if (fp32) hea_slots_kernel<float2><<<grid, 128, 0, st>>>(sp, pairs, npairs, L, (float2 *)slots);
    else if (L >= 4) hea_slots_kernel<int4><<<grid, 128, 0, st>>>(sp, pairs, npairs, L, (int4 *)slots);   // fixed.h
    else hea_slots_kernel<double2><<<grid, 128, 0, st>>>(sp, pairs, npairs, L, (double2 *)slots);
    return cudaGetLastError();
}

cudaError_t launch_merge(const PairInfo *pairs, int npairs, int max_merged, const DevPlan *plans,
                         const MergeItem *items, const MergeRef *refs, const double2 *raw,
                         double2 *merged, cudaStream_t st) {
    if (npairs <= 0 || max_merged <= 0) return cudaSuccess;
    dim3 grid((max_merged + 127) / 128, npairs);
    merge_kernel<<<grid, 128, 0, st>>>(pairs, plans, items, refs, raw, merged);
    return cudaGetLastError();
}

cudaError_t launch_tables(const PairInfo *pairs, int npairs, int max_ops, const DevPlan *plans,
                          const DevRecipe *recipes, const double2 *merged, void *tables, bool fp32,
                          cudaStream_t st) {
    if (npairs <= 0 || max_ops <= 0) return cudaSuccess;
    dim3 grid((max_ops + 127) / 128, npairs);
    if (fp32)
        table_kernel<float2><<<grid, 128, 0, st>>>(pairs, plans, recipes, merged, (float2 *)tables);
    else
        table_kernel<double2><<<grid, 128, 0, st>>>(pairs, plans, recipes, merged, (double2 *)tables);
    return cudaGetLastError();
}

}  // namespace fpk
