// kernels_reduce.cu -- FP64 Monte Carlo moments (K7) and their bootstrap.
//
// x = |Tr|^2 per pair; per group g: N_g, S_k = sum x^k, Q_k = sum x^{2k},
// k = 1..k_max, from which F^(k) = S_k / N and its standard error
// sqrt((Q_k - S_k^2/N) / (N-1) / N) follow (paper: Sec. "Algorithm
// description" for the estimator, Fig. 4 caption for standard errors).
// Deterministic: block b owns a fixed contiguous range of pairs, threads
// stride it in a fixed order, partials are combined by a fixed tree and the
// block partials by one thread in block order with Neumaier compensation.
// The bootstrap (paper: Supplementary, "Bootstrapping for uncertainty
// quantification") resamples each group's stored |Tr|^2 with replacement and
// evaluates F^(k) on every resample: draws counted per member and summed in fixed
// point, a few resamples of a group per CTA (bootstrap_count_kernel); the resamples and
// powers that need it draw by draw in FP64 (bootstrap_kernel).
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "kernels.h"

namespace fpk {
namespace {

constexpr int RT = 256;
constexpr int MAXV = 2 * FP_MAX_KMAX + 1;

__global__ void __launch_bounds__(RT) moments_pass1(const double *__restrict__ tr, const int32_t *__restrict__ group,
                                                    uint64_t count, int k_max, int n_groups, double *__restrict__ partials) {
    __shared__ double sh[RT];
    const int nv = 2 * k_max + 1;
    const uint64_t per = (count + gridDim.x - 1) / gridDim.x;
    const uint64_t lo = (uint64_t)blockIdx.x * per;
    const uint64_t hi = lo + per < count ? lo + per : count;
    for (int g = 0; g < n_groups; ++g) {
        double acc[MAXV];
#pragma unroll
        for (int v = 0; v < MAXV; ++v) acc[v] = 0;
        for (uint64_t i = lo + threadIdx.x; i < hi; i += RT) {
            if (group && group[i] != g) continue;
            if (!group && g != 0) continue;
            double a = tr[2 * i], b = tr[2 * i + 1];
            double x = a * a + b * b, p = 1.0;
            acc[0] += 1.0;
#pragma unroll
            for (int k = 1; k <= FP_MAX_KMAX; ++k) {
                if (k > k_max) break;
                p *= x;
                acc[k] += p;
                acc[k_max + k] += p * p;
            }
        }
        for (int v = 0; v < nv; ++v) {
            sh[threadIdx.x] = acc[v];
            __syncthreads();
            for (int s = RT / 2; s > 0; s >>= 1) {
                if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
                __syncthreads();
            }
            if (threadIdx.x == 0) partials[((size_t)blockIdx.x * n_groups + g) * nv + v] = sh[0];
            __syncthreads();
        }
    }
}

__global__ void moments_pass2(const double *__restrict__ partials, int nblocks, int k_max, int n_groups,
                              double *__restrict__ out) {
    const int nv = 2 * k_max + 1;
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_groups * nv) return;
    int g = t / nv, v = t % nv;
    double s = 0, c = 0;
    for (int b = 0; b < nblocks; ++b) {
        double x = partials[((size_t)b * n_groups + g) * nv + v];
        double y = s + x;
        c += fabs(s) >= fabs(x) ? (s - y) + x : (x - y) + s;
        s = y;
    }
    out[t] = s + c;
}

// Members of every group in increasing pair order, on the device (up to 16 groups): counts per chunk of
// pairs, offsets, and xs = |Tr|^2 of the members group by group.  A CTA takes one (chunk,
// group) and places its members by a scan; the group ids stay in L2 (one CTA per group
// over all 200,000 pairs took 520 us, a counting sort on the host and its copies as much).
constexpr int GT = 256, GP = 4, kChunk = GT * GP;
__device__ __forceinline__ uint32_t group_scan(uint32_t v, uint32_t *total, uint32_t (&sh)[GT / 32]) {   // exclusive
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) sh[wid] = x;
    __syncthreads();
    uint32_t before = 0, all = 0;
    for (int w = 0; w < GT / 32; ++w) {
        if (w < wid) before += sh[w];
        all += sh[w];
    }
    *total = all;
    return before + x - v;
}

// cnt[g nchunks + c]: members of group g = blockIdx.y in chunk c = blockIdx.x (`per` pairs)
__global__ void __launch_bounds__(GT) group_count_kernel(const int32_t *__restrict__ group, uint64_t count, uint64_t per,
                                                         uint32_t *__restrict__ cnt) {
    __shared__ uint32_t sh[GT / 32];
    const uint64_t lo = blockIdx.x * per, hi = lo + per < count ? lo + per : count;
    uint32_t n = 0, all;
    for (uint64_t i = lo + threadIdx.x; i < hi; i += GT) n += group[i] == (int)blockIdx.y;
    group_scan(n, &all, sh);
    if (threadIdx.x == 0) cnt[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = all;
}

// cnt, the same with many groups: a pass over the pairs with an atomic each (cleared before)
__global__ void group_count_many_kernel(const int32_t *__restrict__ group, uint64_t count, uint64_t per, int nchunks,
                                        int n_groups, uint32_t *__restrict__ cnt) {
    const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (i >= count) return;
    const int g = group[i];
    if (g >= 0 && g < n_groups) atomicAdd(&cnt[(size_t)g * nchunks + i / per], 1u);
}

// cnt: from counts to each chunk's first position in its group; off[g + 1] = members of group
// g; exp2 cleared.  A warp per group.
constexpr int kNoScale = 1 << 20;
__device__ __forceinline__ void group_prefix(uint32_t *__restrict__ cnt, int nchunks, int g, uint64_t *__restrict__ off,
                                             int *__restrict__ exp2) {
    const int lane = threadIdx.x & 31;
    uint64_t s = 0;
    for (int c = lane; c - lane < nchunks; c += 32) {
        const uint32_t v = c < nchunks ? cnt[(size_t)g * nchunks + c] : 0;
        uint32_t x = v;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (c < nchunks) cnt[(size_t)g * nchunks + c] = (uint32_t)s + x - v;
        s += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) off[g + 1] = s, exp2[g] = -kNoScale;
}
__global__ void __launch_bounds__(256) group_prefix_kernel(uint32_t *__restrict__ cnt, int nchunks, int n_groups,
                                                           uint64_t *__restrict__ off, int *__restrict__ exp2) {
    const int g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (g < n_groups) group_prefix(cnt, nchunks, g, off, exp2);
}

// inclusive sums over a CTA of 1024 threads
__device__ __forceinline__ uint64_t scan_1024(uint64_t v, uint64_t (&sh)[32]) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    __syncthreads();
    if (lane == 31) sh[wid] = v;
    __syncthreads();
    uint64_t before = 0;
    for (int w = 0; w < wid; ++w) before += sh[w];
    return v + before;
}

// off[g] = first member of group g, off[n_groups] = all members; xoff: the same over the
// groups of at most max_n members (the ones that are counted in shared memory); the list
// `redo` cleared.  prefix: the groups' prefixes first (a few groups), else they are in place.
__global__ void __launch_bounds__(1024) group_offsets_kernel(uint32_t *__restrict__ cnt, int nchunks, int n_groups,
                                                             uint32_t max_n, bool prefix, uint64_t *__restrict__ off,
                                                             uint64_t *__restrict__ xoff, int *__restrict__ exp2,
                                                             unsigned long long *__restrict__ redo) {
    __shared__ uint64_t sh[2][32], base[2];
    if (prefix) {
        for (int g = threadIdx.x >> 5; g < n_groups; g += 32) group_prefix(cnt, nchunks, g, off, exp2);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        *redo = 0;
        off[0] = xoff[0] = base[0] = base[1] = 0;
    }
    __syncthreads();
    for (int g0 = 0; g0 < n_groups; g0 += 1024) {
        const int g = g0 + (int)threadIdx.x;
        const uint64_t n = g < n_groups ? off[g + 1] : 0;
        const uint64_t s = base[0] + scan_1024(n, sh[0]), x = base[1] + scan_1024(n <= max_n ? n : 0, sh[1]);
        if (g < n_groups) off[g + 1] = s, xoff[g + 1] = x;
        __syncthreads();
        if (threadIdx.x == 1023) base[0] = s, base[1] = x;
        __syncthreads();
    }
}

// scale of |t|^2 = x: e with x < 2^e, kNoScale when x^k_max is not finite
__device__ __forceinline__ int scale_of(double x, int k_max) {
    double p = x;
    for (int k = 1; k < k_max; ++k) p *= x;
    return isfinite(p) ? (x > 0 ? ilogb(x) + 1 : -kNoScale) : kNoScale;
}

// xs of the members, and the group's scale: exp2[g] = e with every x < 2^e, or kNoScale
// when a power x^k_max is not finite (such a group takes the FP64 sums below)
__global__ void __launch_bounds__(GT) group_place_kernel(const double *__restrict__ tr, const int32_t *__restrict__ group,
                                                         uint64_t count, uint64_t per, const uint64_t *__restrict__ off,
                                                         const uint32_t *__restrict__ cnt, int k_max,
                                                         double *__restrict__ xs, int *__restrict__ exp2) {
    __shared__ uint32_t sh[GT / 32];
    const uint64_t lo = blockIdx.x * per, hi = lo + per < count ? lo + per : count;
    uint64_t at = off[blockIdx.y] + cnt[(size_t)blockIdx.y * gridDim.x + blockIdx.x];
    int e = -kNoScale;
    for (uint64_t i0 = lo; i0 < hi; i0 += kChunk) {
        const uint64_t i = i0 + (uint64_t)threadIdx.x * GP;
        bool in[GP];
        uint32_t n = 0, all;
#pragma unroll
        for (int j = 0; j < GP; ++j) {
            in[j] = i + j < hi && group[i + j] == (int)blockIdx.y;
            n += in[j];
        }
        uint32_t pos = group_scan(n, &all, sh);
#pragma unroll
        for (int j = 0; j < GP; ++j) {
            if (!in[j]) continue;
            const double a = tr[2 * (i + j)], b = tr[2 * (i + j) + 1], x = a * a + b * b;
            xs[at + pos++] = x;
            e = max(e, scale_of(x, k_max));
        }
        at += all;
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if ((threadIdx.x & 31) == 0 && e > -kNoScale) atomicMax(&exp2[blockIdx.y], e);
}

// The same with many groups: a warp per chunk, 32 pairs at a time, the lanes of one group
// ranked among themselves (in lane order) and placed from the chunk's running position.  A CTA per
// (chunk, group) as above would be 200,000 CTAs for 200,000 pairs in 1,000 groups: 10 resamples of
// them take 272 us this way, 840 that way; at 16 and 17 groups the two take the same.
__global__ void __launch_bounds__(32) group_place_many_kernel(const double *__restrict__ tr, const int32_t *__restrict__ group,
                                                              uint64_t count, uint64_t per, int nchunks, int n_groups,
                                                              const uint64_t *__restrict__ off, uint32_t *__restrict__ cnt,
                                                              int k_max, double *__restrict__ xs, int *__restrict__ exp2) {
    const uint64_t lo = blockIdx.x * per, hi = lo + per < count ? lo + per : count;
    const int lane = threadIdx.x;
    for (uint64_t i0 = lo; i0 < hi; i0 += 32) {
        const uint64_t i = i0 + lane;
        const int id = i < hi ? group[i] : -1, g = id >= 0 && id < n_groups ? id : -1;
        const uint32_t mine = __match_any_sync(0xffffffffu, g), lead = __ffs(mine) - 1;
        uint32_t at = 0;
        if (g >= 0 && lane == (int)lead) at = atomicAdd(&cnt[(size_t)g * nchunks + blockIdx.x], (uint32_t)__popc(mine));
        at = __shfl_sync(0xffffffffu, at, lead) + __popc(mine & ((1u << lane) - 1u));
        if (g >= 0) {
            const double a = tr[2 * i], b = tr[2 * i + 1], x = a * a + b * b;
            xs[off[g] + at] = x;
            const int e = scale_of(x, k_max);
            if (e > exp2[g]) atomicMax(&exp2[g], e);   // (exp2 only grows: a stale read costs an atomic)
        }
        __syncwarp();   // the next 32 see these positions
    }
}

// All of it for a small batch, in one CTA: off and xs, group ids and positions in shared memory.
constexpr int kSmallPairs = 4096, kSmallGroups = 2048;
__global__ void __launch_bounds__(1024) group_small_kernel(const double *__restrict__ tr, const int32_t *__restrict__ group,
                                                           int count, int n_groups, uint64_t *__restrict__ off,
                                                           double *__restrict__ xs) {
    __shared__ int at[kSmallPairs];
    __shared__ uint32_t next[kSmallGroups];
    __shared__ uint64_t sh[32];
    for (int g = threadIdx.x; g < n_groups; g += 1024) next[g] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < count; i += 1024) {
        const int g = group[i];
        at[i] = g >= 0 && g < n_groups ? g : -1;
        if (at[i] >= 0) atomicAdd(&next[at[i]], 1u);
    }
    __syncthreads();
    uint64_t base = 0;
    for (int g0 = 0; g0 < n_groups; g0 += 1024) {
        const int g = g0 + (int)threadIdx.x;
        const uint32_t n = g < n_groups ? next[g] : 0;
        const uint64_t s = base + scan_1024(n, sh);
        if (g < n_groups) off[g + 1] = s, next[g] = (uint32_t)(s - n);
        for (int w = 0; w < 32; ++w) base += sh[w];
    }
    if (threadIdx.x == 0) off[0] = 0;
    __syncthreads();
    if (threadIdx.x < 32)
        for (int i0 = 0; i0 < count; i0 += 32) {
            const int i = i0 + (int)threadIdx.x, g = i < count ? at[i] : -1;
            const uint32_t mine = __match_any_sync(0xffffffffu, g), before = mine & ((1u << threadIdx.x) - 1u);
            if (g >= 0) at[i] = (int)(next[g] + __popc(before));
            __syncwarp();
            if (g >= 0 && !before) next[g] += __popc(mine);
            __syncwarp();
        }
    __syncthreads();
    for (int i = threadIdx.x; i < count; i += 1024)
        if (at[i] >= 0) {
            const double a = tr[2 * i], b = tr[2 * i + 1];
            xs[at[i]] = a * a + b * b;
        }
}

// The powers of every member in fixed point: limbs (low first) of x^k 2^(96 - k e), rounded,
// for group scale e, at xf[((k - 1) n + j) 3], j over the members of the groups of xoff.
// x^k is the product of doubles that the FP64 sums use.
__global__ void powers_kernel(const double *__restrict__ xs, const uint64_t *__restrict__ off,
                              const uint64_t *__restrict__ xoff, int n_groups, int k_max, const int *__restrict__ exp2,
                              uint32_t *__restrict__ xf) {
    const uint64_t n = xoff[n_groups], j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (j >= n) return;
    int g = 0, top = n_groups;   // the last g with xoff[g] <= j
    while (top - g > 1) {
        const int mid = (g + top) / 2;
        (xoff[mid] <= j ? g : top) = mid;
    }
    const int e = exp2[g];
    if (e >= kNoScale) return;
    const double x = xs[off[g] + (j - xoff[g])];
    double p = 1.0;
    for (int k = 1; k <= k_max; ++k) {
        p *= x;
        uint32_t l0 = 0, l1 = 0, l2 = 0;
        if (p > 0 && e > -kNoScale) {
            int pe;
            const uint64_t m = (uint64_t)(frexp(p, &pe) * 0x1.0p53);   // p = m 2^(pe - 53), pe <= k e
            const int sh = 96 + pe - 53 - k * e;                       // <= 43
            if (sh >= 0) {   // m 2^sh over three limbs
                const uint64_t lo = sh < 64 ? m << sh : 0, hi = sh ? m >> (64 - sh) : 0;
                l0 = (uint32_t)lo, l1 = (uint32_t)(lo >> 32), l2 = (uint32_t)hi;
            } else if (sh > -64) {
                const uint64_t lo = (m + (1ull << (-sh - 1))) >> -sh;
                l0 = (uint32_t)lo, l1 = (uint32_t)(lo >> 32);
            }
        }
        uint32_t *o = xf + ((uint64_t)(k - 1) * n + j) * 3;
        o[0] = l0, o[1] = l1, o[2] = l2;
    }
}

// RB resamples of one group per CTA.  A resample's draws are counted per member in
// shared memory (bytes: a count above 255 in N draws of N members has probability
// below 1/256! for N > 255 and cannot occur for fewer), then F^(k) = sum of count x^k / N
// is summed in fixed point: one 32 x 32 -> 64 multiply-add per limb where the
// FP64 pipe, 77 times slower, took a multiplication and an addition per draw and k
// (the whole call, 300 resamples of 200,000 traces, 9 groups, k <= 4: 0.44 ms against
// 2.06 ms with FP64 sums and host-built group lists).  The sums of the integers are exact;
// each term is rounded at half a unit, 2^-97 of the power of the group's largest member.  A
// sum of N terms below N 2^53 units (a resample that missed members far above the rest) would
// hold less than a double: that resample and k goes to bootstrap_kernel, so that every
// F^(k) is within 2^-54 of the sum of its terms.
// Bound: the Philox rounds.
constexpr int CT = 512, RB = 4;
static_assert(FP_MAX_KMAX <= 8, "a bit per power in an entry of the list");
// list of bootstrap_kernel's work: redo[0] entries, entry (g B + b) << 8 | bit per k
__device__ __forceinline__ void redo_add(unsigned long long *redo, uint64_t gb, uint32_t ks) {
    redo[1 + atomicAdd(redo, 1ull)] = gb << 8 | ks;
}
__global__ void __launch_bounds__(CT) bootstrap_count_kernel(const uint32_t *__restrict__ xf,
                                                             const uint64_t *__restrict__ off,
                                                             const uint64_t *__restrict__ xoff, int n_groups, int k_max,
                                                             int B, uint64_t seed, const int *__restrict__ exp2,
                                                             uint32_t max_n, unsigned long long *__restrict__ redo,
                                                             double *__restrict__ out) {
    extern __shared__ uint32_t cnt[];   // [words][RB]: word w holds the counts of members 4w .. 4w+3
    __shared__ uint64_t red[CT / 32][RB][3];
    const int g = blockIdx.y, b0 = blockIdx.x * RB;
    const uint64_t N = off[g + 1] - off[g], o = xoff[g], n = xoff[n_groups];
    if (N == 0 || N > max_n || exp2[g] >= kNoScale) {   // bootstrap_kernel takes these
        if (threadIdx.x < RB && b0 + (int)threadIdx.x < B) redo_add(redo, (uint64_t)g * B + b0 + threadIdx.x, 0xff);
        return;
    }
    const uint32_t words = (uint32_t)((N + 3) / 4);
    for (uint32_t i = threadIdx.x; i < words * RB; i += CT) cnt[i] = 0;
    __syncthreads();
    const uint32_t nq = words, Nn = (uint32_t)N;   // draws come in fours
    for (uint32_t i = threadIdx.x; i < nq * RB; i += CT) {
        const uint32_t r = i / nq, q = i - r * nq;
        if (b0 + (int)r >= B) break;
        const U64x4 x = philox(seed, (uint64_t)(b0 + r), q, (uint64_t)g, 5);
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            if (4 * q + w >= Nn) break;
            const uint32_t pos = __umulhi((uint32_t)(x.x[w] >> 32), Nn);
            atomicAdd(&cnt[(pos >> 2) * RB + r], 1u << (8 * (pos & 3)));
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t again = 0;   // threads below RB: the powers whose sum kept too few bits
    for (int k = 0; k < k_max; ++k) {
        uint64_t s[RB][3];
#pragma unroll
        for (int r = 0; r < RB; ++r) s[r][0] = s[r][1] = s[r][2] = 0;
        const uint32_t *xk = xf + ((uint64_t)k * n + o) * 3;
        for (uint32_t w = threadIdx.x; w < words; w += CT) {
            uint32_t c[RB];
#pragma unroll
            for (int r = 0; r < RB; ++r) c[r] = cnt[w * RB + r];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const uint32_t j = 4 * w + m;
                if (j >= Nn) break;
                const uint32_t l0 = xk[3 * (uint64_t)j], l1 = xk[3 * (uint64_t)j + 1], l2 = xk[3 * (uint64_t)j + 2];
#pragma unroll
                for (int r = 0; r < RB; ++r) {
                    const uint32_t cr = (c[r] >> (8 * m)) & 255u;
                    s[r][0] += (uint64_t)cr * l0;
                    s[r][1] += (uint64_t)cr * l1;
                    s[r][2] += (uint64_t)cr * l2;
                }
            }
        }
#pragma unroll
        for (int r = 0; r < RB; ++r)
#pragma unroll
            for (int l = 0; l < 3; ++l) {
                for (int d = 16; d > 0; d >>= 1) s[r][l] += __shfl_down_sync(0xffffffffu, s[r][l], d);
                if (lane == 0) red[wid][r][l] = s[r][l];
            }
        __syncthreads();
        if (threadIdx.x < RB && b0 + (int)threadIdx.x < B) {
            uint64_t t[3] = {0, 0, 0};
            for (int w = 0; w < CT / 32; ++w)
                for (int l = 0; l < 3; ++l) t[l] += red[w][threadIdx.x][l];
            // t0 + t1 2^32 + t2 2^64, as a high and a low part that double holds to 2^-106
            const uint64_t mid = t[1] + (t[0] >> 32);                  // (< 2^63)
            const uint64_t hi = t[2] + (mid >> 32), lo = (mid << 32) | (t[0] & 0xffffffffu);
            const double v = ((double)hi * 0x1.0p64 + (double)lo) / (double)N;
            out[((size_t)g * k_max + k) * B + b0 + threadIdx.x] =
                exp2[g] > -kNoScale ? ldexp(v, (k + 1) * exp2[g] - 96) : 0.0;
            if (exp2[g] > -kNoScale && v < 0x1.0p53) again |= 1u << k;
        }
        __syncthreads();
    }
    if (again) redo_add(redo, (uint64_t)g * B + b0 + threadIdx.x, again);
}

// In FP64, draw by draw: the groups that the counts do not take (empty, too large for
// shared memory, powers that are not finite) and the sums that they could not hold; redo ==
// nullptr: every resample of every group.  Entry (g, b): resample b of group g.  Draw i takes
// position ((x >> 32) N_g) >> 32 of the group, x = word i % 4 of Philox block
// {b, i / 4, g, 5} (key {seed, 0}); F^(k) of the resample = mean of a^k over
// the draws.  Fixed thread-to-draw mapping and tree: deterministic, whatever the list's order.
constexpr int BT = 256;
__global__ void __launch_bounds__(BT) bootstrap_kernel(const double *__restrict__ xs,
                                                       const uint64_t *__restrict__ goff, int n_groups, int k_max, int B,
                                                       uint64_t seed, const unsigned long long *__restrict__ redo,
                                                       double *__restrict__ out) {
    __shared__ double sh[FP_MAX_KMAX][BT / 32];
    const uint64_t entries = redo ? redo[0] : (uint64_t)n_groups * B;
    for (uint64_t e = blockIdx.x; e < entries; e += gridDim.x) {
        const uint64_t gb = redo ? redo[1 + e] >> 8 : e;
        const uint32_t ks = redo ? (uint32_t)redo[1 + e] & 0xffu : 0xffu;
        const int g = (int)(gb / (uint64_t)B), b = (int)(gb - (uint64_t)g * B);
        const uint64_t off = goff[g], N = goff[g + 1] - off;
        double s[FP_MAX_KMAX];
#pragma unroll
        for (int k = 0; k < FP_MAX_KMAX; ++k) s[k] = 0.0;
        const uint64_t nq = (N + 3) / 4;
        for (uint64_t q = threadIdx.x; q < nq; q += BT) {
            const U64x4 x = philox(seed, (uint64_t)b, q, (uint64_t)g, 5);
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                if (4 * q + w >= N) break;
                const uint64_t pos = ((x.x[w] >> 32) * N) >> 32;
                const double a2 = xs[off + pos];
                double p = 1.0;
#pragma unroll
                for (int k = 0; k < FP_MAX_KMAX; ++k) {
                    if (k < k_max) {
                        p *= a2;
                        s[k] += p;
                    }
                }
            }
        }
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
        for (int k = 0; k < FP_MAX_KMAX; ++k) {
            if (k >= k_max || (uint64_t)wid * 32 >= nq) break;   // (a warp without draws adds nothing)
            double v = s[k];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            if (lane == 0) sh[k][wid] = v;
        }
        __syncthreads();
        if (threadIdx.x < k_max && (ks >> threadIdx.x & 1)) {
            const int k = threadIdx.x;
            double v = 0;
            for (int w = 0; w < BT / 32 && (uint64_t)w * 32 < nq; ++w) v += sh[k][w];
            out[((size_t)g * k_max + k) * B + b] = N ? v / (double)N : __longlong_as_double(0x7ff8000000000000LL);
        }
        __syncthreads();
    }
}

}  // namespace

namespace {
constexpr uint32_t kMaxCounted = 200 * 1024 / RB;   // members whose counts fit shared memory
uint64_t counted_members(uint64_t count, int n_groups) {
    return std::min<uint64_t>(count, (uint64_t)n_groups * kMaxCounted);
}
size_t up16(size_t b) { return (b + 15) / 16 * 16; }
// pairs per chunk: whole passes of a CTA, at most 4096 chunks
uint64_t chunk_pairs(uint64_t count) { return ((count + 4095) / 4096 + kChunk - 1) / kChunk * kChunk; }
constexpr int kFewGroups = 16;   // a CTA per (chunk, group) up to here
constexpr uint64_t kNoWait = 12800;
// small batches: the FP64 sums of this many draws and powers take 20 us, the launches that the
// counts need before they start as much
constexpr uint64_t kSmallSums = 1ull << 22;
int chunks(uint64_t count) { return count ? (int)((count + chunk_pairs(count) - 1) / chunk_pairs(count)) : 0; }
}  // namespace

size_t bootstrap_scratch(uint64_t count, int n_groups, int k_max, int B) {
    return up16((size_t)count * 8) + up16((size_t)(2 * n_groups + 2) * 8) + up16((size_t)n_groups * 4) +
           up16((size_t)n_groups * chunks(count) * 4) + up16((size_t)counted_members(count, n_groups) * k_max * 12) +
           ((size_t)n_groups * B + 1) * 8;
}

cudaError_t launch_bootstrap(const double *tr, const int32_t *group, uint64_t count, int n_groups, int k_max, int B,
                             uint64_t seed, void *scratch, double *out, cudaStream_t st) {
    char *at = (char *)scratch;
    double *xs = (double *)at;
    at += up16((size_t)count * 8);
    uint64_t *off = (uint64_t *)at, *xoff = off + n_groups + 1;
    at += up16((size_t)(2 * n_groups + 2) * 8);
    int *exp2 = (int *)at;
    at += up16((size_t)n_groups * 4);
    uint32_t *cnt = (uint32_t *)at;
    const int nc = chunks(count);
    at += up16((size_t)n_groups * nc * 4);
    const uint64_t nx = counted_members(count, n_groups);
    uint32_t *xf = (uint32_t *)at;
    unsigned long long *redo = (unsigned long long *)(at + up16((size_t)nx * k_max * 12));
    cudaError_t e;
    if (n_groups > 65535) return cudaErrorInvalidValue;
    const uint64_t entries = (uint64_t)B * n_groups;
    const unsigned fgrid = (unsigned)std::min<uint64_t>(entries, 152 * 8);
    if (count <= kSmallPairs && n_groups <= kSmallGroups && count * B * k_max <= kSmallSums) {
        group_small_kernel<<<1, 1024, 0, st>>>(tr, group, (int)count, n_groups, off, xs);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        bootstrap_kernel<<<fgrid, BT, 0, st>>>(xs, off, n_groups, k_max, B, seed, nullptr, out);
        return cudaGetLastError();
    }
    const bool many = n_groups > kFewGroups;
    const uint64_t per = chunk_pairs(count);
    const dim3 cg((unsigned)nc, (unsigned)n_groups);
    if (many) {
        if ((e = cudaMemsetAsync(cnt, 0, (size_t)n_groups * nc * 4, st)) != cudaSuccess) return e;
        if (nc > 0)
            group_count_many_kernel<<<(unsigned)((count + 255) / 256), 256, 0, st>>>(group, count, per, nc, n_groups, cnt);
        group_prefix_kernel<<<(unsigned)((n_groups + 7) / 8), 256, 0, st>>>(cnt, nc, n_groups, off, exp2);
    } else if (nc > 0) {
        group_count_kernel<<<cg, GT, 0, st>>>(group, count, per, cnt);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    group_offsets_kernel<<<1, 1024, 0, st>>>(cnt, nc, n_groups, kMaxCounted, !many, off, xoff, exp2, redo);
    if (nc > 0 && many)
        group_place_many_kernel<<<(unsigned)nc, 32, 0, st>>>(tr, group, count, per, nc, n_groups, off, cnt, k_max, xs, exp2);
    else if (nc > 0)
        group_place_kernel<<<cg, GT, 0, st>>>(tr, group, count, per, off, cnt, k_max, xs, exp2);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // The largest counted group's size sets the shared memory: two CTAs per SM up to 25,600 members, four,
    // which is what their threads allow, up to kNoWait.  A batch of that many pairs in all does not wait for the sizes.
    uint64_t largest = count;
    if (nx > 0) powers_kernel<<<(unsigned)((nx + 255) / 256), 256, 0, st>>>(xs, off, xoff, n_groups, k_max, exp2, xf);
    if (count > kNoWait) {
        std::vector<uint64_t> h((size_t)n_groups + 1);
        if ((e = cudaMemcpyAsync(h.data(), off, h.size() * sizeof(uint64_t), cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
        largest = 0;
        for (int g = 0; g < n_groups; ++g)
            if (h[g + 1] - h[g] <= kMaxCounted) largest = std::max(largest, h[g + 1] - h[g]);
    }
    if (largest > 0) {
        if ((e = allow_smem(bootstrap_count_kernel, kMaxCounted * RB)) != cudaSuccess) return e;
        bootstrap_count_kernel<<<dim3((unsigned)((B + RB - 1) / RB), (unsigned)n_groups), CT,
                                 (size_t)((largest + 3) / 4) * 4 * RB, st>>>(xf, off, xoff, n_groups, k_max, B, seed, exp2,
                                                                             kMaxCounted, redo, out);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    bootstrap_kernel<<<fgrid, BT, 0, st>>>(xs, off, n_groups, k_max, B, seed, largest > 0 ? redo : nullptr, out);
    return cudaGetLastError();
}

int moments_blocks(uint64_t count) {
    uint64_t b = (count + 4095) / 4096;
    if (b < 1) b = 1;
    if (b > 1024) b = 1024;
    return (int)b;
}

cudaError_t launch_moments(const double *tr, const int32_t *group, uint64_t count, int k_max,
                           int n_groups, double *partials, int nblocks, double *out,
                           cudaStream_t st) {
    moments_pass1<<<nblocks, RT, 0, st>>>(tr, group, count, k_max, n_groups, partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    int tot = n_groups * (2 * k_max + 1);
    moments_pass2<<<(tot + 127) / 128, 128, 0, st>>>(partials, nblocks, k_max, n_groups, out);
    return cudaGetLastError();
}

}  // namespace fpk
