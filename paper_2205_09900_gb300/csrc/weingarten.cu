// weingarten.cu -- exact ensemble F^(k) (k = 2, 3) of brickwork circuits of qubits
// or of qudits of local dimension q (Haar U(q^2) gates).
//
// Averaging every Haar U(4) gate of the cyclic U^dagger V circuit over the
// Haar measure turns the k-th moment |Tr(U^dagger V)|^{2k} into a classical
// statistical-mechanics sum (the mapping behind the paper's Eq. theory_eq,
// Sec. "Frame potential"): each gate carries an output and an input pairing
// sigma, tau in S_k with weight Wg(sigma^-1 tau) (the Weingarten function of
// U(4)), and consecutive gates on a qubit wire, output pairing sigma_a then
// input pairing tau_b, meet with weight q^{#cycles(sigma_a^-1 tau_b)}.
//
// After the middle and cyclic merges a depth-l brickwork pair is a cyclic
// brickwork of P = 2(l-1) time positions; bond b holds the gates at the
// positions t with t = b+1 (mod 2).  Give the wire links of any qubit the
// indices t = 0..P-1 (link t joins the gate at position t to the one at t+1).
// Storing a gate's output pairing in slot t and its input pairing in slot
// t-1 (mod P), the variables of one bond occupy every slot exactly once, and
// the transfer across qubit b is
//   (1) the q^{#cycles} link matrix applied to every slot (each link of the
//       qubit pairs one slot of bond b-1 with the same slot of bond b), then
//   (2) the Wg factors of bond b's gates, a diagonal over slot pairs (t, t-1).
// The chain ends close with the links among one bond's gates, slots (t, t+1).
//
// Weights and links depend on sigma^-1 tau only, so the state is unchanged when
// every slot is multiplied from the left by the same permutation: only the
// entries whose last slot is the identity are kept, s^(P-1) of s^P (k = 3: a
// sixth of the FP64 work and of the memory; at l = 6 the 81 MB state stays in
// L2).  A link on a kept slot is unchanged; the link on the last slot mixes the
// s entries {h u} of an orbit (h u: every digit multiplied from the left by h)
// by the same matrix, in place, one thread per orbit.  The state is renormalised
// by a power of two after every bond (exact), the exponents summed at the end.
//
// Bound: the FP64 pipe (about 1.05 TFLOP/s on this part).  The link matrix of
// S_3 is (q^3 - q) I plus a matrix of rank 2 (sums over the even and the odd
// permutations): 14 FP64 operations per 6 entries instead of 36.  Several slots
// run per pass over the state: the low slots on contiguous tiles in shared
// memory, the others in registers.  Measured at n = 50 on a GB300:
// F^(3) at l = 6 in 32 ms against 407 ms with all 6^10 entries and one slot per pass.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "kernels.h"

namespace fpk {
namespace {

constexpr int kMaxSlots = 22;   // k = 2: l <= 12; k = 3 is limited to 12 slots (l <= 7)

struct WgTab {
    int P;                  // slots
    double link[36];        // link[x * s + y] = q^{#cycles(x^-1 y)}
    double wg[36];          // wg[sigma * s + tau] = Wg(sigma^-1 tau)
    double la, lb, lc;      // k = 3: q^3 - q, q, q^2
    uint8_t mul[36];        // mul[a * s + b]: a after b
};

// digits of kept entry c; the last slot is the identity (index 0)
template <int S>
__device__ __forceinline__ void decode(uint64_t c, int P, int *d) {
    if (S == 2) {
        for (int t = 0; t < P - 1; ++t) d[t] = (int)((c >> t) & 1u);
    } else {
        for (int t = 0; t < P - 1; ++t) {
            d[t] = (int)(c % S);
            c /= S;
        }
    }
    d[P - 1] = 0;
}

// x <- link matrix . x.  S_3 in the order 012, 021, 102, 120, 201, 210: the even
// permutations are 0, 3, 4.
template <int S>
__device__ __forceinline__ void apply_link(const WgTab &T, double (&x)[S]) {
    if constexpr (S == 2) {
        const double a = x[0], b = x[1];
        x[0] = fma(T.link[0], a, T.link[2] * b);
        x[1] = fma(T.link[1], a, T.link[3] * b);
    } else {
        const double E = x[0] + x[3] + x[4], O = x[1] + x[2] + x[5];
        const double e = fma(T.lb, E, T.lc * O), o = fma(T.lb, O, T.lc * E);
        x[0] = fma(T.la, x[0], e);
        x[3] = fma(T.la, x[3], e);
        x[4] = fma(T.la, x[4], e);
        x[1] = fma(T.la, x[1], o);
        x[2] = fma(T.la, x[2], o);
        x[5] = fma(T.la, x[5], o);
    }
}

// |x| as the integer that orders like it
__device__ __forceinline__ unsigned long long abs_bits(double x) {
    return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}

__device__ __forceinline__ unsigned long long block_max(unsigned long long v) {   // total in thread 0
    __shared__ unsigned long long red[32];
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
        v = w > v ? w : v;
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int i = 1; i < (int)(blockDim.x >> 5); ++i) v = red[i] > v ? red[i] : v;
    return v;
}

__device__ __forceinline__ double unscale(const double *maxes, int b) {
    const double m = maxes[b];
    return m > 0 ? ldexp(1.0, -ilogb(m)) : 1.0;   // maxes holds the bit patterns of abs_bits
}

// qubit 0: Wg of the bond-0 gates (positions t = 1 mod 2) and the links among them
template <int S>
__device__ __forceinline__ double init_value(const WgTab &T, uint64_t c) {
    int d[kMaxSlots];
    decode<S>(c, T.P, d);
    double p = 1.0;
    for (int t = 1; t < T.P; t += 2) {
        p *= T.wg[d[t] * S + d[t - 1]];
        p *= T.link[d[t] * S + d[(t + 1) % T.P]];
    }
    return p;
}

template <int S>
__global__ void wg_init_kernel(const __grid_constant__ WgTab T, uint64_t N, double *__restrict__ v,
                               double *__restrict__ maxes) {
    unsigned long long mx = 0;
    for (uint64_t c = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; c < N; c += (uint64_t)gridDim.x * blockDim.x) {
        const double p = init_value<S>(T, c);
        v[c] = p;
        const unsigned long long a = abs_bits(p);
        mx = a > mx ? a : mx;
    }
    mx = block_max(mx);
    if (threadIdx.x == 0) atomicMax((unsigned long long *)maxes, mx);
}

// Links on the G slots from stride s^i upwards (stride = s^i), in place: a thread
// holds their s^G values in registers, neighbouring threads neighbouring entries.
template <int S, int G> struct Pow { static constexpr int v = S * Pow<S, G - 1>::v; };
template <int S> struct Pow<S, 0> { static constexpr int v = 1; };

template <int S, int G>
__global__ void __launch_bounds__(256) wg_mid_kernel(const __grid_constant__ WgTab T, uint64_t N, uint64_t stride,
                                                     double *__restrict__ v) {
    constexpr int B = Pow<S, G>::v;
    const uint64_t cols = N / B;
    for (uint64_t col = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; col < cols;
         col += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t hi = col / stride, lo = col - hi * stride;
        double *p = v + hi * stride * B + lo;
        double x[B];
#pragma unroll
        for (int j = 0; j < B; ++j) x[j] = p[j * stride];
#pragma unroll
        for (int g = 0, st = 1; g < G; ++g, st *= S) {
#pragma unroll
            for (int j = 0; j < B; ++j) {
                if ((j / st) % S) continue;
                double y[S];
#pragma unroll
                for (int e = 0; e < S; ++e) y[e] = x[j + e * st];
                apply_link<S>(T, y);
#pragma unroll
                for (int e = 0; e < S; ++e) x[j + e * st] = y[e];
            }
        }
#pragma unroll
        for (int j = 0; j < B; ++j) p[j * stride] = x[j];
    }
}

// Links on the lowest D slots: contiguous tiles of s^D entries in shared memory
// (s = 2: groups of up to 4 slots in registers between barriers; s = 6: one).
constexpr int kLow2 = 12, kLow6 = 4;   // 2^12 and 6^4 entries
template <int S>
__device__ __forceinline__ void low_slots(const WgTab &T, double *tile, int D, uint32_t n) {
    uint32_t st = 1;
    if constexpr (S == 2) {
        for (int t = 0; t < D;) {
            if (D - t >= 4) {
                for (uint32_t i = threadIdx.x; i < n / 16; i += blockDim.x) {
                    double *p = tile + (i / st) * st * 16 + i % st;
                    double x[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) x[j] = p[j * st];
#pragma unroll
                    for (int b = 1; b < 16; b *= 2)
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            if (j & b) continue;
                            double y[2] = {x[j], x[j | b]};
                            apply_link<2>(T, y);
                            x[j] = y[0];
                            x[j | b] = y[1];
                        }
#pragma unroll
                    for (int j = 0; j < 16; ++j) p[j * st] = x[j];
                }
                t += 4;
                st *= 16;
            } else {
                for (uint32_t i = threadIdx.x; i < n / 2; i += blockDim.x) {
                    double *p = tile + (i / st) * st * 2 + i % st;
                    double y[2] = {p[0], p[st]};
                    apply_link<2>(T, y);
                    p[0] = y[0];
                    p[st] = y[1];
                }
                t += 1;
                st *= 2;
            }
            __syncthreads();
        }
    } else {
        for (int t = 0; t < D; ++t, st *= S) {
            for (uint32_t i = threadIdx.x; i < n / S; i += blockDim.x) {
                double *p = tile + (i / st) * st * S + i % st;
                double y[S];
#pragma unroll
                for (int e = 0; e < S; ++e) y[e] = p[e * st];
                apply_link<S>(T, y);
#pragma unroll
                for (int e = 0; e < S; ++e) p[e * st] = y[e];
            }
            __syncthreads();
        }
    }
}

template <int S>
__global__ void __launch_bounds__(256) wg_low_kernel(const __grid_constant__ WgTab T, uint64_t N, int D, uint32_t n,
                                                     double *__restrict__ v) {
    __shared__ double tile[S == 2 ? 1 << kLow2 : 1296];
    for (uint64_t o = (uint64_t)blockIdx.x * n; o < N; o += (uint64_t)gridDim.x * n) {
        for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) tile[i] = v[o + i];
        __syncthreads();
        low_slots<S>(T, tile, D, n);
        for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) v[o + i] = tile[i];
        __syncthreads();
    }
}

// One orbit {h u}, u with first digit 0 (its other digits coded in c): the link on
// the last slot, then Wg of bond b's gates (positions t = par mod 2) times sc.
// Gates that do not touch the last slot weigh the whole orbit alike.
template <int S>
__device__ __forceinline__ void orbit(const WgTab &T, const double *wg, const uint8_t *mul, uint64_t c, int par, double sc, double *v,
                                      unsigned long long &mx) {
    uint64_t r = c, pw = S, idx[S];
    double w = sc;
    int d = 0;   // the digit of slot t
#pragma unroll
    for (int h = 0; h < S; ++h) idx[h] = (uint64_t)h;
    for (int t = 1; t < T.P - 1; ++t, pw *= S) {
        const int prev = d;
        d = (int)(r % S);
        r /= S;
#pragma unroll
        for (int h = 0; h < S; ++h) idx[h] += pw * mul[h * S + d];
        if ((t & 1) == par) w *= wg[d * S + prev];
    }
    double x[S];
#pragma unroll
    for (int h = 0; h < S; ++h) x[h] = v[idx[h]];
    apply_link<S>(T, x);
#pragma unroll
    for (int h = 0; h < S; ++h) {
        // the pair with the last slot (identity): (P-1, P-2) or (0, P-1)
        const int u = par ? mul[h * S + d] : h;
        x[h] *= w * wg[u * S];
        v[idx[h]] = x[h];
        const unsigned long long a = abs_bits(x[h]);
        mx = a > mx ? a : mx;
    }
}

template <int S>
__global__ void __launch_bounds__(256) wg_orbit_kernel(const __grid_constant__ WgTab T, uint64_t N, int par, int b,
                                                       double *__restrict__ v, double *__restrict__ maxes) {
    __shared__ double wg[S * S];
    __shared__ uint8_t mul[S * S];
    for (int i = threadIdx.x; i < S * S; i += blockDim.x) wg[i] = T.wg[i], mul[i] = T.mul[i];
    __syncthreads();
    const double sc = unscale(maxes, b - 1);
    unsigned long long mx = 0;
    for (uint64_t c = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; c < N / S; c += (uint64_t)gridDim.x * blockDim.x)
        orbit<S>(T, wg, mul, c, par, sc, v, mx);
    mx = block_max(mx);
    if (threadIdx.x == 0) atomicMax((unsigned long long *)(maxes + b), mx);
}

// last qubit: links among the last bond's gates
template <int S>
__device__ __forceinline__ double final_value(const WgTab &T, uint64_t c, int par, double p) {
    int d[kMaxSlots];
    decode<S>(c, T.P, d);
    for (int t = par; t < T.P; t += 2) p *= T.link[d[t] * S + d[(t + 1) % T.P]];
    return p;
}

__device__ __forceinline__ double block_sum(double acc) {   // total in thread 0
    __shared__ double red[32];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) red[w] = acc;
    __syncthreads();
    double s = 0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
    return s;
}

// one partial sum per block
template <int S>
__global__ void wg_final_kernel(const __grid_constant__ WgTab T, uint64_t N, int par, int blast,
                                const double *__restrict__ v, const double *__restrict__ maxes,
                                double *__restrict__ partial) {
    const double sc = unscale(maxes, blast);
    double acc = 0;
    for (uint64_t c = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; c < N; c += (uint64_t)gridDim.x * blockDim.x)
        acc += final_value<S>(T, c, par, v[c] * sc);
    acc = block_sum(acc);
    if (threadIdx.x == 0) partial[blockIdx.x] = acc;
}

// The whole sweep in one CTA (states up to kOneCta entries: a pass over them costs
// less than the launches it would take): one launch instead of three per bond.
constexpr uint32_t kOneCta = 512;
template <int S>
__global__ void __launch_bounds__(256) wg_small_kernel(const __grid_constant__ WgTab T, int n, uint32_t N,
                                                       double *__restrict__ out) {
    __shared__ double v[kOneCta];
    __shared__ double wg[S * S];
    __shared__ uint8_t mul[S * S];
    __shared__ unsigned long long top;
    for (int i = threadIdx.x; i < S * S; i += blockDim.x) wg[i] = T.wg[i], mul[i] = T.mul[i];
    unsigned long long mx = 0;
    int e2 = 0;
    for (uint32_t c = threadIdx.x; c < N; c += blockDim.x) {
        v[c] = init_value<S>(T, c);
        const unsigned long long a = abs_bits(v[c]);
        mx = a > mx ? a : mx;
    }
    for (int b = 1; b <= n - 1; ++b) {
        mx = block_max(mx);
        if (threadIdx.x == 0) top = mx;
        __syncthreads();
        const double m = __longlong_as_double((long long)top);
        const double sc = m > 0 ? ldexp(1.0, -ilogb(m)) : 1.0;
        if (m > 0) e2 += ilogb(m);
        if (b == n - 1) {
            double acc = 0;
            for (uint32_t c = threadIdx.x; c < N; c += blockDim.x)
                acc += final_value<S>(T, c, (n - 1) & 1, v[c] * sc);
            acc = block_sum(acc);
            if (threadIdx.x == 0) *out = ldexp(acc * S, e2);
            return;
        }
        low_slots<S>(T, v, T.P - 1, N);
        mx = 0;
        for (uint32_t c = threadIdx.x; c < N / S; c += blockDim.x) orbit<S>(T, wg, mul, c, (b + 1) & 1, sc, v, mx);
    }
}

// fixed-order sum of the partials, times 2^{sum of the per-bond exponents} and
// the s equal shares of the last slot's values
__global__ void __launch_bounds__(256) wg_sum_kernel(const double *__restrict__ partial, int nparts,
                                                     const double *__restrict__ maxes, int nmax, int s,
                                                     double *__restrict__ out) {
    __shared__ int e;
    if (threadIdx.x == 0) e = 0;
    __syncthreads();
    double acc = 0;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) acc += partial[i];
    int my = 0;
    for (int b = threadIdx.x; b < nmax; b += blockDim.x)
        if (maxes[b] > 0) my += ilogb(maxes[b]);
    atomicAdd(&e, my);
    acc = block_sum(acc);   // its barrier also completes e
    if (threadIdx.x == 0) *out = ldexp(acc * s, e);
}

// host: permutations of S_k and their cycle counts
int perms(int k, int (*p)[3]) {
    int np = 0, v[3];
    for (v[0] = 0; v[0] < k; ++v[0])
        for (v[1] = 0; v[1] < (k > 1 ? k : 1); ++v[1])
            for (v[2] = 0; v[2] < (k > 2 ? k : 1); ++v[2]) {
                bool ok = true;
                for (int i = 0; i < k; ++i)
                    for (int j = 0; j < i; ++j) ok = ok && v[i] != v[j];
                if (!ok) continue;
                for (int i = 0; i < 3; ++i) p[np][i] = v[i];
                ++np;
            }
    return np;
}

int cycles(const int *a, const int *b, int k) {   // #cycles of a^-1 b
    int inv[3], seen[3] = {0, 0, 0}, c = 0;
    for (int i = 0; i < k; ++i) inv[a[i]] = i;
    for (int i = 0; i < k; ++i) {
        if (seen[i]) continue;
        ++c;
        for (int j = i; !seen[j]; j = inv[b[j]]) seen[j] = 1;
    }
    return c;
}

template <int S, int G>
cudaError_t run_mid(const WgTab &T, uint64_t N, uint64_t stride, double *v, cudaStream_t st) {
    const uint64_t cols = N / Pow<S, G>::v;
    wg_mid_kernel<S, G><<<(unsigned)std::min<uint64_t>((cols + 255) / 256, 152u * 16u), 256, 0, st>>>(T, N, stride, v);
    return cudaGetLastError();
}

template <int S>
cudaError_t run_sweep(const WgTab &T, int n, uint64_t N, double *v, double *maxes, double *partial, int nparts,
                      double *out, cudaStream_t st) {
    const int threads = 256, slots = T.P - 1;
    if (N <= kOneCta) {
        wg_small_kernel<S><<<1, threads, 0, st>>>(T, n, (uint32_t)N, out);
        return cudaGetLastError();
    }
    const unsigned grid = (unsigned)std::min<uint64_t>((N + threads - 1) / threads, 152u * 16u);
    const unsigned ogrid = (unsigned)std::min<uint64_t>((N / S + threads - 1) / threads, 152u * 16u);
    const int D = std::min(slots, S == 2 ? kLow2 : kLow6);
    uint32_t tile = 1;
    for (int i = 0; i < D; ++i) tile *= S;
    const unsigned lgrid = (unsigned)std::min<uint64_t>(N / tile, 152u * 16u);
    wg_init_kernel<S><<<grid, threads, 0, st>>>(T, N, v, maxes);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    for (int b = 1; b <= n - 2; ++b) {
        wg_low_kernel<S><<<lgrid, threads, 0, st>>>(T, N, D, tile, v);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        uint64_t stride = tile;
        for (int i = D; i < slots;) {
            const int g = std::min(slots - i, S == 2 ? 5 : 2);
            if constexpr (S == 2) {
                e = g == 5 ? run_mid<2, 5>(T, N, stride, v, st) : g == 4 ? run_mid<2, 4>(T, N, stride, v, st)
                  : g == 3 ? run_mid<2, 3>(T, N, stride, v, st) : g == 2 ? run_mid<2, 2>(T, N, stride, v, st)
                           : run_mid<2, 1>(T, N, stride, v, st);
            } else {
                e = g == 2 ? run_mid<6, 2>(T, N, stride, v, st) : run_mid<6, 1>(T, N, stride, v, st);
            }
            if (e != cudaSuccess) return e;
            for (int k = 0; k < g; ++k) stride *= S;
            i += g;
        }
        wg_orbit_kernel<S><<<ogrid, threads, 0, st>>>(T, N, (b + 1) & 1, b, v, maxes);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    wg_final_kernel<S><<<nparts, threads, 0, st>>>(T, N, (n - 1) & 1, n - 2, v, maxes, partial);
    wg_sum_kernel<<<1, 256, 0, st>>>(partial, nparts, maxes, n - 1, S, out);
    return cudaGetLastError();
}

}  // namespace
}  // namespace fpk

extern "C" fp_status fp_exact_brickwork_fkq(int32_t n, int32_t l, int32_t k, int32_t q, void *cuda_stream,
                                             double *F) {
    using namespace fpk;
    if (!F) return api_fail(FP_ERR_ARG, "F is NULL");
    if (n < 2 || n > 1 << 20) return api_fail(FP_ERR_ARG, "n outside [2, 2^20]");
    if (q < 2 || q > 64) return api_fail(FP_ERR_ARG, "local dimension q outside [2, 64]");
    if (k != 2 && k != 3) return api_fail(FP_ERR_ARG, "k must be 2 or 3");
    if (l < 2 || (k == 2 && l > 12) || (k == 3 && l > 7))
        return api_fail(FP_ERR_ARG, "depth l outside [2, 12] (k = 2) or [2, 7] (k = 3)");
    WgTab T;
    T.P = 2 * (l - 1);
    int p[6][3];
    const int s = perms(k, p);
    const double d = (double)q * q;   // Haar U(q^2) gates on neighbouring qudits
    for (int a = 0; a < s; ++a)
        for (int b = 0; b < s; ++b) {
            const int c = cycles(p[a], p[b], k);
            T.link[a * s + b] = std::pow((double)q, c);
            double w;
            if (k == 2) w = c == 2 ? 1.0 / (d * d - 1) : -1.0 / (d * (d * d - 1));
            else w = c == 3 ? (d * d - 2) / (d * (d * d - 1) * (d * d - 4))
                   : c == 2 ? -1.0 / ((d * d - 1) * (d * d - 4))
                            : 2.0 / (d * (d * d - 1) * (d * d - 4));
            T.wg[a * s + b] = w;
        }
    for (int a = 0; a < s; ++a)
        for (int b = 0; b < s; ++b)
            for (int c = 0; c < s; ++c)   // (a after b)(j) = a(b(j))
                if (p[c][0] == p[a][p[b][0]] && p[c][1] == p[a][p[b][1]] && (k < 3 || p[c][2] == p[a][p[b][2]]))
                    T.mul[a * s + b] = (uint8_t)c;
    T.la = (double)q * q * q - q;
    T.lb = q;
    T.lc = (double)q * q;
    uint64_t N = 1;   // entries with the identity in the last slot
    for (int i = 0; i + 1 < T.P; ++i) N *= (uint64_t)s;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    size_t freeb = 0, totb = 0;
    cudaError_t e = cudaMemGetInfo(&freeb, &totb);
    if (e != cudaSuccess) return api_fail(FP_ERR_CUDA, cudaGetErrorString(e));
    const int nparts = (int)std::min<uint64_t>(152 * 4, (N + 255) / 256);
    const size_t bytes = N * sizeof(double) + ((size_t)n + nparts + 1) * sizeof(double);
    if (bytes > freeb) return api_fail(FP_ERR_OOM, "transfer-matrix state does not fit in free device memory");
    double *buf = nullptr;
    if ((e = cudaMalloc(&buf, bytes)) != cudaSuccess) return api_fail(FP_ERR_OOM, cudaGetErrorString(e));
    double *v = buf, *maxes = buf + N, *partial = maxes + n, *out = partial + nparts;
    e = cudaMemsetAsync(maxes, 0, (size_t)n * sizeof(double), st);
    if (e == cudaSuccess) e = k == 2 ? run_sweep<2>(T, n, N, v, maxes, partial, nparts, out, st)
                                     : run_sweep<6>(T, n, N, v, maxes, partial, nparts, out, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(F, out, sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(buf);
    if (e != cudaSuccess) return api_fail(FP_ERR_CUDA, cudaGetErrorString(e));
    return FP_OK;
}

extern "C" fp_status fp_exact_brickwork_fk(int32_t n, int32_t l, int32_t k, void *cuda_stream, double *F) {
    return fp_exact_brickwork_fkq(n, l, k, 2, cuda_stream, F);
}
