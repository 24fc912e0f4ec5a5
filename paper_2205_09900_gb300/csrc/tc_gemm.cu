// tc_gemm.cu -- BF16 GEMM on the sm_103a tensor cores (tcgen05) with fused
// epilogues: the dense layers (forward and backward) of the control-variate MLP.
//
//   C[M x N] = A[M x K] . Bt[N x K]^T (+ bias),  BF16 operands, FP32 accumulate
//
// One CTA per SM walks 128 x NT output tiles (NT <= 256 columns).  The FP32
// accumulators of two tiles live in tensor memory (TMEM: 2 x NT columns x 128
// lanes), so that the epilogue of one tile runs beside the MMAs of the next.  The
// K loop streams stages of 64 columns through a ring of TC_STAGES shared-memory
// buffers, warp-specialised: one lane issues the TMA loads
// (cp.async.bulk.tensor, completing on the stage's "full" mbarrier), one lane
// waits for them and issues four tcgen05.mma (K = 16 each) and a
// tcgen05.commit to the stage's "empty" mbarrier, which the loader waits on
// before it refills the buffer; the tile's last commit signals its accumulator.
// Eight epilogue warps read it back with tcgen05.ld (warp w reaches TMEM lanes
// 32 (w mod 4) .. + 31, i.e. those tile rows; two warps share them by columns),
// add the bias and apply one of
//   mode 0: identity,
//   mode 1: GELU (the pre-activation optionally kept in Z),
//   mode 2: multiply by GELU'(Z) (Z read: the backward pass of a GELU layer),
// then stores FP32 row-major, BF16 row-major and/or BF16 transposed results.
// Tiles are 128-byte rows (64 BF16 of K) in the 128-byte swizzle, one TMA box
// per operand and stage; rows and columns beyond the matrices are zero-filled
// by the TMA unit.
// Bound: 65536 x 256 x 2400 (80 GFLOP, 348 MB) needs 51 us of HBM; the call takes 101 us (335 with
// one tile per CTA and a device error flag allocated per call; 110 with the epilogue's accesses
// a row per lane).  Leaving out the loads of A or the stores saves 18 us each, those of the weights
// 6: shared memory takes in and gives out 48 KB per 64 columns of K beside the epilogue,
// and 512 tiles are four waves of 152 CTAs, the last one a third full.
// Every wait is bounded: on timeout the kernel raises the error flag, waits (bounded)
// for the loads and MMAs that it has in flight, releases its TMEM, and returns;
// launches that find the flag raised return at once.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdint>
#include <mutex>
#include <vector>

#include "fp.h"
#include "kernels.h"

namespace fpk {
namespace {

constexpr int TC_BM = 128, TC_BK = 64, TC_EPI = 8, TC_THREADS = 64 + 32 * TC_EPI, TC_MAXN = 256, TC_STAGES = 4;
constexpr int TC_STG = 4096;   // bytes of an epilogue warp's staging block
constexpr uint64_t TC_DRAIN_NS = 1000000000ull;   // waits for work already issued (after a timeout)

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor (tcgen05) of a K-major tile stored as
// 128-byte rows with the 128-byte swizzle (16-byte chunk c of row r at chunk
// c ^ (r % 8)), tile base 1024-byte aligned: start address >> 4, leading
// offset unused (1), stride offset 1024 bytes (8 rows) >> 4, version 1,
// layout type 2 (128-byte swizzle) in bits 61-63.  Advancing K by 16 BF16
// elements adds 32 bytes to the start address.
__device__ __forceinline__ uint64_t make_desc_sw128(uint32_t saddr) {
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) |
           (2ull << 61);
}

// instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), BF16 A
// (bits 7-9 = 1) and B (bits 10-12 = 1), both K-major, N >> 3 at bit 17, M >> 4 at bit 24
__device__ __forceinline__ uint32_t make_idesc(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ uint64_t gtimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// Poll an mbarrier phase until it completes or `limit_ns` of global time pass.
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t phase, uint64_t limit_ns) {
    const uint64_t t0 = gtimer();
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(mbar), "r"(phase)
            : "memory");
        if (done) return true;
        if (gtimer() - t0 > limit_ns) return false;
    }
}

__device__ __forceinline__ float gelu_f(float v) { return 0.5f * v * (1.0f + erff(v * 0.70710678f)); }
__device__ __forceinline__ float gelu_grad(float z) {
    return 0.5f * (1.0f + erff(z * 0.70710678f)) + z * 0.39894228f * expf(-0.5f * z * z);
}

// A warp's 32 x 32 block of results (lane = row) to and from global memory through its 4 KB of
// shared memory, whole 128-byte (FP32) or 64-byte (BF16) row pieces per instruction: with a row
// per lane every 8- or 16-byte access is a sector of its own.  Chunk c of row r sits at chunk
// c ^ (r mod 8) (BF16: c ^ (r / 2 mod 4)), so that both directions meet all banks.  rows: valid
// rows from the block's first (may be <= 0), nc: valid columns, 16 or 32.
__device__ __forceinline__ void put_rows(unsigned char *s, int lane, const float (&v)[32], float *dst, int ld, int rows, int nc) {
    float4 *b = (float4 *)s;
#pragma unroll
    for (int c = 0; c < 8; ++c)
        b[8 * lane + (c ^ (lane & 7))] = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
    __syncwarp();
    const int c = lane & 7;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = 4 * i + (lane >> 3);
        if (r < rows && 4 * c < nc) *(float4 *)(dst + (size_t)r * ld + 4 * c) = b[8 * r + (c ^ (r & 7))];
    }
    __syncwarp();
}
__device__ __forceinline__ void get_rows(unsigned char *s, int lane, float (&v)[32], const float *src, int ld, int rows, int nc) {
    float4 *b = (float4 *)s;
    const int c = lane & 7;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = 4 * i + (lane >> 3);
        if (r < rows && 4 * c < nc) b[8 * r + (c ^ (r & 7))] = *(const float4 *)(src + (size_t)r * ld + 4 * c);
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const float4 z = b[8 * lane + (q ^ (lane & 7))];
        v[4 * q] = z.x, v[4 * q + 1] = z.y, v[4 * q + 2] = z.z, v[4 * q + 3] = z.w;
    }
    __syncwarp();
}
__device__ __forceinline__ uint32_t bf16_pair(float a, float b) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
    return *(const uint32_t *)&p;
}
// wide: rows start on 16 bytes (else on 8)
__device__ __forceinline__ void put_rows_bf16(unsigned char *s, int lane, const float (&v)[32], __nv_bfloat16 *dst, int ld,
                                              int rows, int nc, bool wide) {
    uint4 *b = (uint4 *)s;
#pragma unroll
    for (int c = 0; c < 4; ++c)
        b[4 * lane + (c ^ ((lane >> 1) & 3))] = make_uint4(bf16_pair(v[8 * c], v[8 * c + 1]), bf16_pair(v[8 * c + 2], v[8 * c + 3]),
                                                           bf16_pair(v[8 * c + 4], v[8 * c + 5]), bf16_pair(v[8 * c + 6], v[8 * c + 7]));
    __syncwarp();
    const int c = lane & 3;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = 8 * i + (lane >> 2);
        if (r >= rows || 8 * c >= nc) continue;
        const uint4 u = b[4 * r + (c ^ ((r >> 1) & 3))];
        __nv_bfloat16 *d = dst + (size_t)r * ld + 8 * c;
        if (wide) {
            *(uint4 *)d = u;
        } else {
            *(uint2 *)d = make_uint2(u.x, u.y);
            *(uint2 *)(d + 4) = make_uint2(u.z, u.w);
        }
    }
    __syncwarp();
}

__device__ __forceinline__ void mbar_init(uint64_t *m, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(m)), "r"(count));
}

// one TMA box (64 BF16 columns = 128 bytes x box rows, first column x, first
// row y) of a 2-D tensor map into shared memory, completing its bytes on the mbarrier
__device__ __forceinline__ void tma_load(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t mbar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            dst),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(mbar)
        : "memory");
}

// Shared memory per stage: the A tile [128 rows x 128 bytes] then the B tile
// [boxn rows x 128 bytes], both written by the TMA unit with the 128-byte
// swizzle that the MMA descriptors declare; stage bases 1024-byte aligned.
// Warp 0: TMA producer, warp 1: MMA issuer, warps 2..9: epilogue.
__global__ void __launch_bounds__(TC_THREADS, 1) tc_gemm_kernel(TcGemm g, const __grid_constant__ CUtensorMap tmA,
                                                                const __grid_constant__ CUtensorMap tmB, int boxn,
                                                                int tiles_n, int tiles) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full[TC_STAGES], empty[TC_STAGES], tfull[2], tempty[2], done;
    __shared__ uint32_t taddr_sh;
    __shared__ volatile int abort_sh;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // an earlier launch timed out: do nothing (one read, so that the whole CTA agrees)
    if (tid == 0) abort_sh = g.err ? *(volatile const int *)g.err : 0;
    __syncthreads();
    if (abort_sh) return;
    unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t ncols = boxn <= 32 ? 32u : (boxn <= 64 ? 64u : (boxn <= 128 ? 128u : 256u));   // per accumulator
    const uint32_t a_bytes = TC_BM * TC_BK * 2, b_bytes = (uint32_t)boxn * TC_BK * 2;
    const uint32_t stage_bytes = a_bytes + TC_MAXN * TC_BK * 2;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&taddr_sh)),
                     "r"(2 * ncols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 32) {
        for (int s = 0; s < TC_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(&tfull[s], 1);
            mbar_init(&tempty[s], TC_EPI);
        }
        mbar_init(&done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
        asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmA) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmB) : "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t taddr = taddr_sh;
    const int nk = (g.K + TC_BK - 1) / TC_BK;
    const uint32_t sbase = smem_u32(smem);
    int it = 0;   // producer, issuer: stages whose loads, MMAs were issued
    if (tid == 0) {
        // producer: TMA loads of a stage once the MMAs TC_STAGES stages earlier have drained the buffer
        for (int t = blockIdx.x; t < tiles && !abort_sh; t += gridDim.x) {
            const int m0 = t / tiles_n * TC_BM, n0 = t % tiles_n * TC_MAXN;
            for (int kt = 0; kt < nk; ++kt, ++it) {
                const int s = it % TC_STAGES, u = it / TC_STAGES;
                if (abort_sh || (u > 0 && !mbar_wait(smem_u32(&empty[s]), (uint32_t)(u - 1) & 1u, g.wait_ns))) {
                    abort_sh = 1;
                    break;
                }
                const uint32_t fb = smem_u32(&full[s]);
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "r"(a_bytes + b_bytes)
                             : "memory");
                const uint32_t sa = sbase + s * stage_bytes, sb = sa + a_bytes;
                tma_load(sa, &tmA, kt * TC_BK, m0, fb);
                tma_load(sb, &tmB, kt * TC_BK, n0, fb);
            }
        }
    } else if (tid == 32) {
        // MMA issuer: four K = 16 steps per stage, then release the buffer
        int i = 0;   // tiles so far
        for (int t = blockIdx.x; t < tiles && !abort_sh; t += gridDim.x, ++i) {
            const int acc = i & 1, n0 = t % tiles_n * TC_MAXN;
            const uint32_t idesc = make_idesc(TC_BM, min(TC_MAXN, g.N - n0)), td = taddr + (uint32_t)acc * ncols;
            // the accumulator's previous tile has been read
            if (i >= 2 && !mbar_wait(smem_u32(&tempty[acc]), (uint32_t)(i / 2 - 1) & 1u, g.wait_ns)) {
                abort_sh = 1;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
            for (int kt = 0; kt < nk; ++kt, ++it) {
                const int s = it % TC_STAGES, u = it / TC_STAGES;
                if (abort_sh || !mbar_wait(smem_u32(&full[s]), (uint32_t)u & 1u, g.wait_ns)) {
                    abort_sh = 1;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;");
                const uint32_t sa = sbase + s * stage_bytes, sb = sa + a_bytes;
#pragma unroll
                for (int kk = 0; kk < TC_BK / 16; ++kk) {
                    const uint64_t ad = make_desc_sw128(sa + kk * 32);
                    const uint64_t bd = make_desc_sw128(sb + kk * 32);
                    const uint32_t accum = (kt > 0 || kk > 0) ? 1u : 0u;
                    asm volatile(
                        "{\n\t.reg .pred p;\n\t"
                        "setp.ne.u32 p, %4, 0;\n\t"
                        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(td),
                        "l"(ad), "l"(bd), "r"(idesc), "r"(accum));
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 smem_u32(&empty[s]))
                             : "memory");
            }
            if (abort_sh) break;
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_u32(&tfull[acc]))
                         : "memory");
        }
    } else if (warp >= 2) {
        const int quarter = warp & 3, half = (warp - 2) >> 2;
        unsigned char *stg = smem + TC_STAGES * stage_bytes + (warp - 2) * TC_STG;
        const bool wide = g.ldcb % 8 == 0 && ((uintptr_t)g.Cb & 15) == 0;
        int i = 0;
        for (int t = blockIdx.x; t < tiles; t += gridDim.x, ++i) {
            const int acc = i & 1, m0 = t / tiles_n * TC_BM, n0 = t % tiles_n * TC_MAXN;
            const int NT = min(TC_MAXN, g.N - n0);   // a multiple of 16
            const bool ok = !abort_sh && mbar_wait(smem_u32(&tfull[acc]), (uint32_t)(i / 2) & 1u, g.wait_ns);
            if (!__all_sync(0xffffffffu, ok)) {   // warp-uniform: the TMEM loads below are warp-collective
                abort_sh = 1;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
            const int row = m0 + quarter * 32 + lane;
            const bool rv = row < g.M;
            for (int c0 = 32 * half; c0 < NT; c0 += 64) {
                uint32_t r[32];
                const uint32_t ta = taddr + ((uint32_t)(quarter * 32) << 16) + (uint32_t)acc * ncols + (uint32_t)c0;
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
                    "%14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                    : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                      "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                      "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
                      "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
                      "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                    : "r"(ta));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                float v[32];
#pragma unroll
                for (int e = 0; e < 32; ++e) v[e] = __uint_as_float(r[e]);
                const int nc = min(32, NT - c0);   // 32 or 16 columns
                if (g.bias) {
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        if (4 * q >= nc) break;
                        const float4 b = *(const float4 *)(g.bias + n0 + c0 + 4 * q);
                        v[4 * q] += b.x, v[4 * q + 1] += b.y, v[4 * q + 2] += b.z, v[4 * q + 3] += b.w;
                    }
                }
                const int r0 = m0 + quarter * 32;
                if (g.mode == 1) {
                    if (g.Z) put_rows(stg, lane, v, g.Z + (size_t)r0 * g.ldz + n0 + c0, g.ldz, g.M - r0, nc);
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] = gelu_f(v[e]);
                } else if (g.mode == 2) {
                    float z[32];
                    get_rows(stg, lane, z, g.Z + (size_t)r0 * g.ldz + n0 + c0, g.ldz, g.M - r0, nc);
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] *= gelu_grad(z[e]);
                }
                if (g.Cf) put_rows(stg, lane, v, g.Cf + (size_t)r0 * g.ldcf + n0 + c0, g.ldcf, g.M - r0, nc);
                if (g.Cb) put_rows_bf16(stg, lane, v, g.Cb + (size_t)r0 * g.ldcb + n0 + c0, g.ldcb, g.M - r0, nc, wide);
                if (g.Cbt && rv) {
#pragma unroll
                    for (int e = 0; e < 32; ++e)
                        if (e < nc) g.Cbt[(size_t)(n0 + c0 + e) * g.ldct + row] = __float2bfloat16(v[e]);
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tempty[acc])) : "memory");
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    // No role runs any more, so every thread reads the same abort_sh here.  Whichever role gave up,
    // the others may have issued all they had to before they could see it (the epilogue waits for
    // a whole tile, the issuer for a stage at a time), so the drain comes after the barrier: the
    // loads of the last phase of each stage buffer, and one more commit, which covers every MMA,
    // so that nothing is in flight when the tensor memory is released and the CTA ends.
    if (abort_sh) {
        if (tid == 0) {
            for (int i = (it > TC_STAGES ? it - TC_STAGES : 0); i < it; ++i)
                mbar_wait(smem_u32(&full[i % TC_STAGES]), (uint32_t)(i / TC_STAGES) & 1u, TC_DRAIN_NS);
            if (g.err) atomicExch_system(g.err, 1);
        } else if (tid == 32 && it > 0) {
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_u32(&done))
                         : "memory");
            mbar_wait(smem_u32(&done), 0u, TC_DRAIN_NS);
        }
        __syncwarp();
        __syncthreads();
    }
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(2 * ncols));
    }
}

bool aligned(const void *p, uintptr_t a) { return ((uintptr_t)p & (a - 1)) == 0; }

}  // namespace

size_t tc_gemm_smem_bytes() { return (size_t)TC_STAGES * (TC_BM + TC_MAXN) * TC_BK * 2 + TC_EPI * TC_STG + 1024; }

const char *tc_gemm_check(const TcGemm &g) {
    if (g.M < 0 || g.N <= 0 || g.N % 16 != 0 || g.K <= 0 || g.K % 8 != 0) return "need N % 16 == 0 and K % 8 == 0";
    if (g.M == 0) return nullptr;   // nothing is read or written
    if (!g.A || !g.Bt || g.lda < g.K || g.ldb < g.K || g.lda % 8 || g.ldb % 8 || !aligned(g.A, 16) ||
        !aligned(g.Bt, 16))
        return "A and Bt need 16-byte alignment and leading dimensions >= K that are multiples of 8";
    if (!g.Cf && !g.Cb && !g.Cbt) return "no output";
    if (g.mode < 0 || g.mode > 2 || (g.mode == 2 && !g.Z)) return "mode must be 0, 1 or 2 (mode 2 needs Z)";
    if (g.Z && (g.ldz < g.N || g.ldz % 4 || !aligned(g.Z, 16)))
        return "Z needs a leading dimension >= N that is a multiple of 4, and 16-byte alignment";
    if (g.bias && !aligned(g.bias, 16)) return "bias needs 16-byte alignment";
    if (g.Cf && (g.ldcf < g.N || g.ldcf % 4 || !aligned(g.Cf, 16)))
        return "C needs a leading dimension >= N that is a multiple of 4, and 16-byte alignment";
    if (g.Cb && (g.ldcb < g.N || g.ldcb % 4 || !aligned(g.Cb, 8)))
        return "C_bf16 needs a leading dimension >= N that is a multiple of 4, and 8-byte alignment";
    if (g.Cbt && (g.ldct < g.M || !aligned(g.Cbt, 2))) return "Ct_bf16 needs a leading dimension >= M";
    return nullptr;
}

namespace {

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static std::once_flag once;
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    });
    return fn;
}

// tensor map of a row-major [rows x ld] BF16 matrix whose first `cols`
// columns are valid; boxes of 64 columns (128 bytes) x box_rows rows, 128-byte swizzle
bool make_map(CUtensorMap *m, const void *base, int rows, int cols, int ld, int box_rows) {
    auto fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {(cuuint32_t)TC_BK, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1u, 1u};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

cudaError_t launch_tc_gemm(const TcGemm &g, cudaStream_t st) {
    if (g.M == 0) return cudaSuccess;
    if (tc_gemm_check(g)) return cudaErrorInvalidValue;
    const int boxn = g.N < TC_MAXN ? g.N : TC_MAXN;
    CUtensorMap ma, mb;
    if (!make_map(&ma, g.A, g.M, g.K, g.lda, TC_BM) || !make_map(&mb, g.Bt, g.N, g.K, g.ldb, boxn))
        return cudaErrorInvalidValue;
    const size_t smem = tc_gemm_smem_bytes();
    // the attribute is set outside stream capture (a launch being captured
    // follows a direct launch on the same device, which has set it)
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(st, &cs);
    if (e != cudaSuccess) return e;
    if (cs == cudaStreamCaptureStatusNone) {
        e = cudaFuncSetAttribute(tc_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const int tiles_n = (g.N + TC_MAXN - 1) / TC_MAXN, tiles = (g.M + TC_BM - 1) / TC_BM * tiles_n;
    TcGemm gk = g;
    gk.wait_ns = wait_limit_ns();
    tc_gemm_kernel<<<std::min(tiles, sms), TC_THREADS, smem, st>>>(gk, ma, mb, boxn, tiles_n, tiles);
    return cudaGetLastError();
}

}  // namespace fpk

namespace fpk {
namespace {

// An error flag of one call in pinned host memory that the kernel reaches through its
// mapped address: nothing to clear, copy or allocate per call (an int from
// cudaMallocAsync, cleared, copied back and freed, took 180 us of a 326 us call).  Flags
// come from a free list that grows to the largest number of calls in flight at once
// (each call waits for its kernel, so a returned flag is idle), at most kMaxFlags; the
// list is portable over devices and threads.
struct ErrorFlag {
    static constexpr size_t kMaxFlags = 256;
    volatile int *host = nullptr;
    int *device = nullptr;
    bool lost = false;   // lost: a kernel may still write it

    static std::mutex &mu() { static std::mutex m; return m; }
    static std::vector<int *> &pool() { static std::vector<int *> *v = new std::vector<int *>(); return *v; }

    ErrorFlag() {
        int *p = nullptr;
        {
            std::lock_guard<std::mutex> lk(mu());
            if (!pool().empty()) {
                p = pool().back();
                pool().pop_back();
            }
        }
        if (!p && cudaHostAlloc((void **)&p, sizeof(int), cudaHostAllocMapped | cudaHostAllocPortable) != cudaSuccess) {
            cudaGetLastError();
            return;
        }
        void *d = nullptr;
        if (cudaHostGetDevicePointer(&d, p, 0) != cudaSuccess) {
            cudaGetLastError();
            cudaFreeHost(p);
            return;
        }
        *p = 0;
        host = p;
        device = (int *)d;
    }
    ~ErrorFlag() {
        if (!host || lost) return;
        int *p = const_cast<int *>(host);
        {
            std::lock_guard<std::mutex> lk(mu());
            if (pool().size() < kMaxFlags) {
                try {
                    pool().push_back(p);
                    p = nullptr;
                } catch (...) {
                }
            }
        }
        if (p) cudaFreeHost(p);
    }
    ErrorFlag(const ErrorFlag &) = delete;
    ErrorFlag &operator=(const ErrorFlag &) = delete;
};

}  // namespace
}  // namespace fpk

extern "C" fp_status fp_gemm_bf16(int32_t M, int32_t N, int32_t K, const void *A, int32_t lda, const void *Bt,
                                  int32_t ldb, const float *bias, int32_t mode, float *Z, float *C, void *C_bf16,
                                  void *Ct_bf16, void *cuda_stream) {
    fpk::TcGemm g{};
    g.M = M, g.N = N, g.K = K;
    g.A = (const __nv_bfloat16 *)A, g.lda = lda;
    g.Bt = (const __nv_bfloat16 *)Bt, g.ldb = ldb;
    g.bias = bias, g.mode = mode;
    g.Z = Z, g.ldz = N;
    g.Cf = C, g.ldcf = N;
    g.Cb = (__nv_bfloat16 *)C_bf16, g.ldcb = N;
    g.Cbt = (__nv_bfloat16 *)Ct_bf16, g.ldct = M;
    if (const char *why = fpk::tc_gemm_check(g)) return fpk::api_fail(FP_ERR_ARG, why);
    if (M == 0) return FP_OK;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    fpk::ErrorFlag flag;
    if (!flag.host) return fpk::api_fail(FP_ERR_OOM, "no pinned memory for the error flag");
    g.err = flag.device;
    cudaError_t e = fpk::launch_tc_gemm(g, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        flag.lost = true;
        return fpk::api_fail(FP_ERR_CUDA, cudaGetErrorString(e));
    }
    if (*flag.host) return fpk::api_fail(FP_ERR_TIMEOUT, "tcgen05 GEMM: an mbarrier wait ran out");
    return FP_OK;
}
