// Tensor-core GEMM for sm_103a: C[M][N] = A[M][K] . B[N][K]^T, BF16 inputs
// (both K-major), FP32 accumulation in tensor memory (TMEM), fused epilogues.
// tc_gemm_split_kernel (end of the file) multiplies FP32-accurate operands
// given as three BF16 copies, with the same stage rows of 128 bytes (64
// 16-bit elements), swizzle and descriptors.
// Two kernels share the pipeline below, both persistent over many tiles:
// tc_gemm_pair_kernel (256 x 256 tiles on CTA pairs) and tc_gemm_persist_kernel
// (128 x 256 tiles, one CTA each; surrogate.cu's use_pairs says when).
//
//   TMA producer:   cp.async.bulk.tensor loads tiles of A and B, 64 values of K
//                   wide (128-byte swizzle), into a ring of stages; each stage
//                   has a `full` mbarrier (transaction bytes) and an `empty`
//                   mbarrier (arrived by tcgen05.commit when the MMAs that
//                   read the stage are done).
//   MMA issuer:     four tcgen05.mma.kind::f16 (K = 16 each) per stage into one
//                   of two FP32 accumulators in TMEM.
//   epilogue warps: tcgen05.ld 32x32b of the other accumulator: warp w reads
//                   TMEM lanes 32 (w % 4) .. + 31 (= output rows).
// Every mbarrier wait has an iteration limit; a wait that runs out sets the
// error word, the CTA still frees its TMEM and returns.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace slos {
namespace tc {

constexpr int BM = 128, BN = 256, BK = 64, STAGES = 4;
constexpr int A_TILE = BM * BK * 2;  // bytes
constexpr int B_TILE = BN * BK * 2;
constexpr int STAGE_BYTES = A_TILE + B_TILE;
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 /*align*/ + 256 /*barriers*/;
constexpr long long kWaitLimit = 1ll << 22;  // tries; a few seconds at most

enum TcEpi : int {
    TC_F32 = 0,        // C = acc                         (float)
    TC_F32_BIAS = 1,   // C = acc + bias[n]               (float)
    TC_GELU = 2,       // Z = acc + bias[n] (bf16, aux), C = gelu(Z) (bf16)
    TC_GELU_BWD = 3,   // C = acc * gelu'(Z), Z = aux (bf16 in), C bf16
    TC_F32_ACCUM = 4,  // C += acc                        (float)
};

struct TcArgs {
    int M, N, K;
    void *C;              // [M][ldc]
    int ldc;
    const float *bias;    // [N]
    __nv_bfloat16 *aux;   // [M][ldc] (Z for TC_GELU out, TC_GELU_BWD in)
    int *err;             // error word (device)
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Bounded wait: true if the phase completed, false if the limit ran out.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity) {
    for (long long i = 0; i < kWaitLimit; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(
            smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y)
        : "memory");
}

// Shared-memory matrix descriptor, K-major operand with 128-byte swizzle:
// start address >> 4 (bits 0-13), leading byte offset 16 B (unused for this
// layout, bits 16-29), stride byte offset 1024 B between 8-row groups
// (bits 32-45), fixed 0b001 (bits 46-48), swizzle mode 2 = 128 B (bits 61-63).
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// Instruction descriptor, kind::f16: FP32 accumulator (bits 4-5 = 1), A and B
// BF16 (bits 7-9 = 1, 10-12 = 1), both K-major, N >> 3 (bits 17-22),
// M >> 4 (bits 24-28).
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(kIdesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// GELU, tanh form, and its derivative (the surrogate's activation).
__device__ __forceinline__ float gelu_f(float z) {
    const float c = 0.7978845608028654f;  // sqrt(2/pi)
    const float u = c * (z + 0.044715f * z * z * z);
    return 0.5f * z * (1.f + tanhf(u));
}
__device__ __forceinline__ float gelu_grad(float z) {
    const float c = 0.7978845608028654f;
    const float u = c * (z + 0.044715f * z * z * z);
    const float t = tanhf(u);
    return 0.5f * (1.f + t) + 0.5f * z * (1.f - t * t) * c * (1.f + 3.f * 0.044715f * z * z);
}

// Epilogue of one 16-column segment of an output row: v holds the
// accumulator values of row `row`, columns col0 .. col0 + 15.
template <int EPI>
__device__ __forceinline__ void tc_store16(const TcArgs &g, int row, int col0, float (&v)[16], bool vec) {
    if (row < g.M && col0 < g.N) {
        const int64_t o0 = (int64_t)row * g.ldc + col0;
        if (EPI == TC_F32_BIAS || EPI == TC_GELU) {
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] += (col0 + i < g.N) ? g.bias[col0 + i] : 0.f;
        }
        if (vec && col0 + 16 <= g.N) {
            if (EPI == TC_F32 || EPI == TC_F32_BIAS || EPI == TC_F32_ACCUM) {
                float4 *dst = reinterpret_cast<float4 *>(reinterpret_cast<float *>(g.C) + o0);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float4 w = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                    if (EPI == TC_F32_ACCUM) {
                        const float4 old = dst[q];
                        w.x += old.x;
                        w.y += old.y;
                        w.z += old.z;
                        w.w += old.w;
                    }
                    dst[q] = w;
                }
            } else {
                __align__(16) __nv_bfloat16 out[16];
                if (EPI == TC_GELU) {
                    __align__(16) __nv_bfloat16 zb[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        zb[i] = __float2bfloat16(v[i]);
                        out[i] = __float2bfloat16(gelu_f(__bfloat162float(zb[i])));
                    }
                    uint4 *za = reinterpret_cast<uint4 *>(g.aux + o0);
                    za[0] = reinterpret_cast<const uint4 *>(zb)[0];
                    za[1] = reinterpret_cast<const uint4 *>(zb)[1];
                } else {  // TC_GELU_BWD
                    __align__(16) __nv_bfloat16 zb[16];
                    const uint4 *zs = reinterpret_cast<const uint4 *>(g.aux + o0);
                    reinterpret_cast<uint4 *>(zb)[0] = zs[0];
                    reinterpret_cast<uint4 *>(zb)[1] = zs[1];
#pragma unroll
                    for (int i = 0; i < 16; ++i) out[i] = __float2bfloat16(v[i] * gelu_grad(__bfloat162float(zb[i])));
                }
                uint4 *dst = reinterpret_cast<uint4 *>(reinterpret_cast<__nv_bfloat16 *>(g.C) + o0);
                dst[0] = reinterpret_cast<const uint4 *>(out)[0];
                dst[1] = reinterpret_cast<const uint4 *>(out)[1];
            }
        } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const int col = col0 + i;
                if (col >= g.N) break;
                const int64_t o = o0 + i;
                const float x = v[i];
                if (EPI == TC_F32 || EPI == TC_F32_BIAS) {
                    reinterpret_cast<float *>(g.C)[o] = x;
                } else if (EPI == TC_F32_ACCUM) {
                    reinterpret_cast<float *>(g.C)[o] += x;
                } else if (EPI == TC_GELU) {
                    const __nv_bfloat16 zb = __float2bfloat16(x);
                    g.aux[o] = zb;
                    reinterpret_cast<__nv_bfloat16 *>(g.C)[o] = __float2bfloat16(gelu_f(__bfloat162float(zb)));
                } else {  // TC_GELU_BWD
                    const float z = __bfloat162float(g.aux[o]);
                    reinterpret_cast<__nv_bfloat16 *>(g.C)[o] = __float2bfloat16(x * gelu_grad(z));
                }
            }
        }
    }
}

// Persistent variant: one CTA per SM walks the output tiles t = blockIdx.x,
// blockIdx.x + gridDim.x, ... (row-major over 128 x 256 tiles, so the CTAs
// running together share A rows in L2).  Six warps:
//   warp 0, lane 0: TMA producer over one stage ring that runs on across tiles;
//   warp 1, lane 0: MMA issuer, alternating between two 128 x 256 FP32
//                   accumulators in TMEM (all 512 columns): tile j uses
//                   accumulator j & 1, after the epilogue has released it
//                   (`tempty`, one arrival per epilogue warp), and commits
//                   `tfull` when its last MMA has completed;
//   warps 2-5:      epilogue; warp w reads TMEM lanes 32 (w % 4) .. + 31, the
//                   quarter its position in the warpgroup gives access to.
// So a tile's epilogue runs while the next tile's loads and MMAs proceed, and
// the ring's fill is paid once per CTA.  Waits are bounded as above; a wait
// that runs out sets the error word and the abort flag, and every role leaves
// its loop.
constexpr int kPersistThreads = 192;
constexpr uint32_t kPersistTmemCols = 2 * BN;

template <int EPI>
__global__ void __launch_bounds__(kPersistThreads, 1)
    tc_gemm_persist_kernel(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb, TcArgs g) {
    extern __shared__ uint8_t smem_tc[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_tc) + 1023) & ~uintptr_t(1023));
    uint8_t *sA = base;
    uint8_t *sB = base + STAGES * A_TILE;
    uint64_t *full = reinterpret_cast<uint64_t *>(sB + STAGES * B_TILE);
    uint64_t *empty = full + STAGES;
    uint64_t *tfull = empty + STAGES;  // [2]
    uint64_t *tempty = tfull + 2;      // [2]
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(tempty + 2);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nk = (g.K + BK - 1) / BK;
    const int ntn = (g.N + BN - 1) / BN;
    const int ntiles = ((g.M + BM - 1) / BM) * ntn;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full + s, 1);
            mbar_init(empty + s, 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(tfull + a, 1);
            mbar_init(tempty + a, 4);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kPersistTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            // producer
            uint32_t it = 0;
            for (int t = blockIdx.x; t < ntiles && !*abort_flag; t += gridDim.x) {
                const int m0 = (t / ntn) * BM, n0 = (t % ntn) * BN;
                for (int kt = 0; kt < nk; ++kt, ++it) {
                    const int s = it % STAGES;
                    const uint32_t ph = (it / STAGES) & 1;
                    if (it >= STAGES && !mbar_wait(empty + s, ph ^ 1)) {
                        atomicExch(g.err, 1);
                        *abort_flag = 1;
                        break;
                    }
                    if (*abort_flag) break;
                    mbar_expect_tx(full + s, STAGE_BYTES);
                    tma_load_2d(sA + s * A_TILE, &ta, kt * BK, m0, full + s);
                    tma_load_2d(sB + s * B_TILE, &tb, kt * BK, n0, full + s);
                }
            }
            // never leave with copies in flight: wait (bounded) for the last loads
            for (uint32_t q = (it > (uint32_t)STAGES ? it - STAGES : 0); q < it; ++q)
                mbar_wait(full + (q % STAGES), (q / STAGES) & 1);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // MMA issuer
            uint32_t it = 0;
            int j = 0;
            for (int t = blockIdx.x; t < ntiles && !*abort_flag; t += gridDim.x, ++j) {
                const int acc = j & 1;
                const int use = j >> 1;  // this accumulator's use count
                if (use > 0 && !mbar_wait(tempty + acc, (use - 1) & 1)) {
                    atomicExch(g.err, 4);
                    *abort_flag = 1;
                    break;
                }
                tc_fence_after();
                const uint32_t d = tmem + (uint32_t)(acc * BN);
                for (int kt = 0; kt < nk; ++kt, ++it) {
                    const int s = it % STAGES;
                    const uint32_t ph = (it / STAGES) & 1;
                    if (*abort_flag || !mbar_wait(full + s, ph)) {
                        atomicExch(g.err, 2);
                        *abort_flag = 1;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t a0 = smem_u32(sA + s * A_TILE), b0 = smem_u32(sB + s * B_TILE);
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk)
                        mma_bf16(d, sw128_desc(a0 + kk * 32), sw128_desc(b0 + kk * 32), (kt > 0 || kk > 0) ? 1u : 0u);
                    mma_commit(empty + s);
                }
                if (*abort_flag) break;
                mma_commit(tfull + acc);  // arrives once this tile's MMAs have completed
            }
        }
    } else {
        // epilogue warps
        const int q = warp & 3;
        // 16-byte stores where every row of C starts on a 16-byte boundary (its epilogues touch only C)
        const bool vec = (g.ldc % 8) == 0 && (reinterpret_cast<uintptr_t>(g.C) & 15) == 0;
        int j = 0;
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++j) {
            const int acc = j & 1;
            const bool ok = __all_sync(0xffffffffu, !*abort_flag && mbar_wait(tfull + acc, (j >> 1) & 1));
            if (!ok) {
                if (lane == 0) {
                    atomicExch(g.err, 3);
                    *abort_flag = 1;
                }
                break;
            }
            tc_fence_after();
            const int m0 = (t / ntn) * BM, n0 = (t % ntn) * BN;
            const int row = m0 + q * 32 + lane;
            const uint32_t src = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN);
#pragma unroll 1
            for (int c = 0; c < BN; c += 16) {
                float v[16];
                tmem_ld16(src + (uint32_t)c, v);
                tc_store16<EPI>(g, row, n0 + c, v, vec);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(tempty + acc);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kPersistTmemCols)
                     : "memory");
    }
}

// ---------------------------------------------------------------- CTA pairs
// tc_gemm_pair_kernel: the persistent pipeline on CTA pairs (cta_group::2).
// A pair shares a 256 x 256 tile: each CTA stages its 128 rows of A and half of
// the 256 rows of B, the pair's MMA reads both halves of B, and each CTA holds
// its 128 rows of the accumulator: 32 KB per CTA and 64 of K, where a 128 x 256
// tile of one CTA takes 48 KB.  What bounds it is the MMAs: 0.36 us per 64 of K (1760 TFLOP/s over 76
// pairs), 0.38 with the loads; four stages instead of six cost 4 %.  A
// thread reads a row of outputs from TMEM; written as it stands that is 16 bytes
// to each of 32 rows an instruction, so the epilogue warps turn their outputs in
// shared memory first (eight warps: four fell behind the MMAs, sixteen were no
// faster).  Measured, us for this kernel / one CTA a tile:
// 16384 x 12376 x 2048 with bias 545 / 632 (1525 TFLOP/s), 12800 x 8000 x 768
// with bias 131 / 242, 16384 x 2048 x 2048 with GELU 116 / 123 and K = 288 60 / 86
// (GELU's arithmetic keeps the epilogue behind the MMAs), 8192^3 684 / 741.
//
// Roles as in tc_gemm_persist_kernel, with these differences: the even CTA
// (rank 0) issues the MMAs of both and owns the `full` barriers, on which the
// loads of both CTAs complete, and the `tempty` ones, on which the epilogue
// warps of both arrive; the MMAs' commits arrive on the `empty` and `tfull`
// barriers of both.  A CTA leaves only after the other has passed its last
// barrier, so no arrival or operand read meets a CTA that is gone.
constexpr int kPairEpiWarps = 8;
constexpr int kPairThreads = 64 + 32 * kPairEpiWarps;
constexpr int kPairStages = 6;
constexpr int kPairStageBytes = 2 * BM * BK * 2;  // per CTA: 128 rows of A, 128 rows of B
constexpr int kPairBox = 32 * 128;                // an epilogue warp's transposition buffer: 32 rows of 128 bytes
constexpr int kPairSmem = kPairStages * kPairStageBytes + kPairEpiWarps * kPairBox + 1024 + 256;
constexpr uint32_t kIdescPair =
    (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(2 * BM >> 4) << 24);

// Address of this CTA's shared variable in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(const void *p, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Bounded wait on a barrier that threads of both CTAs arrive on.
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t *bar, uint32_t parity) {
    for (long long i = 0; i < kWaitLimit; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}
// Load into this CTA's shared memory that completes on a barrier of either CTA of the pair.
__device__ __forceinline__ void tma_load_pair(void *dst, const CUtensorMap *map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], "
        "[%2];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y)
        : "memory");
}
__device__ __forceinline__ void mma_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(kIdescPair), "r"(accumulate)
        : "memory");
}
// Arrival on this barrier of both CTAs once the MMAs issued so far have completed.
__device__ __forceinline__ void mma_commit_pair(uint64_t *bar) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            smem_u32(bar)),
        "h"((uint16_t)3)
        : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&h);
}
__device__ __forceinline__ float2 unpack_bf16(uint32_t x) {
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&x));
}

// What the epilogue of 32 rows x 32 columns reads: Z (four lanes a row) or C
// before the sum (eight lanes a row).  Read a block ahead, the first before
// the wait for the sums, so that its latency is nobody's (us, read where it is
// used / now: accumulating 8192 x 8192 x 2048 330 / 211, 4096 x 12376 x 512 238 / 123;
// GELU' 4096 x 12376 x 512 175 / 116, 4096 x 2048 x 2048 43 / 41; over many
// tiles of a long K GELU' is bound by its arithmetic, 243 at 8192 x 8192 x 2048).
template <int EPI>
constexpr int kPairAhead = EPI == TC_F32_ACCUM ? 8 : (EPI == TC_GELU_BWD ? 4 : 0);
template <int EPI>
__device__ __forceinline__ void pair_load32(const TcArgs &g, int row0, int col0, int lane,
                                            uint4 (&in)[kPairAhead<EPI> + 1]) {
    constexpr int N = kPairAhead<EPI>;  // 16-byte pieces of a row's 32 values, and lanes a row
    if constexpr (N > 0) {
        const size_t bytes = EPI == TC_GELU_BWD ? 2 : 4;
        const char *src = reinterpret_cast<const char *>(EPI == TC_GELU_BWD ? (const void *)g.aux : g.C);
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int r = 32 / N * i + lane / N;
            if (row0 + r < g.M)
                in[i] = *(reinterpret_cast<const uint4 *>(src + ((int64_t)(row0 + r) * g.ldc + col0) * bytes) +
                          lane % N);
        }
    }
}

// Epilogue of 32 rows x 32 columns by a warp, columns col0 .. col0 + 31 all
// inside the matrix, rows and bias 16-byte aligned: v holds row row0 + lane.
// The block is turned in `box` (32 rows of eight 16-byte slots, slot q of row r
// at q ^ (r & 7), free of bank conflicts both ways), so that eight lanes
// write a row's 128 bytes (64 of C and 64 of Z for the bf16 outputs); a thread
// writing its own row sends 16 bytes to each of 32 rows an instruction.
template <int EPI>
__device__ __forceinline__ void pair_store32(const TcArgs &g, int row0, int col0, int lane, float (&v)[32],
                                             const uint4 (&in)[kPairAhead<EPI> + 1], uint4 *box) {
    constexpr bool kBf16 = EPI == TC_GELU || EPI == TC_GELU_BWD;
    if (EPI == TC_F32_BIAS || EPI == TC_GELU) {
        const float4 *b = reinterpret_cast<const float4 *>(g.bias + col0);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float4 x = __ldg(b + i);
            v[4 * i] += x.x;
            v[4 * i + 1] += x.y;
            v[4 * i + 2] += x.z;
            v[4 * i + 3] += x.w;
        }
    }
    const int sw = lane & 7;
    uint4 *mine = box + lane * 8;
    if (EPI == TC_GELU_BWD) {
        // Z of the block: four lanes a row
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = 8 * i + (lane >> 2), q = lane & 3;
            if (row0 + r < g.M) box[r * 8 + (q ^ (r & 7))] = in[i];
        }
        __syncwarp();
    }
    if (!kBf16) {
#pragma unroll
        for (int q = 0; q < 8; ++q)
            mine[q ^ sw] = make_uint4(__float_as_uint(v[4 * q]), __float_as_uint(v[4 * q + 1]),
                                      __float_as_uint(v[4 * q + 2]), __float_as_uint(v[4 * q + 3]));
    } else {
        // slots 0-3: Z, 4-7: C
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t z[4], c[4];
            if (EPI == TC_GELU_BWD) {
                const uint4 zz = mine[q ^ sw];
                z[0] = zz.x;
                z[1] = zz.y;
                z[2] = zz.z;
                z[3] = zz.w;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float a = v[8 * q + 2 * i], b = v[8 * q + 2 * i + 1];
                if (EPI == TC_GELU) z[i] = pack_bf16(a, b);
                const float2 zf = unpack_bf16(z[i]);
                c[i] = EPI == TC_GELU ? pack_bf16(gelu_f(zf.x), gelu_f(zf.y))
                                      : pack_bf16(a * gelu_grad(zf.x), b * gelu_grad(zf.y));
            }
            if (EPI == TC_GELU) mine[q ^ sw] = make_uint4(z[0], z[1], z[2], z[3]);
            mine[(q + 4) ^ sw] = make_uint4(c[0], c[1], c[2], c[3]);
        }
    }
    __syncwarp();
    const int q = lane & 7;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = 4 * i + (lane >> 3);
        if (row0 + r >= g.M) break;
        const int64_t o = (int64_t)(row0 + r) * g.ldc + col0;
        uint4 x = box[r * 8 + (q ^ (r & 7))];
        if (!kBf16) {
            uint4 *dst = reinterpret_cast<uint4 *>(reinterpret_cast<float *>(g.C) + o) + q;
            if (EPI == TC_F32_ACCUM) {
                x.x = __float_as_uint(__uint_as_float(x.x) + __uint_as_float(in[i].x));
                x.y = __float_as_uint(__uint_as_float(x.y) + __uint_as_float(in[i].y));
                x.z = __float_as_uint(__uint_as_float(x.z) + __uint_as_float(in[i].z));
                x.w = __float_as_uint(__uint_as_float(x.w) + __uint_as_float(in[i].w));
            }
            *dst = x;
        } else if (q >= 4) {
            *(reinterpret_cast<uint4 *>(reinterpret_cast<__nv_bfloat16 *>(g.C) + o) + (q - 4)) = x;
        } else if (EPI == TC_GELU) {
            *(reinterpret_cast<uint4 *>(g.aux + o) + q) = x;
        }
    }
    __syncwarp();
}

template <int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
    tc_gemm_pair_kernel(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb, TcArgs g) {
    extern __shared__ uint8_t smem_tc[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_tc) + 1023) & ~uintptr_t(1023));
    uint8_t *boxes = base + kPairStages * kPairStageBytes;
    uint64_t *full = reinterpret_cast<uint64_t *>(boxes + kPairEpiWarps * kPairBox);
    uint64_t *empty = full + kPairStages;
    uint64_t *tfull = empty + kPairStages;  // [2]
    uint64_t *tempty = tfull + 2;           // [2]
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(tempty + 2);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = blockIdx.x & 1, pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
    const int nk = (g.K + BK - 1) / BK;
    const int ntn = (g.N + BN - 1) / BN;
    const int ntiles = ((g.M + 2 * BM - 1) / (2 * BM)) * ntn;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kPairStages; ++s) {
            mbar_init(full + s, 1);
            mbar_init(empty + s, 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(tfull + a, 1);
            mbar_init(tempty + a, 2 * kPairEpiWarps);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kPersistTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // both CTAs' barriers are initialised and their tensor memory is allocated
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            // producer
            uint32_t it = 0;
            for (int t = pair; t < ntiles && !*abort_flag; t += npairs) {
                const int m0 = (t / ntn) * 2 * BM + rank * BM, n0 = (t % ntn) * BN + rank * (BN / 2);
                for (int kt = 0; kt < nk; ++kt, ++it) {
                    const int s = it % kPairStages;
                    const uint32_t ph = (it / kPairStages) & 1;
                    if (it >= (uint32_t)kPairStages && !mbar_wait(empty + s, ph ^ 1)) {
                        atomicExch(g.err, 1);
                        *abort_flag = 1;
                        break;
                    }
                    if (*abort_flag) break;
                    if (rank == 0) mbar_expect_tx(full + s, 2 * kPairStageBytes);
                    const uint32_t bar = cluster_addr(full + s, 0);
                    uint8_t *st = base + s * kPairStageBytes;
                    tma_load_pair(st, &ta, kt * BK, m0, bar);
                    tma_load_pair(st + A_TILE, &tb, kt * BK, n0, bar);
                }
            }
            // never leave with copies in flight: wait (bounded) until the last stages have been consumed
            for (uint32_t q = (it > (uint32_t)kPairStages ? it - kPairStages : 0); q < it; ++q)
                if (!mbar_wait(empty + (q % kPairStages), (q / kPairStages) & 1)) break;
        }
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {
            // MMA issuer of the pair
            uint32_t it = 0;
            int j = 0;
            for (int t = pair; t < ntiles && !*abort_flag; t += npairs, ++j) {
                const int acc = j & 1;
                const int use = j >> 1;  // this accumulator's use count
                if (use > 0 && !mbar_wait_cluster(tempty + acc, (use - 1) & 1)) {
                    atomicExch(g.err, 4);
                    *abort_flag = 1;
                    break;
                }
                tc_fence_after();
                const uint32_t d = tmem + (uint32_t)(acc * BN);
                for (int kt = 0; kt < nk; ++kt, ++it) {
                    const int s = it % kPairStages;
                    const uint32_t ph = (it / kPairStages) & 1;
                    if (*abort_flag || !mbar_wait_cluster(full + s, ph)) {
                        atomicExch(g.err, 2);
                        *abort_flag = 1;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t a0 = smem_u32(base + s * kPairStageBytes), b0 = a0 + A_TILE;
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk)
                        mma_pair(d, sw128_desc(a0 + kk * 32), sw128_desc(b0 + kk * 32), (kt > 0 || kk > 0) ? 1u : 0u);
                    mma_commit_pair(empty + s);
                }
                if (*abort_flag) break;
                mma_commit_pair(tfull + acc);  // arrives once this tile's MMAs have completed
            }
        }
    } else {
        // epilogue warps: this CTA's 128 rows, a quarter of them and a slice of the columns each
        constexpr int kCols = BN * 4 / kPairEpiWarps;
        const int q = warp & 3, c0 = ((warp - 2) >> 2) * kCols;
        const bool vec = (g.ldc % 8) == 0 && ((reinterpret_cast<uintptr_t>(g.C) | reinterpret_cast<uintptr_t>(g.aux) |
                                               reinterpret_cast<uintptr_t>(g.bias)) & 15) == 0;
        uint4 *box = reinterpret_cast<uint4 *>(boxes + (warp - 2) * kPairBox);
        int j = 0;
        for (int t = pair; t < ntiles; t += npairs, ++j) {
            const int acc = j & 1;
            const int row0 = (t / ntn) * 2 * BM + rank * BM + q * 32, n0 = (t % ntn) * BN;
            uint4 ahead[kPairAhead<EPI> + 1];
            if (vec && n0 + c0 + 32 <= g.N) pair_load32<EPI>(g, row0, n0 + c0, lane, ahead);
            const bool ok = __all_sync(0xffffffffu, !*abort_flag && mbar_wait(tfull + acc, (j >> 1) & 1));
            if (!ok) {
                if (lane == 0) {
                    atomicExch(g.err, 3);
                    *abort_flag = 1;
                }
                break;
            }
            tc_fence_after();
            const uint32_t src = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN);
#pragma unroll 1
            for (int c = c0; c < c0 + kCols; c += 32) {
                if (row0 >= g.M || n0 + c >= g.N) break;
                if (vec && n0 + c + 32 <= g.N) {
                    uint4 in[kPairAhead<EPI> + 1];
#pragma unroll
                    for (int i = 0; i < kPairAhead<EPI>; ++i) in[i] = ahead[i];
                    if (c + 32 < c0 + kCols && n0 + c + 64 <= g.N) pair_load32<EPI>(g, row0, n0 + c + 32, lane, ahead);
                    float v[32];
                    tmem_ld32(src + (uint32_t)c, v);
                    pair_store32<EPI>(g, row0, n0 + c, lane, v, in, box);
                } else {
#pragma unroll 1
                    for (int h = 0; h < 32; h += 16) {
                        float v[16];
                        tmem_ld16(src + (uint32_t)(c + h), v);
                        tc_store16<EPI>(g, row0 + lane, n0 + c + h, v, vec);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(cluster_addr(tempty + acc, 0));
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // the other CTA's loads, arrivals and tensor-memory reads are done too
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kPersistTmemCols)
                     : "memory");
    }
}

}  // namespace tc
}  // namespace slos

namespace slos {
namespace tc {

// ---------------------------------------------------------------- split operands
// tc_gemm_split_kernel: FP32-accurate products on the 16-bit tensor path.  Each
// operand value is scaled by a power of two of its row and split into three
// BF16 numbers, v = p0 + p1 + p2 (24 significant bits at any size), and the
// product is p0 q0 + p0 q1 + p1 q0 + p1 q1 + p0 q2 + p2 q0, taken smallest
// first (the dropped terms are ~2^-24 of it).  Columns 2t and 2t + 1 are re and
// im of output t: psi(row, t) = rowscale[row] colscale[t] (re + i im) 2^(-2
// kSplitTarget); stored as |psi|^2, or as psi (complex64).
//
// CTA pairs as in tc_gemm_pair_kernel, tiles of 256 x bn; a stage holds the
// three parts of both operands for 64 values of K and feeds all six products
// from them (24 MMAs), so two stages of 96 KB a CTA keep the loads a stage
// ahead.  Bound by the MMAs, so what is left to choose is how evenly the tiles
// fill the pairs: bn (split_columns) is the multiple of 32 up to 256 with the
// least waves x columns (2 x 2002 columns in tiles of 224 fill 3.8 of 4 waves,
// of 256 3.4).
//
// The tensor core's FP32 accumulation does not round to nearest: over the
// ~1500 MMAs of a long K its errors pile up in one direction (measured:
// |psi|^2 of the amplitude-encoding GEMM biased low by 4e-5 when one
// accumulator took all of them).  So the K sum is taken in chunks of
// kSpChunkStages stages: each chunk accumulates into one of two TMEM buffers
// while the epilogue warps move the other buffer's finished chunk into FP32
// registers (half a row, up to 128 columns, per thread; round-to-nearest adds).
// Roles: warp 0 TMA producer, warp 1 MMA issuer (of the even CTA), warps 2-9
// epilogue (TMEM lane quarter = warp % 4, the first half of the columns for
// warps 2-5 and the second for warps 6-9).  Waits are bounded as above.
constexpr int kSplitTarget = 50;   // exponent of a scaled row's largest magnitude
constexpr int kSpParts = 3;        // BF16 numbers per value
constexpr int kSpStages = 2;
constexpr int kSpChunkStages = 1;  // 24 MMAs per chunk
constexpr int kSpThreads = 320;
constexpr int kSpEpiWarps = 8;
constexpr int kSpTile = BM * 128;             // bytes of 128 rows of an operand
constexpr int kSpStageBytes = 2 * kSpParts * kSpTile;  // the parts of A, then those of B
constexpr int kSpBox = 32 * 9 * 8;            // an epilogue warp's block of 32 rows x 8 outputs, padded
constexpr int kSpSmem = kSpStages * kSpStageBytes + kSpEpiWarps * kSpBox + 1024 + 256;
constexpr uint32_t kSpTmemCols = 2 * BN;

struct SplitArgs {
    int M, N, K;  // N = 2 x outputs
    int bn;       // columns of a tile: a multiple of 32, at most 256
    void *C;      // [M][N / 2] float or complex64
    int amps;
    const float *colscale, *rowscale;
    int part_rows_a, part_rows_b;  // rows from one part of an operand to the next
    int *err;
};

// Columns of a tile for M x N outputs on `pairs` CTA pairs: the least time of
// waves x (columns + 32; the fixed cost of a wave in columns), the widest of equals.
inline int split_columns(int M, int N, int pairs) {
    int best = BN;
    int64_t least = INT64_MAX;
    for (int bn = BN; bn >= 32; bn -= 32) {
        const int64_t tiles = (int64_t)((N + bn - 1) / bn) * ((M + 2 * BM - 1) / (2 * BM));
        const int64_t cost = (tiles + pairs - 1) / pairs * (bn + 32);
        if (cost < least) {
            least = cost;
            best = bn;
        }
    }
    return best;
}

__device__ __forceinline__ void mma_split_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// 32 rows x 16 columns (8 outputs) by a warp: v holds row row0 + lane.  Turned
// in `box` so that eight lanes write a row's eight outputs.
__device__ __forceinline__ void split_store(const SplitArgs &g, int row0, int col0, int lane, const float *v,
                                            float2 *box) {
    const int t0 = col0 / 2, outs = g.N / 2;
    const float rs = row0 + lane < g.M ? __ldg(g.rowscale + row0 + lane) : 0.f;
    constexpr float unscale = 1.f / ((float)(1ull << kSplitTarget) * (float)(1ull << kSplitTarget));
    float *boxf = reinterpret_cast<float *>(box);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float c = t0 + i < outs ? __ldg(g.colscale + t0 + i) : 0.f;
        // rs and unscale are powers of two; the sums reach 2^118, so unscale comes first
        const float re = v[2 * i] * unscale * rs * c, im = v[2 * i + 1] * unscale * rs * c;
        if (g.amps) box[lane * 9 + i] = make_float2(re, im);
        else boxf[lane * 9 + i] = re * re + im * im;
    }
    __syncwarp();
    const int i = lane & 7;
#pragma unroll
    for (int p = 0; p < 8; ++p) {
        const int r = 4 * p + (lane >> 3);
        if (row0 + r < g.M && t0 + i < outs) {
            const int64_t o = (int64_t)(row0 + r) * outs + t0 + i;
            if (g.amps) reinterpret_cast<float2 *>(g.C)[o] = box[r * 9 + i];
            else reinterpret_cast<float *>(g.C)[o] = boxf[r * 9 + i];
        }
    }
    __syncwarp();
}

static __global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kSpThreads, 1)
    tc_gemm_split_kernel(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb, SplitArgs g) {
    extern __shared__ uint8_t smem_tc[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_tc) + 1023) & ~uintptr_t(1023));
    uint8_t *boxes = base + kSpStages * kSpStageBytes;
    uint64_t *full = reinterpret_cast<uint64_t *>(boxes + kSpEpiWarps * kSpBox);
    uint64_t *empty = full + kSpStages;
    uint64_t *cfull = empty + kSpStages;  // [2] a chunk's MMAs are done
    uint64_t *cempty = cfull + 2;         // [2] the epilogue warps of both CTAs have taken the chunk
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(cempty + 2);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = blockIdx.x & 1, pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
    const int bn = g.bn;
    const int nk = (g.K + BK - 1) / BK;
    const int nchunks = (nk + kSpChunkStages - 1) / kSpChunkStages;
    const int ntn = (g.N + bn - 1) / bn;
    const int ntiles = ((g.M + 2 * BM - 1) / (2 * BM)) * ntn;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kSpStages; ++s) {
            mbar_init(full + s, 1);
            mbar_init(empty + s, 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(cfull + a, 1);
            mbar_init(cempty + a, 2 * kSpEpiWarps);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kSpTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            // producer: every stage of every tile, in order
            const uint32_t bytes = 2u * kSpParts * (uint32_t)(kSpTile + bn / 2 * 128);  // of both CTAs
            uint32_t it = 0;
            for (int t = pair; t < ntiles && !*abort_flag; t += npairs) {
                const int m0 = (t / ntn) * 2 * BM + rank * BM, n0 = (t % ntn) * bn + rank * (bn / 2);
                for (int kt = 0; kt < nk; ++kt, ++it) {
                    const int s = it % kSpStages;
                    const uint32_t ph = (it / kSpStages) & 1;
                    if (it >= (uint32_t)kSpStages && !mbar_wait(empty + s, ph ^ 1)) {
                        atomicExch(g.err, 1);
                        *abort_flag = 1;
                        break;
                    }
                    if (*abort_flag) break;
                    if (rank == 0) mbar_expect_tx(full + s, bytes);
                    const uint32_t bar = cluster_addr(full + s, 0);
                    uint8_t *st = base + s * kSpStageBytes;
                    // rows past a part's last are another part's: they meet outputs that are not stored
#pragma unroll
                    for (int p = 0; p < kSpParts; ++p) {
                        tma_load_pair(st + p * kSpTile, &ta, kt * BK, m0 + p * g.part_rows_a, bar);
                        tma_load_pair(st + (kSpParts + p) * kSpTile, &tb, kt * BK, n0 + p * g.part_rows_b, bar);
                    }
                }
            }
            // never leave with copies in flight: wait (bounded) until the last stages have been consumed
            for (uint32_t q = (it > (uint32_t)kSpStages ? it - kSpStages : 0); q < it; ++q)
                if (!mbar_wait(empty + (q % kSpStages), (q / kSpStages) & 1)) break;
        }
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {
            // as kIdescPair, with the tile's own width
            const uint32_t idesc =
                (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(2 * BM >> 4) << 24);
            uint32_t it = 0, c = 0;  // stages and chunks over all tiles
            for (int t = pair; t < ntiles && !*abort_flag; t += npairs) {
                for (int ch = 0; ch < nchunks; ++ch, ++c) {
                    const int b = c & 1;
                    const uint32_t use = c >> 1;
                    if (use > 0 && !mbar_wait_cluster(cempty + b, (use - 1) & 1)) {
                        atomicExch(g.err, 4);
                        *abort_flag = 1;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t d = tmem + (uint32_t)(b * BN);
                    const int k1 = min(nk, (ch + 1) * kSpChunkStages);
                    for (int kt = ch * kSpChunkStages; kt < k1; ++kt, ++it) {
                        const int s = it % kSpStages;
                        const uint32_t ph = (it / kSpStages) & 1;
                        if (*abort_flag || !mbar_wait_cluster(full + s, ph)) {
                            atomicExch(g.err, 2);
                            *abort_flag = 1;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t a0 = smem_u32(base + s * kSpStageBytes), b0 = a0 + kSpParts * kSpTile;
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {
                            uint64_t p[kSpParts], q[kSpParts];
#pragma unroll
                            for (int i = 0; i < kSpParts; ++i) {
                                p[i] = sw128_desc(a0 + i * kSpTile + kk * 32);
                                q[i] = sw128_desc(b0 + i * kSpTile + kk * 32);
                            }
                            mma_split_pair(d, p[2], q[0], idesc, (kt > ch * kSpChunkStages || kk > 0) ? 1u : 0u);
                            mma_split_pair(d, p[0], q[2], idesc, 1u);
                            mma_split_pair(d, p[1], q[1], idesc, 1u);
                            mma_split_pair(d, p[1], q[0], idesc, 1u);
                            mma_split_pair(d, p[0], q[1], idesc, 1u);
                            mma_split_pair(d, p[0], q[0], idesc, 1u);
                        }
                        mma_commit_pair(empty + s);
                    }
                    if (*abort_flag) break;
                    mma_commit_pair(cfull + b);
                }
            }
        }
    } else {
        // epilogue warps: each thread sums half of its row's columns over the chunks
        constexpr int HC = BN / 2;
        const int hn = bn / 2;  // columns of a half, a multiple of 16
        const int q = warp & 3;
        const int hc = (warp - 2) >> 2;  // column half
        float2 *box = reinterpret_cast<float2 *>(boxes + (warp - 2) * kSpBox);
        uint32_t c = 0;
        bool ok = true;
        for (int t = pair; t < ntiles && ok; t += npairs) {
            float acc[HC];
#pragma unroll
            for (int i = 0; i < HC; ++i) acc[i] = 0.f;
            for (int ch = 0; ch < nchunks; ++ch, ++c) {
                const int b = c & 1;
                ok = __all_sync(0xffffffffu, !*abort_flag && mbar_wait(cfull + b, (c >> 1) & 1));
                if (!ok) {
                    if (lane == 0) {
                        atomicExch(g.err, 3);
                        *abort_flag = 1;
                    }
                    break;
                }
                tc_fence_after();
                const uint32_t src = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * BN + hc * hn);
#pragma unroll
                for (int c16 = 0; c16 < HC; c16 += 16) {
                    if (c16 < hn) {
                        float v[16];
                        tmem_ld16(src + (uint32_t)c16, v);
#pragma unroll
                        for (int i = 0; i < 16; ++i) acc[c16 + i] += v[i];
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(cluster_addr(cempty + b, 0));
            }
            if (!ok) break;
            const int row0 = (t / ntn) * 2 * BM + rank * BM + q * 32, n0 = (t % ntn) * bn + hc * hn;
#pragma unroll
            for (int c16 = 0; c16 < HC; c16 += 16)
                if (c16 < hn && n0 + c16 < g.N && row0 < g.M) split_store(g, row0, n0 + c16, lane, acc + c16, box);
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kSpTmemCols) : "memory");
    }
}

}  // namespace tc
}  // namespace slos
