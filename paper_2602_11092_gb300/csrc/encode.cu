// Amplitude-encoded input (Sec. II-C, amplitude encoding): the input is a
// state vector |x> = sum_s x_s |s> over the plan's basis (n photons), the
// output is U|x>, with amplitudes
//     psi(t) = sum_s <t|U|s> x_s = sum_s Phi[t][s] x_s,
// Phi the n-photon transfer matrix of U.  Phi is built layer by layer with
// the photon-by-photon recursion of Sec. II-A.2/II-A.3 applied to every input
// column at once: for a k-photon input s with highest occupied mode c,
//     A_k[s][t] = sum_{j : t_j > 0} U[j][c] A_{k-1}[s - e_c][t - e_j],
// A_0 = 1, so A_n[s][t] = Per(U[rows t, cols s]) / prod t!, and
// <t|U|s> = A_n[s][t] sqrt(prod t!) / sqrt(prod s!).  The rows t use the
// plan's fixed-width parent slots; the columns a per-state (s - e_c, c)
// table.  Then one complex GEMM applies Phi to every input vector of the
// batch (U is shared by the batch, as the layer's weights are).
//
// The GEMM runs on the tensor cores as one real GEMM with K' = 2K:
//     [Yr | Yi](b, t) = sum_s  xr_s [Ar | Ai](s, t) + xi_s [-Ai | Ar](s, t),
// x_s = X[b][s] / g_s, A = A_n, its output columns interleaved (2t = re,
// 2t + 1 = im of output t) so the epilogue forms g_t (Yr + i Yi) and its
// |.|^2 from adjacent columns of one row.  For FP32-accurate products on the
// 16-bit tensor path (tc_gemm_split_kernel) every operand value is split into
// three BF16 numbers, which hold an FP32 value's 24 significant bits whatever
// its size: a component of a state vector keeps its relative accuracy however
// small it is beside the others (a map that does not mix hands it straight to
// its output).  A power of two per row of X and one per output t first brings
// the row's largest magnitude to [2^50, 2^51), so that products of small
// vectors and small outputs stay far above FP32's subnormals; the epilogue
// undoes both.  The batch runs in chunks of kEncodeChunk rows, so the split
// copy of X needs a fixed workspace.  (Bases of a few states: encode_small_kernel.)
//
// One call, 4096 states of 2002 amplitudes: 818 us with TF32 pairs on single
// CTAs (GEMM 645, splits and their clearing 110, transfer matrix 47), now
// 577 us (GEMM 427, splits 100, transfer matrix 50).  FP16 pairs (three products instead of six) take 369 us, but share
// an exponent range of 2^-40 over a row and lose what lies below it.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <string>

#include "../../include/slos.h"
#include "common.cuh"
#include "plan.h"
#include "profile.h"
#include "tab_launch.h"
#include "tc_gemm.cuh"

namespace slos {
slos_status_t fail(slos_status_t st, const std::string &msg);

constexpr int kTransferThreads = 256;
constexpr int kTransferRows = 4;  // input columns per block: they share the slot rows of the outputs

// Layer k of the transfer matrix.  colmax (the last layer): per output t the
// largest |re|, |im| over the inputs, as the bits of a non-negative float; the
// layer before clears it (`clear`, nclear entries: a memset of its own cost 3 us
// a call).
template <int KW>
__global__ void __launch_bounds__(kTransferThreads)
    transfer_kernel(const float2 *U, int m, const uint32_t *slots, const uint32_t *colinfo, int64_t Fk, int64_t Fp,
                    const float2 *prev, float2 *cur, int first, unsigned int *colmax, unsigned int *clear,
                    int64_t nclear) {
    __shared__ float2 uc[kTransferRows][32];  // column c of U, zero past m (padding slots name mode kMaxModes)
    __shared__ int64_t from[kTransferRows];
    const int64_t s0 = (int64_t)blockIdx.y * kTransferRows;
    const int rows = (int)min((int64_t)kTransferRows, Fk - s0);
    if (clear) {
        const int64_t step = (int64_t)gridDim.x * gridDim.y * kTransferThreads;
        for (int64_t i = ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * kTransferThreads + threadIdx.x; i < nclear; i += step)
            clear[i] = 0u;
    }
    if (threadIdx.x < kTransferRows * 32) {
        const int r = threadIdx.x >> 5, j = threadIdx.x & 31;
        if (r < rows) {
            const uint32_t ci = __ldg(colinfo + s0 + r);
            uc[r][j] = j < m ? U[j * m + (int)(ci & 31u)] : make_float2(0.f, 0.f);
            if (j == 0) from[r] = (int64_t)(ci >> 5) * Fp;
        }
    }
    __syncthreads();
    const int64_t t = (int64_t)blockIdx.x * kTransferThreads + threadIdx.x;
    if (t >= Fk) return;
    uint32_t e[KW];
    const uint4 *sl = reinterpret_cast<const uint4 *>(slots) + t * (KW / 4);
#pragma unroll
    for (int q4 = 0; q4 < KW / 4; ++q4) {
        const uint4 w4 = __ldg(sl + q4);
        e[4 * q4] = w4.x;
        e[4 * q4 + 1] = w4.y;
        e[4 * q4 + 2] = w4.z;
        e[4 * q4 + 3] = w4.w;
    }
    unsigned int top = 0u;
#pragma unroll
    for (int r = 0; r < kTransferRows; ++r) {
        if (r >= rows) break;
        float2 acc;
        if (first) {
            acc = uc[r][e[0] & 31u];  // one photon: <e_j|U|e_c> = U[j][c]
        } else {
            const float2 *pv = prev + from[r];
            acc = make_float2(0.f, 0.f);
#pragma unroll
            for (int q = 0; q < KW; ++q) acc = cfma(uc[r][e[q] & 31u], pv[e[q] >> 5], acc);
        }
        cur[(s0 + r) * Fk + t] = acc;
        // as unsigned integers non-negative floats order like their values, NaN above infinity
        top = max(top, max(__float_as_uint(fabsf(acc.x)), __float_as_uint(fabsf(acc.y))));
    }
    if (colmax) atomicMax(colmax + t, top);
}

// Exponent of the power of two that brings a row whose largest magnitude has
// these bits to [2^kSplitTarget, 2^(kSplitTarget + 1)); 0 for rows of zeros and
// of values that are not finite (their products are not either, whatever the
// scale).  Sums of 2^16 products stay below 2^118, and a value keeps its three
// parts normal down to 2^-160 of its row's largest.
__device__ __forceinline__ int split_exponent(unsigned int bits) {
    if (bits == 0u || bits >= 0x7f800000u) return 0;
    return min(126, tc::kSplitTarget - ilogbf(__uint_as_float(bits)));
}
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }

// v = p[0] + p[1] + p[2] in BF16.
constexpr int kParts = tc::kSpParts;
__device__ __forceinline__ void bf16_split(float v, __nv_bfloat16 (&p)[kParts]) {
#pragma unroll
    for (int i = 0; i < kParts; ++i) {
        p[i] = __float2bfloat16_rn(v);
        v -= __bfloat162float(p[i]);
    }
}

constexpr int kEncodeChunk = 4096;  // batch rows per GEMM launch
constexpr int kEncodeKAlign = 64;   // K' padded to whole 128-byte stage rows

// Real-form operand B of the GEMM, [N = 2K rows][K2 cols], K-major:
//   row 2t:     cols s -> Ar[s][t],  K + s -> -Ai[s][t],  2K .. K2-1 -> 0
//   row 2t + 1: cols s -> Ai[s][t],  K + s ->  Ar[s][t]
// scaled and split into kParts copies, each 2K rows after the one before;
// 32 x 32 tiles of A through shared memory, so both the read (along t) and the
// writes (along s) are coalesced.  colscale[t] = g_t times t's share of the
// scale's inverse.
__global__ void __launch_bounds__(256) encode_split_b_kernel(const float2 *A, int64_t K, int64_t K2,
                                                             const unsigned int *colmax, const float *g,
                                                             __nv_bfloat16 *bsplit, float *colscale) {
    __shared__ float2 tile[32][33];
    const int64_t s0 = (int64_t)blockIdx.y * 32, t0 = (int64_t)blockIdx.x * 32;
    const int64_t part = 2 * K * K2;
    for (int i = threadIdx.y; i < 32; i += 8) {
        const int64_t ss = s0 + i, tt = t0 + threadIdx.x;
        tile[i][threadIdx.x] = (ss < K && tt < K) ? A[ss * K + tt] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += 8) {
        const int64_t tt = t0 + i, ss = s0 + threadIdx.x;
        if (tt >= K) continue;
        const int ex = split_exponent(__ldg(colmax + tt));
        if (blockIdx.y == 0 && threadIdx.x == 0) colscale[tt] = g[tt] * pow2f(tc::kSplitTarget - ex);
        if (blockIdx.y + 1 == gridDim.y) {
            for (int64_t c = 2 * K + threadIdx.x; c < K2; c += 32)
#pragma unroll
                for (int p = 0; p < kParts; ++p)
                    bsplit[p * part + 2 * tt * K2 + c] = bsplit[p * part + (2 * tt + 1) * K2 + c] =
                        __float2bfloat16_rn(0.f);
        }
        if (ss >= K) continue;
        const float sc = pow2f(ex);
        const float2 v = tile[threadIdx.x][i];  // A[ss][tt]
        __nv_bfloat16 re[kParts], im[kParts];
        bf16_split(v.x * sc, re);
        bf16_split(v.y * sc, im);
#pragma unroll
        for (int p = 0; p < kParts; ++p) {
            __nv_bfloat16 *o = bsplit + p * part + 2 * tt * K2 + ss;
            o[0] = re[p];
            o[K] = __hneg(im[p]);
            o[K2] = im[p];
            o[K2 + K] = re[p];
        }
    }
}

// Real-form operand A of the GEMM for batch rows [b0, b0 + rows), T threads
// per row: [rows][K2], cols s -> Re X[b][s] / g_s, K + s -> Im X[b][s] / g_s,
// the padding columns 2K .. K2-1 zero; scaled and split into kParts copies,
// each kEncodeChunk rows after the one before.  rowscale[r] = the row's share
// of its scale's inverse.  T = 32 (a warp per row, no barrier)
// up to kSplitWarpRow values, a block per row beyond (1657 rows of 56: a block
// each cost 3 us more than a warp each).
constexpr int kSplitThreads = 256;
constexpr int kSplitKeep = 8;  // values per thread kept in registers between the maximum and the split
constexpr int64_t kSplitWarpRow = 32 * kSplitKeep;
template <int T>
__global__ void __launch_bounds__(kSplitThreads) encode_split_a_kernel(const float2 *X, const float *g, int64_t b0,
                                                                       int rows, int64_t K, int64_t K2,
                                                                       __nv_bfloat16 *asplit, float *rowscale) {
    __shared__ unsigned int red[kSplitThreads / 32];
    const int64_t r = (int64_t)blockIdx.x * (kSplitThreads / T) + threadIdx.x / T;
    if (r >= rows) return;  // whole warps (T = 32) or nobody
    const int tid = threadIdx.x % T;
    const float2 *x = X + (b0 + r) * K;
    auto value = [&](int64_t s) {
        const float2 v = x[s];
        const float gs = __ldg(g + s);
        return make_float2(v.x / gs, v.y / gs);
    };
    auto bits = [](float2 v) { return max(__float_as_uint(fabsf(v.x)), __float_as_uint(fabsf(v.y))); };
    float2 keep[kSplitKeep];
    unsigned int top = 0u;
#pragma unroll
    for (int i = 0; i < kSplitKeep; ++i) {
        const int64_t s = tid + (int64_t)i * T;
        keep[i] = s < K ? value(s) : make_float2(0.f, 0.f);
        top = max(top, bits(keep[i]));
    }
    const int64_t rest = tid + (int64_t)kSplitKeep * T;
    for (int64_t s = rest; s < K; s += T) top = max(top, bits(value(s)));
    top = __reduce_max_sync(0xffffffffu, top);
    if (T > 32) {
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = top;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < T / 32; ++w) top = max(top, red[w]);
    }
    const int ex = split_exponent(top);
    const float sc = pow2f(ex);
    const int64_t part = (int64_t)kEncodeChunk * K2;
    __nv_bfloat16 *o = asplit + r * K2;
    auto put = [&](int64_t s, float2 v) {
        __nv_bfloat16 re[kParts], im[kParts];
        bf16_split(v.x * sc, re);
        bf16_split(v.y * sc, im);
#pragma unroll
        for (int p = 0; p < kParts; ++p) {
            o[p * part + s] = re[p];
            o[p * part + K + s] = im[p];
        }
    };
#pragma unroll
    for (int i = 0; i < kSplitKeep; ++i) {
        const int64_t s = tid + (int64_t)i * T;
        if (s < K) put(s, keep[i]);
    }
    for (int64_t s = rest; s < K; s += T) put(s, value(s));
    for (int64_t c = 2 * K + tid; c < K2; c += T)
#pragma unroll
        for (int p = 0; p < kParts; ++p) o[p * part + c] = __float2bfloat16_rn(0.f);
    if (tid == 0) rowscale[r] = pow2f(tc::kSplitTarget - ex);
}

// Bases of up to kSmallStates states: the whole product in FP32 on the CUDA
// cores, thread = one output of one vector, Phi (at most 32 KB) and a CTA's
// vectors in shared memory.  Bound by launch latency up to a few thousand
// vectors; what it saves is two launches and the tensor pipeline's start.
// One call, us, split GEMM / this: 4096 states of 10 17.1 / 6.4, 16 of 56
// 20.5 / 10.3, 8192 of 56 33.0 / 19.6.
constexpr int kSmallStates = 64;
constexpr int kSmallThreads = 256;
__global__ void __launch_bounds__(kSmallThreads) encode_small_kernel(const float2 *A, const float *g, const float2 *X,
                                                                     int K, int64_t batch, int amps, void *out) {
    __shared__ float2 phi[kSmallStates * kSmallStates];  // A[s][t]
    __shared__ float2 x[kSmallThreads];                  // the rows' vectors over g
    for (int i = threadIdx.x; i < K * K; i += kSmallThreads) phi[i] = A[i];
    const int rows = kSmallThreads / K, r = threadIdx.x / K, t = threadIdx.x % K;
    const float gt = __ldg(g + t);
    for (int64_t b0 = (int64_t)blockIdx.x * rows; b0 < batch; b0 += (int64_t)gridDim.x * rows) {
        const bool own = r < rows && b0 + r < batch;
        const int64_t o = b0 * K + threadIdx.x;
        __syncthreads();
        if (own) {
            const float2 v = X[o];
            x[threadIdx.x] = make_float2(v.x / gt, v.y / gt);
        }
        __syncthreads();
        if (!own) continue;
        float2 acc = make_float2(0.f, 0.f);
        for (int s = 0; s < K; ++s) acc = cfma(x[r * K + s], phi[s * K + t], acc);
        acc = cscale(acc, gt);
        if (amps) reinterpret_cast<float2 *>(out)[o] = acc;
        else reinterpret_cast<float *>(out)[o] = cabs2(acc);
    }
}

// BF16 matrix [rows][cols] (row stride ld elements, a multiple of 8), box
// 64 x box_rows, 128-byte swizzle: the operand layout of tc_gemm.cuh.
static PFN_cuTensorMapEncodeTiled_v12000 encode_map_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *q = nullptr;
        cudaDriverEntryPointQueryResult r;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &q, 12000, cudaEnableDefault, &r) ==
                cudaSuccess &&
            r == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(q);
    });
    return fn;
}
static bool make_map_bf16(CUtensorMap *map, const __nv_bfloat16 *ptr, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
    auto fn = encode_map_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)(ld * 2)};
    cuuint32_t box[2] = {(cuuint32_t)tc::BK, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16 *>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static bool encodable(const slos_plan_s *p) {
    if (!p->tab.enabled || !p->tab.gfact || p->K > kMaxEncodeStates) return false;
    for (int k = 1; k <= p->n; ++k)
        if (!p->tab.layer[k].colinfo) return false;
    return true;
}

static size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

static int64_t encode_k2(const slos_plan_s *p) {
    return (2 * p->K + kEncodeKAlign - 1) / kEncodeKAlign * kEncodeKAlign;
}

// workspace: the transfer matrices of layers n and n-1, the split operands
// B [kParts][2K][K2] and A [kParts][kEncodeChunk][K2], then the largest
// magnitude and the scale of each output and the scale of each row of a chunk
struct EncodeLayout {
    size_t a, b, bsplit, asplit, colmax, colscale, rowscale, total;
};
static EncodeLayout encode_layout(const slos_plan_s *p) {
    const int n = p->n;
    const size_t K = (size_t)p->K, K2 = (size_t)encode_k2(p);
    EncodeLayout L;
    size_t at = 0;
    auto take = [&](size_t bytes) {
        const size_t o = at;
        at += align256(bytes);
        return o;
    };
    L.a = take((size_t)p->F[n] * p->F[n] * sizeof(float2));
    L.b = take(n >= 2 ? (size_t)p->F[n - 1] * p->F[n - 1] * sizeof(float2) : 0);
    L.bsplit = take(kParts * 2 * K * K2 * sizeof(__nv_bfloat16));
    L.asplit = take(kParts * kEncodeChunk * K2 * sizeof(__nv_bfloat16));
    L.colmax = take(K * sizeof(unsigned int));
    L.colscale = take(K * sizeof(float));
    L.rowscale = take(kEncodeChunk * sizeof(float));
    L.total = at;
    return L;
}

}  // namespace slos

using namespace slos;

extern "C" {

slos_status_t slos_encoded_workspace_bytes(slos_plan_t p, size_t *bytes) {
    if (!p || p->kind != 0 || !bytes) return fail(SLOS_ERR_INVALID_ARG, "slos_encoded_workspace_bytes: bad argument");
    if (!encodable(p))
        return fail(SLOS_ERR_UNSUPPORTED, "slos_encoded_workspace_bytes: amplitude encoding needs a PNR plan with at "
                                          "most 32768 outputs");
    *bytes = encode_layout(p).total;
    return SLOS_OK;
}

slos_status_t slos_encoded_forward(slos_plan_t p, const void *U, const void *X, int batch, slos_output_t output,
                                   void *out, void *workspace, size_t workspace_bytes, void *stream) {
    if (!p || p->kind != 0) return fail(SLOS_ERR_INVALID_ARG, "slos_encoded_forward: not a single-shape plan");
    if (!encodable(p))
        return fail(SLOS_ERR_UNSUPPORTED, "slos_encoded_forward: amplitude encoding needs a PNR plan with at most "
                                          "32768 outputs");
    if (batch < 0) return fail(SLOS_ERR_INVALID_ARG, "slos_encoded_forward: negative batch");
    if (output != SLOS_OUT_PROBS && output != SLOS_OUT_AMPS)
        return fail(SLOS_ERR_INVALID_ARG, "slos_encoded_forward: bad output");
    if (!U || (batch > 0 && (!X || !out))) return fail(SLOS_ERR_INVALID_ARG, "slos_encoded_forward: NULL pointer");
    const EncodeLayout L = encode_layout(p);
    if (!workspace || workspace_bytes < L.total)
        return fail(SLOS_ERR_INVALID_ARG, "slos_encoded_forward: workspace too small (slos_encoded_workspace_bytes)");
    cudaStream_t s = (cudaStream_t)stream;
    const int n = p->n, m = p->m;
    char *ws = reinterpret_cast<char *>(workspace);
    float2 *buf[2] = {reinterpret_cast<float2 *>(ws + L.a), reinterpret_cast<float2 *>(ws + L.b)};
    unsigned int *colmax = reinterpret_cast<unsigned int *>(ws + L.colmax);
    const float2 *Ud = reinterpret_cast<const float2 *>(U);
    cudaError_t e;
    const bool small = p->K <= kSmallStates;
    if (!small && n == 1 && (e = cudaMemsetAsync(colmax, 0, (size_t)p->K * sizeof(unsigned int), s)) != cudaSuccess)
        return fail(SLOS_ERR_CUDA, std::string("slos_encoded_forward: ") + cudaGetErrorString(e));
    {
        ProfScope ps("slos_transfer", 0.0, s);
        for (int k = 1; k <= n; ++k) {
            const int64_t Fk = p->F[k], Fp = p->F[k - 1];
            float2 *cur = buf[(n - k) & 1];
            const float2 *prev = k >= 2 ? buf[(n - k + 1) & 1] : nullptr;
            dim3 grid((unsigned)((Fk + kTransferThreads - 1) / kTransferThreads),
                      (unsigned)((Fk + kTransferRows - 1) / kTransferRows));
            unsigned int *top = !small && k == n ? colmax : nullptr, *clr = !small && k == n - 1 ? colmax : nullptr;
            const uint32_t *sl = p->tab.layer[k].slots, *ci = p->tab.layer[k].colinfo;
            switch (p->tab.layer[k].kw) {
                case 4: transfer_kernel<4><<<grid, kTransferThreads, 0, s>>>(Ud, m, sl, ci, Fk, Fp, prev, cur, k == 1, top, clr, p->K); break;
                case 8: transfer_kernel<8><<<grid, kTransferThreads, 0, s>>>(Ud, m, sl, ci, Fk, Fp, prev, cur, k == 1, top, clr, p->K); break;
                default: transfer_kernel<12><<<grid, kTransferThreads, 0, s>>>(Ud, m, sl, ci, Fk, Fp, prev, cur, k == 1, top, clr, p->K); break;
            }
            if ((e = cudaGetLastError()) != cudaSuccess)
                return fail(SLOS_ERR_CUDA, std::string("slos_encoded_forward: ") + cudaGetErrorString(e));
        }
    }
    if (batch == 0) return SLOS_OK;
    const int64_t K = p->K, K2 = encode_k2(p);
    if (small) {
        const int64_t rows = kSmallThreads / K, ctas = (batch + rows - 1) / rows;
        ProfScope ps("slos_encode_gemm", 8.0 * batch * (double)K * K, s);  // flops
        encode_small_kernel<<<(unsigned)std::min<int64_t>(ctas, (int64_t)p->sm_count * 4), kSmallThreads, 0, s>>>(
            buf[0], p->tab.gfact, reinterpret_cast<const float2 *>(X), (int)K, batch, output == SLOS_OUT_AMPS, out);
        if ((e = cudaGetLastError()) != cudaSuccess)
            return fail(SLOS_ERR_CUDA, std::string("slos_encoded_forward: ") + cudaGetErrorString(e));
        return SLOS_OK;
    }
    __nv_bfloat16 *bsplit = reinterpret_cast<__nv_bfloat16 *>(ws + L.bsplit);
    __nv_bfloat16 *asplit = reinterpret_cast<__nv_bfloat16 *>(ws + L.asplit);
    float *colscale = reinterpret_cast<float *>(ws + L.colscale), *rowscale = reinterpret_cast<float *>(ws + L.rowscale);
    {
        ProfScope ps("slos_encode_split", 0.0, s);
        dim3 grid((unsigned)((K + 31) / 32), (unsigned)((K + 31) / 32));
        encode_split_b_kernel<<<grid, dim3(32, 8), 0, s>>>(buf[0], K, K2, colmax, p->tab.gfact, bsplit, colscale);
        if ((e = cudaGetLastError()) != cudaSuccess)
            return fail(SLOS_ERR_CUDA, std::string("slos_encoded_forward: ") + cudaGetErrorString(e));
    }
    static bool attr_done[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_done[dev]) {
        if ((e = cudaFuncSetAttribute(tc::tc_gemm_split_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      tc::kSpSmem)) != cudaSuccess)
            return fail(SLOS_ERR_CUDA, std::string("slos_encoded_forward: ") + cudaGetErrorString(e));
        attr_done[dev] = true;
    }
    CUtensorMap ma;
    if (!make_map_bf16(&ma, asplit, (int64_t)kParts * kEncodeChunk, K2, K2, tc::BM))
        return fail(SLOS_ERR_CUDA, "slos_encoded_forward: cuTensorMapEncodeTiled failed");
    const float2 *Xd = reinterpret_cast<const float2 *>(X);
    for (int b0 = 0; b0 < batch; b0 += kEncodeChunk) {
        const int rows = std::min(kEncodeChunk, batch - b0);
        {
            ProfScope ps("slos_encode_split", 0.0, s);
            if (K <= kSplitWarpRow)
                encode_split_a_kernel<32><<<(unsigned)((rows + 7) / 8), kSplitThreads, 0, s>>>(
                    Xd, p->tab.gfact, b0, rows, K, K2, asplit, rowscale);
            else
                encode_split_a_kernel<kSplitThreads><<<(unsigned)rows, kSplitThreads, 0, s>>>(
                    Xd, p->tab.gfact, b0, rows, K, K2, asplit, rowscale);
            if ((e = cudaGetLastError()) != cudaSuccess)
                return fail(SLOS_ERR_CUDA, std::string("slos_encoded_forward: ") + cudaGetErrorString(e));
        }
        const int pairs = std::max(1, p->sm_count / 2);
        tc::SplitArgs g;
        memset(&g, 0, sizeof(g));
        g.M = rows;
        g.N = (int)(2 * K);
        g.K = (int)K2;
        g.bn = tc::split_columns(g.M, g.N, pairs);
        g.C = output == SLOS_OUT_AMPS ? (void *)(reinterpret_cast<float2 *>(out) + (int64_t)b0 * K)
                                      : (void *)(reinterpret_cast<float *>(out) + (int64_t)b0 * K);
        g.colscale = colscale;
        g.rowscale = rowscale;
        g.amps = output == SLOS_OUT_AMPS ? 1 : 0;
        g.err = p->d_status + 2;
        g.part_rows_a = kEncodeChunk;
        g.part_rows_b = (int)(2 * K);
        CUtensorMap mb;
        if (!make_map_bf16(&mb, bsplit, kParts * 2 * K, K2, K2, g.bn / 2))
            return fail(SLOS_ERR_CUDA, "slos_encoded_forward: cuTensorMapEncodeTiled failed");
        const int64_t tiles = (int64_t)((g.N + g.bn - 1) / g.bn) * ((rows + 2 * tc::BM - 1) / (2 * tc::BM));
        const unsigned grid = 2 * (unsigned)std::min<int64_t>(tiles, pairs);
        ProfScope ps("slos_encode_gemm", 6.0 * 2.0 * rows * (double)g.N * (double)K2, s);  // flops
        tc::tc_gemm_split_kernel<<<grid, tc::kSpThreads, tc::kSpSmem, s>>>(ma, mb, g);
        if ((e = cudaGetLastError()) != cudaSuccess)
            return fail(SLOS_ERR_CUDA, std::string("slos_encoded_forward: ") + cudaGetErrorString(e));
    }
    return SLOS_OK;
}

}  // extern "C"
