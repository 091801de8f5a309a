// Measurement strategies on top of an output distribution (Sec. II-A.3,
// QuantumLayer: per-mode photon-number expectations) and renormalisation onto
// the plan's space, each with its backward.  Caller buffers only; every sum is
// taken in a fixed order (within a thread, over the warp, the warps, then the
// CTAs of a cluster in rank order), so every value is reproducible.
//
// All four move a few bytes per output and are bound by memory once enough of
// it is in flight; what held them back was one 256-thread CTA per instance
// walking its row 1 KB at a time, and 16 one-byte table loads per output and
// instance.  The reductions now split an instance's row over a thread-block
// cluster (partial sums meet in distributed shared memory, so no workspace),
// the renormalisation keeps its row in registers between its sum and its
// division, and the expectations read an output's occupations as 32-bit words
// once for several instances.  512 instances of 8008 outputs, 16 modes:
// renormalise 15.0 -> 10.1 us, its backward 21.9 -> 13.6 us, expectations 44.2 -> 15 us,
// their backward 35.8 -> 9.5 us.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <string>

#include "../../include/slos.h"
#include "common.cuh"
#include "dfloat.cuh"
#include "plan.h"
#include "profile.h"

namespace slos {
slos_status_t fail(slos_status_t st, const std::string &msg);

namespace cg = cooperative_groups;

constexpr int kMaxCluster = 8;

// Occupations of one output, MW words of 4 modes, as floats (0x4b000000 + n is
// the float 2^23 + n, so a byte permute and a subtraction convert exactly).
template <int MW>
__device__ __forceinline__ void occ_floats(const uint32_t *__restrict__ row, float (&f)[4 * MW]) {
#pragma unroll
    for (int w = 0; w < MW; ++w) {
        const uint32_t x = __ldg(row + w);
#pragma unroll
        for (int q = 0; q < 4; ++q) f[4 * w + q] = __uint_as_float(__byte_perm(x, 0x4b000000u, 0x7440u | q)) - 8388608.f;
    }
}

// out[b][j] = sum_t occ[t][j] p[b][t]: a cluster of CTAs per NI instances,
// each CTA a slice of the outputs.
constexpr int kExpThreads = 256;
constexpr int kExpWarps = kExpThreads / 32;
template <int MW, int NI>
__global__ void __launch_bounds__(kExpThreads, 2) expect_fwd_kernel(const float *p, const uint32_t *occ, int64_t K,
                                                                    int m, int B, float *out) {
    constexpr int N = (NI * 4 * MW + 31) / 32 * 32;  // values reduced over the warp, padded
    __shared__ float red[kExpWarps][N];
    __shared__ float part[N];
    cg::cluster_group cluster = cg::this_cluster();
    const int C = gridDim.x, rank = blockIdx.x;
    const int b0 = blockIdx.y * NI;
    const int64_t per = (K + C - 1) / C;
    const int64_t hi = min(K, per * (rank + 1));
    float v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = 0.f;
#pragma unroll 2
    for (int64_t c = per * rank + threadIdx.x; c < hi; c += kExpThreads) {
        float x[NI], f[4 * MW];
#pragma unroll
        for (int i = 0; i < NI; ++i) x[i] = b0 + i < B ? __ldg(p + (size_t)(b0 + i) * K + c) : 0.f;
        occ_floats<MW>(occ + (size_t)c * MW, f);
#pragma unroll
        for (int i = 0; i < NI; ++i)
#pragma unroll
            for (int j = 0; j < 4 * MW; ++j) v[i * 4 * MW + j] += f[j] * x[i];
    }
    // reduce-scatter over the warp: at each step a lane keeps the half of the
    // values its bit selects, so N values cost about N shuffles instead of 5 N
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int at = 0;
    {
        int n = N;
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) {
            n /= 2;
            const bool up = (lane & s) != 0;
#pragma unroll
            for (int i = 0; i < N / 2; ++i) {
                if (i < n) {
                    const float send = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
                    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
                }
            }
            at += up ? n : 0;
        }
    }
#pragma unroll
    for (int i = 0; i < N / 32; ++i) red[warp][at + i] = v[i];
    __syncthreads();
    for (int i = threadIdx.x; i < NI * 4 * MW; i += kExpThreads) {
        float s = 0.f;
        for (int w = 0; w < kExpWarps; ++w) s += red[w][i];
        part[i] = s;
    }
    cluster.sync();
    if (rank == 0) {
        for (int i = threadIdx.x; i < NI * 4 * MW; i += kExpThreads) {
            const int b = b0 + i / (4 * MW), j = i % (4 * MW);
            if (b >= B || j >= m) continue;
            float s = 0.f;
#pragma unroll
            for (int r = 0; r < kMaxCluster; ++r) s += r < C ? cluster.map_shared_rank(part, r)[i] : 0.f;
            out[(size_t)b * m + j] = s;
        }
    }
    cluster.sync();  // no CTA leaves while its partial sums are read
}

// dp[b][t] = sum_j occ[t][j] dout[b][j]: thread = output, kExpBwdInst instances
// in turn with the output's occupations in registers.
constexpr int kExpBwdInst = 8;
template <int MW>
__global__ void __launch_bounds__(kExpThreads) expect_bwd_kernel(const float *dout, const uint32_t *occ, int64_t K,
                                                                 int m, int B, float *dp) {
    __shared__ float4 d[kExpBwdInst][MW];
    const int b0 = blockIdx.y * kExpBwdInst;
    for (int i = threadIdx.x; i < kExpBwdInst * 4 * MW; i += kExpThreads) {
        const int b = b0 + i / (4 * MW), j = i % (4 * MW);
        reinterpret_cast<float *>(d)[i] = (b < B && j < m) ? dout[(size_t)b * m + j] : 0.f;
    }
    __syncthreads();
    const int64_t c = (int64_t)blockIdx.x * kExpThreads + threadIdx.x;
    if (c >= K) return;
    float f[4 * MW];
    occ_floats<MW>(occ + (size_t)c * MW, f);
    const int nb = min(kExpBwdInst, B - b0);
#pragma unroll 4
    for (int i = 0; i < nb; ++i) {
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < MW; ++w) {
            const float4 x = d[i][w];
            v += f[4 * w] * x.x;
            v += f[4 * w + 1] * x.y;
            v += f[4 * w + 2] * x.z;
            v += f[4 * w + 3] * x.w;
        }
        dp[(size_t)(b0 + i) * K + c] = v;
    }
}

constexpr int kRenThreads = 512;
constexpr int kRenKeep = 16;  // values per thread kept in registers between the two passes

// Cluster-wide sum of one double-float per thread, fixed order (a tree over
// the lanes, the warps and the ranks); every thread gets it.
__device__ __forceinline__ dfl warp_sum(dfl v, int width) {
    for (int o = width / 2; o > 0; o >>= 1) {
        const dfl w = {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
        v = df_add(v, w);
    }
    return v;
}
__device__ dfl cluster_sum(dfl v, dfl *red, dfl *part) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    v = warp_sum(v, 32);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    v = warp_sum(lane < kRenThreads / 32 ? red[lane] : df_zero(), 32);
    if (gridDim.x == 1) return v;
    cg::cluster_group cluster = cg::this_cluster();
    if (threadIdx.x == 0) *part = v;
    cluster.sync();
    v = df_zero();
    if (lane < (int)gridDim.x) v = *cluster.map_shared_rank(part, lane);
    v = warp_sum(v, kMaxCluster);  // lanes 0..7; the others hold zeros and are not used
    v = {__shfl_sync(0xffffffffu, v.hi, 0), __shfl_sync(0xffffffffu, v.lo, 0)};
    cluster.sync();  // no CTA leaves while its partial sum is read
    return v;
}

// Z = sum_t p[t]; q[t] = p[t] / Z  (sums in double-float, dfloat.cuh).  q may be p.
__global__ void __launch_bounds__(kRenThreads, 3) renorm_fwd_kernel(const float *p, int64_t K, float *q, float *Z) {
    __shared__ dfl red[kRenThreads / 32], part;
    const int b = blockIdx.y;
    const int64_t per = (K + gridDim.x - 1) / gridDim.x;
    const int64_t lo = per * blockIdx.x;
    const int n = (int)(min(K, lo + per) - lo);  // at most K < 2^31
    const float *pb = p + (size_t)b * K + lo;
    float keep[kRenKeep];
#pragma unroll
    for (int i = 0; i < kRenKeep; ++i) {
        const int64_t c = threadIdx.x + (int64_t)i * kRenThreads;
        keep[i] = c < n ? pb[c] : 0.f;
    }
    // pairs first (exact), in four independent chains: the additions of one
    // chain wait 20 instructions for each other
    dfl part4[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) part4[i] = two_sum(keep[4 * i], keep[4 * i + 1]);
#pragma unroll
    for (int i = 0; i < 4; ++i) part4[i] = df_add(part4[i], two_sum(keep[4 * i + 2], keep[4 * i + 3]));
    dfl acc = df_add(df_add(part4[0], part4[1]), df_add(part4[2], part4[3]));
    const int64_t rest = threadIdx.x + (int64_t)kRenKeep * kRenThreads;
#pragma unroll 4
    for (int64_t c = rest; c < n; c += kRenThreads) acc = df_add_f(acc, pb[c]);
    const float z = df_float(cluster_sum(acc, red, &part));
    const float inv = z > 0.f ? 1.f / z : 0.f;
    float *qb = q + (size_t)b * K + lo;
#pragma unroll
    for (int i = 0; i < kRenKeep; ++i) {
        const int64_t c = threadIdx.x + (int64_t)i * kRenThreads;
        if (c < n) qb[c] = keep[i] * inv;
    }
    for (int64_t c = rest; c < n; c += kRenThreads) qb[c] = pb[c] * inv;
    if (blockIdx.x == 0 && threadIdx.x == 0) Z[b] = z;
}

// dp[t] = (dq[t] - sum_s dq[s] q[s]) / Z.  dp may be dq.
__global__ void __launch_bounds__(kRenThreads, 2) renorm_bwd_kernel(const float *q, const float *Z, const float *dq,
                                                                    int64_t K, float *dp) {
    __shared__ dfl red[kRenThreads / 32], part;
    const int b = blockIdx.y;
    const int64_t per = (K + gridDim.x - 1) / gridDim.x;
    const int64_t lo = per * blockIdx.x;
    const int n = (int)(min(K, lo + per) - lo);
    const float *qb = q + (size_t)b * K + lo, *dqb = dq + (size_t)b * K + lo;
    float keep[kRenKeep], qv[kRenKeep];
#pragma unroll
    for (int i = 0; i < kRenKeep; ++i) {
        const int64_t c = threadIdx.x + (int64_t)i * kRenThreads;
        keep[i] = c < n ? dqb[c] : 0.f;
        qv[i] = c < n ? qb[c] : 0.f;
    }
    const float z = Z[b];
    dfl part4[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) part4[i] = two_prod(keep[i], qv[i]);
#pragma unroll
    for (int i = 4; i < kRenKeep; ++i) part4[i & 3] = df_add(part4[i & 3], two_prod(keep[i], qv[i]));
    dfl acc = df_add(df_add(part4[0], part4[1]), df_add(part4[2], part4[3]));
    const int64_t rest = threadIdx.x + (int64_t)kRenKeep * kRenThreads;
#pragma unroll 4
    for (int64_t c = rest; c < n; c += kRenThreads) acc = df_add(acc, two_prod(dqb[c], qb[c]));
    const float sdot = df_float(cluster_sum(acc, red, &part));
    const float inv = z > 0.f ? 1.f / z : 0.f;
    float *dpb = dp + (size_t)b * K + lo;
#pragma unroll
    for (int i = 0; i < kRenKeep; ++i) {
        const int64_t c = threadIdx.x + (int64_t)i * kRenThreads;
        if (c < n) dpb[c] = (keep[i] - sdot) * inv;
    }
    for (int64_t c = rest; c < n; c += kRenThreads) dpb[c] = (dqb[c] - sdot) * inv;
}

// A kernel launched with clusters of `cluster` CTAs along x (the grid's width).
template <typename... P, typename... A>
static cudaError_t launch_clusters(void (*kernel)(P...), int cluster, int rows, int threads, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cluster, rows);
    cfg.blockDim = dim3(threads);
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = cluster;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// The renormalisation's CTAs per row: one while the row fits its registers
// (8192 outputs; a cluster costs two cluster barriers: 16.9 us against
// 10.1 us on 512 rows of 8008), then clusters until a slice does.
static int renorm_cluster(const slos_plan_s *p) {
    int c = 1;
    while (c < kMaxCluster && p->K > (int64_t)c * kRenThreads * kRenKeep) c *= 2;
    return c;
}

template <int MW>
static cudaError_t launch_expect_fwd(const slos_plan_s *p, const float *probs, int batch, float *out, cudaStream_t s) {
    const uint32_t *occ = reinterpret_cast<const uint32_t *>(p->tab.occ);
    // four instances share an output's occupations once that still leaves a
    // CTA for every other SM; the row is split until there are four per SM
    const int ni = batch >= 2 * p->sm_count ? 4 : 1;
    const int rows = (batch + ni - 1) / ni;
    int c = 1;
    while (c < kMaxCluster && (int64_t)rows * c < 4 * p->sm_count && p->K / (2 * c) >= 1024) c *= 2;
    return ni == 4 ? launch_clusters(expect_fwd_kernel<MW, 4>, c, rows, kExpThreads, s, probs, occ, p->K, p->m, batch, out)
                   : launch_clusters(expect_fwd_kernel<MW, 1>, c, rows, kExpThreads, s, probs, occ, p->K, p->m, batch, out);
}

template <int MW>
static cudaError_t launch_expect_bwd(const slos_plan_s *p, const float *dout, int batch, float *dprobs, cudaStream_t s) {
    dim3 grid((unsigned)((p->K + kExpThreads - 1) / kExpThreads), (batch + kExpBwdInst - 1) / kExpBwdInst);
    expect_bwd_kernel<MW><<<grid, kExpThreads, 0, s>>>(dout, reinterpret_cast<const uint32_t *>(p->tab.occ), p->K, p->m,
                                                       batch, dprobs);
    return cudaGetLastError();
}

static slos_status_t check(slos_plan_t p, int batch, const char *who) {
    if (!p || p->kind != 0) return fail(SLOS_ERR_INVALID_ARG, std::string(who) + ": not a single-shape plan");
    if (batch < 0) return fail(SLOS_ERR_INVALID_ARG, std::string(who) + ": negative batch");
    if (batch > 65535) return fail(SLOS_ERR_UNSUPPORTED, std::string(who) + ": at most 65535 instances per call");
    return SLOS_OK;
}

static slos_status_t launched(cudaError_t e, const char *who) {
    if (e != cudaSuccess) return fail(SLOS_ERR_CUDA, std::string(who) + ": " + cudaGetErrorString(e));
    return SLOS_OK;
}

}  // namespace slos

using namespace slos;

extern "C" {

slos_status_t slos_expectations(slos_plan_t p, const float *probs, int batch, float *out, void *stream) {
    slos_status_t st = check(p, batch, "slos_expectations");
    if (st != SLOS_OK) return st;
    if (!p->tab.occ) return fail(SLOS_ERR_UNSUPPORTED, "slos_expectations: plan too large for its occupation table");
    if (batch == 0) return SLOS_OK;
    if (!probs || !out) return fail(SLOS_ERR_INVALID_ARG, "slos_expectations: NULL pointer");
    cudaStream_t s = (cudaStream_t)stream;
    ProfScope ps("slos_expectations", (double)batch * (4.0 * p->K + 4.0 * p->m), s);
    cudaError_t e;
    switch (occ_row(p->m) / 4) {
        case 1: e = launch_expect_fwd<1>(p, probs, batch, out, s); break;
        case 2: e = launch_expect_fwd<2>(p, probs, batch, out, s); break;
        case 3: e = launch_expect_fwd<3>(p, probs, batch, out, s); break;
        case 4: e = launch_expect_fwd<4>(p, probs, batch, out, s); break;
        case 5: e = launch_expect_fwd<5>(p, probs, batch, out, s); break;
        default: e = launch_expect_fwd<6>(p, probs, batch, out, s); break;
    }
    return launched(e, "slos_expectations");
}

slos_status_t slos_expectations_backward(slos_plan_t p, const float *dout, int batch, float *dprobs, void *stream) {
    slos_status_t st = check(p, batch, "slos_expectations_backward");
    if (st != SLOS_OK) return st;
    if (!p->tab.occ)
        return fail(SLOS_ERR_UNSUPPORTED, "slos_expectations_backward: plan too large for its occupation table");
    if (batch == 0) return SLOS_OK;
    if (!dout || !dprobs) return fail(SLOS_ERR_INVALID_ARG, "slos_expectations_backward: NULL pointer");
    cudaStream_t s = (cudaStream_t)stream;
    ProfScope ps("slos_expectations_bwd", (double)batch * (4.0 * p->K + 4.0 * p->m), s);
    cudaError_t e;
    switch (occ_row(p->m) / 4) {
        case 1: e = launch_expect_bwd<1>(p, dout, batch, dprobs, s); break;
        case 2: e = launch_expect_bwd<2>(p, dout, batch, dprobs, s); break;
        case 3: e = launch_expect_bwd<3>(p, dout, batch, dprobs, s); break;
        case 4: e = launch_expect_bwd<4>(p, dout, batch, dprobs, s); break;
        case 5: e = launch_expect_bwd<5>(p, dout, batch, dprobs, s); break;
        default: e = launch_expect_bwd<6>(p, dout, batch, dprobs, s); break;
    }
    return launched(e, "slos_expectations_backward");
}

slos_status_t slos_renormalise(slos_plan_t p, const float *pr, int batch, float *q, float *Z, void *stream) {
    slos_status_t st = check(p, batch, "slos_renormalise");
    if (st != SLOS_OK) return st;
    if (batch == 0) return SLOS_OK;
    if (!pr || !q || !Z) return fail(SLOS_ERR_INVALID_ARG, "slos_renormalise: NULL pointer");
    cudaStream_t s = (cudaStream_t)stream;
    ProfScope ps("slos_renormalise", (double)batch * 8.0 * p->K, s);
    return launched(launch_clusters(renorm_fwd_kernel, renorm_cluster(p), batch, kRenThreads, s, pr, p->K, q, Z),
                    "slos_renormalise");
}

slos_status_t slos_renormalise_backward(slos_plan_t p, const float *q, const float *Z, const float *dq, int batch,
                                        float *dp, void *stream) {
    slos_status_t st = check(p, batch, "slos_renormalise_backward");
    if (st != SLOS_OK) return st;
    if (batch == 0) return SLOS_OK;
    if (!q || !Z || !dq || !dp) return fail(SLOS_ERR_INVALID_ARG, "slos_renormalise_backward: NULL pointer");
    cudaStream_t s = (cudaStream_t)stream;
    ProfScope ps("slos_renormalise_bwd", (double)batch * 12.0 * p->K, s);
    return launched(launch_clusters(renorm_bwd_kernel, renorm_cluster(p), batch, kRenThreads, s, q, Z, dq, p->K, dp),
                    "slos_renormalise_backward");
}

}  // extern "C"
