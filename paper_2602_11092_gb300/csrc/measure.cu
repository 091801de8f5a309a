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
// expectations 44.2 -> 15 us, their backward 35.8 -> 9.5 us.
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

// Renormalisation: T threads a row, KEEP values of it per thread in registers
// between the sum and the division (what is left of longer rows is read again),
// rows of fewer than 128 threads sharing a CTA.  A row's sum is a chain of
// double-float additions (20 instructions each) per thread and one over its
// lanes and warps, so short rows want few threads (many rows in flight, no
// barrier) and long ones want many; renorm_launch has the lines.
constexpr int kRenLong = 512;  // threads of the longest rows, which may also split over a cluster

// Sum of one double-float per thread over a row's T threads (and its cluster),
// fixed order (a tree over the lanes, the warps and the ranks); every thread
// of the row gets it.
__device__ __forceinline__ dfl warp_sum(dfl v, int width) {
    for (int o = width / 2; o > 0; o >>= 1) {
        const dfl w = {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
        v = df_add(v, w);
    }
    return v;
}
__device__ __forceinline__ dfl lane0(dfl v) {
    return {__shfl_sync(0xffffffffu, v.hi, 0), __shfl_sync(0xffffffffu, v.lo, 0)};
}
template <int T>
__device__ __forceinline__ dfl row_sum(dfl v, dfl *red, dfl *part) {
    v = warp_sum(v, 32);
    if constexpr (T > 32) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        if (lane == 0) red[warp] = v;
        __syncthreads();
        // the row's T / 32 warps are the CTA's
        v = lane0(warp_sum(lane < T / 32 ? red[lane] : df_zero(), T / 32));
        if (T == kRenLong && gridDim.x > 1) {
            cg::cluster_group cluster = cg::this_cluster();
            if (threadIdx.x == 0) *part = v;
            cluster.sync();
            v = df_zero();
            if (lane < (int)gridDim.x) v = *cluster.map_shared_rank(part, lane);
            v = lane0(warp_sum(v, kMaxCluster));
            cluster.sync();  // no CTA leaves while its partial sum is read
        }
    }
    return v;
}

// The slice of a row that this thread's CTA of the cluster (or its part of the CTA) takes.
template <int T>
struct RenRow {
    static constexpr int kThreads = T < 128 ? 128 : T;
    int b, tid;
    int64_t lo, n;  // first value, values (none for rows past the batch)
    __device__ RenRow(int64_t K, int B) {
        tid = threadIdx.x % T;
        b = blockIdx.y * (kThreads / T) + threadIdx.x / T;
        const int64_t per = (K + gridDim.x - 1) / gridDim.x;
        lo = per * blockIdx.x;
        n = b < B ? min(K, lo + per) - lo : 0;
    }
};

// Z = sum_t p[t]; q[t] = p[t] / Z  (sums in double-float, dfloat.cuh).  q may be p.
template <int T, int KEEP>
__global__ void __launch_bounds__(RenRow<T>::kThreads) renorm_fwd_kernel(const float *p, int64_t K, int B, float *q,
                                                                         float *Z) {
    __shared__ dfl red[RenRow<T>::kThreads / 32], part;
    const RenRow<T> r(K, B);
    const float *pb = p + (size_t)r.b * K + r.lo;
    float keep[KEEP];
#pragma unroll
    for (int i = 0; i < KEEP; ++i) {
        const int64_t c = r.tid + (int64_t)i * T;
        keep[i] = c < r.n ? pb[c] : 0.f;
    }
    // pairs first (exact), in independent chains: the additions of one chain
    // wait 20 instructions for each other
    constexpr int kChains = KEEP >= 8 ? 4 : 1;
    dfl chain[kChains];
#pragma unroll
    for (int i = 0; i < KEEP / 2; ++i) {
        const dfl pair = two_sum(keep[2 * i], keep[2 * i + 1]);
        chain[i % kChains] = i < kChains ? pair : df_add(chain[i % kChains], pair);
    }
    dfl acc = chain[0];
    if constexpr (kChains == 4) acc = df_add(df_add(chain[0], chain[1]), df_add(chain[2], chain[3]));
    const int64_t rest = r.tid + (int64_t)KEEP * T;
#pragma unroll 4
    for (int64_t c = rest; c < r.n; c += T) acc = df_add_f(acc, pb[c]);
    const float z = df_float(row_sum<T>(acc, red, &part));
    const float inv = z > 0.f ? 1.f / z : 0.f;
    float *qb = q + (size_t)r.b * K + r.lo;
#pragma unroll
    for (int i = 0; i < KEEP; ++i) {
        const int64_t c = r.tid + (int64_t)i * T;
        if (c < r.n) qb[c] = keep[i] * inv;
    }
    for (int64_t c = rest; c < r.n; c += T) qb[c] = pb[c] * inv;
    if (blockIdx.x == 0 && r.tid == 0 && r.b < B) Z[r.b] = z;
}

// dp[t] = (dq[t] - sum_s dq[s] q[s]) / Z.  dp may be dq.
template <int T, int KEEP>
__global__ void __launch_bounds__(RenRow<T>::kThreads) renorm_bwd_kernel(const float *q, const float *Z, const float *dq,
                                                                         int64_t K, int B, float *dp) {
    __shared__ dfl red[RenRow<T>::kThreads / 32], part;
    const RenRow<T> r(K, B);
    const float *qb = q + (size_t)r.b * K + r.lo, *dqb = dq + (size_t)r.b * K + r.lo;
    float keep[KEEP], qv[KEEP];
#pragma unroll
    for (int i = 0; i < KEEP; ++i) {
        const int64_t c = r.tid + (int64_t)i * T;
        keep[i] = c < r.n ? dqb[c] : 0.f;
        qv[i] = c < r.n ? qb[c] : 0.f;
    }
    const float z = r.b < B ? Z[r.b] : 0.f;
    constexpr int kChains = KEEP >= 8 ? 4 : 1;
    dfl chain[kChains];
#pragma unroll
    for (int i = 0; i < KEEP; ++i) {
        const dfl prod = two_prod(keep[i], qv[i]);
        chain[i % kChains] = i < kChains ? prod : df_add(chain[i % kChains], prod);
    }
    dfl acc = chain[0];
    if constexpr (kChains == 4) acc = df_add(df_add(chain[0], chain[1]), df_add(chain[2], chain[3]));
    const int64_t rest = r.tid + (int64_t)KEEP * T;
#pragma unroll 4
    for (int64_t c = rest; c < r.n; c += T) acc = df_add(acc, two_prod(dqb[c], qb[c]));
    const float sdot = df_float(row_sum<T>(acc, red, &part));
    const float inv = z > 0.f ? 1.f / z : 0.f;
    float *dpb = dp + (size_t)r.b * K + r.lo;
#pragma unroll
    for (int i = 0; i < KEEP; ++i) {
        const int64_t c = r.tid + (int64_t)i * T;
        if (c < r.n) dpb[c] = (keep[i] - sdot) * inv;
    }
    for (int64_t c = rest; c < r.n; c += T) dpb[c] = (dqb[c] - sdot) * inv;
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
    cfg.numAttrs = cluster > 1 ? 1 : 0;  // a grid of single CTAs launches without
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// Calls f.run<T, KEEP>(cluster, CTAs) with the shape for rows of K outputs.
// Measured, us, forward / backward (a warp a row, 128, 256 and 512 threads):
//   65,535 rows of 10: warp x 2 values 16 / 18, x 8 25 / 31, 512 x 16 629 / 811
//   65,535 of 120: x 8 24 / 31, x 16 33 / 46;  of 330: x 16 37 / 50, x 32 56 / 81
//   65,535 of 1001: x 32 76 / 117, 128 x 16 145 / 190;  16,384 of 2002: 61 / 96, 44 / 60
//   4096 of 4368: 256 x 16 29 / 39, 512 x 16 43 / 59;  of 8008: 256 x 32 43 / 61, 512 x 16 48 / 71
//   4096 of 12,376: 512 x 16, the rest read again, 77 / 118, two CTAs 113 / 161
// Clusters pay where a CTA would walk more than 32,768 values (1000 rows of
// 54,264: one CTA 173 / 251, two 112 / 167) and for few rows (one of 54,264:
// 20 / 25, eight CTAs 4.7 / 5.2).
template <typename F>
static cudaError_t renorm_launch(const slos_plan_s *p, int batch, F f) {
    const int64_t K = p->K;
    if (K <= 64) return f.template run<32, 2>(1, (batch + 3) / 4);
    if (K <= 256) return f.template run<32, 8>(1, (batch + 3) / 4);
    if (K <= 512) return f.template run<32, 16>(1, (batch + 3) / 4);
    if (K <= 1024) return f.template run<32, 32>(1, (batch + 3) / 4);
    if (K <= 2048) return f.template run<128, 16>(1, batch);
    if (K <= 4608) return f.template run<256, 16>(1, batch);
    if (K <= 8192) return f.template run<256, 32>(1, batch);
    int c = 1;
    while (c < kMaxCluster &&
           (K / c > 32768 || ((int64_t)2 * c * batch <= p->sm_count && K / (2 * c) >= 4096)))
        c *= 2;
    return f.template run<kRenLong, 16>(c, batch);
}
struct RenormFwd {
    const float *p;
    int64_t K;
    int B;
    float *q, *Z;
    cudaStream_t s;
    template <int T, int KEEP>
    cudaError_t run(int cluster, int rows) const {
        return launch_clusters(renorm_fwd_kernel<T, KEEP>, cluster, rows, RenRow<T>::kThreads, s, p, K, B, q, Z);
    }
};
struct RenormBwd {
    const float *q, *Z, *dq;
    int64_t K;
    int B;
    float *dp;
    cudaStream_t s;
    template <int T, int KEEP>
    cudaError_t run(int cluster, int rows) const {
        return launch_clusters(renorm_bwd_kernel<T, KEEP>, cluster, rows, RenRow<T>::kThreads, s, q, Z, dq, K, B, dp);
    }
};

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
    return launched(renorm_launch(p, batch, RenormFwd{pr, p->K, batch, q, Z, s}), "slos_renormalise");
}

slos_status_t slos_renormalise_backward(slos_plan_t p, const float *q, const float *Z, const float *dq, int batch,
                                        float *dp, void *stream) {
    slos_status_t st = check(p, batch, "slos_renormalise_backward");
    if (st != SLOS_OK) return st;
    if (batch == 0) return SLOS_OK;
    if (!q || !Z || !dq || !dp) return fail(SLOS_ERR_INVALID_ARG, "slos_renormalise_backward: NULL pointer");
    cudaStream_t s = (cudaStream_t)stream;
    ProfScope ps("slos_renormalise_bwd", (double)batch * 12.0 * p->K, s);
    return launched(renorm_launch(p, batch, RenormBwd{q, Z, dq, p->K, batch, dp, s}), "slos_renormalise_backward");
}

}  // extern "C"
