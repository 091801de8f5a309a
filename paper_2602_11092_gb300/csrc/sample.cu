// Shot sampling from output distributions (the hardware-aware design
// section: MerlinProcessor returns counts of a finite number of shots).
//
// Exact integer inversion of the cumulative distribution: weights are fixed
// point, P(t) = floor(p(t) 2^32); C(t) = P(0) + ... + P(t) and the total T are
// exact 64-bit integers (K < 2^31 weights below 2^32 + 1 each), so no
// summation order can change a decision.  A draw u in [0, 1) becomes the
// target floor(floor(u 2^32) T / 2^32) (a 96-bit product) and the outcome is
// the first t with C(t) > target.  Three kernels: sums of runs of 32 weights,
// an in-place inclusive scan of the run sums per instance, and eight lanes per
// shot that search the run prefix nine ways at a time and then resolve the
// run's 32 weights, four per lane.  Rows of few outcomes take one kernel
// instead (sample_small_kernel).
//
// What bounds it: the shots' dependent reads.  One thread per shot that
// bisected sums of 256 weights and then walked its run took 127 us for 256 x
// 1000 shots over 12,376 outcomes (148 us a call): 32 lanes in 32 different
// rows of memory, up to 256 dependent steps each.  With runs of 32 a run is
// one 128-byte line that eight lanes read at once (51 us a call, most of it
// the host's); the finer prefix costs 8 bytes per 32 weights.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <string>

#include "../../include/slos.h"
#include "plan.h"
#include "profile.h"

namespace slos {
slos_status_t fail(slos_status_t st, const std::string &msg);

constexpr int kSampleRun = 32;                              // weights per entry of the prefix
constexpr int kShotLanes = 8;                               // lanes per shot
constexpr int kLaneWeights = kSampleRun / kShotLanes;       // weights a lane resolves
constexpr int kSumThreads = 256;
constexpr int kSumWeights = 8;                              // consecutive weights per thread of the sums
constexpr int kSumLanes = kSampleRun / kSumWeights;         // threads per run
constexpr int kScanThreads = 1024;
constexpr int kShotThreads = 256;
constexpr int kSmallWeights = 4;                            // weights per thread of the one-kernel form
constexpr int64_t kSmallOutcomes = kShotThreads * kSmallWeights;

__device__ __forceinline__ uint64_t fixed32(float x) {
    return x > 0.f ? __float2ull_rz(x * 4294967296.0f) : 0ull;  // NaN and negatives weigh nothing
}

// floor(floor(x 2^32) T / 2^32)
__device__ __forceinline__ uint64_t shot_target(float x, uint64_t T) {
    const uint64_t U32 = x > 0.f ? (uint64_t)__float2uint_rz(x * 4294967296.0f) : 0ull;  // saturates at 2^32 - 1
    const uint64_t lo64 = T * U32, hi64 = __umul64hi(T, U32);
    return (hi64 << 32) | (lo64 >> 32);
}

// sums[b][r] = weights of run r; clears the counts of the same outcomes.
// Memory-bound: every weight read once (16-byte loads where the rows allow),
// every count written once.
__global__ void __launch_bounds__(kSumThreads) run_sum_kernel(const float *p, int64_t K, int64_t nruns, bool vec,
                                                              uint64_t *sums, int32_t *counts) {
    const int b = blockIdx.y;
    const int64_t c = ((int64_t)blockIdx.x * kSumThreads + threadIdx.x) * kSumWeights;
    const float *pb = p + (size_t)b * K + c;
    int32_t *cb = counts ? counts + (size_t)b * K + c : nullptr;
    uint64_t v = 0;
    if (vec && c + kSumWeights <= K) {
        const float4 x = reinterpret_cast<const float4 *>(pb)[0], y = reinterpret_cast<const float4 *>(pb)[1];
        v = fixed32(x.x) + fixed32(x.y) + fixed32(x.z) + fixed32(x.w) + fixed32(y.x) + fixed32(y.y) + fixed32(y.z) +
            fixed32(y.w);
        if (cb) {
            reinterpret_cast<int4 *>(cb)[0] = make_int4(0, 0, 0, 0);
            reinterpret_cast<int4 *>(cb)[1] = make_int4(0, 0, 0, 0);
        }
    } else {
#pragma unroll
        for (int i = 0; i < kSumWeights; ++i) {
            if (c + i < K) {
                v += fixed32(pb[i]);
                if (cb) cb[i] = 0;
            }
        }
    }
#pragma unroll
    for (int o = kSumLanes / 2; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o, kSumLanes);
    if (threadIdx.x % kSumLanes == 0 && c < K) sums[(size_t)b * nruns + c / kSampleRun] = v;
}

// Inclusive scan of one instance's run sums, in place: tiles of one entry per
// thread (coalesced), scanned by warp shuffles, the warps' totals by warp 0.
__global__ void __launch_bounds__(kScanThreads) run_scan_kernel(uint64_t *sums, int64_t nruns) {
    __shared__ uint64_t tot[kScanThreads / 32];
    uint64_t *row = sums + (size_t)blockIdx.x * nruns;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t carry = 0;
    for (int64_t i0 = 0; i0 < nruns; i0 += kScanThreads) {
        const int64_t i = i0 + threadIdx.x;
        uint64_t v = i < nruns ? row[i] : 0ull;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t w = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += w;
        }
        if (lane == 31) tot[warp] = v;
        __syncthreads();
        if (warp == 0) {
            uint64_t s = tot[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint64_t w = __shfl_up_sync(0xffffffffu, s, o);
                if (lane >= o) s += w;
            }
            tot[lane] = s;
        }
        __syncthreads();
        v += carry + (warp > 0 ? tot[warp - 1] : 0ull);
        if (i < nruns) row[i] = v;
        carry += tot[kScanThreads / 32 - 1];
        __syncthreads();
    }
}

// Eight lanes per shot (a group of the warp; groups run their own loops).
__global__ void __launch_bounds__(kShotThreads) sample_kernel(const float *p, int64_t K, int64_t nruns,
                                                              const uint64_t *prefix, const float *u, int shots,
                                                              int32_t *samples, int32_t *counts) {
    const int b = blockIdx.y;
    const int g = threadIdx.x % kShotLanes;
    const unsigned group = 0xffu << (threadIdx.x & 24);
    const int64_t shot = (int64_t)blockIdx.x * (kShotThreads / kShotLanes) + threadIdx.x / kShotLanes;
    if (shot >= shots) return;
    const size_t idx = (size_t)b * shots + shot;
    const uint64_t *pre = prefix + (size_t)b * nruns;
    const uint64_t T = pre[nruns - 1];
    if (T == 0) {
        if (g == 0) samples[idx] = -1;  // no outcome carries any weight
        return;
    }
    const uint64_t target = shot_target(u[idx], T);
    // first run whose inclusive prefix exceeds the target: [l, h] is cut into
    // nine parts, the lanes read the last entry of the first eight
    int64_t l = 0, h = nruns - 1;
    while (l < h) {
        const int64_t step = (h - l + 9) / 9;
        const int64_t at = l + step * (g + 1) - 1;
        const bool past = at >= h || pre[at] > target;
        const int below = kShotLanes - __popc(__ballot_sync(group, past));
        l += step * below;
        h = min(h, l + step - 1);
    }
    // the run's weights, four per lane, scanned over the group
    const int64_t t0 = l * kSampleRun + g * kLaneWeights;
    const float *pb = p + (size_t)b * K;
    uint64_t w[kLaneWeights], sum = 0;
#pragma unroll
    for (int i = 0; i < kLaneWeights; ++i) {
        w[i] = t0 + i < K ? fixed32(pb[t0 + i]) : 0ull;
        sum += w[i];
    }
    uint64_t incl = sum;
#pragma unroll
    for (int o = 1; o < kShotLanes; o <<= 1) {
        const uint64_t v = __shfl_up_sync(group, incl, o, kShotLanes);
        if (g >= o) incl += v;
    }
    const uint64_t before = (l > 0 ? pre[l - 1] : 0ull) + incl - sum;
    // the run's prefix exceeds the target, so exactly one lane holds the
    // outcome (unless the weights' sum passed 2^64: the run's last state then)
    const bool mine = before <= target && before + sum > target;
    if (__ballot_sync(group, mine) == 0u) {
        const int64_t t = min((l + 1) * (int64_t)kSampleRun, K) - 1;
        if (g == 0) {
            samples[idx] = (int32_t)t;
            if (counts) atomicAdd(counts + (size_t)b * K + t, 1);
        }
    } else if (mine) {
        uint64_t acc = before;
        int t = 0;
#pragma unroll
        for (int i = 0; i < kLaneWeights; ++i) {
            acc += w[i];
            if (acc <= target) t = i + 1;
        }
        samples[idx] = (int32_t)(t0 + t);
        if (counts) atomicAdd(counts + (size_t)b * K + t0 + t, 1);
    }
}

// Rows of up to kSmallOutcomes outcomes: each CTA scans its row into shared
// memory and takes `per` shots, a thread each, by bisection; the counts are
// gathered in shared memory.  One launch instead of three, and no lanes wasted
// on short searches: what bounds it is the shots' reads and writes.  Measured,
// us a call, eight lanes a shot over the prefix in memory / this form: 16 x
// 1,000,000 shots of 10 outcomes 1022 / 54, with counts 5467 / 58; 256 x 1000
// of 330 35 / 4.8; 4096 x 100 of 330 80 / 10.
__global__ void __launch_bounds__(kShotThreads) sample_small_kernel(const float *p, int K, const float *u, int shots,
                                                                    int per, int32_t *samples, int32_t *counts) {
    __shared__ uint64_t C[kSmallOutcomes];
    __shared__ int hist[kSmallOutcomes];
    __shared__ uint64_t tot[kShotThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int b = blockIdx.y;
    const float *pb = p + (size_t)b * K;
    uint64_t w[kSmallWeights], sum = 0;
#pragma unroll
    for (int i = 0; i < kSmallWeights; ++i) {
        const int t = threadIdx.x * kSmallWeights + i;
        w[i] = t < K ? fixed32(pb[t]) : 0ull;
        sum += w[i];
    }
    uint64_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) tot[warp] = incl;
    __syncthreads();
    uint64_t acc = incl - sum;
    for (int q = 0; q < warp; ++q) acc += tot[q];
#pragma unroll
    for (int i = 0; i < kSmallWeights; ++i) {
        const int t = threadIdx.x * kSmallWeights + i;
        acc += w[i];
        if (t < K) {
            C[t] = acc;
            hist[t] = 0;
        }
    }
    __syncthreads();
    const uint64_t T = C[K - 1];
    const int64_t s0 = (int64_t)blockIdx.x * per, s1 = min(s0 + per, (int64_t)shots);
    const size_t row = (size_t)b * shots;
    for (int64_t s = s0 + threadIdx.x; s < s1; s += kShotThreads) {
        if (T == 0) {
            samples[row + s] = -1;  // no outcome carries any weight
            continue;
        }
        const uint64_t target = shot_target(u[row + s], T);
        int l = 0, h = K - 1;
        while (l < h) {
            const int mid = (l + h) >> 1;
            if (C[mid] > target) h = mid;
            else l = mid + 1;
        }
        samples[row + s] = l;
        if (counts) atomicAdd(hist + l, 1);
    }
    if (!counts) return;
    __syncthreads();
    for (int t = threadIdx.x; t < K; t += kShotThreads) {
        int32_t *c = counts + (size_t)b * K + t;
        if (gridDim.x == 1) *c = hist[t];
        else if (hist[t] > 0) atomicAdd(c, hist[t]);
    }
}

static int64_t runs_of(const slos_plan_s *p) { return (p->K + kSampleRun - 1) / kSampleRun; }

}  // namespace slos

using namespace slos;

extern "C" {

slos_status_t slos_sample_workspace_bytes(slos_plan_t p, int batch, size_t *bytes) {
    if (!p || p->kind != 0 || !bytes) return fail(SLOS_ERR_INVALID_ARG, "slos_sample_workspace_bytes: bad argument");
    if (batch < 0) return fail(SLOS_ERR_INVALID_ARG, "slos_sample_workspace_bytes: negative batch");
    *bytes = (size_t)batch * runs_of(p) * sizeof(uint64_t);
    return SLOS_OK;
}

slos_status_t slos_sample(slos_plan_t p, const float *probs, int batch, int shots, const float *uniforms,
                          int32_t *samples, int32_t *counts, void *workspace, size_t workspace_bytes, void *stream) {
    if (!p || p->kind != 0) return fail(SLOS_ERR_INVALID_ARG, "slos_sample: not a single-shape plan");
    if (batch < 0 || shots < 0) return fail(SLOS_ERR_INVALID_ARG, "slos_sample: negative batch or shots");
    if (batch > 65535) return fail(SLOS_ERR_UNSUPPORTED, "slos_sample: at most 65535 instances per call");
    if (batch == 0) return SLOS_OK;
    if (!probs || (shots > 0 && (!uniforms || !samples)))
        return fail(SLOS_ERR_INVALID_ARG, "slos_sample: NULL pointer");
    const int64_t nruns = runs_of(p);
    if (!workspace || workspace_bytes < (size_t)batch * nruns * sizeof(uint64_t))
        return fail(SLOS_ERR_INVALID_ARG, "slos_sample: workspace too small (slos_sample_workspace_bytes)");
    cudaStream_t s = (cudaStream_t)stream;
    uint64_t *pre = reinterpret_cast<uint64_t *>(workspace);
    ProfScope ps("slos_sample", (double)batch * (4.0 * p->K) + (double)batch * shots * 8.0, s);
    cudaError_t e;
    if (p->K <= kSmallOutcomes) {
        // as many CTAs a row as fill the GPU, each with a block of shots at least
        const int blocks = (int)std::min<int64_t>(((int64_t)shots + kShotThreads - 1) / kShotThreads,
                                                  (int64_t)p->sm_count * (2048 / kShotThreads) / batch);
        const int g = std::max(1, blocks);
        if (counts && g > 1 &&
            (e = cudaMemsetAsync(counts, 0, (size_t)batch * p->K * sizeof(int32_t), s)) != cudaSuccess)
            return fail(SLOS_ERR_CUDA, std::string("slos_sample: ") + cudaGetErrorString(e));
        if (shots > 0 || counts)
            sample_small_kernel<<<dim3((unsigned)g, batch), kShotThreads, 0, s>>>(
                probs, (int)p->K, uniforms, shots, (int)(((int64_t)shots + g - 1) / g), samples, counts);
        if ((e = cudaGetLastError()) != cudaSuccess)
            return fail(SLOS_ERR_CUDA, std::string("slos_sample: ") + cudaGetErrorString(e));
        return SLOS_OK;
    }
    // 16-byte accesses where every row starts on a 16-byte boundary
    const bool vec = p->K % 4 == 0 && reinterpret_cast<uintptr_t>(probs) % 16 == 0 &&
                     reinterpret_cast<uintptr_t>(counts) % 16 == 0;
    const int64_t per = (int64_t)kSumThreads * kSumWeights;
    run_sum_kernel<<<dim3((unsigned)((p->K + per - 1) / per), batch), kSumThreads, 0, s>>>(probs, p->K, nruns, vec, pre,
                                                                                           counts);
    run_scan_kernel<<<batch, kScanThreads, 0, s>>>(pre, nruns);
    if (shots > 0) {
        constexpr int kPerBlock = kShotThreads / kShotLanes;
        sample_kernel<<<dim3((unsigned)((shots + kPerBlock - 1) / kPerBlock), batch), kShotThreads, 0, s>>>(
            probs, p->K, nruns, pre, uniforms, shots, samples, counts);
    }
    if ((e = cudaGetLastError()) != cudaSuccess)
        return fail(SLOS_ERR_CUDA, std::string("slos_sample: ") + cudaGetErrorString(e));
    return SLOS_OK;
}

}  // extern "C"
