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
// run's 32 weights, four per lane.
//
// What bounds it: the shots' dependent reads.  One thread per shot that
// bisected sums of 256 weights and then walked its run took 127 us for 256 x
// 1000 shots over 12,376 outcomes (148 us a call): 32 lanes in 32 different
// rows of memory, up to 256 dependent steps each.  With runs of 32 a run is
// one 128-byte line that eight lanes read at once (51 us a call, most of it
// the host's); the finer prefix costs 8 bytes per 32 weights.
#include <cuda_runtime.h>
#include <stdint.h>

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

__device__ __forceinline__ uint64_t fixed32(float x) {
    return x > 0.f ? __float2ull_rz(x * 4294967296.0f) : 0ull;  // NaN and negatives weigh nothing
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
    const float x = u[idx];
    const uint64_t U32 = x > 0.f ? (uint64_t)__float2uint_rz(x * 4294967296.0f) : 0ull;  // saturates at 2^32 - 1
    const uint64_t lo64 = T * U32, hi64 = __umul64hi(T, U32);
    const uint64_t target = (hi64 << 32) | (lo64 >> 32);  // floor(U32 T / 2^32)
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
