// Forward layers of small and middling batches (inference on slot-table plans):
// lane = state.
//
// The two-group walk of slos_pair.cu gives a warp one state of 64 instances,
// so a batch of one pays for 64: 256-byte rows of which 8 bytes are used, and
// 184 us for the 735,000 states of m=16, n=8, whatever the batch up to 64
// (25 us here for one instance, 77 us for 16).
// Here layer k of a group of W = 1, 2 or 4 instances is complex64 [F_k][W] and
// a thread sums one state for its W instances from the same parent slots
// (tables.h): a_k(t) = sum over the parents of U[j, c_k] a_{k-1}(t - e_j)
// (Sec. II-A.2/II-A.3).  Neighbouring states have neighbouring parents (t - e_j
// moves all ranks of a run by the same offset), so a warp's gathers share
// sectors, outputs leave the lanes coalesced without a transposition, and the
// slot rows are read once per W instances.  Bound by L2 gathers and slot-row
// bytes; W = 4 fills a 32-byte sector per parent.
//
// Threshold detection: the final layer's positions are its pattern-grouped
// list order; a warp takes a run of whole patterns (PlanTables::lseg) and adds
// each pattern's states in a fixed order.
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"
#include "slos_kernels.cuh"
#include "tab_launch.h"

namespace slos {

constexpr int kNwThreads = 256;
constexpr int kNwWarps = kNwThreads / 32;
constexpr int kNwUsRow = kMaxModes + 1;  // U column, a zero row past the last mode
constexpr int kNwSum = 64;               // positions of a window whose patterns are summed from shared memory

template <int W>
__device__ __forceinline__ void nw_load(const float2 *p, float2 (&v)[W]) {
    if constexpr (W == 1) {
        v[0] = __ldg(p);
    } else {
#pragma unroll
        for (int i = 0; i < W; i += 2) {
            const float4 x = __ldg(reinterpret_cast<const float4 *>(p) + i / 2);
            v[i] = make_float2(x.x, x.y);
            v[i + 1] = make_float2(x.z, x.w);
        }
    }
}
template <int W>
__device__ __forceinline__ void nw_store(float2 *p, const float2 (&v)[W]) {
    if constexpr (W == 1) {
        p[0] = v[0];
    } else {
#pragma unroll
        for (int i = 0; i < W; i += 2)
            reinterpret_cast<float4 *>(p)[i / 2] = make_float4(v[i].x, v[i].y, v[i + 1].x, v[i + 1].y);
    }
}

// U[j, c_k] of the group's instances, zero past the last mode and the batch.
template <int W>
__device__ __forceinline__ void nw_stage_u(const FwdArgs &a, int g, float2 (*us)[W]) {
    for (int i = threadIdx.x; i < kNwUsRow * W; i += kNwThreads) {
        const int j = i / W, b = g * W + i % W;
        us[j][i % W] =
            (b < a.B && j < a.m) ? a.U[((int64_t)b * a.m + j) * a.m + a.col] : make_float2(0.f, 0.f);
    }
    __syncthreads();
}

// Amplitudes of the state (or list position) c for the group's W instances.
template <int KW, int W>
__device__ __forceinline__ void nw_state(const FwdArgs &a, const uint4 *slots, const float2 (*us)[W], const float2 *prev,
                                         uint32_t c, float2 (&acc)[W]) {
    uint32_t e[KW];
#pragma unroll
    for (int q4 = 0; q4 < KW / 4; ++q4) {
        const uint4 w4 = __ldg(slots + (size_t)c * (KW / 4) + q4);
        e[4 * q4] = w4.x;
        e[4 * q4 + 1] = w4.y;
        e[4 * q4 + 2] = w4.z;
        e[4 * q4 + 3] = w4.w;
    }
    if (a.k == 1) {
#pragma unroll
        for (int i = 0; i < W; ++i) acc[i] = us[e[0] & 31u][i];  // one photon: a_1(e_j) = U[j, c_1]
        return;
    }
#pragma unroll
    for (int i = 0; i < W; ++i) acc[i] = make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < KW; ++q) {
        if (e[q] != kSlotEmpty) {
            float2 v[W];
            nw_load<W>(prev + (size_t)SLOS_IDX(e[q] >> 5, (uint32_t)a.Fprev, a.status) * W, v);
#pragma unroll
            for (int i = 0; i < W; ++i) acc[i] = cfma(us[e[q] & 31u][i], v[i], acc[i]);
        }
    }
}

template <int EPI, int KW, int W>
__global__ void __launch_bounds__(kNwThreads) slos_fwd_narrow_kernel(FwdArgs a, TabArgs t) {
    __shared__ __align__(16) float2 us[kNwUsRow][W];
    const int g = blockIdx.y;
    nw_stage_u<W>(a, g, us);
    const uint32_t c = blockIdx.x * kNwThreads + threadIdx.x;
    if (c >= (uint32_t)a.Fk) return;
    float2 acc[W];
    nw_state<KW, W>(a, reinterpret_cast<const uint4 *>(t.slots), us, a.prev + (size_t)g * a.Fprev * W, c, acc);
    if (EPI == EPI_STORE) {
        nw_store<W>(a.next + ((size_t)g * a.Fk + c) * W, acc);
        return;
    }
    const float w = __ldg(t.w + c);
#pragma unroll
    for (int i = 0; i < W; ++i) {
        const int b = g * W + i;
        if (b >= a.B) break;
        if (EPI == EPI_PROBS)
            reinterpret_cast<float *>(a.out)[(size_t)b * a.K + c] = w * cabs2(acc[i]);
        else
            reinterpret_cast<float2 *>(a.out)[(size_t)b * a.K + c] = cscale(acc[i], sqrtf(w));
    }
}

template <int KW, int W>
__global__ void __launch_bounds__(kNwThreads) slos_fwd_narrow_thresh_kernel(FwdArgs a, TabArgs t) {
    __shared__ __align__(16) float2 us[kNwUsRow][W];
    __shared__ float p[kNwWarps][W][kNwSum], wt[kNwWarps][kNwSum];  // |a_n|^2 and weight of a window of positions
    const int g = blockIdx.y;
    nw_stage_u<W>(a, g, us);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int item = blockIdx.x * kNwWarps + warp;
    if (item >= t.nseg) return;
    const int lo = __ldg(t.lseg + item), n = __ldg(t.lseg + item + 1) - lo;
    const int pat0 = __ldg(t.lpat + lo), npat = __ldg(t.lpat + lo + n - 1) - pat0 + 1;
    const float2 *prev = a.prev + (size_t)g * a.Fprev * W;
    float *out = reinterpret_cast<float *>(a.out);
    // an item of more than one window is one pattern; lane i < W sums instance i
    float run = 0.f;
    for (int s0 = 0; s0 < n; s0 += kNwSum) {
        const int ns = min(kNwSum, n - s0);
        for (int s = lane; s < ns; s += 32) {
            float2 acc[W];
            const uint32_t c = (uint32_t)(lo + s0 + s);
            nw_state<KW, W>(a, reinterpret_cast<const uint4 *>(t.slots), us, prev, c, acc);
            wt[warp][s] = __ldg(t.w + c);
#pragma unroll
            for (int i = 0; i < W; ++i) p[warp][i][s] = cabs2(acc[i]);
        }
        __syncwarp();
        // each pattern's states in list order, the sum the two-group walk takes
        if (n <= kNwSum) {
            const int cnt = n / npat;  // the patterns of an item have the same number of states
            for (int x = lane; x < npat * W; x += 32) {
                const int i = x / npat, q = x % npat, b = g * W + i;
                if (b >= a.B) break;
                float s = 0.f;
                for (int r = 0; r < cnt; ++r) s = __fmaf_rn(wt[warp][q * cnt + r], p[warp][i][q * cnt + r], s);
                out[(size_t)b * a.K + pat0 + q] = s;
            }
        } else if (lane < W) {
            for (int r = 0; r < ns; ++r) run = __fmaf_rn(wt[warp][r], p[warp][lane][r], run);
        }
        __syncwarp();
    }
    if (n > kNwSum && lane < W && g * W + lane < a.B) out[(size_t)(g * W + lane) * a.K + pat0] = run;
}

template <int KW, int W>
static cudaError_t launch_narrow(const FwdArgs &a, const TabArgs &t, int epi, cudaStream_t s) {
    const unsigned groups = (unsigned)((a.B + W - 1) / W);
    const dim3 grid((unsigned)((a.Fk + kNwThreads - 1) / kNwThreads), groups);
    switch (epi) {
        case EPI_STORE: slos_fwd_narrow_kernel<EPI_STORE, KW, W><<<grid, kNwThreads, 0, s>>>(a, t); break;
        case EPI_PROBS: slos_fwd_narrow_kernel<EPI_PROBS, KW, W><<<grid, kNwThreads, 0, s>>>(a, t); break;
        case EPI_AMPS: slos_fwd_narrow_kernel<EPI_AMPS, KW, W><<<grid, kNwThreads, 0, s>>>(a, t); break;
        case EPI_THRESH:
            slos_fwd_narrow_thresh_kernel<KW, W>
                <<<dim3((unsigned)((t.nseg + kNwWarps - 1) / kNwWarps), groups), kNwThreads, 0, s>>>(a, t);
            break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <int W>
static cudaError_t launch_narrow_kw(const FwdArgs &a, const TabArgs &t, int epi, cudaStream_t s) {
    switch (t.kw) {
        case 4: return launch_narrow<4, W>(a, t, epi, s);
        case 8: return launch_narrow<8, W>(a, t, epi, s);
        case 12: return launch_narrow<12, W>(a, t, epi, s);
        default: return cudaErrorInvalidValue;
    }
}

int slos_narrow_width(int batch) { return batch == 1 ? 1 : (batch == 2 ? 2 : 4); }

cudaError_t slos_launch_fwd_narrow(const FwdArgs &a, const TabArgs &t, int epi, int width, cudaStream_t s) {
    switch (width) {
        case 1: return launch_narrow_kw<1>(a, t, epi, s);
        case 2: return launch_narrow_kw<2>(a, t, epi, s);
        case 4: return launch_narrow_kw<4>(a, t, epi, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace slos
