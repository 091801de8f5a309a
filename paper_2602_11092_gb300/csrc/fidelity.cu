// Fidelity kernel (kernel-methods section): with the embedding
// |phi(x)> = U(x)|s> of a Fock input s,
//     K[i][j] = |<phi_a(i)|phi_b(j)>|^2 = |<s|Ua[i]^dag Ub[j]|s>|^2,
// and for a Fock state <s|V|s> = Per(W) / prod_i s_i! with the n x n matrix
// W[a][b] = V[c_a][c_b] = sum_k conj(Ua[i][k][c_a]) Ub[j][k][c_b] over the
// photon columns c_1 <= ... <= c_n.
//
// The photon columns of a tile's 16 + 16 unitaries are staged in shared memory;
// W is formed in FP32 (each entry an m-term inner product) and kept in
// registers, one pair per thread.  The permanent runs in
// double-float arithmetic (dfloat.cuh, about 44 bits on the FP32 pipe), and the
// FP32 pipe's instruction rate is what bounds the kernel: W costs about 1,700
// instructions a pair at n = 6, the permanent several times that.  Two forms:
//
// * n <= 6 (fid_subset_kernel): Laplace's expansion over the two halves of the
//   rows, Per(W) = sum_S Per(W[top, S]) Per(W[bottom, not S]) over the column
//   subsets S of size floor(n / 2), each half's permanents built row by row
//   (Per over S = sum over c in S of W[r][c] Per over S - c).  At n = 6 that is
//   200 complex products against 160 for Glynn's formula, but all but 20 have
//   a float factor, and sums keep their rounding errors in a second float
//   (two_sum) renormalised once per sum: about 8,600 operations a pair
//   against 16,600.  The top half's permanents wait in shared memory.
// * n = 7, 8 (fidelity_kernel), where the subsets outgrow the registers:
//   Glynn's formula
//     Per(W) = 2^(1-n) sum_{delta in {+-1}^n, delta_1 = 1} (prod_a delta_a)
//              prod_b (sum_a delta_a W[a][b])
//   walked in Gray-code order (one row sum update per term).  Its terms reach
//   about n^n / 2^(n-1) while the permanent of a block of a unitary is at most
//   1, so FP32 sums would lose the result.  The updates add +-2 W[r][c], exact
//   in float.
//
// A set against itself (Ub the same array as Ua) is symmetric: only the tiles
// on and above the diagonal are computed and each is written twice.  1024
// points, m = 12, n = 6: 625 us with Glynn's formula on every tile, 257 us with
// the subset expansion in scalar code (waiting for instruction fetch), 229 us
// with packed pairs, 214 us with the warps of a CTA kept together by barriers
// (the FP32 pipe 59 % busy).
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <string>
#include <utility>

#include "../../include/slos.h"
#include "common.cuh"
#include "dfloat.cuh"
#include "profile.h"

namespace slos {
slos_status_t fail(slos_status_t st, const std::string &msg);

constexpr int kFidTile = 16;
constexpr int kFidMaxPhotons = 8;

struct FidArgs {
    const float2 *Ua, *Ub;
    float *K;
    int m, Na, Nb;
    int cols[kFidMaxPhotons];
    float inv_sf2;   // 1 / (prod s_i!)^2
    bool sym;        // Ub is Ua: tiles on and above the diagonal, written twice
};

__device__ __forceinline__ void fid_tile(int Nb, bool sym, uint32_t b, int &ti, int &tj);
// blockIdx.x, read anew at each use (the compiler keeps nothing derived from it)
__device__ __forceinline__ uint32_t fid_block() {
    uint32_t b;
    asm volatile("mov.u32 %0, %%ctaid.x;" : "=r"(b));
    return b;
}

template <int N>
__global__ void __launch_bounds__(kFidTile *kFidTile) fidelity_kernel(FidArgs a) {
    extern __shared__ float2 sm[];
    const int m = a.m;
    float2 *wa = sm;                              // [16][m][N]
    float2 *wb = sm + (size_t)kFidTile * m * N;   // [16][m][N]
    int ti, tj;
    fid_tile(a.Nb, a.sym, fid_block(), ti, tj);
    const int i0 = ti * kFidTile, j0 = tj * kFidTile;
    const int tid = threadIdx.y * kFidTile + threadIdx.x;
    const int per = m * N;
    for (int idx = tid; idx < kFidTile * per; idx += kFidTile * kFidTile) {
        const int t = idx / per, r = idx % per, k = r / N, c = r % N;
        const int col = a.cols[c];
        wa[idx] = (i0 + t < a.Na) ? a.Ua[((size_t)(i0 + t) * m + k) * m + col] : make_float2(0.f, 0.f);
        wb[idx] = (j0 + t < a.Nb) ? a.Ub[((size_t)(j0 + t) * m + k) * m + col] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    if (i0 + (int)threadIdx.y >= a.Na || j0 + (int)threadIdx.x >= a.Nb) return;
    const float2 *pa = wa + (size_t)threadIdx.y * per, *pb = wb + (size_t)threadIdx.x * per;
    float2 W[N][N];
#pragma unroll
    for (int r = 0; r < N; ++r)
#pragma unroll
        for (int c = 0; c < N; ++c) W[r][c] = make_float2(0.f, 0.f);
    for (int k = 0; k < m; ++k) {
#pragma unroll
        for (int r = 0; r < N; ++r) {
            const float2 x = pa[k * N + r];
#pragma unroll
            for (int c = 0; c < N; ++c) W[r][c] = cfma_conj_a(x, pb[k * N + c], W[r][c]);
        }
    }
    // Glynn, Gray-code order over delta_2..delta_N (bit q-1 of d: delta_{q+1} = -1)
    cdfl S[N];
#pragma unroll
    for (int c = 0; c < N; ++c) {
        S[c] = {df_zero(), df_zero()};
#pragma unroll
        for (int r = 0; r < N; ++r) {
            S[c].re = df_add_f(S[c].re, W[r][c].x);
            S[c].im = df_add_f(S[c].im, W[r][c].y);
        }
    }
    auto product = [&]() {
        cdfl pr = S[0];
#pragma unroll
        for (int c = 1; c < N; ++c) pr = cdf_mul(pr, S[c]);
        return pr;
    };
    cdfl t = product();
    uint32_t d = 0;
    for (uint32_t g = 1; g < (1u << (N - 1)); ++g) {
        const int q = __ffs(g);  // flips delta_{q+1}, row q of W (1-based bit index q)
        d ^= 1u << (q - 1);
        const float sgn = ((d >> (q - 1)) & 1u) ? -2.f : 2.f;
#pragma unroll
        for (int r = 1; r < N; ++r) {
            if (r == q) {
#pragma unroll
                for (int c = 0; c < N; ++c) {
                    S[c].re = df_add_f(S[c].re, sgn * W[r][c].x);
                    S[c].im = df_add_f(S[c].im, sgn * W[r][c].y);
                }
            }
        }
        const cdfl pr = product();
        t = (__popc(d) & 1) ? cdf_sub(t, pr) : cdf_add(t, pr);
    }
    const float scale = 1.f / (float)(1u << (N - 1));
    const float tr = df_float(t.re) * scale, tim = df_float(t.im) * scale;
    const float v = (tr * tr + tim * tim) * a.inv_sf2;
    // the tile once more: its two registers held through the sums cost 2-6 %
    // (one pair, n = 8: 113 us, now 107)
    fid_tile(a.Nb, a.sym, fid_block(), ti, tj);
    const int i = ti * kFidTile + threadIdx.y, j = tj * kFidTile + threadIdx.x;
    if (a.sym && i > j) return;  // the mirrored entry of a diagonal tile
    a.K[(size_t)i * a.Nb + j] = v;
    if (a.sym && i < j) a.K[(size_t)j * a.Nb + i] = v;
}

// Tile (row, column) of block `b` (a grid's x extent is below 2^31): all tiles,
// or the upper triangle row by row (row r of the triangle starts at
// r T - r (r - 1) / 2 for T tiles a side).
__device__ __forceinline__ void fid_tile(int Nb, bool sym, uint32_t b, int &ti, int &tj) {
    const uint32_t T = (uint32_t)(Nb + kFidTile - 1) / kFidTile;
    if (!sym) {
        ti = (int)(b / T);
        tj = (int)(b % T);
        return;
    }
    uint32_t lo = 0, hi = T - 1;  // the last row that starts at or before b
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) / 2;
        if ((uint64_t)mid * T - (uint64_t)mid * (mid - 1) / 2 <= b) lo = mid;
        else hi = mid - 1;
    }
    ti = (int)lo;
    tj = (int)(lo + (b - (uint32_t)((uint64_t)lo * T - (uint64_t)lo * (lo - 1) / 2)));
}

// ------------------------------------------------------------ subsets of columns
constexpr int fid_popc(int mask) {
    int c = 0;
    for (; mask; mask &= mask - 1) ++c;
    return c;
}
constexpr int fid_binom(int n, int k) {
    int r = 1;
    for (int i = 1; i <= k; ++i) r = r * (n - k + i) / i;
    return r;
}
// The r-th k-subset of n columns as a bitmask (increasing), and its inverse.
constexpr int fid_subset(int n, int k, int r) {
    for (int mask = 0; mask < (1 << n); ++mask)
        if (fid_popc(mask) == k && r-- == 0) return mask;
    return 0;
}
constexpr int fid_rank(int mask) {
    int r = 0;
    for (int q = 0; q < mask; ++q) r += fid_popc(q) == fid_popc(mask) ? 1 : 0;
    return r;
}
constexpr int fid_column(int mask, int i) {
    for (int c = 0;; ++c)
        if ((mask >> c) & 1)
            if (i-- == 0) return c;
}

// The two parts of a complex value take the same operations, so they travel as
// packed pairs (add/sub/mul/fma.f32x2, each part rounded to nearest): half the
// instructions of scalar code, which had the kernel waiting for instruction
// fetch (its body is straight-line code for every subset).
__device__ __forceinline__ uint64_t f2_pack(float2 a) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
    return r;
}
__device__ __forceinline__ float2 f2_unpack(uint64_t a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
}
__device__ __forceinline__ uint64_t f2_swap(uint64_t a) {
    const float2 v = f2_unpack(a);
    return f2_pack(make_float2(v.y, v.x));
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t f2_sub(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Complex double-float, the parts packed: (re, im) = hi + lo.
struct FidVal {
    uint64_t hi, lo;
};
// A sum with the rounding errors of hi's additions collected in lo.
struct FidSum {
    uint64_t s, c;
};
// A factor f as pairs for f.re * (re, im) and f.im * (-im, re), and negated.
struct FidFactor {
    uint64_t re, nre, im, nim;
};
__device__ __forceinline__ FidFactor fid_factor(float2 f) {
    return {f2_pack(make_float2(f.x, f.x)), f2_pack(make_float2(-f.x, -f.x)), f2_pack(make_float2(-f.y, f.y)),
            f2_pack(make_float2(f.y, -f.y))};
}
// a += f * (hi + lo), part by part (f exact floats, nf = -f); LO: lo is not zero
template <bool FIRST, bool LO>
__device__ __forceinline__ void fid_mac(FidSum &a, uint64_t f, uint64_t nf, uint64_t hi, uint64_t lo) {
    const uint64_t p = f2_mul(f, hi);
    uint64_t ne = f2_fma(nf, hi, p);  // p - f hi: minus the product's rounding error
    if (LO) ne = f2_fma(nf, lo, ne);
    if (FIRST) {
        a.s = p;
        a.c = f2_sub(0ull, ne);
    } else {
        const uint64_t s = f2_add(a.s, p);
        const uint64_t bb = f2_sub(s, a.s);
        const uint64_t e = f2_add(f2_sub(a.s, f2_sub(s, bb)), f2_sub(p, bb));  // two_sum's error
        a.s = s;
        a.c = f2_add(a.c, f2_sub(e, ne));
    }
}
__device__ __forceinline__ FidVal fid_value(FidSum a) {
    const uint64_t s = f2_add(a.s, a.c);
    const uint64_t bb = f2_sub(s, a.s);
    return {s, f2_add(f2_sub(a.s, f2_sub(s, bb)), f2_sub(a.c, bb))};
}
// a += f * v
template <bool FIRST, bool LO>
__device__ __forceinline__ void fid_cmac(FidSum &a, const FidFactor &f, FidVal v) {
    fid_mac<FIRST, LO>(a, f.re, f.nre, v.hi, v.lo);
    fid_mac<false, LO>(a, f.im, f.nim, f2_swap(v.hi), LO ? f2_swap(v.lo) : 0ull);
}

// Permanents over the column subsets of one half's rows 0..K-1.
template <int N, int K>
struct FidLevel {
    FidVal v[fid_binom(N, K)];
};

// Subset R of level K from the permanents of level K - 1 and row `w`, or (two
// rows of floats) from the row before.
template <int N, int K, int R, int... I>
__device__ __forceinline__ FidVal fid_expand(const FidFactor (&w)[N], const FidLevel<N, K - 1> &prev,
                                             std::integer_sequence<int, I...>) {
    constexpr int mask = fid_subset(N, K, R);
    FidSum a;
    (fid_cmac<I == 0, true>(a, w[fid_column(mask, I)], prev.v[fid_rank(mask ^ (1 << fid_column(mask, I)))]), ...);
    return fid_value(a);
}
template <int N, int R>
__device__ __forceinline__ FidVal fid_pair(const uint64_t (&w0)[N], const FidFactor (&w1)[N]) {
    constexpr int mask = fid_subset(N, 2, R);
    constexpr int c0 = fid_column(mask, 0), c1 = fid_column(mask, 1);
    FidSum a;
    fid_cmac<true, false>(a, w1[c0], {w0[c1], 0ull});
    fid_cmac<false, false>(a, w1[c1], {w0[c0], 0ull});
    return fid_value(a);
}
template <int N, int... R>
__device__ __forceinline__ void fid_level2(const uint64_t (&w0)[N], const FidFactor (&w1)[N], FidLevel<N, 2> &out,
                                           std::integer_sequence<int, R...>) {
    ((out.v[R] = fid_pair<N, R>(w0, w1)), ...);
}
// Permanent of subset R over ROWS >= 1 rows: w0 the first row, last the last
// one, prev the level before (ROWS >= 3).
template <int N, int ROWS, int R>
__device__ __forceinline__ FidVal fid_perm(const uint64_t (&w0)[N], const FidFactor (&last)[N],
                                           const FidLevel<N, ROWS - 1> &prev) {
    if constexpr (ROWS == 1) return {w0[fid_column(fid_subset(N, 1, R), 0)], 0ull};
    else if constexpr (ROWS == 2) return fid_pair<N, R>(w0, last);
    else return fid_expand<N, ROWS, R>(last, prev, std::make_integer_sequence<int, ROWS>());
}

// total += a * b in double-float
__device__ __forceinline__ void fid_total(cdfl &total, FidVal a, FidVal b) {
    const float2 ah = f2_unpack(a.hi), al = f2_unpack(a.lo), bh = f2_unpack(b.hi), bl = f2_unpack(b.lo);
    total = cdf_add(total, cdf_mul({{ah.x, al.x}, {ah.y, al.y}}, {{bh.x, bl.x}, {bh.y, bl.y}}));
}

constexpr int kFidThreads = 256;  // a 16 x 16 tile, one pair per thread
constexpr int kFidSync = 4;       // subsets between the barriers that keep the CTA's warps together

// Half of the expansion over ROWS rows: the top half leaves its permanents in
// `kept` (one column per thread), the bottom half multiplies them with its own
// (of the complementary columns) into the total.
template <int N, int ROWS, int R>
__device__ __forceinline__ void fid_term(const uint64_t (&w0)[N], const FidFactor (&last)[N],
                                         const FidLevel<N, ROWS - 1> &prev, bool top, ulonglong2 *kept, cdfl &total) {
    if (N >= 5 && R > 0 && R % kFidSync == 0) __syncthreads();
    const FidVal v = fid_perm<N, ROWS, R>(w0, last, prev);
    if (top) {
        kept[R * kFidThreads] = make_ulonglong2(v.hi, v.lo);
    } else {
        constexpr int other = fid_rank(((1 << N) - 1) ^ fid_subset(N, ROWS, R));
        const ulonglong2 k = kept[other * kFidThreads];
        fid_total(total, {k.x, k.y}, v);
    }
}
template <int N, int ROWS, int... R>
__device__ __forceinline__ void fid_half(const uint64_t (&w0)[N], const FidFactor (&last)[N],
                                         const FidLevel<N, ROWS - 1> &prev, bool top, ulonglong2 *kept, cdfl &total,
                                         std::integer_sequence<int, R...>) {
    (fid_term<N, ROWS, R>(w0, last, prev, top, kept, total), ...);
}

// Rows r0 .. r0 + ROWS - 1 of W, then their permanents.
template <int N, int ROWS>
__device__ __forceinline__ void fid_rows(const float2 *pa, const float2 *pb, int m, int r0, bool top, ulonglong2 *kept,
                                         cdfl &total) {
    if constexpr (ROWS == 0) {
        kept[0] = make_ulonglong2(f2_pack(make_float2(1.f, 0.f)), 0ull);
    } else {
        float2 W[ROWS][N];
#pragma unroll
        for (int r = 0; r < ROWS; ++r)
#pragma unroll
            for (int c = 0; c < N; ++c) W[r][c] = make_float2(0.f, 0.f);
        for (int k = 0; k < m; ++k) {
            float2 y[N];
#pragma unroll
            for (int c = 0; c < N; ++c) y[c] = pb[k * N + c];
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const float2 x = pa[k * N + r0 + r];
#pragma unroll
                for (int c = 0; c < N; ++c) W[r][c] = cfma_conj_a(x, y[c], W[r][c]);
            }
        }
        static_assert(ROWS <= 3, "halves of at most three rows");
        uint64_t w0[N];
        FidFactor f[N];
#pragma unroll
        for (int c = 0; c < N; ++c) w0[c] = f2_pack(W[0][c]);
        FidLevel<N, ROWS - 1> prev;
        if constexpr (ROWS == 3) {
#pragma unroll
            for (int c = 0; c < N; ++c) f[c] = fid_factor(W[1][c]);
            fid_level2<N>(w0, f, prev, std::make_integer_sequence<int, fid_binom(N, 2)>());
        }
#pragma unroll
        for (int c = 0; c < N; ++c) f[c] = fid_factor(W[ROWS - 1][c]);
        fid_half<N, ROWS>(w0, f, prev, top, kept, total, std::make_integer_sequence<int, fid_binom(N, ROWS)>());
    }
}

template <int N>
__global__ void __launch_bounds__(kFidThreads, 2) fid_subset_kernel(FidArgs a) {
    constexpr int TOP = N / 2, BOT = N - TOP;
    extern __shared__ float4 fid_sm[];
    const int m = a.m;
    const int per = (m * N) | 1;  // odd rows: the 16 columns' reads fall into distinct banks
    ulonglong2 *kept = reinterpret_cast<ulonglong2 *>(fid_sm) + threadIdx.x;            // [C(N, TOP)][threads]
    float2 *wa = reinterpret_cast<float2 *>(fid_sm + fid_binom(N, TOP) * kFidThreads);  // [16][per]
    float2 *wb = wa + kFidTile * per;
    int ti, tj;
    fid_tile(a.Nb, a.sym, blockIdx.x, ti, tj);
    const int i0 = ti * kFidTile, j0 = tj * kFidTile;
    for (int idx = threadIdx.x; idx < kFidTile * m * N; idx += kFidThreads) {
        const int t = idx / (m * N), r = idx % (m * N), k = r / N, c = r % N;
        const int col = a.cols[c];
        wa[t * per + r] = (i0 + t < a.Na) ? a.Ua[((size_t)(i0 + t) * m + k) * m + col] : make_float2(0.f, 0.f);
        wb[t * per + r] = (j0 + t < a.Nb) ? a.Ub[((size_t)(j0 + t) * m + k) * m + col] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    const int tx = threadIdx.x % kFidTile, ty = threadIdx.x / kFidTile;
    const float2 *pa = wa + ty * per, *pb = wb + tx * per;
    cdfl total = {df_zero(), df_zero()};
    if constexpr (TOP == BOT) {
        // one copy of the code serves both halves
#pragma unroll 1
        for (int half = 0; half < 2; ++half) fid_rows<N, TOP>(pa, pb, m, half * TOP, half == 0, kept, total);
    } else {
        fid_rows<N, TOP>(pa, pb, m, 0, true, kept, total);
        fid_rows<N, BOT>(pa, pb, m, TOP, false, kept, total);
    }
    const float tr = df_float(total.re), tim = df_float(total.im);
    const float v = (tr * tr + tim * tim) * a.inv_sf2;
    const int i = i0 + ty, j = j0 + tx;
    if (i < a.Na && j < a.Nb && (!a.sym || i <= j)) a.K[(size_t)i * a.Nb + j] = v;
    if (!a.sym) return;
    // the mirrored entries, turned in shared memory
    __syncthreads();
    float *tile = reinterpret_cast<float *>(fid_sm);
    tile[tx * (kFidTile + 1) + ty] = v;
    __syncthreads();
    const int r = j0 + ty, c = i0 + tx;
    if (r < a.Nb && c < a.Na && c < r) a.K[(size_t)r * a.Nb + c] = tile[ty * (kFidTile + 1) + tx];
}

static int64_t fid_tiles(const FidArgs &a) {
    const int64_t ta = (a.Na + kFidTile - 1) / kFidTile, tb = (a.Nb + kFidTile - 1) / kFidTile;
    return a.sym ? ta * (ta + 1) / 2 : ta * tb;
}

template <int N>
static cudaError_t launch_fid(const FidArgs &a, cudaStream_t s) {
    const size_t sm = 2 * (size_t)kFidTile * a.m * N * sizeof(float2);
    fidelity_kernel<N><<<(unsigned)fid_tiles(a), dim3(kFidTile, kFidTile), sm, s>>>(a);
    return cudaGetLastError();
}

template <int N>
static cudaError_t launch_fid_subset(const FidArgs &a, cudaStream_t s) {
    const auto bytes = [](int m) {
        return (size_t)fid_binom(N, N / 2) * kFidThreads * sizeof(float4) +
               2 * (size_t)kFidTile * ((m * N) | 1) * sizeof(float2);
    };
    // the attribute belongs to the current device's context: set once per device
    static std::mutex mu;
    static bool attr_set[64] = {false};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lk(mu);
        if (!attr_set[dev]) {
            const cudaError_t e = cudaFuncSetAttribute(
                fid_subset_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes(kMaxModes));
            if (e != cudaSuccess) return e;
            attr_set[dev] = true;
        }
    }
    fid_subset_kernel<N><<<(unsigned)fid_tiles(a), kFidThreads, bytes(a.m), s>>>(a);
    return cudaGetLastError();
}

}  // namespace slos

using namespace slos;

extern "C" {

slos_status_t slos_fidelity_kernel(int m, const int *input_state, const void *Ua, int Na, const void *Ub, int Nb,
                                   float *K, void *stream) {
    if (!input_state) return fail(SLOS_ERR_INVALID_ARG, "slos_fidelity_kernel: NULL input_state");
    if (m < 1 || m > kMaxModes) return fail(SLOS_ERR_UNSUPPORTED, "slos_fidelity_kernel: m must be in [1, 24]");
    if (Na < 0 || Nb < 0) return fail(SLOS_ERR_INVALID_ARG, "slos_fidelity_kernel: negative count");
    FidArgs a;
    int n = 0;
    double sf = 1.0;
    for (int i = 0; i < m; ++i) {
        if (input_state[i] < 0) return fail(SLOS_ERR_INVALID_ARG, "slos_fidelity_kernel: negative occupation");
        for (int q = 0; q < input_state[i]; ++q) {
            if (n >= kFidMaxPhotons)
                return fail(SLOS_ERR_UNSUPPORTED, "slos_fidelity_kernel: at most 8 photons");
            a.cols[n++] = i;
            sf *= (double)(q + 1);
        }
    }
    if (n == 0) return fail(SLOS_ERR_INVALID_ARG, "slos_fidelity_kernel: the input state holds no photon");
    if ((int64_t)(Na + kFidTile - 1) / kFidTile > 65535)
        return fail(SLOS_ERR_UNSUPPORTED, "slos_fidelity_kernel: at most 65535 * 16 rows");
    if (Na == 0 || Nb == 0) return SLOS_OK;
    if (!Ua || !Ub || !K) return fail(SLOS_ERR_INVALID_ARG, "slos_fidelity_kernel: NULL pointer");
    a.Ua = reinterpret_cast<const float2 *>(Ua);
    a.Ub = reinterpret_cast<const float2 *>(Ub);
    a.K = K;
    a.m = m;
    a.Na = Na;
    a.Nb = Nb;
    a.inv_sf2 = 1.0 / (sf * sf);
    a.sym = Ua == Ub && Na == Nb;
    cudaStream_t s = (cudaStream_t)stream;
    ProfScope ps("slos_fidelity", 8.0 * m * n * ((double)Na + Nb) + 4.0 * Na * Nb, s);
    cudaError_t e;
    switch (n) {
        case 1: e = launch_fid_subset<1>(a, s); break;
        case 2: e = launch_fid_subset<2>(a, s); break;
        case 3: e = launch_fid_subset<3>(a, s); break;
        case 4: e = launch_fid_subset<4>(a, s); break;
        case 5: e = launch_fid_subset<5>(a, s); break;
        case 6: e = launch_fid_subset<6>(a, s); break;
        case 7: e = launch_fid<7>(a, s); break;
        default: e = launch_fid<8>(a, s); break;
    }
    if (e != cudaSuccess) return fail(SLOS_ERR_CUDA, std::string("slos_fidelity_kernel: ") + cudaGetErrorString(e));
    return SLOS_OK;
}

}  // extern "C"
