// Variance-optimal level placement (paper Section 3): a one-pass per-feature histogram over equal
// bins of the normalised range ("Discretization"), then the dynamic programme
//   T(k, m) = min_j T(k-1, j) + V(j, m)
// over the bin edges ("Dynamic Programming with Candidate Points"), exact: integers below 2^53, held in doubles.
#include "common.cuh"
#include "internal.h"

namespace zipml {

// ---------------------------------------------------------------------------------------------
// Histogram.  A block owns 32 features and a chunk of rows and keeps 32 x bins counters in shared
// memory (row stride bins+1, so that lanes hitting the same bin of different features fall into
// different banks).  blockDim = (32, 32): a warp reads 128 contiguous bytes of a row; the counters leave room
// for one block per SM, so a thread requests eight of its rows before it counts the first (with 8 warps and a row
// at a time the kernel waited for memory: 1,046 us on 500,000 x 512, now 350 us).
// ---------------------------------------------------------------------------------------------
constexpr int kHistWarps = 32, kHistAhead = 8;

__global__ void __launch_bounds__(32 * kHistWarps) histogram_kernel(const float* __restrict__ A, int64_t m, int64_t n, int64_t lda,
                                                                    int bins, int64_t rows_per_block,
                                                                    const float* __restrict__ lo, const float* __restrict__ inv,
                                                                    uint32_t* __restrict__ counts) {
    extern __shared__ uint32_t s_hist[];
    const int stride = bins + 1;
    const int t = threadIdx.y * 32 + threadIdx.x;
    for (int i = t; i < 32 * stride; i += 32 * kHistWarps) s_hist[i] = 0u;
    __syncthreads();
    const int64_t j = (int64_t)blockIdx.x * 32 + threadIdx.x;
    if (j < n) {
        const float flo = __ldg(lo + j), finv = __ldg(inv + j);
        const int64_t r0 = (int64_t)blockIdx.y * rows_per_block;
        const int64_t r1 = min(m, r0 + rows_per_block);
        uint32_t* mine = s_hist + threadIdx.x * stride;
        for (int64_t r = r0 + threadIdx.y; r < r1; r += kHistWarps * kHistAhead) {
            float v[kHistAhead];
#pragma unroll
            for (int u = 0; u < kHistAhead; ++u) v[u] = r + u * kHistWarps < r1 ? __ldg(A + (r + u * kHistWarps) * lda + j) : 0.0f;
#pragma unroll
            for (int u = 0; u < kHistAhead; ++u) {
                uint32_t cell;
                float p;
                uniform_cell(v[u], flo, finv, bins, cell, p);
                if (r + u * kHistWarps < r1) atomicAdd(mine + cell, 1u);
            }
        }
    }
    __syncthreads();
    for (int i = t; i < 32 * bins; i += 32 * kHistWarps) {
        const int f = i / bins, c = i - f * bins;
        const int64_t jj = (int64_t)blockIdx.x * 32 + f;
        const uint32_t v = s_hist[f * stride + c];
        if (jj < n && v) atomicAdd(counts + jj * bins + c, v);
    }
}

int launch_histogram(zipml_ctx* ctx, const float* A, int64_t m, int64_t n, int64_t lda, int bins, const float* lo,
                     const float* inv, uint32_t* counts) {
    cudaError_t e = cudaMemsetAsync(counts, 0, sizeof(uint32_t) * (size_t)(n * bins), ctx->stream);
    if (e != cudaSuccess) return cuda_status(e);
    const size_t smem = sizeof(uint32_t) * 32 * (size_t)(bins + 1);
    if (smem > (size_t)ctx->smem_optin) return ZIPML_ERR_WORKSPACE;
    e = cudaFuncSetAttribute(histogram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_status(e);
    // one block per SM at a time: the number of row chunks that leaves the last wave fullest, fewest first (every
    // chunk flushes its counters), of at least 512 rows
    const int64_t col_tiles = (n + 31) / 32;
    int64_t chunks = 1;
    double best = 0.0;
    for (int64_t c = 1; c <= ctx->sm_count && (c == 1 || m / c >= 512); ++c) {
        const int64_t blocks = col_tiles * c, waves = (blocks + ctx->sm_count - 1) / ctx->sm_count;
        const double full = (double)blocks / (double)(waves * ctx->sm_count);
        if (full > best * 1.03) { best = full; chunks = c; }
    }
    int64_t rows_per_block = (m + chunks - 1) / chunks;
    chunks = (m + rows_per_block - 1) / rows_per_block;
    histogram_kernel<<<dim3((unsigned)col_tiles, (unsigned)chunks), dim3(32, kHistWarps), smem, ctx->stream>>>(
        A, m, n, lda, bins, rows_per_block, lo, inv, counts);
    ctx->launches += 1;
    return cuda_status(cudaGetLastError());
}

// ---------------------------------------------------------------------------------------------
// Level DP: one block per feature.  With bin centres at odd positions x_i = 2i+1 (units of 1/(2M))
// and edges at even positions, the variance of the points of [d_j, d_m] is
//   4 M^2 V(j, m) = sum_{j <= i < m} c_i (2m - x_i)(x_i - 2j) = C_j - C_m + m D_j - j D_m,
//   C_j = sum_{i < j} c_i x_i (x_i - 2j),   D_j = sum_{i < j} c_i (4j - 2 x_i),
// so with E_k(m) = T(k, m) + C_m the recursion becomes
//   E_1 = 0,   E_k(m) = min_j E_{k-1}(j) + m D_j - j D_m,   T(s, M) = E_s(M) - C_M:
// two multiply-adds per candidate.  Every quantity is an integer below 2^53 (at most 10^9 points, 1024 bins:
// 0 <= m D_j <= 4 * 1024^2 * 10^9, -1024^2 * 10^9 <= E <= 0), so double arithmetic is exact and the result does not
// depend on the order of evaluation.  Ties go to the smallest j.
// The interval cost satisfies the quadrangle inequality (a point of [b,c) adds (2d-2c)(2b-2a) >= 0 to
// w(a,d) + w(b,c) - w(a,c) - w(b,d), points left and right of it add non-negative amounts too), so the
// leftmost minimiser j*(m) does not decrease with m.  The edges m are taken in five rounds, every 256th (and M), then
// every 64th, 16th, 4th and all: one of a round scans only from the minimiser of its neighbour below among the
// rounds before to that of its neighbour above, so a round looks at about M candidates, spread
// over groups of lanes (32 down to 4 a group: the ranges get shorter; 8 in the last round 15 % slower, 2 as fast on
// short tails, 1 slower).  The minima, and with
// ascending scans and strict comparisons the leftmost minimisers, are those of the full scan.
// Measured, a call on 3,000 rows (512 features of 1,024 bins): 7 intervals 536 -> 210 us, 15 intervals 1,228 -> 452;
// bound by the chain of the rounds (load, two multiply-adds, compare, a few shuffles, barrier).
// ---------------------------------------------------------------------------------------------
constexpr int kDpThreads = 256;

// E_k(mm) and its leftmost minimiser over j_lo .. j_hi by a group of G lanes; every lane of the warp takes part.
template <int G>
__device__ __forceinline__ void dp_minimise(const double* D, const double* prev, double* cur, unsigned short* ak, bool valid, int mm,
                                            int j_lo, int j_hi) {
    const int lane = threadIdx.x & 31;
    double best = INFINITY;
    int bj = 0x7fffffff;
    if (valid) {
        const double dm = D[mm], md = (double)mm;
        int j = j_lo + (lane & (G - 1));
        double jd = -(double)j;                                     // (counted along: conversions are slow)
#pragma unroll 4
        for (; j <= j_hi; j += G, jd -= (double)G) {
            const double c = fma(jd, dm, fma(md, D[j], prev[j]));
            if (c < best) { best = c; bj = j; }
        }
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
        if (ob < best || (ob == best && oj < bj)) { best = ob; bj = oj; }
    }
    if (valid && (lane & (G - 1)) == 0) { cur[mm] = best; ak[mm] = (unsigned short)bj; }
}

// One round of a layer: the multiples of S that are not multiples of 4 S.
template <int G, int S>
__device__ __forceinline__ void dp_round(const double* D, const double* prev, double* cur, unsigned short* ak, int k, int M) {
    constexpr int kGroups = kDpThreads / G;
    const int items = (M / (4 * S)) * 3 + (M % (4 * S)) / S;
    for (int q0 = 0; q0 < items; q0 += kGroups) {
        const int q = q0 + (int)threadIdx.x / G;
        const int mm = S * (q / 3 * 4 + q % 3 + 1);
        const bool valid = q < items && mm >= k && mm < M;
        int j_lo = k - 1, j_hi = 0;
        if (valid) {
            const int below = mm / (4 * S) * (4 * S), above = min(below + 4 * S, M);
            if (below >= k) j_lo = ak[below];
            j_hi = min((int)ak[above], mm - 1);
        }
        dp_minimise<G>(D, prev, cur, ak, valid, mm, j_lo, j_hi);
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kDpThreads) levels_dp_kernel(const uint32_t* __restrict__ counts, int bins, int s,
                                                               const float* __restrict__ lo,
                                                               const float* __restrict__ hi,
                                                               float* __restrict__ levels_out,
                                                               unsigned long long* __restrict__ objective_out) {
    extern __shared__ double s_mem[];
    const int M = bins, M1 = bins + 1;
    double* D = s_mem;
    double* prev = D + M1;
    double* cur = prev + M1;
    unsigned short* arg = reinterpret_cast<unsigned short*>(cur + M1);   // (s+1) x M1
    __shared__ int s_idx[17];
    __shared__ unsigned long long tot[3][kDpThreads / 32];
    const int64_t j_feat = blockIdx.x;
    const uint32_t* cnt = counts + j_feat * M;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long S0, S1, S2;                                  // sums of c, c x, c x^2 over all bins
    {
        // exclusive prefix sums of c and c x: every thread sums a run of bins, the runs' totals are scanned by warps
        const int per = (M + kDpThreads - 1) / kDpThreads;
        const int i_begin = min(M, (int)threadIdx.x * per), i_end = min(M, i_begin + per);
        unsigned long long a0 = 0, a1 = 0, a2 = 0;
        for (int i = i_begin; i < i_end; ++i) {
            const unsigned long long c = cnt[i], x = 2ull * i + 1ull;
            a0 += c; a1 += c * x; a2 += c * x * x;
        }
        const unsigned long long own0 = a0, own1 = a1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long b0 = __shfl_up_sync(0xffffffffu, a0, o), b1 = __shfl_up_sync(0xffffffffu, a1, o);
            const unsigned long long b2 = __shfl_up_sync(0xffffffffu, a2, o);
            if (lane >= o) { a0 += b0; a1 += b1; a2 += b2; }
        }
        if (lane == 31) { tot[0][warp] = a0; tot[1][warp] = a1; tot[2][warp] = a2; }
        a0 -= own0; a1 -= own1;
        __syncthreads();
        S0 = S1 = S2 = 0;
#pragma unroll
        for (int w = 0; w < kDpThreads / 32; ++w) {
            if (w == warp) { a0 += S0; a1 += S1; }
            S0 += tot[0][w]; S1 += tot[1][w]; S2 += tot[2][w];
        }
        for (int i = i_begin; i < i_end; ++i) {
            D[i] = (double)(4ull * i * a0 - 2ull * a1);
            prev[i] = 0.0;                                          // E_1
            const unsigned long long c = cnt[i], x = 2ull * i + 1ull;
            a0 += c; a1 += c * x;
        }
        if (threadIdx.x == 0) { D[M] = (double)(4ull * M * S0 - 2ull * S1); prev[M] = 0.0; }
        for (int mm = 1 + threadIdx.x; mm <= M; mm += kDpThreads) arg[M1 + mm] = 0;
    }
    __syncthreads();
    for (int k = 2; k <= s; ++k) {
        unsigned short* ak = arg + k * M1;
        const int items = M / 256 + (M % 256 != 0 ? 1 : 0);         // multiples of 256, and M
        for (int q = warp; q < items; q += kDpThreads / 32) {
            const int mm = q < M / 256 ? (q + 1) * 256 : M;
            dp_minimise<32>(D, prev, cur, ak, mm >= k, mm, k - 1, mm - 1);
        }
        __syncthreads();
        dp_round<32, 64>(D, prev, cur, ak, k, M);
        dp_round<16, 16>(D, prev, cur, ak, k, M);
        dp_round<8, 4>(D, prev, cur, ak, k, M);
        dp_round<4, 1>(D, prev, cur, ak, k, M);
        double* t = prev; prev = cur; cur = t;
    }
    if (threadIdx.x == 0) {
        // T(s, M) = E_s(M) - C_M, C_M = sum c x (x - 2 M)
        if (objective_out) objective_out[j_feat] = (unsigned long long)((long long)prev[M] - ((long long)S2 - 2ll * M * (long long)S1));
        int mm = M;
        for (int k = s; k >= 1; --k) { s_idx[k] = mm; mm = arg[k * M1 + mm]; }
        s_idx[0] = 0;
    }
    __syncthreads();
    if (threadIdx.x <= s) {
        const float flo = lo[j_feat], fhi = hi[j_feat];
        const float range = __fsub_rn(fhi, flo);
        const float frac = __fdiv_rn((float)s_idx[threadIdx.x], (float)M);
        float v = __fadd_rn(flo, __fmul_rn(range, frac));
        if (threadIdx.x == 0) v = flo;
        if (threadIdx.x == s) v = fhi;
        levels_out[j_feat * (s + 1) + threadIdx.x] = v;
    }
}

int launch_levels_dp(zipml_ctx* ctx, const uint32_t* counts, int64_t n, int bins, int s, const float* lo,
                     const float* hi, float* levels_out, uint64_t* objective_out) {
    const size_t smem = sizeof(double) * 3 * (size_t)(bins + 1) + sizeof(unsigned short) * (size_t)(s + 1) * (bins + 1);
    if (smem > (size_t)ctx->smem_optin) return ZIPML_ERR_WORKSPACE;
    cudaError_t e = cudaFuncSetAttribute(levels_dp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_status(e);
    if (n > 0x7fffffffLL) return ZIPML_ERR_WORKSPACE;
    levels_dp_kernel<<<(unsigned)n, kDpThreads, smem, ctx->stream>>>(
        counts, bins, s, lo, hi, levels_out, reinterpret_cast<unsigned long long*>(objective_out));
    ctx->launches += 1;
    return cuda_status(cudaGetLastError());
}

}  // namespace zipml
