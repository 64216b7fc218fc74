// Variance-optimal level placement (paper Section 3): a one-pass per-feature histogram over equal
// bins of the normalised range ("Discretization"), then the dynamic programme
//   T(k, m) = min_j T(k-1, j) + V(j, m)
// over the bin edges ("Dynamic Programming with Candidate Points"), exact: integers below 2^53, held in doubles.
#include "common.cuh"
#include "internal.h"

namespace zipml {

// ---------------------------------------------------------------------------------------------
// Histogram.  A block owns 32 features, a lane each, and keeps their counters in shared memory as [bin][feature]: a
// warp reads 128 contiguous bytes of a row and counts without bank conflicts whatever the bins are.  The row chunks of a column tile
// take groups of kHistWarps * kHistAhead rows in turn, from the last to the first (the range pass has left the end of A in L2);
// a thread has kHistAhead rows requested, each asked for as soon as its register is counted.
// Bound by HBM: 500,000 x 512 at 1,024 bins 380 -> 155 us ([feature][bin + 1] counters before, whose conflicts took three
// wavefronts a warp, and 43 instructions a sample, mostly row numbers and addresses in 64 bits).
// ---------------------------------------------------------------------------------------------
constexpr int kHistWarps = 32, kHistAhead = 16;

// Offset: unsigned where kHistWarps rows span less than 4 GB, else 64 bits.
template <typename Offset>
__global__ void __launch_bounds__(32 * kHistWarps) histogram_kernel(const float* __restrict__ A, int64_t m, int64_t n, int64_t lda,
                                                                    int bins, const float* __restrict__ lo, const float* __restrict__ inv,
                                                                    uint32_t* __restrict__ counts) {
    extern __shared__ uint32_t s_hist[];
    const int lane = threadIdx.x, warp = threadIdx.y, t = warp * 32 + lane;
    for (int i = t; i < 32 * bins; i += 32 * kHistWarps) s_hist[i] = 0u;
    __syncthreads();
    const int64_t j = (int64_t)blockIdx.x * 32 + lane;
    if (j < n) {
        const float flo = __ldg(lo + j), finv = __ldg(inv + j);
        const uint32_t last = (uint32_t)(bins - 1);
        uint32_t* mine = s_hist + lane;
        // floor((v - lo) * inv), the product rounded as the grid prescribes (the conversion saturates, NaN and negative values at 0)
        auto count = [&](float v) { atomicAdd(mine + 32u * min(__float2uint_rd(__fmul_rn(__fsub_rn(v, flo), finv)), last), 1u); };
        constexpr int kGroup = kHistWarps * kHistAhead;
        const int64_t groups = m / kGroup;                          // whole ones
        const Offset at = ((Offset)warp * (Offset)lda + (Offset)lane) * (Offset)sizeof(float);
        const char* column = reinterpret_cast<const char*>(A + (int64_t)blockIdx.x * 32);
        const int64_t part = kHistWarps * lda * (int64_t)sizeof(float);
        float v[kHistAhead];
        int64_t q = groups - 1 - blockIdx.y;
        if (q >= 0) {
            const char* p = column + q * kHistAhead * part;
#pragma unroll
            for (int u = 0; u < kHistAhead; ++u, p += part) v[u] = __ldg(reinterpret_cast<const float*>(p + at));
        }
        for (; q >= (int64_t)gridDim.y; q -= gridDim.y) {
            const char* p = column + (q - gridDim.y) * kHistAhead * part;
#pragma unroll
            for (int u = 0; u < kHistAhead; ++u, p += part) {
                count(v[u]);
                v[u] = __ldg(reinterpret_cast<const float*>(p + at));
            }
        }
        if (q >= 0) {
#pragma unroll
            for (int u = 0; u < kHistAhead; ++u) count(v[u]);
        }
        if (blockIdx.y == gridDim.y - 1)
            for (int64_t r = groups * kGroup + warp; r < m; r += kHistWarps) count(__ldg(A + r * lda + j));
    }
    __syncthreads();
    uint32_t* out = counts + (int64_t)blockIdx.x * 32 * bins;
    for (int i = t; i < 32 * bins; i += 32 * kHistWarps) {
        const uint32_t v = s_hist[i];
        if (gridDim.y == 1) out[i] = v;
        else if (v) atomicAdd(out + i, v);
    }
}

int launch_histogram(zipml_ctx* ctx, const float* A, int64_t m, int64_t n, int64_t lda, int bins, const float* lo,
                     const float* inv, uint32_t* counts) {
    const size_t smem = sizeof(uint32_t) * 32 * (size_t)bins;
    if (smem > (size_t)ctx->smem_optin) return ZIPML_ERR_WORKSPACE;
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
    if (chunks > 1) {
        const cudaError_t e = cudaMemsetAsync(counts, 0, sizeof(uint32_t) * histogram_count(n, bins), ctx->stream);
        if (e != cudaSuccess) return cuda_status(e);
    }
    auto launch = [&](auto kernel) -> int {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return cuda_status(e);
        kernel<<<dim3((unsigned)col_tiles, (unsigned)chunks), dim3(32, kHistWarps), smem, ctx->stream>>>(A, m, n, lda, bins, lo, inv, counts);
        ctx->launches += 1;
        return cuda_status(cudaGetLastError());
    };
    return lda < (1ll << 32) / (kHistWarps * (int64_t)sizeof(float)) ? launch(histogram_kernel<uint32_t>) : launch(histogram_kernel<uint64_t>);
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
// The three edges between two neighbours are searched together, on one load of a candidate (7 intervals 155 -> 145 us), but for few bins of
// many features, whose edges have a group each and whose idle warps rest (20,000 features, 15 intervals: 17 bins 1,067 -> 683 us, 256 bins 2,665 -> 2,265;
// in one kernel with the other form both took 1.2 to 1.9 times as long).
// Measured, a call on 3,000 rows (512 features of 1,024 bins) against the full scan: 7 intervals 536 -> 210 us, 15 intervals
// 1,228 -> 452; bound by the chain of the rounds (load, two multiply-adds, compare, a few shuffles, barrier).
// ---------------------------------------------------------------------------------------------
constexpr int kDpThreads = 256;
constexpr int kDpRun = 1024 / kDpThreads;       // bins that a thread sums, at most

// E_k and its leftmost minimiser for the N edges first, first + S, .. over j_lo .. j_hi by a group of G lanes; every lane of the warp
// takes part.  N edges share the loads of a candidate.  Of several edges, one counts where it is at least k, and a candidate where it
// lies below the edge.
template <int G, int N, int S>
__device__ __forceinline__ void dp_minimise(const double* D, const double* prev, double* cur, unsigned short* ak, bool valid, int k, int first,
                                            int j_lo, int j_hi) {
    const int lane = threadIdx.x & 31;
    double best[N];
    int bj[N];
#pragma unroll
    for (int u = 0; u < N; ++u) { best[u] = INFINITY; bj[u] = 0x7fffffff; }
    if (valid) {
        double dm[N], md[N];
#pragma unroll
        for (int u = 0; u < N; ++u) { dm[u] = D[first + u * S]; md[u] = (double)(first + u * S); }
        int j = j_lo + (lane & (G - 1));
        double jd = -(double)j;                                     // (counted along: conversions are slow)
#pragma unroll 2
        for (; j <= j_hi; j += G, jd -= (double)G) {
            const double dj = D[j], pj = prev[j];
#pragma unroll
            for (int u = 0; u < N; ++u) {
                const double c = fma(jd, dm[u], fma(md[u], dj, pj));
                if (c < best[u] && (N == 1 || j < first + u * S)) { best[u] = c; bj[u] = j; }
            }
        }
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1)
#pragma unroll
        for (int u = 0; u < N; ++u) {
            const double ob = __shfl_xor_sync(0xffffffffu, best[u], o);
            const int oj = __shfl_xor_sync(0xffffffffu, bj[u], o);
            if (ob < best[u] || (ob == best[u] && oj < bj[u])) { best[u] = ob; bj[u] = oj; }
        }
#pragma unroll
    for (int u = 0; u < N; ++u)
        if (valid && (lane & (G - 1)) == u % G && first + u * S >= k) { cur[first + u * S] = best[u]; ak[first + u * S] = (unsigned short)bj[u]; }
}

// One round of a layer: the multiples of S that are not multiples of 4 S, the three between two neighbours of the rounds before at once.
// FEW (bins): a group for every edge, and the warps that are left over rest.
template <int G, int S, bool FEW>
__device__ __forceinline__ void dp_round(const double* D, const double* prev, double* cur, unsigned short* ak, int k, int M) {
    constexpr int kGroups = kDpThreads / G;
    if constexpr (FEW) {
        const int edges = M / (4 * S) * 3 + M % (4 * S) / S;        // (the last may be M itself)
        for (int q0 = 0; q0 < edges; q0 += kGroups) {
            const int q = q0 + (int)threadIdx.x / G, below = q / 3 * (4 * S), mm = below + (q % 3 + 1) * S;
            const bool valid = q < edges && mm >= k && mm < M;
            if (__any_sync(0xffffffffu, valid)) {
                const int j_lo = valid && below >= k ? (int)ak[below] : k - 1;
                dp_minimise<G, 1, S>(D, prev, cur, ak, valid, k, mm, j_lo, valid ? min((int)ak[min(below + 4 * S, M)], mm - 1) : 0);
            }
        }
        __syncthreads();
        return;
    }
    const int items = M / (4 * S);                                  // whole intervals; M itself may end a shorter one
    for (int q0 = 0; q0 < items; q0 += kGroups) {
        const int q = q0 + (int)threadIdx.x / G, below = q * 4 * S, above = below + 4 * S;
        const bool valid = q < items && below + 3 * S >= k;
        const int j_lo = valid && below >= k ? (int)ak[below] : k - 1;
        dp_minimise<G, 3, S>(D, prev, cur, ak, valid, k, below + S, j_lo, valid ? min((int)ak[above], below + 3 * S - 1) : 0);
    }
    const int rest = (M % (4 * S) + S - 1) / S - 1;                 // edges of that one (at most 3): a group each
    if ((int)threadIdx.x / 32 * 32 < rest * G) {
        const int q = (int)threadIdx.x / G, below = items * 4 * S, mm = below + (q + 1) * S;
        const bool valid = q < rest && mm >= k;
        const int j_lo = valid && below >= k ? (int)ak[below] : k - 1;
        dp_minimise<G, 1, S>(D, prev, cur, ak, valid, k, mm, j_lo, valid ? min((int)ak[M], mm - 1) : 0);
    }
    __syncthreads();
}

template <bool FEW>
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
    const uint32_t* cnt = counts + j_feat / 32 * 32 * M + j_feat % 32;   // bin i at 32 i
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long S0, S1, S2;                                  // sums of c, c x, c x^2 over all bins
    {
        // exclusive prefix sums of c and c x: every thread sums a run of bins, the runs' totals are scanned by warps
        const int per = (M + kDpThreads - 1) / kDpThreads;
        const int i_begin = min(M, (int)threadIdx.x * per), i_end = min(M, i_begin + per);
        uint32_t c_run[kDpRun];
#pragma unroll
        for (int u = 0; u < kDpRun; ++u) c_run[u] = i_begin + u < i_end ? cnt[(int64_t)(i_begin + u) * 32] : 0u;
        unsigned long long a0 = 0, a1 = 0, a2 = 0;
#pragma unroll
        for (int u = 0; u < kDpRun; ++u) {
            const unsigned long long c = c_run[u], x = 2ull * (i_begin + u) + 1ull;
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
#pragma unroll
        for (int u = 0; u < kDpRun; ++u) {
            const int i = i_begin + u;
            if (i >= i_end) break;
            D[i] = (double)(4ull * i * a0 - 2ull * a1);
            prev[i] = 0.0;                                          // E_1
            const unsigned long long c = c_run[u], x = 2ull * i + 1ull;
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
            dp_minimise<32, 1, 1>(D, prev, cur, ak, mm >= k, k, mm, k - 1, mm - 1);
        }
        __syncthreads();
        dp_round<32, 64, FEW>(D, prev, cur, ak, k, M);
        dp_round<16, 16, FEW>(D, prev, cur, ak, k, M);
        dp_round<8, 4, FEW>(D, prev, cur, ak, k, M);
        dp_round<4, 1, FEW>(D, prev, cur, ak, k, M);
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
    if (n > 0x7fffffffLL) return ZIPML_ERR_WORKSPACE;
    auto kernel = bins <= 256 && n >= 8ll * ctx->sm_count ? levels_dp_kernel<true> : levels_dp_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_status(e);
    kernel<<<(unsigned)n, kDpThreads, smem, ctx->stream>>>(
        counts, bins, s, lo, hi, levels_out, reinterpret_cast<unsigned long long*>(objective_out));
    ctx->launches += 1;
    return cuda_status(cudaGetLastError());
}

}  // namespace zipml
