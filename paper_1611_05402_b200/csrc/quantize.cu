// Column range scan and the quantize + pack kernel (paper Section 2.1; Supplement "Randomized
// Quantization" and "Column Scaling"): two independent unbiased stochastic roundings of every
// sample element onto its feature's level grid, written as two bit-packed planes.
#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace zipml {

// ---------------------------------------------------------------------------------------------
// Column range.  A block of 256 threads takes tx * VEC columns (tx a power of two, at least the row's as far as it
// goes) and 256 / tx rows at a time, up to 4 KB of consecutive memory; a thread keeps its VEC columns, kRangeAhead rows in flight.
// The row chunks of a column tile take groups of rows in turn, so that the pass as a whole goes through A from front to back and
// leaves the end of A in L2.  Their results meet in order-preserving integer keys (a maximum of the value's key, a maximum
// of the complement for the minimum: exact and order independent); the tile's last block turns the keys into the grid
// and clears keys and counter for the next pass: no launch before this one to set them, none after it.
// Bound by HBM.  500,000 x 512 230 -> 148 us (one row in flight a thread before), 100,003 x 1,001 70 -> 63, and what follows finds more of
// A in L2: the whole call on 250,000 x 1,000 at 4 bits 664 -> 567 us, 4,096 x 64 19 -> 12.
// ---------------------------------------------------------------------------------------------
struct RangeArgs {
    const float* A;
    int64_t m, n, lda;                         // n: columns of this launch
    uint32_t *lo_key, *hi_key;                 // 0 between passes
    unsigned* done;                            // blocks that have finished, per column tile; 0 between passes
    DeviceStatus* status;
    int s;                                     // intervals of the grid
    int symmetric;
    float *lo, *hi, *inv, *step;               // results; all but lo may be null
};

__device__ __forceinline__ void range_results(const RangeArgs& a, int64_t j, uint32_t lo_key, uint32_t hi_key) {
    float lo = float_from_order_key(~lo_key), hi = float_from_order_key(hi_key);
    if (a.symmetric) {                         // the grid [-M_j, M_j], M_j = max |value| (Supplement "Column Scaling")
        hi = fmaxf(fabsf(lo), fabsf(hi));
        lo = -hi;
    }
    const float range = __fsub_rn(hi, lo);
    a.lo[j] = lo;
    if (a.hi) a.hi[j] = hi;
    if (a.inv) a.inv[j] = range > 0.0f ? __fdiv_rn((float)a.s, range) : 0.0f;
    if (a.step) a.step[j] = __fdiv_rn(range, (float)a.s);
}

// Called by every thread of a block once its keys are on their way: the tile's last block writes the results of columns j0 .. j0 +
// count - 1 and clears what the pass has used.
__device__ __forceinline__ void range_finish(const RangeArgs& a, unsigned tile, unsigned blocks, int64_t j0, int count) {
    const int t = threadIdx.y * blockDim.x + threadIdx.x;
    __shared__ bool last_s;
    __threadfence();
    __syncthreads();
    if (t == 0) last_s = atomicAdd(a.done + tile, 1u) == blocks - 1;
    __syncthreads();
    if (!last_s) return;
    __threadfence();
    for (int64_t j = j0 + t; j < min(a.n, j0 + count); j += 256) {
        range_results(a, j, __ldcg(a.lo_key + j), __ldcg(a.hi_key + j));
        a.lo_key[j] = 0u;
        a.hi_key[j] = 0u;
    }
    if (t == 0) a.done[tile] = 0u;
}

template <int VEC>
__global__ void __launch_bounds__(256, 4) range_scan_kernel(const RangeArgs a) {
    constexpr int kRangeAhead = VEC == 4 ? 4 : 16;
    __shared__ float lo_s[256 * VEC], hi_s[256 * VEC];
    const int tx = blockDim.x, ty = blockDim.y, t = threadIdx.y * tx + threadIdx.x;
    const int64_t first = (int64_t)blockIdx.x * tx * VEC, j0 = first + threadIdx.x * VEC;
    float lo[VEC], hi[VEC], probe = 0.0f;                          // probe: NaN once a value is not finite
#pragma unroll
    for (int v = 0; v < VEC; ++v) { lo[v] = INFINITY; hi[v] = -INFINITY; }
    if (j0 < a.n) {
        const int nv = (int)min((int64_t)VEC, a.n - j0);
        const int64_t group = (int64_t)ty * kRangeAhead;
        for (int64_t r0 = blockIdx.y * group; r0 < a.m; r0 += gridDim.y * group) {
            const float* src = a.A + (r0 + threadIdx.y) * a.lda + j0;
            if (r0 + group <= a.m && nv == VEC) {
                float val[kRangeAhead][VEC];
#pragma unroll
                for (int u = 0; u < kRangeAhead; ++u, src += ty * a.lda) {
                    if constexpr (VEC == 4) {
                        const float4 q = __ldg(reinterpret_cast<const float4*>(src));
                        val[u][0] = q.x; val[u][1] = q.y; val[u][2] = q.z; val[u][3] = q.w;
                    } else {
                        val[u][0] = __ldg(src);
                    }
                }
#pragma unroll
                for (int u = 0; u < kRangeAhead; ++u)
#pragma unroll
                    for (int v = 0; v < VEC; ++v) {
                        probe = fmaf(val[u][v], 0.0f, probe);
                        lo[v] = fminf(lo[v], val[u][v]);
                        hi[v] = fmaxf(hi[v], val[u][v]);
                    }
            } else {
                for (int64_t r = r0 + threadIdx.y; r < min(a.m, r0 + group); r += ty, src += ty * a.lda)
#pragma unroll
                    for (int v = 0; v < VEC; ++v)
                        if (v < nv) {
                            const float val = __ldg(src + v);
                            probe = fmaf(val, 0.0f, probe);
                            lo[v] = fminf(lo[v], val);
                            hi[v] = fmaxf(hi[v], val);
                        }
            }
        }
    }
    if (!(probe == 0.0f)) set_status(a.status, ZIPML_ERR_NONFINITE, 1);
#pragma unroll
    for (int v = 0; v < VEC; ++v) { lo_s[t * VEC + v] = lo[v]; hi_s[t * VEC + v] = hi[v]; }
    __syncthreads();
    for (int c = t; c < tx * VEC; c += 256) {
        float x = lo_s[c], y = hi_s[c];
        for (int k = 1; k < ty; ++k) { x = fminf(x, lo_s[k * tx * VEC + c]); y = fmaxf(y, hi_s[k * tx * VEC + c]); }
        if (first + c < a.n && x <= y) {                           // at least one row seen
            atomicMax(a.lo_key + first + c, ~float_order_key(x));
            atomicMax(a.hi_key + first + c, float_order_key(y));
        }
    }
    range_finish(a, blockIdx.x, gridDim.y, first, tx * VEC);
}

int launch_column_range(zipml_ctx* ctx, const float* A, int64_t m, int64_t n, int64_t lda, int s, bool symmetric, float* lo_out, float* hi_out,
                        float* inv_out, float* step_out) {
    const bool vec = (lda % 4 == 0) && ((reinterpret_cast<uintptr_t>(A) & 15) == 0);
    const int per = vec ? 4 : 1;
    for (int64_t j0 = 0; j0 < n; j0 += kRangeColumns) {            // (the keys hold so many columns at a time)
        RangeArgs a{};
        a.A = A + j0; a.m = m; a.n = n - j0 < kRangeColumns ? n - j0 : kRangeColumns; a.lda = lda;
        a.lo_key = ctx->range_keys; a.hi_key = a.lo_key + kRangeColumns; a.done = a.hi_key + kRangeColumns;
        a.status = ctx->d_status; a.s = s; a.symmetric = symmetric;
        a.lo = lo_out + j0;
        a.hi = hi_out ? hi_out + j0 : nullptr;
        a.inv = inv_out ? inv_out + j0 : nullptr;
        a.step = step_out ? step_out + j0 : nullptr;
        int tx = 8;
        while (tx < 256 && tx * per < a.n) tx *= 2;
        const int ty = 256 / tx;
        const int64_t tiles = (a.n + tx * per - 1) / (tx * per);
        // four blocks per SM, of at least 64 rows each
        int64_t chunks = (int64_t)ctx->sm_count * 4 / tiles;
        const int64_t most = (m + 63) / 64;
        chunks = chunks > most ? most : chunks;
        chunks = chunks < 1 ? 1 : chunks;
        const dim3 grid((unsigned)tiles, (unsigned)chunks), block((unsigned)tx, (unsigned)ty);
        if (vec) range_scan_kernel<4><<<grid, block, 0, ctx->stream>>>(a);
        else range_scan_kernel<1><<<grid, block, 0, ctx->stream>>>(a);
        ctx->launches += 1;
    }
    return cuda_status(cudaGetLastError());
}

// ---------------------------------------------------------------------------------------------
// Quantize + pack.  A thread owns four consecutive features (8, 16 or 32 bits of a plane's row) and kQuantRows
// consecutive rows per pass: the features' lo and inv are loaded once, the rows' loads and Philox chains are
// independent and overlap, and the next pass's samples are on their way while this pass draws.
//   Cell and threshold.  With t = (v - lo) * inv rounded as the grid prescribes and tc = clamp(t, 0, s), p = tc - floor tc:
//     up <=> (word >> 8) < ceil(2^24 p) (u24 * 2^-24 < p is exact in fp32, u24 an integer; p <= 0 or NaN: never up).
//     Cell and threshold together, floor(tc) << 24 plus ceil(2^24 p), are ceil(2^24 tc): one conversion.  A draw is an
//     addition whose carry reaches the cell in the upper byte, from where byte permutes collect the codes.  t >= s lands in
//     code s with p = 0: no special case for the upper end.
//   Draws.  One Philox block serves a feature pair: counter (row, row's upper half, pair, draw), words {first feature copy
//     1, copy 2, second feature copy 1, copy 2}, the top 24 bits of a word the uniform integer.  The round keys depend on
//     the seed alone and arrive as kernel parameters (an operand of the xor).  The 32 x 32 -> 64-bit products are what
//     the rounds cost (half of the FMA pipe takes them): of the first two rounds' four, two depend only on the pair
//     (kept for the thread's life) and two only on the row (shared by the thread's pairs): 17 a block, not 20.
//   Sparse rows.  A pair whose two values lie on grid points (5 % non-zeros: nine pairs in ten) has no draw to make.
//     Where at most a quarter of a warp's pairs are anything else, the lanes put those thresholds in a queue in shared
//     memory and share them out evenly, one Philox block per 32 pairs instead of eight per lane; the four answers of a pair go to its
//     owner's word, whose bits a shift and a mask add to the codes.  (Queueing the samples, with cells and thresholds
//     done by whoever draws, saves conversions and loses more to shared memory, which was 87 % busy: 148 us per
//     4,096 x 32,768, now 134.)
// Level tables: the block's tables are staged in shared memory as [feature of the thread][level][thread column], so
// that a warp's look-ups are free of bank conflicts whatever its codes are (from 32 thread columns on; of fewer, two rows' lanes share a column's bank); the cell is found by bisection, whose offset is the cell's
// number times 256, and p by a multiplication with the staged reciprocal of the cell's width, corrected (quotient below).
// Blocks with a cell too narrow or too wide for that divide instead; a quotient too small for it is between 0 and
// 2^-24 anyway, and its threshold is 1 if the numerator lies above the staged one from which on the division does not round to 0 and 0 if not
// (a numerator of exactly width 2^-150, half of the smallest number, comes out of the correction as 0 or not).  No calls, and no branch a
// sample: 85 -> 71 instructions a sample, 890 -> 655 us on 500,000 x 512 at 3 bits.  Such a
// call needs no range pass before this kernel: the feature's extremes, which it returns and which carry the check for
// non-finite values, are gathered on the way.
// What bounds it: dense rows, the integer products (that pipe 73 % busy, issue slots 62 %; 24 warps per SM: fewer
// registers per thread spill, more leave too few warps); sparse rows, issue slots (75 %) and DRAM (60 %) together.
// Measured, whole call with the range pass, samples queued and conversions of their own for cell and threshold ->
// now: 100,003 x 1,001 at 8 bits 279 -> 251 us, 65,536 x 4,096 of 5 % non-zeros at 4 bits 484 -> 415.
// ---------------------------------------------------------------------------------------------
constexpr int kQuantRows = 4;                  // rows per thread and pass
constexpr int kQuantTableCols = 64;            // thread columns per block with level tables
constexpr int kNarrowGroups = 16;              // of four features, in rows that pad themselves (level tables)
constexpr int kQuantQueue = 64;                // pairs that a warp shares out (of the 256 of a pass); more: each lane does its own
constexpr uint32_t kPhiloxM0 = 0xD2511F53u, kPhiloxM1 = 0xCD9E8D57u;

struct PhiloxKeys {                            // the ten round keys of one seed
    uint32_t k0[10], k1[10];
};

static PhiloxKeys philox_keys(uint64_t seed) {
    PhiloxKeys k;
    uint32_t a = (uint32_t)seed, b = (uint32_t)(seed >> 32);
    for (int r = 0; r < 10; ++r) { k.k0[r] = a; k.k1[r] = b; a += 0x9E3779B9u; b += 0xBB67AE85u; }
    return k;
}

// Rounds FIRST .. 9 of philox4x32_10() with its key schedule given.
template <int FIRST>
__device__ __forceinline__ Philox4 philox_rounds(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, const PhiloxKeys& key) {
#pragma unroll
    for (int r = FIRST; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)kPhiloxM0 * c0, p1 = (uint64_t)kPhiloxM1 * c2;
        c0 = (uint32_t)(p1 >> 32) ^ c1 ^ key.k0[r];
        c1 = (uint32_t)p1;
        c2 = (uint32_t)(p0 >> 32) ^ c3 ^ key.k1[r];
        c3 = (uint32_t)p0;
    }
    Philox4 out;
    out.v[0] = c0; out.v[1] = c1; out.v[2] = c2; out.v[3] = c3;
    return out;
}

// A decision (cell << 24 plus threshold) and its draw: the code in the upper byte.  The uniform integer u below the threshold
// carries into the cell: threshold + 2^24 - 1 - u >= 2^24.
__device__ __forceinline__ uint32_t with_draw(uint32_t decision, uint32_t word) { return decision + 0xFFFFFFu - (word >> 8); }

// The upper bytes of four words side by side, CB bits each; what lies above is undefined.
template <int CB>
__device__ __forceinline__ uint32_t pack_codes(const uint32_t (&c)[4]) {
    if constexpr (CB == 8) return __byte_perm(__byte_perm(c[0], c[1], 0x0073), __byte_perm(c[2], c[3], 0x0073), 0x5410);
    else {
        const uint32_t w = __byte_perm(c[0], c[2], 0x0073) + (__byte_perm(c[1], c[3], 0x0073) << CB);
        return CB == 4 ? w : w + (w >> 4);
    }
}

// num / width rounded to nearest, from rw = 1 / width rounded to nearest: two residual corrections (Markstein, "Computation
// of elementary functions on the IBM RISC System/6000 processor", 1990: a faithful quotient corrected once with the
// correctly rounded reciprocal is the correctly rounded quotient, where nothing underflows).  For widths in [2^-40, 2^40] the
// residuals of quotients from 2^-60 on are multiples of 2^(-60 - 23 - 40 - 23) and cannot underflow; smaller ones
// come out wrong by at most 2^-110.
// Compared with CUDA's division on 2 x 10^10 pairs (widths 2^-40 .. 2^40, quotients 2^-60 .. 2): equal.
__device__ __forceinline__ float quotient(float num, float width, float rw) {
    float q = __fmul_rn(num, rw);
    q = __fmaf_rn(__fmaf_rn(-q, width, num), rw, q);
    return __fmaf_rn(__fmaf_rn(-q, width, num), rw, q);
}

template <int CB> struct QuantWord;
template <> struct QuantWord<8> { using type = uint32_t; };
template <> struct QuantWord<4> { using type = uint16_t; };
template <> struct QuantWord<2> { using type = uint8_t; };

// Sparse rows: a lane's 32 answers (4 rows, 2 planes, 4 features) in one word.  A row's four answers of a plane lie CB bits
// apart from bit answer_shift() on, where they are added to its codes.
template <int CB>
__host__ __device__ constexpr int answer_shift(int row, int plane) {
    return CB == 8 ? 4 * plane + row : CB == 4 ? 16 * plane + row : 16 * (row >> 1) + 8 * plane + (row & 1);
}

// TB: 0 for a uniform grid of `bits` bits, else the bits of the level table.  NARROW: level tables, rows of at most kNarrowGroups groups.
template <int CB, int TB, bool NARROW>
__global__ void __launch_bounds__(256, 3) quantize_kernel(const float* __restrict__ A, int64_t m, int64_t n, int64_t lda, int bits,
                                                          const float* __restrict__ lo, const float* __restrict__ inv,
                                                          const float* __restrict__ levels, const RangeArgs range, const PhiloxKeys key,
                                                          uint32_t draw,
                                                          uint8_t* __restrict__ plane1, uint8_t* __restrict__ plane2, int64_t row_bytes,
                                                          bool vec_ok, int passes, unsigned col_blocks, unsigned row_blocks, int64_t group0) {
    using Word = typename QuantWord<CB>::type;
    constexpr bool TABLE = TB > 0;
    constexpr int L = 1 << TB;                                     // TABLE: levels
    // TABLE: where level k of the feature i of thread column c is staged, floats: k * kCols + i * kFeature + c, or with i * L * kCols
    constexpr int kCols = kQuantTableCols, kFeature = NARROW ? kNarrowGroups : L * kCols;
    __shared__ uint2 queue_s[8][kQuantQueue];                      // pairs to draw: {threshold, lane * 8 + row * 2 + pair in the upper byte}, {threshold}
    __shared__ uint32_t answer_s[8][32];                           // and what came out, per lane
    extern __shared__ float4 cell_s[];                             // TABLE: level, width of its cell, 1 / width, least numerator
    float* lev_s = reinterpret_cast<float*>(cell_s + (NARROW ? 1 : 4) * L * kCols);   // TABLE: levels
    const int tx = blockDim.x, tid = threadIdx.y * tx + threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int col = NARROW ? tid & (kNarrowGroups - 1) : threadIdx.x;   // TABLE: the thread's column as it is staged
    const unsigned row_block = blockIdx.x / col_blocks, col_block = blockIdx.x - row_block * col_blocks;
    const int64_t g = group0 + (int64_t)col_block * tx + threadIdx.x;   // this thread's group of four features (group0: the launch's first)
    const int64_t groups = row_bytes * 8 / (4 * CB);
    const int64_t j0 = g * 4;
    const int nf = (int)max((int64_t)0, min((int64_t)4, n - j0));  // real features of the group (0: padding)
    bool divide = false;                                           // TABLE: a cell of the block needs the division itself
    if constexpr (TABLE) {
        const int64_t jb = (group0 + (int64_t)col_block * tx) * 4; // first feature of the block
        const int cols = NARROW ? kNarrowGroups : tx;              // (NARROW: the row's columns over and over)
        for (int idx = tid; idx < cols * 4 * L; idx += 256) {      // consecutive threads read consecutive floats of the table
            const int fc = idx / L, k = idx - fc * L, f = NARROW ? fc & (4 * tx - 1) : fc;
            const bool have = jb + f < n;
            const float val = have ? __ldg(levels + (jb + f) * L + k) : 0.0f;
            const float next = have && k < L - 1 ? __ldg(levels + (jb + f) * L + k + 1) : val;
            const float width = __fsub_rn(next, val);
            // An empty cell, and one whose width overflows, takes no value up: its reciprocal is stored as 0, and so are its quotients.
            const bool takes = width > 0.0f && width <= 3.402823466e+38f;
            if (takes && !(width >= 9.1e-13f && width <= 1.09e12f)) divide = true;
            const int at = (fc & 3) * kFeature + k * kCols + (fc >> 2);
            lev_s[at] = k < L - 1 ? val : INFINITY;
            // (a numerator above width 2^-150 has a quotient that is not rounded to 0; at and below it it is)
            cell_s[at] = make_float4(val, takes ? width : 1.0f, takes ? __frcp_rn(width) : 0.0f,
                                     takes ? __fmul_rd(__fmul_rn(width, 0x1p-75f), 0x1p-75f) : INFINITY);
        }
        divide = __syncthreads_or(divide);
    }
    float flo[4] = {0.0f, 0.0f, 0.0f, 0.0f}, finv[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    float seen_lo[4], seen_hi[4], probe = 0.0f;                    // TABLE: the extremes of this thread's rows; NaN once a value is not finite
    float mid[4];                                                  // TABLE: where the bisection starts
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if constexpr (!TABLE) {
            if (i < nf) { flo[i] = __ldg(lo + j0 + i); finv[i] = __ldg(inv + j0 + i); }
        } else {
            seen_lo[i] = INFINITY; seen_hi[i] = -INFINITY;
            mid[i] = lev_s[i * kFeature + L / 2 * kCols + col];
        }
    }
    const uint32_t top = ((1u << bits) - 1u) << 24;
    // the blocks run from the last rows to the first: the range pass has left the end of A in L2
    const int64_t row_first = ((int64_t)(row_blocks - 1 - row_block) * blockDim.y + threadIdx.y) * kQuantRows * passes;
    // (rows above 2^32: a block holds a power of two of them, at its multiple, so all its rows have the same upper half)
    const uint32_t row_hi = (uint32_t)((uint64_t)row_first >> 32), pair0 = (uint32_t)(j0 >> 1);
    uint32_t row0 = (uint32_t)row_first;
    int left = (int)max((int64_t)0, min((int64_t)kQuantRows * passes, m - row_first));   // rows from this pass on
    const float* src = A + row_first * lda + j0;                   // the row that is requested next
    uint8_t* out1 = plane1 + row_first * row_bytes + g * (int64_t)sizeof(Word);
    uint8_t* out2 = plane2 + row_first * row_bytes + g * (int64_t)sizeof(Word);
    // the part of the Philox rounds 0 and 1 that depends on the pair alone
    uint32_t pair_lo[2];
    uint64_t pair_p[2];
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const uint64_t a = (uint64_t)kPhiloxM1 * (pair0 + p);
        pair_lo[p] = (uint32_t)a ^ key.k0[1];
        pair_p[p] = (uint64_t)kPhiloxM0 * ((uint32_t)(a >> 32) ^ row_hi ^ key.k0[0]);
    }
    // The rows of a warp, with everything that depends on the matrix's edges compiled out where it lies inside.
    auto run = [&](auto inside, auto divides) {
        constexpr bool kInside = decltype(inside)::value;
        [[maybe_unused]] constexpr bool kDivide = decltype(divides)::value;
        // cell << 24 plus threshold of value x of feature i
        auto decide = [&](float x, int i) -> uint32_t {
            if constexpr (!TABLE) {
                // (the conversion saturates: negative values and NaN at 0, large ones and infinity at 2^32 - 1)
                return min(__float2uint_ru(__fmul_rn(__fmul_rn(__fsub_rn(x, flo[i]), finv[i]), 16777216.0f)), top);
            } else {
                // level k of the thread's feature i lies kCols floats after level k - 1: byte 1 of the offset is k (the last
                // level is staged as infinity); the search ends at the largest k <= L - 2 whose level is <= x
                static_assert(kCols * sizeof(float) == 256, "a level's offset is its number in byte 1");
                uint32_t at = col * 4u;
                const char* lev = reinterpret_cast<const char*>(lev_s + i * kFeature);
                if (mid[i] <= x) at += L / 2 * 256;
#pragma unroll
                for (int half = L >> 2; half > 0; half >>= 1)
                    if (*reinterpret_cast<const float*>(lev + at + half * 256) <= x) at += half * 256;
                const float4 c = *reinterpret_cast<const float4*>(reinterpret_cast<const char*>(cell_s + i * kFeature) + 4 * at);
                const float num = __fsub_rn(x, c.x);
                const float p = kDivide ? (c.z != 0.0f ? __fdiv_rn(num, c.y) : 0.0f) : quotient(num, c.y, c.z);
                // the upper end (a quotient of 1 or more) is always up
                uint32_t threshold = __float2uint_ru(fminf(__fmul_rn(p, 16777216.0f), 16777216.0f));
                if (!kDivide) threshold = num > c.w ? max(threshold, 1u) : 0u;
                return __byte_perm(at, 0u, 0x1444) + threshold;
            }
        };
        float v[kQuantRows][4];
        auto request = [&](int have) {                             // the next kQuantRows rows, of which `have` exist
            if (kInside && vec_ok) {
#pragma unroll
                for (int r = 0; r < kQuantRows; ++r, src += lda) {
                    const float4 t = __ldg(reinterpret_cast<const float4*>(src));
                    v[r][0] = t.x; v[r][1] = t.y; v[r][2] = t.z; v[r][3] = t.w;
                }
            } else {                                               // (what does not exist is certain)
#pragma unroll
                for (int r = 0; r < kQuantRows; ++r, src += lda)
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[r][i] = kInside || (r < have && i < nf) ? __ldg(src + i) : TABLE ? -INFINITY : flo[i];
            }
        };
        request(left);
#pragma unroll 1
        for (int pass = 0; pass < passes; ++pass, left -= kQuantRows, row0 += kQuantRows) {
            if (!kInside && !__any_sync(0xffffffffu, left > 0)) break;
            uint32_t t[kQuantRows][4];
#pragma unroll
            for (int r = 0; r < kQuantRows; ++r)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (TABLE && (kInside || (r < left && i < nf))) {
                        seen_lo[i] = fminf(seen_lo[i], v[r][i]);
                        seen_hi[i] = fmaxf(seen_hi[i], v[r][i]);
                        probe = fmaf(v[r][i], 0.0f, probe);
                    }
                    t[r][i] = decide(v[r][i], i);
                    if (TABLE && !kInside && i >= nf) t[r][i] = 0u;
                }
            if (pass + 1 < passes) request(left - kQuantRows);
            // a guess from the first row (dense or sparse data look alike in every row), the count where it says sparse
            int total = 4 * kQuantQueue, count = 0;
            uint32_t need = 0u;                                    // bit 2 r + p: pair p of row r has a draw to make
            if (__popc(__ballot_sync(0xffffffffu, ((t[0][0] | t[0][1] | t[0][2] | t[0][3]) & 0xFFFFFFu) != 0u)) <= 20) {
#pragma unroll
                for (int r = 0; r < kQuantRows; ++r)
#pragma unroll
                    for (int p = 0; p < 2; ++p)
                        if (((t[r][2 * p] | t[r][2 * p + 1]) & 0xFFFFFFu) != 0u) need |= 1u << (2 * r + p);
                count = __popc(need);
                total = __reduce_add_sync(0xffffffffu, count);
            }
            uint32_t w1[kQuantRows], w2[kQuantRows];
            if (total > kQuantQueue) {
#pragma unroll
                for (int r = 0; r < kQuantRows; ++r) {
                    const uint64_t a = (uint64_t)kPhiloxM0 * (row0 + r);
                    const uint64_t b = (uint64_t)kPhiloxM1 * ((uint32_t)(a >> 32) ^ draw ^ key.k1[0]);
                    Philox4 rnd[2];
#pragma unroll
                    for (int p = 0; p < 2; ++p)
                        rnd[p] = philox_rounds<2>((uint32_t)(b >> 32) ^ pair_lo[p], (uint32_t)b,
                                                  (uint32_t)(pair_p[p] >> 32) ^ (uint32_t)a ^ key.k1[1], (uint32_t)pair_p[p], key);
                    uint32_t c1[4], c2[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        c1[i] = with_draw(t[r][i], rnd[i >> 1].v[2 * (i & 1)]);
                        c2[i] = with_draw(t[r][i], rnd[i >> 1].v[2 * (i & 1) + 1]);
                    }
                    w1[r] = pack_codes<CB>(c1);
                    w2[r] = pack_codes<CB>(c2);
                }
            } else {
                uint32_t answers = 0u;
                if (total > 0) {                                   // (integers on a grid of integers: no draw at all)
                    answer_s[warp][lane] = 0u;
                    int at = count;                                // exclusive prefix sum over the warp
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int up = __shfl_up_sync(0xffffffffu, at, o);
                        if (lane >= o) at += up;
                    }
                    at -= count;
#pragma unroll
                    for (int k = 0; k < 2 * kQuantRows; ++k)
                        if (need >> k & 1u)
                            queue_s[warp][at++] = make_uint2(__byte_perm(t[k >> 1][2 * (k & 1)], (uint32_t)(lane * 2 * kQuantRows + k), 0x4210),
                                                             t[k >> 1][2 * (k & 1) + 1] & 0xFFFFFFu);
                    __syncwarp();
#pragma unroll 1
                    for (int e0 = 0; e0 < total; e0 += 32) {
                        const uint2 q = queue_s[warp][min(e0 + lane, total - 1)];  // (lanes past the end repeat the last: or-ing twice is harmless)
                        const int owner = q.x >> 27, r = (q.x >> 25) & 3, p = (q.x >> 24) & 1;
                        const uint32_t row = __shfl_sync(0xffffffffu, row0, owner) + r, pair = __shfl_sync(0xffffffffu, pair0, owner) + p;
                        const Philox4 rnd = philox_rounds<0>(row, row_hi, pair, draw, key);
                        const uint32_t t0 = q.x & 0xFFFFFFu, t1 = q.y;
                        const uint32_t up1 = (with_draw(t0, rnd.v[0]) >> 24) | (with_draw(t1, rnd.v[2]) >> 24 << CB);
                        const uint32_t up2 = (with_draw(t0, rnd.v[1]) >> 24) | (with_draw(t1, rnd.v[3]) >> 24 << CB);
                        const int shift = answer_shift<CB>(r, 0) + 2 * p * CB;
                        atomicOr(&answer_s[warp][owner], (up1 | up2 << answer_shift<CB>(0, 1)) << shift);
                    }
                    __syncwarp();
                    answers = answer_s[warp][lane];
                }
                constexpr uint32_t kEach = CB == 8 ? 0x01010101u : CB == 4 ? 0x1111u : 0x55u;
#pragma unroll
                for (int r = 0; r < kQuantRows; ++r) {
                    const uint32_t w = pack_codes<CB>(t[r]);
                    w1[r] = w + (answers >> answer_shift<CB>(r, 0) & kEach);
                    w2[r] = w + (answers >> answer_shift<CB>(r, 1) & kEach);
                }
            }
#pragma unroll
            for (int r = 0; r < kQuantRows; ++r, out1 += row_bytes, out2 += row_bytes)
                if (kInside || (r < left && g < groups)) {
                    *reinterpret_cast<Word*>(out1) = (Word)w1[r];
                    *reinterpret_cast<Word*>(out2) = (Word)w2[r];
                }
        }
    };
    if (TABLE && divide) run(std::false_type{}, std::true_type{});
    else if (__all_sync(0xffffffffu, nf == 4 && left == kQuantRows * passes)) run(std::true_type{}, std::false_type{});
    else run(std::false_type{}, std::false_type{});
    if constexpr (NARROW) {                                        // padding past the block's groups
        out1 = plane1 + row_first * row_bytes;
        out2 = plane2 + row_first * row_bytes;
        const int rows = (int)max((int64_t)0, min((int64_t)kQuantRows * passes, m - row_first));
#pragma unroll 1
        for (int r = 0; r < rows; ++r, out1 += row_bytes, out2 += row_bytes)
#pragma unroll 1
            for (int64_t h = g + tx; h < groups; h += tx) {
                *reinterpret_cast<Word*>(out1 + h * (int64_t)sizeof(Word)) = (Word)0;
                *reinterpret_cast<Word*>(out2 + h * (int64_t)sizeof(Word)) = (Word)0;
            }
    }
    if constexpr (TABLE) {
        if (!(probe == 0.0f)) set_status(range.status, ZIPML_ERR_NONFINITE, 1);
        // (a value that is beaten already needs no atomic: after the first blocks hardly any does)
        const int64_t jk = j0 - group0 * 4;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (i < nf && seen_lo[i] <= seen_hi[i]) {
                const uint32_t a = ~float_order_key(seen_lo[i]), b = float_order_key(seen_hi[i]);
                if (a > *reinterpret_cast<volatile uint32_t*>(range.lo_key + jk + i)) atomicMax(range.lo_key + jk + i, a);
                if (b > *reinterpret_cast<volatile uint32_t*>(range.hi_key + jk + i)) atomicMax(range.hi_key + jk + i, b);
            }
        range_finish(range, col_block, row_blocks, (int64_t)col_block * tx * 4, tx * 4);
    }
}

int launch_quantize(zipml_ctx* ctx, const float* A, int64_t m, int64_t n, int64_t lda, int bits, int level_mode,
                    const float* lo, const float* inv, const float* levels, uint64_t seed, uint32_t draw, uint8_t* plane1,
                    uint8_t* plane2, int64_t row_bytes, float* lo_out, float* step_out) {
    const int cb = container_bits(bits);
    const bool table = level_mode == ZIPML_LEVELS_TABLE;
    const bool vec_ok = (lda % 4 == 0) && ((reinterpret_cast<uintptr_t>(A) & 15) == 0);
    const PhiloxKeys key = philox_keys(seed);
    const int64_t all_groups = row_bytes * 8 / (4 * cb);
    // (level tables: as many columns at a time as the range keys hold)
    const int64_t slab = table ? kRangeColumns / 4 : all_groups;
    for (int64_t group0 = 0; group0 < all_groups; group0 += slab) {
        const int64_t groups = all_groups - group0 < slab ? all_groups - group0 : slab;
        // 256 threads: as many feature groups as the row has (a power of two from 4 to 256; 64 with level tables), the
        // rest row groups.  More passes per thread share the loads of lo and inv (the staging of the tables), as
        // long as the grid still covers the SMs several times over.
        // Narrow rows on level tables that pad themselves to twice their features and more leave the padding out (of a warp's lanes up to seven in eight
        // looked up cells of nothing): 13,421,772 x 5 at 2 bits 1,779 -> 955 us, 4,194,304 x 8 570 -> 321, 2,097,152 x 16 332 -> 171;
        // where nothing is saved this form takes 4 to 15 % longer (24 to 64 features), but for 4 bits, whose tables take 80 KB a block otherwise:
        // 524,288 x 64 207 -> 179.
        int tx = 4;
        while (tx < kNarrowGroups && tx < (n + 3) / 4) tx *= 2;
        const bool narrow = table && all_groups <= kNarrowGroups && (tx < all_groups || bits == 4);
        while (!narrow && tx < (table ? kQuantTableCols : 256) && tx < groups) tx *= 2;
        const int ty = 256 / tx;
        const int64_t col_blocks = narrow ? 1 : (groups + tx - 1) / tx;
        int passes = 1;
        while (passes < (table ? 16 : 8) && (m / (ty * kQuantRows * passes * 2)) * col_blocks >= (int64_t)ctx->sm_count * 16) passes *= 2;
        const size_t smem = table ? (sizeof(float4) + sizeof(float)) * ((size_t)(narrow ? 1 : 4) << bits) * kQuantTableCols : 0;
        auto blocks_of_rows = [&]() { return (m + (int64_t)ty * kQuantRows * passes - 1) / ((int64_t)ty * kQuantRows * passes); };
        while (blocks_of_rows() > 0x7fffffffLL / col_blocks && passes < (1 << 20)) passes *= 2;      // the grid is one-dimensional, columns first
        const int64_t row_blocks = blocks_of_rows();
        if (row_blocks > 0x7fffffffLL / col_blocks) return ZIPML_ERR_WORKSPACE;
        const dim3 grid((unsigned)(row_blocks * col_blocks)), block((unsigned)tx, (unsigned)ty);
        RangeArgs range{};
        if (table) {
            const int64_t j0 = group0 * 4;
            range.n = n - j0 < kRangeColumns ? n - j0 : kRangeColumns;
            range.lo_key = ctx->range_keys; range.hi_key = range.lo_key + kRangeColumns; range.done = range.hi_key + kRangeColumns;
            range.s = (1 << bits) - 1;
            range.lo = lo_out + j0;
            range.step = step_out ? step_out + j0 : nullptr;
        }
        range.status = ctx->d_status;
        auto launch = [&](auto kernel) -> int {
            // (the kernel's own 5 KB of shared memory count towards the 48 KB that need no opt-in)
            if (smem > 40 * 1024) {
                const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
                if (e != cudaSuccess) return cuda_status(e);
            }
            kernel<<<grid, block, smem, ctx->stream>>>(A, m, n, lda, bits, lo, inv, levels, range, key, draw, plane1, plane2, row_bytes, vec_ok,
                                                       passes, (unsigned)col_blocks, (unsigned)row_blocks, group0);
            return ZIPML_OK;
        };
        int rc;
        if (!table) rc = cb == 2 ? launch(quantize_kernel<2, 0, false>) : cb == 4 ? launch(quantize_kernel<4, 0, false>) : launch(quantize_kernel<8, 0, false>);
        else if (narrow)
            rc = bits == 1   ? launch(quantize_kernel<2, 1, true>)
                 : bits == 2 ? launch(quantize_kernel<2, 2, true>)
                 : bits == 3 ? launch(quantize_kernel<4, 3, true>)
                             : launch(quantize_kernel<4, 4, true>);
        else
            rc = bits == 1   ? launch(quantize_kernel<2, 1, false>)
                 : bits == 2 ? launch(quantize_kernel<2, 2, false>)
                 : bits == 3 ? launch(quantize_kernel<4, 3, false>)
                             : launch(quantize_kernel<4, 4, false>);
        if (rc != ZIPML_OK) return rc;
        ctx->launches += 1;
    }
    return cuda_status(cudaGetLastError());
}

// ---------------------------------------------------------------------------------------------
// Layout conversion: row-major planes <-> 128-byte column blocks ([block][row][128 B]).  One thread moves
// 16 bytes; a warp covers four 128-byte pieces (four consecutive rows of one block): 512 contiguous bytes
// on the blocked side, four runs of 128 bytes on the row-major side.  Bytes of a block past the end of
// the row are written as zero (to blocks) or skipped (to rows).
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) convert_layout_kernel(const uint4* __restrict__ in1, const uint4* __restrict__ in2,
                                                             uint4* __restrict__ out1, uint4* __restrict__ out2, int64_t m,
                                                             int64_t row_bytes, int64_t nblk, bool to_blocks) {
    const int64_t pieces = nblk * m;                      // 128-byte pieces of a plane
    const int64_t row16 = row_bytes / 16;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < pieces * 8; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t piece = i >> 3, blk = piece / m, row = piece - blk * m;
        const int64_t c16 = blk * 8 + (i & 7);            // 16-byte column of the row
        const bool inside = c16 < row16;
        const int64_t r_idx = row * row16 + c16;
        if (to_blocks) {
            const uint4 z = make_uint4(0u, 0u, 0u, 0u);
            out1[i] = inside ? __ldg(in1 + r_idx) : z;
            out2[i] = inside ? __ldg(in2 + r_idx) : z;
        } else if (inside) {
            out1[r_idx] = __ldg(in1 + i);
            out2[r_idx] = __ldg(in2 + i);
        }
    }
}

int launch_convert_layout(zipml_ctx* ctx, const zipml_dataset* d, int to_layout, uint8_t* out1, uint8_t* out2) {
    const int64_t nblk = (d->row_bytes + 127) / 128;
    const int64_t units = nblk * d->m * 8;
    int64_t blocks = (units + 255) / 256;
    if (blocks > (int64_t)ctx->sm_count * 32) blocks = (int64_t)ctx->sm_count * 32;
    convert_layout_kernel<<<(unsigned)blocks, 256, 0, ctx->stream>>>(
        reinterpret_cast<const uint4*>(d->plane1), reinterpret_cast<const uint4*>(d->plane2), reinterpret_cast<uint4*>(out1),
        reinterpret_cast<uint4*>(out2), d->m, d->row_bytes, nblk, to_layout == ZIPML_LAYOUT_COLUMN_BLOCKS);
    ctx->launches += 1;
    return cuda_status(cudaGetLastError());
}

}  // namespace zipml
