// Cluster engine of zipml_sgd_epoch on uniform grids, int8 tensor cores, split by rows: one thread-block cluster of nb <= 16 CTAs, the
// minibatch cut into row parts, the packed row into slices that the CTAs own (Supplement "Double Sampling", footnote
// form; "End-to-end Quantization").
//
// A small step is a chain of hand-overs; its arithmetic is little.  So everything that crosses a warp is kept to what
// has to cross:
//   * the model travels as what the dots need of it: the owner of a slice turns its w = step * x~ into fixed point with the
//     slice's own power of two and stores the bytes (four balanced base-256 digits per entry: W + 0x80808080, xor
//     0x80808080), as B fragments, into every CTA's shared memory (st.async, 16 bytes a thread), with the scale and the
//     slice's part of lo^T x~ behind them;
//   * a warp waits for its slice alone, multiplies its 32-byte slabs of the codes (mma.sync m16n8k32 u8 x s8: exact
//     integer sums) and leaves 16 rows x 2 planes of partial dots;                                            barrier
//   * a warp per 16 rows adds them up, subtracts the labels and writes the residuals' digits: 16 rows of plane 1 with
//     r2 and 16 rows of plane 2 with r1 are the 32 entries of one contraction;                                barrier
//   * a warp takes 16-byte columns of one slice (transposing ldmatrix), multiplies, centres the sums (codes less half
//     the top code) and bulk-copies its part of the gradient, a low and a high integer per feature, behind the sum of its
//     residuals, into the owner's shared memory;
//   * the owner adds the nb parts in a fixed order, in double from the integers on (the centred sums and the residuals' sum cancel on
//     rows that are mostly zeros: joined in fp32 the gradient lost 10 to 25 times its precision there), applies Q4, updates its
//     fp32 slice, applies Q3;                                                                                 barrier
//     and publishes.
// Codes of less than 8 bits are masked where they lie in their byte: the shift is in the digits (dots) or comes off the
// sums (gradient).
// The code tiles come a few steps ahead, one tensor copy per plane whose box is as wide as the distance of the rows in
// shared memory, an odd number of 16-byte units (rows above 2 KB: a bulk copy each).
// Larger minibatches take several clusters and several chunks of rows per CTA.  A CTA holds whole rows, so a chunk's dots,
// residuals and gradient need nothing from the others: the codes are read once, and the gradient's parts add up in
// shared memory until the last chunk: as integers, whose unit the first chunk's residuals choose with two bits to spare (sums of fp32 lost
// what the centre adds, sums of doubles cost 6 % at 8,192 x 1,999 at 8 bits), or as doubles over more rows than the integers hold.  The clusters hold replicas of the model: the owners of the same slice hand each
// other their sums through L2 (self-validating 8-byte words, two buffers in turn) and add them in the same order.
// Buffer reuse: a CTA sends its part of step t after its warps have read the digits of step t (first barrier), and an
// owner publishes after all parts have arrived: digits, parts and their sources are free when they are written again.
// The step's machine code has to stay small: what does not fit the instruction cache is fetched again every step (with
// everything inlined and unrolled, 64 to 78 KB, the kernel took twice as long).  So loops are rolled, rare paths and
// random draws are out of line, and nothing is divided inside the loop.
// Every wait is bounded; when one gives up the CTA records ZIPML_ERR_TIMEOUT, skips its later waits, still issues every
// store and copy, and all CTAs meet at a cluster barrier before they exit.
#include <cuda.h>
#include <string.h>

#include "cluster.cuh"
#include "int_digits.cuh"

namespace zipml {

struct SliceArgs {
    const uint8_t* p1;
    const uint8_t* p2;
    const float* lo;
    const float* step;
    const float* b;
    float* x;
    float* grad_out;             // null or 2n
    float* model_out;            // null or n: the model the last executed step's gradient saw
    const int32_t* order;        // device copy of the batch order, or null
    unsigned long long* trace;
    DeviceStatus* status;
    int64_t m, batch, first_step, num_steps, row_bytes;
    uint64_t seed;
    uint32_t epoch;
    float lr;
    int reg;                     // ZIPML_REG_* and its fp32 constant
    float reg_cst;
    int n, bits;
    int model_bits, grad_bits;
    int whole, rows_last;        // batches below `whole` are full, that one has rows_last rows
    double full_scale, last_scale;   // 1 / (2 rows)
    int clusters, chunks;        // clusters; chunks of rows per CTA and step
    int nb, rc, cr, rb;          // CTAs per cluster, rows per CTA, rows per chunk, blocks of 16 rows in a chunk
    unsigned long long* exchange;    // [2][clusters][owners SF][2] words {fp32, tag} between the clusters
    uint32_t tag;                // of the first step; greater than any that the buffer holds
    int owners, sps;             // CTAs that own a slice, 32-byte slabs per slice
    int slabs, cols;             // 32-byte slabs and 16-byte columns that hold features
    int a_parts, a_inv, spw;     // dots: parts of a slice, slabs per part (a warp takes a part and RBC row blocks at a time)
    int b_parts, b_inv, cpw;     // gradient: parts of a slice, 16-byte columns per part
    int p_shift;                 // 2^p_shift lanes share the sum of one owned feature
    int pitch, slots, use_tmap;
    int trace_steps;
};

struct alignas(16) SliceShared {
    double base[16];             // owner: per-warp parts of lo^T x~ (entries past the warps stay zero, here and below)
    double red[2][16];           // owner: per-warp parts of the squared norms of gradient and model
    double nrm_g[kSliceMaxCtas]; // squared norms of the owners' gradients and models
    double nrm_x[kSliceMaxCtas];
    uint64_t full[kSliceMaxSlots], empty[kSliceMaxSlots];
    uint64_t w_bar[kSliceMaxCtas];   // a slice's digits have arrived
    uint64_t part_bar, gn_bar, xn_bar;
    float delta_r;               // value of a unit of the residuals' fixed point, not a number where a residual is none
    int k_r;                     // else it is 2^-k_r
    float wmax[32];              // owner: per-warp maxima of |w|
    uint32_t rmax[16];           // maxima of |residual| of a row block, as bit patterns
    int gave_up;
};

// Shared memory after SliceShared; SF = 32 sps NG features of a slice:
//   wd[owners][sps NG 32 + 4]  words: digits of w [slab][group][t][half][digit], then the scale and lo^T x~ (doubles)
//   psum[owners a_parts][rb][32]  doubles: partial dots in the order of the residuals' contraction
//   rdig[rb][32]  words: digits of the residuals [t][half][digit... ] as B fragments
//   gpart[owners][4 + 2 SF]  this CTA's part of the gradient, slice by slice, behind its sum of residuals and the sums' unit, two
//                          doubles: integers, or (MODE 2) doubles without a unit
//   gbuf[nb][4 + 2 SF]       the parts of the own slice
//   wv[SF]                 w of the own slice
//   ring[slots]: codes [2][16 rb][pitch], 128 bytes of slack
// MODE: 0 = one chunk in one cluster, else several: 1 = of at most fifteen row blocks together, 2 = of more.
template <int CB, int RBC, int MODE>
__global__ void __launch_bounds__(kSliceThreads + 32, 1) sgd_slice_kernel(const SliceArgs a, const __grid_constant__ CUtensorMap tm1,
                                                                     const __grid_constant__ CUtensorMap tm2) {
    constexpr bool MANY = MODE > 0;
    constexpr int NG = IntPath<CB>::NG, NS = IntPath<CB>::NS;
    constexpr int CT = NG == 1 ? 2 : 1;                  // columns that a warp takes at once in the gradient
    static_assert(NS == 4, "a thread stores four digits at once");
    extern __shared__ __align__(16) unsigned char s_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cl = MANY ? blockIdx.x / a.nb : 0, bi = MANY ? blockIdx.x - cl * a.nb : blockIdx.x;
    const int n = a.n, sps = a.sps, owners = a.owners, rb = a.rb, SF = 32 * sps * NG;
    const int wd_words = sps * NG * 32 + 4, part_words = 2 * SF + 4;
    SliceShared* sh = reinterpret_cast<SliceShared*>(s_raw);
    uint32_t* wd = reinterpret_cast<uint32_t*>(s_raw + sizeof(SliceShared));
    double* psum = reinterpret_cast<double*>(wd + owners * wd_words);
    uint32_t* rdig = reinterpret_cast<uint32_t*>(psum + owners * a.a_parts * rb * 32);
    int* gpart = reinterpret_cast<int*>(rdig + rb * 32);
    int* gbuf = gpart + owners * part_words;
    float* wv = reinterpret_cast<float*>(gbuf + a.nb * part_words);
    unsigned char* ring = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(wv + SF) + 127) & ~(uintptr_t)127);
    const int plane_bytes = (16 * rb * a.pitch + 127) & ~127, slot_bytes = 2 * plane_bytes + 128;
    const bool owner = bi < owners;
    const uint32_t part_bytes = 4u * a.nb * (4 + (owner ? min(2 * sps, a.cols - bi * 2 * sps) : 0) * 32 * NG);

    if (tid < a.slots) {
        mbar_init(sh->full + tid, 1);
        mbar_init(sh->empty + tid, kSliceWarps);
    } else if (tid >= 32 && tid < 32 + owners) {
        mbar_init(sh->w_bar + tid - 32, 1);
        mbar_arrive_expect_tx(sh->w_bar + tid - 32, 4u * wd_words);
    } else if (tid == 64) {
        mbar_init(&sh->part_bar, 1);
        mbar_arrive_expect_tx(&sh->part_bar, part_bytes);
    } else if (tid == 65) {
        mbar_init(&sh->gn_bar, 1);
        mbar_arrive_expect_tx(&sh->gn_bar, 8u * owners);
    } else if (tid == 66) {
        mbar_init(&sh->xn_bar, 1);
        mbar_arrive_expect_tx(&sh->xn_bar, 8u * owners);
    } else if (tid == 67) {
        sh->gave_up = 0;
    } else if (tid >= 96 && tid < 128) {
        sh->wmax[tid - 96] = 0.0f;
    } else if (tid >= 128 && tid < 144) {
        const int c = tid - 128;
        sh->nrm_g[c] = sh->nrm_x[c] = sh->base[c] = sh->red[0][c] = sh->red[1][c] = 0.0;
    }
    mbar_fence_init();
    __syncthreads();
    slice_cluster_sync();                                // every CTA's barriers exist before anyone writes into it
    after_previous_kernel(a.num_steps);

    // steps are counted from the call's first one; a batch is named by its index
    const int steps = (int)a.num_steps, whole = a.whole;
    auto batch_at = [&](int k) { return k < steps ? (a.order ? a.order[a.first_step + k] : (int)a.first_step + k) : 0; };
    const int row_base = (cl * a.nb + bi) * a.rc, chunks = MANY ? a.chunks : 1;
    const int rows_full = min(a.rc, (int)a.batch - row_base), rows_last = min(a.rc, a.rows_last - row_base);
    auto rows_of = [&](int batch, int chunk) { return max(0, min(a.cr, (batch < whole ? rows_full : rows_last) - chunk * a.cr)); };
    if (warp == kSliceWarps) {
        // -------------------------------------------------------------------- the copying warp
        int slot = 0;
        uint32_t parity = 1;                             // of the slots' emptiness: all are empty at first
#pragma unroll 1
        for (int k = 0; k < steps; ++k) {
            const int batch = batch_at(k);
#pragma unroll 1
            for (int chunk = 0; chunk < chunks; ++chunk) {
                const int64_t r0 = batch * a.batch + row_base + chunk * a.cr;
                unsigned char* dst = ring + slot * slot_bytes;
                slice_wait(sh, sh->empty + slot, parity, a.status, 84);
                if (a.use_tmap) {                        // (boxes that reach past the last row are filled up and count in full)
                    if (lane == 0) {
                        mbar_arrive_expect_tx(sh->full + slot, 2u * (uint32_t)(a.cr * a.pitch));
                        slice_tensor_copy(dst, &tm1, 0, (int)r0, sh->full + slot);
                        slice_tensor_copy(dst + plane_bytes, &tm2, 0, (int)r0, sh->full + slot);
                    }
                } else {
                    const int rows = rows_of(batch, chunk);
                    if (lane == 0) mbar_arrive_expect_tx(sh->full + slot, 2u * (uint32_t)rows * (uint32_t)a.row_bytes);
                    for (int i = lane; i < 2 * rows; i += 32)
                        bulk_copy_g2s(dst + (i & 1) * plane_bytes + (i >> 1) * a.pitch, (i & 1 ? a.p2 : a.p1) + (r0 + (i >> 1)) * a.row_bytes,
                                      (uint32_t)a.row_bytes, sh->full + slot);
                }
                if (++slot == a.slots) { slot = 0; parity ^= 1u; }
            }
        }
        __syncwarp();
        slice_cluster_sync();
        return;
    }

    int batch = batch_at(0), batch_next = batch_at(1);
    // labels: a lane of the first rb warps forms one residual, of this row of the CTA
    const int res_row = warp * 16 + 2 * ((lane >> 2) & 3) + (lane & 1) + 8 * ((lane >> 1) & 1);
    // (MANY: where the load stands suits it, moved it costs 1 % a step: 8,192 x 1,999 at 6 bits 643 -> 648 us an epoch; else it has to move: 2 bits
    // 500 x 256 3.53 -> 3.34 us)
    const float* labels = MANY ? a.b : from_here_on(a.b);
    auto label_of = [&](int batch, int chunk) {
        if constexpr (MANY) return warp < rb && res_row < rows_of(batch, chunk) ? a.b[batch * a.batch + row_base + chunk * a.cr + res_row] : 0.0f;
        else return warp < rb && res_row < rows_of(batch, chunk) ? load_freely(labels + batch * a.batch + row_base + chunk * a.cr + res_row) : 0.0f;
    };
    float label = label_of(batch, 0);

    // ------------------------------------------------------------------------ the steps
    const int gl = lane >> 2, tl = lane & 3, lm = lane >> 3, l8 = lane & 7;
    // dots: units of a part of a slice and RBC row blocks, dealt to the warps
    const int a_all = owners * a.a_parts;
    const int ws_first = warp % a_all, rb_first = warp / a_all * RBC, ws_more = kSliceWarps % a_all, rb_more = kSliceWarps / a_all * RBC;
    // owner: the pieces of its digits and their destinations, dealt to the threads; feature of this thread
    const int items = 8 * sps * NG, item_first = tid % items, dest_first = tid / items, item_more = kSliceThreads % items, dest_more = kSliceThreads / items;
    const int P = 1 << a.p_shift, pp = tid & (P - 1), k_own = tid >> a.p_shift;
    const int f_own = bi * SF + k_own;
    const bool mine = owner && k_own < SF && f_own < n;
    const int c0 = 1 << (a.bits - 1);
    const float st = mine ? a.step[f_own] : 0.0f, lof = mine ? a.lo[f_own] : 0.0f;
    const double mid = fma((double)c0, (double)st, (double)lof);
    const double st_low = (double)st / (double)(1 << (CB * (k_own % NG)));    // (codes were multiplied where they lie in their byte)
    float x = mine ? a.x[f_own] : 0.0f;
    auto draw = [&](int k, uint32_t stream) { return slice_draw(a.seed, a.epoch, (uint32_t)a.first_step + (uint32_t)k, (uint32_t)f_own, stream); };

    const int marked = blockIdx.x == 0 && tid == 0 && a.trace ? a.trace_steps : -1;
    int slot = 0;
    uint32_t parity = 0, w_parity = 0, part_parity = 0, gn_parity = 0, xn_parity = 0;
    int k_sum = 0;                                       // MODE 1: the unit of the sums over a step's chunks is 2^-k_sum
#pragma unroll 1
    for (int step = -1; step < steps; ++step) {
        const bool last = step == steps - 1;
        uint32_t u_x = 0u, u_g = 0u;
        if (step >= 0) {
            if (step < marked) slice_mark(a.trace, step, 0);
            bool batch_full = true;
#pragma unroll 1
            for (int chunk = 0; chunk < chunks; ++chunk) {
            const bool final_chunk = chunk == chunks - 1;
            const uint32_t tile_addr = smem_u32(ring) + (uint32_t)(slot * slot_bytes);
            slice_wait(sh, sh->full + slot, parity, a.status, 6);
            // -------------------------------------------------------------- dots
#pragma unroll 1
            for (int ws = ws_first, rb0 = rb_first; rb0 < rb;) {
                const int a_slice = (ws * a.a_inv) >> 16;           // ws / a_parts
                const int slab0 = (ws - a_slice * a.a_parts) * a.spw, slab1 = min(min(sps, a.slabs - a_slice * sps), slab0 + a.spw);
                const bool keeper = slab0 == 0 && rb0 == 0 && chunk == 0;         // re-arms the slice's barrier
                slice_wait(sh, sh->w_bar + a_slice, w_parity, a.status, 4);
                if (keeper && lane == 0 && !last) mbar_arrive_expect_tx(sh->w_bar + a_slice, 4u * wd_words);
                if (step < marked) slice_mark(a.trace, step, 1);
                const uint32_t* wsl = wd + a_slice * wd_words;
                const double delta = *reinterpret_cast<const double*>(wsl + wd_words - 4);
                const double base = slab0 == 0 ? *reinterpret_cast<const double*>(wsl + wd_words - 2) : 0.0;
                {
                    int c[2][RBC][4];
#pragma unroll
                    for (int pl = 0; pl < 2; ++pl)
#pragma unroll
                        for (int i = 0; i < RBC; ++i)
#pragma unroll
                            for (int e = 0; e < 4; ++e) c[pl][i][e] = 0;
                    // lane's address of a fragment: row l8 (+ 8 for the odd matrices), bytes 0 or 16 of the slab
                    uint32_t addr = tile_addr + (uint32_t)((rb0 * 16 + l8 + (lm & 1) * 8) * a.pitch) + (uint32_t)((a_slice * sps + slab0) * 32 + (lm >> 1) * 16);
                    const uint32_t* wq = wsl + slab0 * NG * 32 + tl * 8 + (gl & 3);
#pragma unroll 1
                    for (int ks = slab0; ks < slab1; ++ks, addr += 32u, wq += NG * 32) {
                        uint32_t bf[NG][2];
#pragma unroll
                        for (int g = 0; g < NG; ++g) {
                            bf[g][0] = gl < NS ? wq[g * 32] : 0u;
                            bf[g][1] = gl < NS ? wq[g * 32 + 4] : 0u;
                        }
#pragma unroll
                        for (int i = 0; i < RBC; ++i) {
                            if (RBC == 1 || rb0 + i < rb) {
                                uint32_t a1[4], a2[4];
                                ldsm_x4(a1, addr + (uint32_t)(i * 16 * a.pitch));
                                ldsm_x4(a2, addr + (uint32_t)(i * 16 * a.pitch + plane_bytes));
#pragma unroll
                                for (int g = 0; g < NG; ++g) {
                                    mma_u8s8(c[0][i], slice_dot_codes<CB>(a1[0], g), slice_dot_codes<CB>(a1[1], g), slice_dot_codes<CB>(a1[2], g),
                                             slice_dot_codes<CB>(a1[3], g), bf[g][0], bf[g][1]);
                                    mma_u8s8(c[1][i], slice_dot_codes<CB>(a2[0], g), slice_dot_codes<CB>(a2[1], g), slice_dot_codes<CB>(a2[2], g),
                                             slice_dot_codes<CB>(a2[3], g), bf[g][0], bf[g][1]);
                                }
                            }
                        }
                    }
                    // lane t = 0 has digits 0, 1 of rows g and g + 8, lane t = 1 digits 2, 3: the first takes row g, the
                    // other row g + 8.  Plane 1's dot belongs to r1, which meets plane 2's codes: entries 16 .. 31.
#pragma unroll
                    for (int i = 0; i < RBC; ++i) {
                        if (RBC == 1 || rb0 + i < rb) {
#pragma unroll
                            for (int pl = 0; pl < 2; ++pl) {
                                const long long upper = c[pl][i][0] + 256ll * c[pl][i][1], lower = c[pl][i][2] + 256ll * c[pl][i][3];
                                const long long got = __shfl_xor_sync(0xffffffffu, tl == 0 ? lower : upper, 1);
                                const long long v = tl == 0 ? upper + 65536ll * got : got + 65536ll * lower;
                                const int k = (pl == 0 ? 16 : 0) + 4 * (gl >> 1) + (gl & 1) + 2 * tl;
                                if (tl < 2) psum[(ws * rb + rb0 + i) * 32 + k] = (double)v * delta + base;
                            }
                        }
                    }
                }
                ws += ws_more; rb0 += rb_more;
                if (ws >= a_all) { ws -= a_all; rb0 += RBC; }
            }
            if (a.grad_bits > 0 && mine && pp == 0 && chunk == 0) u_g = draw(step, 4u);
            if (a.model_bits > 0 && mine && pp == 0 && chunk == 0) u_x = draw(step + 1, 3u);
            slice_bar();

            // -------------------------------------------------------------- residuals and their digits
            if (warp < rb) {
                double d[4] = {-(double)label, 0.0, 0.0, 0.0};
                const double* ps = psum + warp * 32 + lane;
#pragma unroll 1
                for (int w = 0; w < a_all; w += 4)
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (w + i < a_all) d[i] += ps[(w + i) * rb * 32];
                const float r = res_row < rows_of(batch, chunk) ? (float)((d[0] + d[1]) + (d[2] + d[3])) : 0.0f;
                // (largest as bit patterns: a residual that is not a number wins, and the gradient is none either)
                uint32_t top_bits = __reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(r)));
                if (rb > 1) {                            // one scale for all row blocks
                    if (lane == 0) sh->rmax[warp] = top_bits;
                    asm volatile("bar.sync 2, %0;" ::"r"(32 * rb) : "memory");
#pragma unroll 1
                    for (int w2 = 0; w2 < rb; ++w2) top_bits = max(top_bits, sh->rmax[w2]);
                }
                const float top = __uint_as_float(top_bits);
                int k_r = slice_exponent(top, 0);
                if constexpr (MODE == 1) k_r = chunk > 0 && k_r >= k_sum ? k_sum : slice_exponent(top, 2);   // (two bits for the chunks to come)
                if (tid == 0) { sh->delta_r = top <= 3.402823466e+38f ? slice_pow2(-k_r) : __int_as_float(0x7fffffff); sh->k_r = k_r; }
                const uint32_t digits = ((uint32_t)__float2int_rn(r * slice_pow2(k_r)) + 0x80808080u) ^ 0x80808080u;
                unsigned char* out = reinterpret_cast<unsigned char*>(rdig + warp * 32) + ((lane >> 2) & 3) * 32 + (lane >> 4) * 16 + (lane & 3);
#pragma unroll
                for (int s = 0; s < NS; ++s) out[4 * s] = (unsigned char)(digits >> (8 * s));
            }
            if (final_chunk) {
                batch_full = batch < whole;
                batch = batch_next;
                batch_next = batch_at(step + 2);
            }
            label = label_of(batch, final_chunk ? 0 : chunk + 1);
            slice_bar();
            if (step < marked) slice_mark(a.trace, step, 2);

            // -------------------------------------------------------------- the rows' part of the gradient
            const double unit_r = (double)sh->delta_r;
            const int k_r = sh->k_r, coarser = MODE == 1 && chunk > 0 ? min(63, k_sum - k_r) : 0;    // bits that the sums so far come down
            k_sum = k_r;
#pragma unroll 1
            for (int unit = warp; unit < owners * a.b_parts; unit += kSliceWarps) {
                const int b_slice = (unit * a.b_inv) >> 16, bj = unit - b_slice * a.b_parts;     // unit / b_parts
                const int col_begin = bj * a.cpw, col_end = min(min(2 * sps, a.cols - b_slice * 2 * sps), col_begin + a.cpw);
                if (col_begin >= col_end) continue;
                int* part = gpart + b_slice * part_words;
                const uint32_t row_addr = tile_addr + (uint32_t)((lane >> 4) * plane_bytes + (lane & 15) * a.pitch + b_slice * sps * 32);
                const uint32_t* rq = rdig + tl * 8 + (gl & 3);
                int ones[4] = {0, 0, 0, 0};              // the digits' sums
#pragma unroll 1
                for (int kb = 0; kb < rb; ++kb)
                    mma_u8s8(ones, 0x01010101u, 0x01010101u, 0x01010101u, 0x01010101u, gl < NS ? rq[kb * 32] : 0u, gl < NS ? rq[kb * 32 + 4] : 0u);
                if (bj == 0) {                           // the sum of the residuals, and the unit of the features' sums
                    const int s = ones[0] + 256 * ones[1], upper = __shfl_down_sync(0xffffffffu, s, 1);
                    if (lane == 0) {
                        double2* head = reinterpret_cast<double2*>(part);
                        *head = make_double2(fma(slice_double(s, upper), unit_r, MANY && chunk > 0 ? head->x : 0.0), __hiloint2double((1023 - k_r) << 20, 0));
                    }
                }
                if (MODE == 1 && coarser > 0) {          // (seldom: a chunk's largest residual is four times the earlier ones')
#pragma unroll 1
                    for (int w = 4 + col_begin * 32 * NG + 2 * lane; w < 4 + col_end * 32 * NG; w += 64) {
                        int2* pair = reinterpret_cast<int2*>(part + w);
                        const long long v = (pair->x + 65536ll * pair->y) >> coarser;
                        *pair = make_int2((int)(v & 0xffff), (int)(v >> 16));
                    }
                    __syncwarp();
                }
#pragma unroll 1
                for (int col0 = col_begin; col0 < col_end; col0 += CT) {
                    int acc[CT][NG][4];
#pragma unroll 1
                    for (int kb = 0; kb < rb; ++kb) {
                        const uint32_t b0 = gl < NS ? rq[kb * 32] : 0u, b1 = gl < NS ? rq[kb * 32 + 4] : 0u;
#pragma unroll
                        for (int ti = 0; ti < CT; ++ti) {
                            if (col0 + ti < col_end) {
                                uint32_t r4[4];
                                ldsm_x4_trans(r4, row_addr + (uint32_t)(kb * 16 * a.pitch + (col0 + ti) * 16));
                                const uint32_t pel = __byte_perm(r4[0], r4[1], 0x6420), pol = __byte_perm(r4[0], r4[1], 0x7531);
                                const uint32_t peh = __byte_perm(r4[2], r4[3], 0x6420), poh = __byte_perm(r4[2], r4[3], 0x7531);
#pragma unroll
                                for (int g = 0; g < NG; ++g) {
                                    // sums of (code - c0) * residual, codes where they lie: c0 times the digits' sums come off first
                                    const int from = -(c0 << (CB * g));
                                    if (RBC == 1 || kb == 0)
                                        slice_mma_from(acc[ti][g], slice_codes<CB>(pel, g), slice_codes<CB>(pol, g), slice_codes<CB>(peh, g),
                                                       slice_codes<CB>(poh, g), b0, b1, from * ones[0], from * ones[1]);
                                    else
                                        mma_u8s8(acc[ti][g], slice_codes<CB>(pel, g), slice_codes<CB>(pol, g), slice_codes<CB>(peh, g),
                                                 slice_codes<CB>(poh, g), b0, b1);
                                }
                            }
                        }
                    }
                    // rows g, g + 8 of the accumulators are bytes 2g, 2g + 1 of the column
#pragma unroll
                    for (int ti = 0; ti < CT; ++ti) {
                        if (col0 + ti < col_end) {
#pragma unroll
                            for (int g = 0; g < NG; ++g) {
                                int* out = part + 4 + 2 * (((col0 + ti) * 16 + 2 * gl) * NG + g) + tl;
                                // lane t = 0 has the lower digits, t = 1 the upper ones (fifteen row blocks at most: below 2^31)
                                const int first = acc[ti][g][0] + 256 * acc[ti][g][1], second = acc[ti][g][2] + 256 * acc[ti][g][3];
                                if constexpr (MODE == 2) {         // (chunks with scales of their own, a feature to a lane)
                                    const int got = __shfl_xor_sync(0xffffffffu, tl == 0 ? second : first, 1);
                                    double* sum = reinterpret_cast<double*>(out - tl + 2 * NG * tl);
                                    if (tl < 2) *sum = fma(slice_double(tl == 0 ? first : got, tl == 0 ? got : second), unit_r, chunk > 0 ? *sum : 0.0);
                                } else if (tl < 2) {
                                    out[0] = (MODE == 1 && chunk > 0 ? out[0] : 0) + first;
                                    out[2 * NG] = (MODE == 1 && chunk > 0 ? out[2 * NG] : 0) + second;
                                }
                            }
                        }
                    }
                }
                if (!final_chunk) continue;
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    const int w0 = bj == 0 ? 0 : 4 + col_begin * 32 * NG, w1 = 4 + col_end * 32 * NG;
                    slice_copy(slice_peer(gbuf + bi * part_words + w0, b_slice), part + w0, 4u * (w1 - w0), slice_peer(&sh->part_bar, b_slice));
                }
            }
            if (lane == 0) mbar_arrive(sh->empty + slot);
            if (++slot == a.slots) { slot = 0; parity ^= 1u; }
            }
            w_parity ^= 1u;
            if (step < marked) slice_mark(a.trace, step, 3);

            // -------------------------------------------------------------- the owner sums the parts and updates
            if (owner) {
                slice_wait(sh, &sh->part_bar, part_parity, a.status, 2);
                part_parity ^= 1u;
                if (tid == 0 && !last) mbar_arrive_expect_tx(&sh->part_bar, part_bytes);
                double t = 0.0, all = 0.0;               // sums of the codes and of the residuals
                if (mine)
#pragma unroll 2
                    for (int w = pp; w < a.nb; w += P) {
                        const int* part = gbuf + w * part_words;
                        const double2 h = *reinterpret_cast<const double2*>(part);
                        if constexpr (MODE == 2) {
                            t += reinterpret_cast<const double*>(part)[2 + k_own];
                        } else {
                            const int2 v = *reinterpret_cast<const int2*>(part + 4 + 2 * k_own);
                            t = fma(slice_double(v.x, v.y), h.y, t);
                        }
                        all += h.x;
                    }
                t = fma(st_low, t, mid * all);
#pragma unroll 1
                for (int o = 1; o < P; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                if (MANY && a.clusters > 1) {
                    const uint32_t tag = a.tag + (uint32_t)step;
                    unsigned long long* box = a.exchange + ((size_t)(step & 1) * a.clusters * owners * SF + f_own) * 2;
                    const size_t stride = (size_t)owners * SF * 2;
                    const float hi = (float)t, low = (float)(t - (double)hi);
                    if (mine && pp == 0) slice_post(box + cl * stride, hi, low, tag);
                    t = 0.0;
                    if (mine)
#pragma unroll 1
                        for (int c = pp; c < a.clusters; c += P) t += c == cl ? (double)hi + (double)low : slice_collect(sh, box + c * stride, tag, a.status);
#pragma unroll 1
                    for (int o = 1; o < P; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                }
                float g = (float)(t * (batch_full ? a.full_scale : a.last_scale));
                const bool writes = mine && pp == 0;
                if (last && a.grad_out && writes && cl == 0) a.grad_out[f_own] = g;
                if (step < marked) slice_mark(a.trace, step, 4);
                if (a.grad_bits > 0) {
                    const float M = slice_norm(writes ? (double)g * (double)g : 0.0, P, bi, sh->red[0], sh->nrm_g, &sh->gn_bar, gn_parity, owners, sh, a.status, 3);
                    gn_parity ^= 1u;
                    g = slice_quantize(g, M, a.grad_bits, u_g);
                }
                if (last && a.grad_out && writes && cl == 0) a.grad_out[n + f_own] = g;
                const float y = fmaf(-a.lr, g, x);
                x = a.reg == ZIPML_REG_NONE ? y : slice_regularise(y, x, a.reg, a.reg_cst);
            }
        } else if (a.model_bits > 0 && mine && pp == 0) {
            u_x = draw(step + 1, 3u);
        }
        if (last) break;

        // ------------------------------------------------------------------ publish what the next step sees
        if (owner) {
            float xt = x;
            if (a.model_bits > 0) {
                const float M = slice_norm(mine && pp == 0 ? (double)x * (double)x : 0.0, P, bi, sh->red[1], sh->nrm_x, &sh->xn_bar, xn_parity, owners, sh, a.status, 8);
                xn_parity ^= 1u;
                xt = slice_quantize(x, M, a.model_bits, u_x);
            }
            const bool writes = mine && pp == 0;
            if (a.model_out && step + 2 == steps && writes && cl == 0) a.model_out[f_own] = xt;
            const float w = writes ? st * xt : 0.0f;
            if (pp == 0 && k_own < SF) wv[k_own] = w;
            const float top = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(w))));
            double bpart = writes ? (double)lof * (double)xt : 0.0;
#pragma unroll 1
            for (int o = 16; o >= P; o >>= 1) bpart += __shfl_xor_sync(0xffffffffu, bpart, o);
            if (lane == 0) { sh->wmax[warp] = top; sh->base[warp] = bpart; }
            slice_bar();
            const float wmax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(sh->wmax[lane])));
            const int k_w = slice_exponent(wmax, SliceShift<CB>::kMost);
            const float inv = slice_pow2(k_w);
#pragma unroll 1
            for (int item = item_first, dest = dest_first; dest < a.nb;) {
                const int half = item & 1, t = (item >> 1) & 3, gs = item >> 3, g = gs % NG, q = (gs / NG) * 8 + half * 4 + t;
                const float* src = wv + q * 4 * NG + g;
                const float up = inv * (float)(1 << SliceShift<CB>::of(g));
                uint32_t d[4];
                transpose4x4((uint32_t)__float2int_rn(src[0] * up) + 0x80808080u, (uint32_t)__float2int_rn(src[NG] * up) + 0x80808080u,
                             (uint32_t)__float2int_rn(src[2 * NG] * up) + 0x80808080u, (uint32_t)__float2int_rn(src[3 * NG] * up) + 0x80808080u, d);
                slice_store16(slice_peer(wd + bi * wd_words + 4 * item, dest),
                              make_uint4(d[0] ^ 0x80808080u, d[1] ^ 0x80808080u, d[2] ^ 0x80808080u, d[3] ^ 0x80808080u), slice_peer(sh->w_bar + bi, dest));
                item += item_more; dest += dest_more;
                if (item >= items) { item -= items; ++dest; }
            }
            if (tid >= kSliceThreads - a.nb) {           // the scale and lo^T x~
                const int dest = tid - (kSliceThreads - a.nb);
                const unsigned long long s = wmax <= 3.402823466e+38f ? (unsigned long long)(1023 - k_w - SliceShift<CB>::kMost) << 52   // 2^-(k_w + kMost)
                                                                      : 0x7fffffffffffffffull;
                const unsigned long long l = (unsigned long long)__double_as_longlong(slice_sum16(sh->base));
                slice_store16(slice_peer(wd + bi * wd_words + wd_words - 4, dest), make_uint4((uint32_t)s, (uint32_t)(s >> 32), (uint32_t)l, (uint32_t)(l >> 32)),
                              slice_peer(sh->w_bar + bi, dest));
            }
        }
        if (step >= 0 && step < marked) slice_mark(a.trace, step, 5);
    }
    if (mine && pp == 0 && cl == 0) a.x[f_own] = x;
    __syncwarp();
    slice_cluster_sync();                                // nobody leaves while a copy may still target it
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
struct SlicePlan {
    int clusters, chunks, nb, rc, cr, rb, owners, sps, slabs, cols, a_parts, spw, b_parts, cpw, p_shift, pitch, slots;
    size_t smem;
};

static size_t slice_smem_bytes(const SlicePlan& r, int ng, int slots) {
    const size_t sf = (size_t)32 * r.sps * ng;
    size_t bytes = sizeof(SliceShared) + 4 * (size_t)r.owners * ((size_t)r.sps * ng * 32 + 4) + 8 * (size_t)r.owners * r.a_parts * r.rb * 32 +
                   4 * (size_t)r.rb * 32 + 4 * (size_t)(r.owners + r.nb) * (2 * sf + 4) + 4 * sf + 128;
    return bytes + (size_t)slots * (2 * (((size_t)16 * r.rb * r.pitch + 127) & ~(size_t)127) + 128);
}

// How many clusters (most: as many as can be resident at once): one for 16 rows per CTA where a step has the work to pay
// for their exchange (about 1.2 us), batch x (features + 128).  Measured, us per step with 1 / 2 / 4 / 8 clusters: 8 bits 512 x 1,000
// 4.6 / 4.8 / 5.0 / 6.6, 1,024 x 1,000 8.5 / 6.1 / 5.1 / 5.6, 4,096 x 1,000 28.9 / 16.7 / 10.2 / 8.7, 2,400 x 287 7.1 / 6.6 / 6.2 / 5.3; 4 bits
// 1,024 x 64 3.7 / 4.4 / 4.1 / 4.2, 4,096 x 64 7.5 / 5.4 / 5.0 / 5.0, 512 x 512 3.8 / 4.2 / 4.3 / 4.9, 384 x 4,035 10.8 / 8.2 / 8.7 / 10.5; 2 bits 1,024 x
// 2,048 7.8 / 7.5 / 6.3 / 7.3.
static int slice_clusters(int64_t B, int64_t n, int most) {
    if (B * (n + 128) < 650000) return 1;
    const int64_t want = (B + 16 * kSliceMaxCtas - 1) / (16 * kSliceMaxCtas);
    return (int)(want > most ? most : want);
}

static int make_slice_plan(const zipml_ctx* ctx, const zipml_dataset* d, const zipml_sgd_params* p, int most_clusters, SlicePlan* plan) {
    const int cb = container_bits(d->bits), ng = 8 / cb;
    const int64_t B = p->batch < d->m ? p->batch : d->m;
    const int64_t used = (d->n * cb + 7) / 8, slabs = (used + 31) / 32;
    if (d->n > kSliceMaxCtas * kSliceThreads) return ZIPML_ERR_WORKSPACE;      // (a thread per feature of a slice)
    if (d->level_mode != ZIPML_LEVELS_UNIFORM || (d->m + B - 1) / B > 0x7ffffff0 || slabs > 1024 || d->row_bytes > (1 << 16) || B > (1 << 24)) return ZIPML_ERR_WORKSPACE;
    int64_t clusters = p->grid_feature_parts > 0 ? p->grid_feature_parts : slice_clusters(B, d->n, most_clusters);
    if (clusters > most_clusters) clusters = most_clusters;
    const int64_t Bc = (B + clusters - 1) / clusters;
    int64_t nb = p->grid_row_parts > 0 ? p->grid_row_parts : (Bc + 15) / 16;    // automatic: 16 rows per CTA
    if (nb > kSliceMaxCtas) nb = kSliceMaxCtas;
    if (nb > Bc) nb = Bc;
    for (; nb <= kSliceMaxCtas && nb <= Bc; ++nb) {      // (more parts than asked for where a tile or a slice does not fit)
        SlicePlan r;
        r.clusters = (int)clusters;
        r.rc = (int)((Bc + nb - 1) / nb);
        r.nb = (int)((Bc + r.rc - 1) / r.rc);
        r.sps = (int)((slabs + r.nb - 1) / r.nb);
        r.owners = (int)((slabs + r.sps - 1) / r.sps);
        r.slabs = (int)slabs; r.cols = (int)((used + 15) / 16);
        if (32 * r.sps * ng > kSliceThreads) continue;
        const int per = r.owners < kSliceWarps ? kSliceWarps / r.owners : 1;
        r.spw = (r.sps + per - 1) / per;
        r.a_parts = (r.sps + r.spw - 1) / r.spw;
        r.cpw = (2 * r.sps + per - 1) / per;
        r.b_parts = (2 * r.sps + r.cpw - 1) / r.cpw;
        r.p_shift = 0;
        while (r.p_shift < 4 && (32 * r.sps * ng) << (r.p_shift + 1) <= kSliceThreads && (1 << r.p_shift) < r.nb) ++r.p_shift;
        const int units = (int)(d->row_bytes / 16);
        r.pitch = 16 * (units | 1);
        // as few chunks as leave two slots, equally long
        const int blocks = (r.rc + 15) / 16;
        for (r.chunks = (blocks + 14) / 15; r.chunks <= blocks; ++r.chunks) {
            r.rb = (blocks + r.chunks - 1) / r.chunks;
            if (slice_smem_bytes(r, ng, 2) <= (size_t)ctx->smem_optin) break;
        }
        if (r.chunks > blocks) continue;
        r.chunks = (blocks + r.rb - 1) / r.rb;
        r.cr = r.chunks == 1 ? r.rc : 16 * r.rb;
        r.slots = kSliceMaxSlots;
        while (slice_smem_bytes(r, ng, r.slots) > (size_t)ctx->smem_optin) --r.slots;
        r.smem = slice_smem_bytes(r, ng, r.slots);
        *plan = r;
        return ZIPML_OK;
    }
    return ZIPML_ERR_WORKSPACE;
}

template <int CB, int RBC>
static const void* slice_kernel(int mode) {
    return mode == 0 ? (const void*)sgd_slice_kernel<CB, RBC, 0> : mode == 1 ? (const void*)sgd_slice_kernel<CB, RBC, 1> : (const void*)sgd_slice_kernel<CB, RBC, 2>;
}
template <int CB>
static const void* slice_kernel(const SlicePlan& r) {
    const int mode = r.clusters == 1 && r.chunks == 1 ? 0 : (r.rc + 15) / 16 <= 15 ? 1 : 2;
    return r.rb == 1 ? slice_kernel<CB, 1>(mode) : slice_kernel<CB, 2>(mode);
}

int launch_sgd_slice(zipml_ctx* ctx, const zipml_dataset* d, const float* b, float* x, const zipml_sgd_params* p, int64_t first_step,
                     int64_t num_steps, float* grad_out) {
    const int cb = container_bits(d->bits);
    if (cb == 0) return ZIPML_ERR_UNSUPPORTED;
    SlicePlan plan;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    const void* kernel = nullptr;
    int rc;
    // (clusters are taken back until all of them can be resident at once: they wait for one another)
    for (int most = kSliceMaxClusters;;) {
        rc = make_slice_plan(ctx, d, p, ctx->cooperative ? most : 1, &plan);
        if (rc != ZIPML_OK) return rc;
        kernel = cb == 2 ? slice_kernel<2>(plan) : cb == 4 ? slice_kernel<4>(plan) : slice_kernel<8>(plan);
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plan.smem);
        if (e == cudaSuccess && plan.nb > 8) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return cuda_status(e);
        memset(&cfg, 0, sizeof(cfg));
        cfg.gridDim = dim3((unsigned)(plan.nb * plan.clusters));
        cfg.blockDim = dim3(kSliceThreads + 32);
        cfg.dynamicSmemBytes = plan.smem;
        cfg.stream = ctx->stream;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)plan.nb;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeCooperative;
        attr[1].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int fit = 0;
        e = cudaOccupancyMaxActiveClusters(&fit, kernel, &cfg);
        if (e != cudaSuccess) { (void)cudaGetLastError(); return ZIPML_ERR_WORKSPACE; }
        if (fit < 1) return ZIPML_ERR_WORKSPACE;
        if (fit >= plan.clusters) break;
        most = fit;
    }
    if (plan.clusters > 1 || early_start(ctx, num_steps, attr + 1)) cfg.numAttrs = 2;      // (a cooperative launch, or one that starts early)
    const int64_t T = (d->m + p->batch - 1) / p->batch;
    SliceArgs a;
    memset(&a, 0, sizeof(a));
    if (p->batch_order) {
        rc = ws_reserve(ctx, carve_size(sizeof(int32_t) * (size_t)T));
        if (rc != ZIPML_OK) return rc;
        const cudaError_t e = cudaMemcpyAsync(ctx->ws, p->batch_order, sizeof(int32_t) * (size_t)T, cudaMemcpyHostToDevice, ctx->stream);
        if (e != cudaSuccess) return cuda_status(e);
        a.order = reinterpret_cast<const int32_t*>(ctx->ws);
    }
    a.p1 = d->plane1; a.p2 = d->plane2; a.lo = d->feat_lo; a.step = d->feat_step;
    a.b = b; a.x = x; a.grad_out = grad_out; a.model_out = p->model_out;
    a.trace = reinterpret_cast<unsigned long long*>(p->trace);
    a.trace_steps = p->trace ? p->trace_steps : 0;
    a.status = ctx->d_status;
    a.m = d->m; a.batch = p->batch < d->m ? p->batch : d->m; a.row_bytes = d->row_bytes;
    a.first_step = first_step; a.num_steps = num_steps;
    a.whole = (int)(d->m / a.batch); a.rows_last = (int)(d->m - a.whole * a.batch);
    a.full_scale = 1.0 / (2.0 * (double)a.batch); a.last_scale = 1.0 / (2.0 * (double)(a.rows_last > 0 ? a.rows_last : 1));
    a.seed = p->seed; a.epoch = (uint32_t)p->epoch; a.lr = p->lr; a.reg = p->reg; a.reg_cst = reg_constant(p);
    a.n = (int)d->n; a.bits = d->bits; a.model_bits = p->model_bits; a.grad_bits = p->grad_bits;
    a.clusters = plan.clusters; a.chunks = plan.chunks; a.nb = plan.nb; a.rc = plan.rc; a.cr = plan.cr; a.rb = plan.rb; a.owners = plan.owners; a.sps = plan.sps; a.slabs = plan.slabs; a.cols = plan.cols;
    a.a_parts = plan.a_parts; a.a_inv = 65536 / plan.a_parts + 1; a.spw = plan.spw; a.b_parts = plan.b_parts; a.b_inv = 65536 / plan.b_parts + 1; a.cpw = plan.cpw;
    CUtensorMap tmaps[2];
    memset(tmaps, 0, sizeof(tmaps));
    a.use_tmap = d->m < (1ll << 31) - 4096 && encode_plane_maps(ctx, d, plan.pitch / 4, plan.cr, true, tmaps) == ZIPML_OK;
    a.p_shift = plan.p_shift; a.pitch = plan.pitch; a.slots = plan.slots;
    void* params[] = {&a, &tmaps[0], &tmaps[1]};
    if (plan.clusters > 1) {
        rc = exchange_tags(ctx, (size_t)2 * plan.clusters * plan.owners * 32 * plan.sps * (8 / cb) * 16, num_steps, &a.exchange, &a.tag);
        if (rc != ZIPML_OK) return rc;
    }
    cudaError_t e = cudaLaunchKernelExC(&cfg, kernel, params);
    if (e != cudaSuccess) return cuda_status(e);
    ctx->launches += 1;
    ctx->ran(ZIPML_ENGINE_CLUSTER, "sgd_slice_kernel");
    return ZIPML_OK;
}

}  // namespace zipml
