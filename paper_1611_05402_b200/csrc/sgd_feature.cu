// Cluster engine of zipml_sgd_epoch on uniform grids, int8 tensor cores, split by features: nb <= 16 CTAs of a thread-block cluster, each of
// which owns the features of a few 16-byte columns of the packed row and reads all of the cluster's rows there (Supplement "Double Sampling",
// footnote form; "End-to-end Quantization").
//
// A small step is a chain of hand-overs; its arithmetic is little.  Split by features the model and the gradient stay in the CTA that owns
// them; what travels is a row's two dots to the row's owner, as integers, and its two residuals back:
//   * dots: a warp takes 16 rows of the own columns (mma.sync m16n8k32 u8 x s8 against the digits of w = step * x~: exact integer sums)
//     and stores the two of a row into its owner's shared memory (st.async, 16 bytes);
//   * the owner of a row adds the nb parts, 16 lanes a row, in the largest of the CTAs' units, and what the copying warp has made of
//     lo^T x~ and the row's label meanwhile, an integer in the same unit; each lane stores the residuals of two rows into one CTA;
//   * every CTA takes the largest residual of all rows for the scale and writes their digits: 16 rows of plane 1 with r2 and 16 rows of
//     plane 2 with r1 are the 32 entries of one contraction;                                                  barrier
//   * gradient: a warp takes a column and a part of the row blocks (transposing ldmatrix) and leaves a low and a high integer per feature;
//                                                                                                             barrier
//   * sums over the parts, exact integers until they meet lo and step in double (codes less a constant centre in fp32 lost 10 to 37 times
//     the precision on rows that are mostly zeros: 1.2e-6 of the gradient at 256 x 1,000, 4e-8 now); Q4, update, Q3, w;   barrier
//     and the digits of w, four balanced base-256 digits per entry, with the power of two of the CTA's largest.            barrier
// Bound by the chain of dependent instructions: some 680 a warp and step at 50 % of the issue slots (8 bits 256 x 1,000: dots 1.1 k cycles,
// hand-overs 0.8 k and 0.2 k, digits of the residuals 0.7 k, gradient 0.7 k, update 0.6 k, digits of w 0.6 k); a quantized gradient and
// model add a norm over the CTAs each, 2.1 k.  Measured against the form split by rows, us per step: 8 bits 256 x 1,000 3.3 -> 2.9, 2 bits
// 1,024 x 2,048 with both quantized 9.0 -> 7.6, 8 bits 512 x 2,000 5.9 -> 4.6, 4 bits 128 x 4,000 5.9 -> 3.5; against the column engine 8 bits
// 1,024 x 4,000 12.3 -> 6.1, 4 bits 16 x 8,000 7.6 -> 3.4.
// Codes of less than 8 bits are masked where they lie in their byte: the shift is in the digits (dots) or comes off the sums (gradient).
// Larger minibatches take several clusters, each with its rows and a replica of the model: the owners of the same features hand each other
// their sums through L2 (self-validating 8-byte words, two buffers in turn) and add them in the same order.
// Buffer reuse: a CTA sends the dots of step t + 1 after it has used all residuals of step t, whose owners had read all dots of step t;
// and residuals of step t + 1 leave when every CTA has sent its dots of that step.  Rows past a short batch travel too (their residuals are
// 0): every phase of every barrier counts the same bytes.
// Every wait is bounded; when one gives up the CTA records ZIPML_ERR_TIMEOUT, skips its later waits, still issues every store and copy,
// and all CTAs meet at a cluster barrier before they exit.
#include <cuda.h>
#include <string.h>

#include "cluster.cuh"
#include "int_digits.cuh"

namespace zipml {

struct FeatureArgs {
    const float* lo;
    const float* step;
    const float* b;
    float* x;
    float* grad_out;             // null or 2n
    float* model_out;            // null or n: the model the last executed step's gradient saw
    const int32_t* order;        // device copy of the batch order, or null
    unsigned long long* trace;
    DeviceStatus* status;
    int64_t first_step, num_steps, batch;
    uint64_t seed;
    uint32_t epoch;
    float lr;
    int reg;                     // ZIPML_REG_* and its fp32 constant
    float reg_cst;
    int n, bits;
    int model_bits, grad_bits;
    int whole, rows_last;        // batches below `whole` are full, that one has rows_last rows
    double full_scale, last_scale;   // 1 / (2 rows)
    int clusters, rows;          // clusters, rows per cluster
    unsigned long long* exchange;    // [2][clusters][nb F][2] words {fp32, tag} between the clusters
    uint32_t tag;                // of the first step; greater than any that the buffer holds
    int nb, cols, cols_inv;      // CTAs per cluster, 16-byte columns per CTA
    int rb, kpp, parts;          // blocks of 16 rows; of a part; parts
    int rpo;                     // rows per owner
    uint32_t rpo_inv;            // 2^31 / rpo: row r is owner ((2r + 1) rpo_inv) >> 32's
    int boxes, box_rows;         // tensor copies per plane and rows of each
    int p_shift;                 // 2^p_shift lanes share the sum of one feature
    int pitch, plane_bytes, slot_bytes, slots;
    int trace_steps;
};

struct alignas(16) FeatureBase {
    double base;                 // a CTA's part of lo^T x~ (not a number where w is none)
    int k, pad;                  // its dots' unit is 2^-k
};
struct alignas(16) FeatureRest {
    long long rest;              // of an own row: lo^T x~ less the label, in units of 2^-k
    int k;
    float unit;                  // 2^-k (not a number where the rest is none)
};
struct alignas(128) FeatureShared {
    FeatureBase base[kSliceMaxCtas];
    double red[2][16];           // per-warp parts of the squared norms of gradient and model
    double nrm_g[kSliceMaxCtas]; // squared norms of the owners' gradients and models (entries past the CTAs stay zero)
    double nrm_x[kSliceMaxCtas];
    int2 rsum[2];                // sums of the residuals' integers, lower 16 bits and the rest; two steps in turn
    uint64_t full[kSliceMaxSlots], empty[kSliceMaxSlots];
    uint64_t base_bar, rest_bar, dot_bar, res_bar, gn_bar, xn_bar;
    float wmax[32];              // per-warp maxima of |w| (entries past the warps stay zero)
    int gave_up;
};

__device__ __forceinline__ uint4 feature_pair(long long a, long long b) { return make_uint4((uint32_t)a, (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32)); }

// Shared memory after FeatureShared; F = 16 cols NG features of the CTA, SF the same in whole 32-byte slabs:
//   wd[SF]                 words: digits of w [slab][group][t][half][digit]
//   wv[SF]                 w of the own features, zero past them
//   lox[F]                 doubles: lo * x~ of the own features
//   rdig[rb][32]           words: digits of the residuals [t][half][digit] as B fragments
//   gsum[parts][2 F + 4]   the parts of the gradient, a low and a high integer per feature
//   dsum[nb][rpo + odd]    pairs of integers: the CTAs' dots of the own rows, in their units
//   rest[rpo]              what the own rows' residuals take besides the dots
//   res[16 rb]             pairs of floats: residuals of all rows, zero past the batch
//   ring[slots]: codes [2][rows][pitch], labels of the own rows
template <int CB, bool MANY>
__global__ void __launch_bounds__(kSliceThreads + 32, 1) sgd_feature_kernel(const FeatureArgs a, const __grid_constant__ CUtensorMap tm1,
                                                                            const __grid_constant__ CUtensorMap tm2) {
    constexpr int NG = IntPath<CB>::NG;
    extern __shared__ __align__(128) unsigned char s_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cl = MANY ? blockIdx.x / a.nb : 0, bi = MANY ? blockIdx.x - cl * a.nb : blockIdx.x;
    const int n = a.n, F = 16 * a.cols * NG, sps = (a.cols + 1) / 2, SF = 32 * sps * NG, part_words = 2 * F + 4;
    const int row_base = cl * a.rows;
    const int B = max(0, min(a.rows, (int)a.batch - row_base) + 1) & ~1;       // the cluster's rows (they travel in pairs)
    FeatureShared* sh = reinterpret_cast<FeatureShared*>(s_raw);
    uint32_t* wd = reinterpret_cast<uint32_t*>(s_raw + sizeof(FeatureShared));
    float* wv = reinterpret_cast<float*>(wd + SF);
    double* lox = reinterpret_cast<double*>(wv + SF);
    uint32_t* rdig = reinterpret_cast<uint32_t*>(lox + F);
    int* gsum = reinterpret_cast<int*>(rdig + a.rb * 32);
    const int dstride = a.rpo | 1;                       // (the CTAs' dots of a row in different banks)
    longlong2* dsum = reinterpret_cast<longlong2*>(gsum + a.parts * part_words);
    FeatureRest* rest = reinterpret_cast<FeatureRest*>(dsum + a.nb * dstride);
    float2* res = reinterpret_cast<float2*>(rest + a.rpo);
    unsigned char* ring = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(res + 16 * a.rb) + 127) & ~(uintptr_t)127);
    const int own = max(0, min(a.rpo, B - bi * a.rpo));          // rows whose residuals this CTA forms
    const uint32_t dot_bytes = 16u * a.nb * own;

    if (tid < a.slots) {
        mbar_init(sh->full + tid, 33);                           // the tile's byte count and the 32 lanes that copy labels
        mbar_init(sh->empty + tid, kSliceWarps);
    } else if (tid == 32) {
        mbar_init(&sh->dot_bar, 1);
        mbar_arrive_expect_tx(&sh->dot_bar, dot_bytes);
    } else if (tid == 33) {
        mbar_init(&sh->res_bar, 1);
        mbar_arrive_expect_tx(&sh->res_bar, 8u * B);
    } else if (tid == 34) {
        mbar_init(&sh->gn_bar, 1);
        mbar_arrive_expect_tx(&sh->gn_bar, 8u * a.nb);
    } else if (tid == 35) {
        mbar_init(&sh->xn_bar, 1);
        mbar_arrive_expect_tx(&sh->xn_bar, 8u * a.nb);
    } else if (tid == 36) {
        mbar_init(&sh->base_bar, 1);
        mbar_arrive_expect_tx(&sh->base_bar, 16u * a.nb);
    } else if (tid == 37) {
        mbar_init(&sh->rest_bar, 32);
    } else if (tid == 38) {
        sh->gave_up = 0;
    } else if (tid >= 64 && tid < 80) {
        sh->nrm_g[tid - 64] = sh->nrm_x[tid - 64] = 0.0;
        sh->wmax[tid - 48] = 0.0f;
        sh->base[tid - 64] = FeatureBase{0.0, 0x7fffffff, 0};
        if (tid < 66) sh->rsum[tid - 64] = make_int2(0, 0);
    }
#pragma unroll 1
    for (int k = tid; k < SF; k += kSliceThreads + 32) {
        wv[k] = 0.0f;
        if (k < F) lox[k] = 0.0;
    }
#pragma unroll 1
    for (int r = tid; r < 16 * a.rb; r += kSliceThreads + 32) res[r] = make_float2(0.0f, 0.0f);
    mbar_fence_init();
    __syncthreads();
    slice_cluster_sync();                                // every CTA's barriers exist before anyone writes into it
    after_previous_kernel(a.num_steps);

    // steps are counted from the call's first one; a batch is named by its index
    const int steps = (int)a.num_steps, whole = a.whole;
    auto batch_at = [&](int k) { return k < steps ? (a.order ? a.order[a.first_step + k] : (int)a.first_step + k) : 0; };
    auto own_of = [&](int batch) { return max(0, min(own, (batch < whole ? (int)a.batch : a.rows_last) - row_base - bi * a.rpo)); };
    if (warp == kSliceWarps) {
        // -------------------------------------------------------------------- the copying warp, which also sees to lo^T x~
        int slot = 0, used = 0;                          // slots to fill and to read labels from
        uint32_t parity = 1, used_parity = 0, base_parity = 0;   // (of the slots' emptiness: all are empty at first)
        const int owners = (B + a.rpo - 1) / a.rpo;
#pragma unroll 1
        for (int k = 0; k < steps + a.slots; ++k) {
            if (k >= a.slots) {                          // step k - slots: its lo^T x~, once the owners have it
                slice_bar_all();
                double v = 0.0;
#pragma unroll 1
                for (int f = lane; f < F; f += 32) v += lox[f];
                v = warp_sum(v);
                const float wmax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(sh->wmax[lane])));
                if (!(wmax <= 3.402823466e+38f)) v = __longlong_as_double(0x7fffffffffffffffll);
                if (lane < owners)
                    slice_store16(slice_peer(sh->base + bi, lane), feature_pair(__double_as_longlong(v), slice_exponent(wmax, SliceShift<CB>::kMost) + SliceShift<CB>::kMost),
                                  slice_peer(&sh->base_bar, lane));
                if (own > 0) {
                    // less the label, as an integer in the largest of the CTAs' units or one that holds it in 61 bits: the residuals
                    // are exact sums of integers but for what a part has below that unit
                    slice_wait(sh, &sh->base_bar, base_parity, a.status, 7);
                    if (lane == 0 && k + 1 < steps + a.slots) mbar_arrive_expect_tx(&sh->base_bar, 16u * a.nb);
                    const FeatureBase part = sh->base[lane & 15];
                    const int k_min = __reduce_min_sync(0xffffffffu, part.k);
                    double base = part.base;
#pragma unroll
                    for (int o = 1; o < 16; o <<= 1) base += __shfl_xor_sync(0xffffffffu, base, o);
                    slice_wait(sh, sh->full + used, used_parity, a.status, 6);
                    const float* labels = reinterpret_cast<const float*>(ring + used * a.slot_bytes + 2 * a.plane_bytes);
                    const int rows = own_of(batch_at(k - a.slots));
#pragma unroll 1
                    for (int i = lane; i < rows; i += 32) {
                        const double v = base - (double)labels[i];
                        const int e = min(k_min, 60 + 1023 - ((__double2hiint(v) >> 20) & 0x7ff));
                        rest[i] = FeatureRest{__double2ll_rn(v * __longlong_as_double((long long)(1023 + e) << 52)), e, v - v == 0.0 ? slice_pow2(-e) : __int_as_float(0x7fffffff)};
                    }
                    mbar_arrive(&sh->rest_bar);
                }
                base_parity ^= 1u;
                if (++used == a.slots) { used = 0; used_parity ^= 1u; }
            }
            if (k >= steps) continue;
            const int batch = batch_at(k);
            const int64_t r0 = batch * a.batch + row_base;
            unsigned char* dst = ring + slot * a.slot_bytes;
            slice_wait(sh, sh->empty + slot, parity, a.status, 84);
            if (lane == 0) {                             // (boxes that reach past the last row are filled up and count in full)
                mbar_arrive_expect_tx(sh->full + slot, 2u * (uint32_t)(a.boxes * a.box_rows * a.pitch));
#pragma unroll 1
                for (int i = 0; i < a.boxes; ++i) {
                    slice_tensor_copy(dst + i * a.box_rows * a.pitch, &tm1, 2 * bi * a.cols, (int)r0 + i * a.box_rows, sh->full + slot);
                    slice_tensor_copy(dst + a.plane_bytes + i * a.box_rows * a.pitch, &tm2, 2 * bi * a.cols, (int)r0 + i * a.box_rows, sh->full + slot);
                }
            }
            const uint32_t labels = smem_u32(dst + 2 * a.plane_bytes);
            const int rows = own_of(batch);
#pragma unroll 1
            for (int i = lane; i < rows; i += 32)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(labels + 4u * i), "l"(a.b + r0 + bi * a.rpo + i) : "memory");
            asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(sh->full + slot)) : "memory");
            if (++slot == a.slots) { slot = 0; parity ^= 1u; }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
        slice_cluster_sync();
        return;
    }

    // ------------------------------------------------------------------------ the steps
    const int gl = lane >> 2, tl = lane & 3, lm = lane >> 3, l8 = lane & 7;
    const int P = 1 << a.p_shift, pp = tid & (P - 1), k_own = tid >> a.p_shift, f_own = bi * F + k_own;
    const bool mine = k_own < F && f_own < n, writes = mine && pp == 0;
    const float st = mine ? a.step[f_own] : 0.0f, lof = mine ? a.lo[f_own] : 0.0f;
    const double lo_double = lof, st_low = (double)st / (double)(1 << (CB * (k_own % NG)));     // (codes were multiplied where they lie in their byte)
    float x = mine ? a.x[f_own] : 0.0f;
    auto draw = [&](int k, uint32_t stream) { return slice_draw(a.seed, a.epoch, (uint32_t)a.first_step + (uint32_t)k, (uint32_t)f_own, stream); };

    const int marked = blockIdx.x == 0 && tid == 0 && a.trace ? a.trace_steps : -1;
    int batch = batch_at(0), batch_next = batch_at(1);
    int slot = 0;
    uint32_t parity = 0, step_parity = 0, gn_parity = 0, xn_parity = 0;
#pragma unroll 1
    for (int step = -1; step < steps; ++step) {
        const bool last = step == steps - 1;
        uint32_t u_x = 0u, u_g = 0u;
        if (step >= 0) {
            const unsigned char* tile = ring + slot * a.slot_bytes;
            const uint32_t tile_addr = smem_u32(tile);
            if (step < marked) slice_mark(a.trace, step, 0);
            // -------------------------------------------------------------- dots (the tile has come: see the last barrier)
#pragma unroll 1
            for (int blk = warp; blk < a.rb; blk += kSliceWarps) {
                // lane t < 2 of a group sends row g + 8 t
                const int r = blk * 16 + gl + 8 * tl, owner = (int)__umulhi(2u * (uint32_t)r + 1u, a.rpo_inv);
                const bool sends = tl < 2 && r < B;
                const uint32_t to = sends ? slice_peer(dsum + bi * dstride + r - owner * a.rpo, owner) : 0u, to_bar = sends ? slice_peer(&sh->dot_bar, owner) : 0u;
                int c[2][4];
#pragma unroll
                for (int e = 0; e < 4; ++e) c[0][e] = c[1][e] = 0;
                // lane's address of a fragment: row l8 (+ 8 for the odd matrices), bytes 0 or 16 of the slab
                uint32_t addr = tile_addr + (uint32_t)((blk * 16 + l8 + (lm & 1) * 8) * a.pitch) + (uint32_t)((lm >> 1) * 16);
                const uint32_t* wq = wd + tl * 8 + (gl & 3);
#pragma unroll 1
                for (int ks = 0; ks < sps; ++ks, addr += 32u, wq += NG * 32) {
                    uint32_t a1[4], a2[4];
                    ldsm_x4(a1, addr);
                    ldsm_x4(a2, addr + (uint32_t)a.plane_bytes);
#pragma unroll
                    for (int g = 0; g < NG; ++g) {
                        const uint32_t b0 = gl < 4 ? wq[g * 32] : 0u, b1 = gl < 4 ? wq[g * 32 + 4] : 0u;
                        mma_u8s8(c[0], slice_dot_codes<CB>(a1[0], g), slice_dot_codes<CB>(a1[1], g), slice_dot_codes<CB>(a1[2], g), slice_dot_codes<CB>(a1[3], g), b0, b1);
                        mma_u8s8(c[1], slice_dot_codes<CB>(a2[0], g), slice_dot_codes<CB>(a2[1], g), slice_dot_codes<CB>(a2[2], g), slice_dot_codes<CB>(a2[3], g), b0, b1);
                    }
                }
                // lane t = 0 has digits 0, 1 of rows g and g + 8, lane t = 1 digits 2, 3: the first takes row g, the other row g + 8
                long long d[2];
#pragma unroll
                for (int pl = 0; pl < 2; ++pl) {
                    const long long upper = c[pl][0] + 256ll * c[pl][1], lower = c[pl][2] + 256ll * c[pl][3];
                    const long long got = __shfl_xor_sync(0xffffffffu, tl == 0 ? lower : upper, 1);
                    d[pl] = tl == 0 ? upper + 65536ll * got : got + 65536ll * lower;
                }
                if (sends) slice_store16(to, feature_pair(d[0], d[1]), to_bar);
            }
            if (a.grad_bits > 0 && writes) u_g = draw(step, 4u);
            if (a.model_bits > 0 && writes) u_x = draw(step + 1, 3u);
            if (step < marked) slice_mark(a.trace, step, 1);
            // -------------------------------------------------------------- residuals of the own rows
            const bool batch_full = batch < whole;
            if (2 * warp < own) {
                const int rows = own_of(batch), p16 = lane & 15;
                const uint32_t to = lane < a.nb ? slice_peer(res + bi * a.rpo, lane) : 0u, to_bar = lane < a.nb ? slice_peer(&sh->res_bar, lane) : 0u;
                slice_wait(sh, &sh->rest_bar, step_parity, a.status, 8);
                const int k_part = sh->base[p16].k;
                slice_wait(sh, &sh->dot_bar, step_parity, a.status, 4);
                if (tid == 0 && !last) mbar_arrive_expect_tx(&sh->dot_bar, dot_bytes);
#pragma unroll 1
                for (int i0 = 2 * warp; i0 < own; i0 += 2 * kSliceWarps) {
                    const int i = i0 + (lane >> 4);
                    const longlong2 d = i < own && p16 < a.nb ? dsum[p16 * dstride + i] : make_longlong2(0, 0);
                    const FeatureRest more = rest[i];
                    const int down = min(63, k_part - more.k);
                    const long long d1 = d.x >> down, d2 = d.y >> down;
                    long long v = (lane & 1 ? d2 : d1) + __shfl_xor_sync(0xffffffffu, lane & 1 ? d1 : d2, 1);
#pragma unroll
                    for (int o = 2; o < 16; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                    const float r = i < rows ? __ll2float_rn(v + more.rest) * more.unit : 0.0f;
                    // lane p < nb gets both rows' residuals for CTA p (the odd lanes of a row have plane 2)
                    const float other = __shfl_xor_sync(0xffffffffu, r, 1);
                    const float r1 = lane & 1 ? other : r, r2 = lane & 1 ? r : other;
                    const float n1 = __shfl_down_sync(0xffffffffu, r1, 16), n2 = __shfl_down_sync(0xffffffffu, r2, 16);
                    if (lane < a.nb)
                        slice_store16(to + 8u * (uint32_t)i, make_uint4(__float_as_uint(r1), __float_as_uint(r2), __float_as_uint(n1), __float_as_uint(n2)), to_bar);
                }
            }
            batch = batch_next;
            batch_next = batch_at(step + 2);
            if (step < marked) slice_mark(a.trace, step, 2);
            slice_wait(sh, &sh->res_bar, step_parity, a.status, 5);
            if (tid == 0 && !last) mbar_arrive_expect_tx(&sh->res_bar, 8u * B);
            step_parity ^= 1u;
            if (step < marked) slice_mark(a.trace, step, 3);
            // -------------------------------------------------------------- digits of the residuals, one scale for all rows
            // (largest as bit patterns: a residual that is not a number wins, and the gradient is none either)
            uint32_t top_bits = 0u;
#pragma unroll 4
            for (int i = lane; i < 8 * a.rb; i += 32) {
                const uint4 v = reinterpret_cast<const uint4*>(res)[i];
                top_bits = max(max(top_bits, max(v.x & 0x7fffffffu, v.y & 0x7fffffffu)), max(v.z & 0x7fffffffu, v.w & 0x7fffffffu));
            }
            const float top = __uint_as_float(__reduce_max_sync(0xffffffffu, top_bits));
            const int k_r = slice_exponent(top, 0);
            const float up_r = slice_pow2(k_r), delta_r = top <= 3.402823466e+38f ? slice_pow2(-k_r) : __int_as_float(0x7fffffff);
            int r_low = 0, r_high = 0;                   // sums of the integers' halves (some 2,000 entries a warp at most)
            const int entry_row = 2 * ((lane >> 2) & 3) + (lane & 1) + 8 * ((lane >> 1) & 1);
#pragma unroll 1
            for (int blk = warp; blk < a.rb; blk += kSliceWarps) {
                const float r = reinterpret_cast<const float*>(res + blk * 16 + entry_row)[lane < 16 ? 1 : 0];
                const int whole_r = __float2int_rn(r * up_r);
                r_low += whole_r & 0xffff;
                r_high += whole_r >> 16;
                const uint32_t digits = ((uint32_t)whole_r + 0x80808080u) ^ 0x80808080u;
                unsigned char* out = reinterpret_cast<unsigned char*>(rdig + blk * 32) + ((lane >> 2) & 3) * 32 + (lane >> 4) * 16 + (lane & 3);
#pragma unroll
                for (int s = 0; s < 4; ++s) out[4 * s] = (unsigned char)(digits >> (8 * s));
            }
            r_low = __reduce_add_sync(0xffffffffu, r_low);
            r_high = __reduce_add_sync(0xffffffffu, r_high);
            if (lane == 0) {
                atomicAdd(&sh->rsum[step & 1].x, r_low);
                atomicAdd(&sh->rsum[step & 1].y, r_high);
            }
            slice_bar();
            if (step < marked) slice_mark(a.trace, step, 4);
            // -------------------------------------------------------------- gradient of the own features
#pragma unroll 1
            for (int task = warp; task < a.cols * a.parts; task += kSliceWarps) {
                const int part = (task * a.cols_inv) >> 16, col = task - part * a.cols;         // task / cols
                const int kb0 = part * a.kpp, kb1 = min(a.rb, kb0 + a.kpp);
                const uint32_t* rq = rdig + kb0 * 32 + tl * 8 + (gl & 3);
                uint32_t addr = tile_addr + (uint32_t)((lane >> 4) * a.plane_bytes + (kb0 * 16 + (lane & 15)) * a.pitch + col * 16);
                int acc[NG][4];
#pragma unroll
                for (int g = 0; g < NG; ++g)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[g][e] = 0;
#pragma unroll 1
                for (int kb = kb0; kb < kb1; ++kb, rq += 32, addr += 16u * (uint32_t)a.pitch) {
                    const uint32_t b0 = gl < 4 ? rq[0] : 0u, b1 = gl < 4 ? rq[4] : 0u;
                    uint32_t r4[4];
                    ldsm_x4_trans(r4, addr);
                    const uint32_t pel = __byte_perm(r4[0], r4[1], 0x6420), pol = __byte_perm(r4[0], r4[1], 0x7531);
                    const uint32_t peh = __byte_perm(r4[2], r4[3], 0x6420), poh = __byte_perm(r4[2], r4[3], 0x7531);
#pragma unroll
                    for (int g = 0; g < NG; ++g)
                        mma_u8s8(acc[g], slice_codes<CB>(pel, g), slice_codes<CB>(pol, g), slice_codes<CB>(peh, g), slice_codes<CB>(poh, g), b0, b1);
                }
                // rows g, g + 8 of the accumulators are bytes 2g, 2g + 1 of the column; lane t = 0 has the lower digits, t = 1 the upper
                // ones (seven row blocks at most: below 2^31)
#pragma unroll
                for (int g = 0; g < NG; ++g) {
                    int* out = gsum + part * part_words + 2 * ((col * 16 + 2 * gl) * NG + g) + tl;
                    if (tl < 2) {
                        out[0] = acc[g][0] + 256 * acc[g][1];
                        out[2 * NG] = acc[g][2] + 256 * acc[g][3];
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(sh->empty + slot);
            if (++slot == a.slots) { slot = 0; parity ^= 1u; }
            if (step < marked) slice_mark(a.trace, step, 5);
            slice_bar();

            // -------------------------------------------------------------- sums over the parts, update
            long long sum = 0;
            if (mine)
#pragma unroll 2
                for (int w = pp; w < a.parts; w += P) {
                    const int2 v = *reinterpret_cast<const int2*>(gsum + w * part_words + 2 * k_own);
                    sum += v.x + 65536ll * v.y;
                }
#pragma unroll 1
            for (int o = 1; o < P; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            const int2 halves = sh->rsum[step & 1];
            if (tid == 0) sh->rsum[(step + 1) & 1] = make_int2(0, 0);
            double t = fma(st_low, (double)sum, lo_double * slice_double(halves.x, halves.y)) * (double)delta_r;
            if constexpr (MANY) {
                const uint32_t tag = a.tag + (uint32_t)step;
                unsigned long long* box = a.exchange + ((size_t)(step & 1) * a.clusters * a.nb * F + f_own) * 2;
                const size_t stride = (size_t)a.nb * F * 2;
                const float hi = (float)t, low = (float)(t - (double)hi);
                if (writes) slice_post(box + cl * stride, hi, low, tag);
                t = 0.0;
                if (mine)
#pragma unroll 1
                    for (int c = pp; c < a.clusters; c += P) t += c == cl ? (double)hi + (double)low : slice_collect(sh, box + c * stride, tag, a.status);
#pragma unroll 1
                for (int o = 1; o < P; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            }
            float g = (float)(t * (batch_full ? a.full_scale : a.last_scale));
            if (last && a.grad_out && writes && cl == 0) a.grad_out[f_own] = g;
            if (step < marked) slice_mark(a.trace, step, 6);
            if (a.grad_bits > 0) {
                const float M = slice_norm(writes ? (double)g * (double)g : 0.0, P, bi, sh->red[0], sh->nrm_g, &sh->gn_bar, gn_parity, a.nb, sh, a.status, 3);
                gn_parity ^= 1u;
                g = slice_quantize(g, M, a.grad_bits, u_g);
            }
            if (last && a.grad_out && writes && cl == 0) a.grad_out[n + f_own] = g;
            const float y = fmaf(-a.lr, g, x);
            x = a.reg == ZIPML_REG_NONE ? y : slice_regularise(y, x, a.reg, a.reg_cst);
        } else if (a.model_bits > 0 && writes) {
            u_x = draw(step + 1, 3u);
        }
        if (last) break;

        // ------------------------------------------------------------------ what the next step sees: Q3, digits of w
        float xt = x;
        if (a.model_bits > 0) {
            const float M = slice_norm(writes ? (double)x * (double)x : 0.0, P, bi, sh->red[1], sh->nrm_x, &sh->xn_bar, xn_parity, a.nb, sh, a.status, 8);
            xn_parity ^= 1u;
            xt = slice_quantize(x, M, a.model_bits, u_x);
        }
        if (a.model_out && step + 2 == steps && writes && cl == 0) a.model_out[f_own] = xt;
        const float w = writes ? st * xt : 0.0f;
        if (writes) wv[k_own] = w;
        if (writes) lox[k_own] = (double)lof * (double)xt;
        const float top_w = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(w))));
        if (lane == 0) sh->wmax[warp] = top_w;
        slice_bar_all();
        const float wmax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(sh->wmax[lane])));
        const int k_w = slice_exponent(wmax, SliceShift<CB>::kMost);
        if (tid < SF / 4) {
            const int half = tid & 1, t = (tid >> 1) & 3, gs = tid >> 3, g = gs % NG, q = (gs / NG) * 8 + half * 4 + t;
            const float* src = wv + q * 4 * NG + g;
            const float up = slice_pow2(k_w) * (float)(1 << SliceShift<CB>::of(g));
            uint32_t d[4];
            transpose4x4((uint32_t)__float2int_rn(src[0] * up) + 0x80808080u, (uint32_t)__float2int_rn(src[NG] * up) + 0x80808080u,
                         (uint32_t)__float2int_rn(src[2 * NG] * up) + 0x80808080u, (uint32_t)__float2int_rn(src[3 * NG] * up) + 0x80808080u, d);
            *reinterpret_cast<uint4*>(wd + 4 * tid) = make_uint4(d[0] ^ 0x80808080u, d[1] ^ 0x80808080u, d[2] ^ 0x80808080u, d[3] ^ 0x80808080u);
        }
        if (warp == kSliceWarps - 1) slice_wait(sh, sh->full + slot, parity, a.status, 6);      // (for all: the barrier hands it on)
        slice_bar();
        if (step >= 0 && step < marked) slice_mark(a.trace, step, 7);
    }
    if (writes && cl == 0) a.x[f_own] = x;
    __syncwarp();
    slice_cluster_sync();                                // nobody leaves while a store may still target it
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
template <int CB>
static const void* feature_kernel(bool many) {
    return many ? (const void*)sgd_feature_kernel<CB, true> : (const void*)sgd_feature_kernel<CB, false>;
}

// The parts of a plan that follow from the clusters; false where it does not fit.
static bool feature_plan(const zipml_ctx* ctx, const zipml_dataset* d, const zipml_sgd_params* p, int64_t clusters, FeatureArgs* a, size_t* smem) {
    const int cb = container_bits(d->bits), ng = 8 / cb;
    const int64_t B = p->batch < d->m ? p->batch : d->m;
    const int64_t cols = (d->n * cb + 127) / 128;
    a->rows = 2 * (int)((B + 2 * clusters - 1) / (2 * clusters));      // (even: rows travel in pairs)
    a->clusters = (int)((B + a->rows - 1) / a->rows);             // none without rows
    const int64_t most = p->grid_row_parts > 0 && p->grid_row_parts < kSliceMaxCtas ? p->grid_row_parts : kSliceMaxCtas;
    a->cols = (int)((cols + most - 1) / most);
    const int F = 16 * a->cols * ng;
    if (F > kSliceThreads) return false;
    a->nb = (int)((cols + a->cols - 1) / a->cols);
    a->cols_inv = 65536 / a->cols + 1;
    a->rb = (a->rows + 15) / 16;
    const int want = a->cols < kSliceWarps ? kSliceWarps / a->cols : 1;
    a->kpp = (a->rb + want - 1) / want;
    if (a->kpp > 7) a->kpp = (a->rb + (a->rb + 6) / 7 - 1) / ((a->rb + 6) / 7);
    a->parts = (a->rb + a->kpp - 1) / a->kpp;
    if (a->parts * a->cols > 1024) return false;
    a->rpo = 2 * ((a->rows + 2 * a->nb - 1) / (2 * a->nb));       // (even: rows travel in pairs)
    a->rpo_inv = (uint32_t)((1ull << 31) / (uint64_t)a->rpo);
    a->boxes = (a->rows + 255) / 256;
    a->box_rows = (a->rows + a->boxes - 1) / a->boxes;
    if (a->boxes > 1) a->box_rows = (a->box_rows + 7) / 8 * 8;    // (a copy starts on 128 bytes)
    a->p_shift = 0;
    while (a->p_shift < 4 && F << (a->p_shift + 1) <= kSliceThreads && (1 << a->p_shift) < a->parts) ++a->p_shift;
    a->pitch = 16 * (a->cols | 1);
    const int tile_rows = a->boxes * a->box_rows > 16 * a->rb ? a->boxes * a->box_rows : 16 * a->rb;
    a->plane_bytes = (tile_rows * a->pitch + 127) / 128 * 128;
    a->slot_bytes = 2 * a->plane_bytes + (4 * a->rpo + 127) / 128 * 128;
    const size_t sf = (size_t)32 * ((a->cols + 1) / 2) * ng;
    const size_t fixed = sizeof(FeatureShared) + 8 * sf + 8 * (size_t)F + 128 * (size_t)a->rb + 4 * (size_t)a->parts * (2 * F + 4) + 16 * (size_t)a->nb * (a->rpo | 1) + 16 * (size_t)a->rpo +
                         128 * (size_t)a->rb + 128;
    a->slots = kSliceMaxSlots;
    while (a->slots > 1 && fixed + (size_t)a->slots * a->slot_bytes > (size_t)ctx->smem_optin) --a->slots;
    *smem = fixed + (size_t)a->slots * a->slot_bytes;
    return a->slots >= 2;
}

int launch_sgd_feature(zipml_ctx* ctx, const zipml_dataset* d, const float* b, float* x, const zipml_sgd_params* p, int64_t first_step,
                       int64_t num_steps, float* grad_out) {
    const int cb = container_bits(d->bits);
    const int64_t B = p->batch < d->m ? p->batch : d->m;
    const int64_t T = (d->m + p->batch - 1) / p->batch;
    if (d->level_mode != ZIPML_LEVELS_UNIFORM || B > 65536 || d->n > 65536 || d->m >= (1ll << 31) - 16384 || T > 0x7ffffff0) return ZIPML_ERR_WORKSPACE;
    FeatureArgs a;
    memset(&a, 0, sizeof(a));
    size_t smem = 0;
    // As few clusters as hold the rows, or as many as asked for; four from 448 rows, whose exchange (some 1.2 us) costs less than the other
    // rows, eight where those are of few CTAs.  us per step with 1 / 2 / 4 / 8: 8 bits n 1,000 x 384 3.80 / 3.91 / 3.83, x 512 4.37 / 4.07 /
    // 3.86, x 1,024 - / 5.33 / 4.42; n 300 (10 CTAs) x 1,024 - / 4.60 / 4.01 / 3.83, x 2,048 - / - / 4.84 / 4.12; 2 bits n 2,048 x 1,024 5.73 /
    // 5.72 / 4.84.  (Eight of sixteen CTAs are seldom resident at once.)
    const int64_t cols_all = (d->n * cb + 127) / 128;
    int64_t clusters = p->grid_feature_parts > 0 ? p->grid_feature_parts : B < 448 ? 1 : B >= 1024 && (cols_all + (cols_all + 15) / 16 - 1) / ((cols_all + 15) / 16) <= 12 ? 8 : 4;
    const void* kernel = nullptr;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    cudaError_t e;
    // (clusters are taken back until all of them can be resident at once: they wait for one another)
    for (int most = ctx->cooperative ? kSliceMaxClusters : 1;;) {
        if (clusters > most) clusters = most;
        while (!feature_plan(ctx, d, p, clusters, &a, &smem))
            if (++clusters > most) return ZIPML_ERR_WORKSPACE;
        const bool many = a.clusters > 1;
        kernel = cb == 2 ? feature_kernel<2>(many) : cb == 4 ? feature_kernel<4>(many) : feature_kernel<8>(many);
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess && a.nb > 8) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return cuda_status(e);
        memset(&cfg, 0, sizeof(cfg));
        cfg.gridDim = dim3((unsigned)(a.nb * a.clusters));
        cfg.blockDim = dim3(kSliceThreads + 32);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = ctx->stream;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)a.nb;
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
        if (fit >= a.clusters) break;
        most = fit;
    }
    if (a.clusters > 1 || early_start(ctx, num_steps, attr + 1)) cfg.numAttrs = 2;      // (a cooperative launch, or one that starts early)
    CUtensorMap tmaps[2];
    memset(tmaps, 0, sizeof(tmaps));
    int rc = encode_plane_maps(ctx, d, a.pitch / 4, a.box_rows, true, tmaps);
    if (rc != ZIPML_OK) return ZIPML_ERR_WORKSPACE;              // (also where a box would be wider than 256 elements)
    if (p->batch_order) {
        rc = ws_reserve(ctx, carve_size(sizeof(int32_t) * (size_t)T));
        if (rc != ZIPML_OK) return rc;
        e = cudaMemcpyAsync(ctx->ws, p->batch_order, sizeof(int32_t) * (size_t)T, cudaMemcpyHostToDevice, ctx->stream);
        if (e != cudaSuccess) return cuda_status(e);
        a.order = reinterpret_cast<const int32_t*>(ctx->ws);
    }
    a.lo = d->feat_lo; a.step = d->feat_step;
    a.b = b; a.x = x; a.grad_out = grad_out; a.model_out = p->model_out;
    a.trace = reinterpret_cast<unsigned long long*>(p->trace);
    a.trace_steps = p->trace ? p->trace_steps : 0;
    a.status = ctx->d_status;
    a.batch = B;
    a.first_step = first_step; a.num_steps = num_steps;
    a.whole = (int)(d->m / B); a.rows_last = (int)(d->m - a.whole * B);
    a.full_scale = 1.0 / (2.0 * (double)B); a.last_scale = 1.0 / (2.0 * (double)(a.rows_last > 0 ? a.rows_last : 1));
    a.seed = p->seed; a.epoch = (uint32_t)p->epoch; a.lr = p->lr; a.reg = p->reg; a.reg_cst = reg_constant(p);
    a.n = (int)d->n; a.bits = d->bits; a.model_bits = p->model_bits; a.grad_bits = p->grad_bits;
    if (a.clusters > 1) {
        rc = exchange_tags(ctx, (size_t)2 * a.clusters * a.nb * 16 * a.cols * (8 / cb) * 16, num_steps, &a.exchange, &a.tag);
        if (rc != ZIPML_OK) return rc;
    }
    void* params[] = {&a, &tmaps[0], &tmaps[1]};
    e = cudaLaunchKernelExC(&cfg, kernel, params);
    if (e != cudaSuccess) return cuda_status(e);
    ctx->launches += 1;
    ctx->ran(ZIPML_ENGINE_CLUSTER, "sgd_feature_kernel");
    return ZIPML_OK;
}

}  // namespace zipml
