// Cluster engine of zipml_sgd_epoch on level tables: one thread-block cluster of nb <= 16 CTAs, each of which owns the features of a few
// 16-byte units of the packed row and reads all rows of the minibatch there (Supplement "Double Sampling", footnote form, on the levels of
// "Optimal quantization"; "End-to-end Quantization").
//
// A level table is looked up, and what it costs is building it and looking things up.  Split by features a CTA needs the tables of its own
// features alone, 1 KB each, and builds them from its own slice of the model: the model never leaves the CTA, nor does the gradient.
// What travels is two floats per row and CTA, and the residuals back:
//   * dots: WL lanes take a row, a word of codes each, whose codes become bytes that are the entries' offsets (a shift and a masking OR
//     per register); a look-up is one byte permute into the table's address, the load and the sum.  4 words x 8 levels (2 x 16) of a slot fill
//     the 32 banks: lanes meet different ones or the same word.  The row's two sums go to the row's owner (st.async, 8 bytes);
//   * the owner of nb-th part of the rows adds the CTAs' sums in double, 16 lanes a row, subtracts the label, and each lane stores the
//     two residuals into one CTA;
//   * gradient: the same lanes and look-ups on the levels themselves, against the residuals; a transposing butterfly over the rows of the
//     warp, then one sum over the warps in double: the owner's 16 lanes of a feature all hold it, update the model entry and write a
//     level's product each.                                                                                    two barriers
// Large batches take the dots with a lane per row and whole units: nothing to exchange, and the look-ups of a warp, of one word, broadcast.
// Bound by instructions: a look-up is three and its share of the offsets, 128 a lane and step at 3 bits n 512 batch 512 (977 instructions of
// a warp and step before that form, 50 % of the issue slots), and by the chain of two hand-overs, of about 700 and 300 cycles.
// Measured there, us per step: 6.3 split by rows -> 4.5 -> 4.3 (four lanes a feature in the update) -> 4.05 (offsets as bytes; a shift, an
// OR and an add per look-up before) -> 3.85 (a lane per row) -> 3.45 (two rows to a 16-byte store).  Batch 64: 4.1 -> 2.1.
// Buffer reuse: a CTA sends the dots of step t + 1 after it has used all residuals of step t, whose owners had read all dots of step t;
// and residuals of step t + 1 leave when every CTA has sent its dots of that step.  Rows past a short batch travel too (their residuals are
// 0): every phase of every barrier counts the same bytes.
// Every wait is bounded; when one gives up the CTA records ZIPML_ERR_TIMEOUT, skips its later waits, still issues every store and copy,
// and all CTAs meet at a cluster barrier before they exit.
#include <cuda.h>
#include <string.h>

#include "cluster.cuh"

namespace zipml {

// Rows from which a lane takes a whole row's dots (us per step at 3 bits n 512, four lanes a row / one: 64 rows 2.11 / 2.28, 128 2.39 / 2.57,
// 256 2.87 / 2.81, 512 4.14 / 3.85).
constexpr int kTableRowLanes = 256;

struct TableArgs {
    const float* levels;
    const float* b;
    float* x;
    float* grad_out;             // null or 2n
    float* model_out;            // null or n: the model the last executed step's gradient saw
    const int32_t* order;        // device copy of the batch order, or null
    unsigned long long* trace;
    DeviceStatus* status;
    int64_t first_step, num_steps;
    uint64_t seed;
    uint32_t epoch;
    float lr;
    int reg;                     // ZIPML_REG_* and its fp32 constant
    float reg_cst;
    int n, real_levels;          // levels per feature in memory (1-bit codes: 2, looked up in tables of 4)
    int model_bits, grad_bits;
    int64_t batch;
    int whole, rows_last;        // batches below `whole` are full, that one has rows_last rows
    double full_scale, last_scale;   // 1 / (2 rows)
    int nb, units;               // CTAs, 16-byte units per CTA
    int rpo;                     // rows per owner
    uint32_t rpo_inv;            // 2^31 / rpo: row r is owner ((2r + 1) rpo_inv) >> 32's
    int boxes, box_rows;         // tensor copies per plane and rows of each
    int pitch, plane_bytes, slot_bytes, slots;
    int trace_steps;
};

struct alignas(256) TableShared {
    double red[2][16];           // per-warp parts of the squared norms of gradient and model
    double nrm_g[kSliceMaxCtas]; // squared norms of the owners' gradients and models (entries past the CTAs stay zero)
    double nrm_x[kSliceMaxCtas];
    uint64_t full[kSliceMaxSlots], empty[kSliceMaxSlots];
    uint64_t dot_bar, res_bar, gn_bar, xn_bar;
    int gave_up;
};

__device__ __forceinline__ double table_pair(float a, float b) {
    return __longlong_as_double((long long)((unsigned long long)__float_as_uint(b) << 32 | __float_as_uint(a)));
}
__device__ __forceinline__ uint4 table_four(float a, float b, float c, float d) {
    return make_uint4(__float_as_uint(a), __float_as_uint(b), __float_as_uint(c), __float_as_uint(d));
}
__device__ __forceinline__ float table_load(uint32_t addr) {
    float v;                                             // (not volatile: the address comes from a code that was read after the barriers)
    asm("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint32_t table_word(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

__device__ __forceinline__ void table_words(uint32_t (&v)[4], uint32_t addr) {
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(addr));
}

// The codes of a word, each as the byte offset of its entry (lane word w of WL): four to a register, slot CB-wise apart.  A table has
// L x WL entries of 4 bytes, levels WL apart.
template <int BITS>
struct TableOffsets {
    static constexpr int CB = BITS == 2 ? 2 : 4, PER = 8 / CB;           // slots per byte
    static constexpr int UP = BITS == 4 ? 3 : 4;                         // a level's offset is code << UP
    static constexpr uint32_t MASK = 0x01010101u * (((1u << BITS) - 1) << UP);
    uint32_t v[PER];
    __device__ __forceinline__ TableOffsets(uint32_t word, uint32_t lane_offsets) {
#pragma unroll
        for (int k = 0; k < PER; ++k) v[k] = ((CB * k <= UP ? word << (UP - CB * k) : word >> (CB * k - UP)) & MASK) | lane_offsets;
    }
    // address of slot i's entry: the offset is the low byte of an address in a table region on 256 bytes
    __device__ __forceinline__ uint32_t at(int i, uint32_t region) const {
        return __byte_perm(v[i % PER], region, 0x7650 + i / PER) + (uint32_t)(i * (1 << BITS) * (BITS == 4 ? 2 : 4) * 4);
    }
};

// Shared memory after TableShared; F = features of the CTA's units, L levels:
//   tab[F L]  level * x~ and lev[F L]  levels, both [unit][words of a lane][slot][level][lane word]
//   xown[F], gsub[F]   master model and gradient of the step, in the order of the tables without their levels
//   gsum[F][16]        the warps' sums of the gradient, 16-byte pieces swapped with bits 1 and 2 of the feature
//   dsum[nb][rpo + 2]  float pairs: the CTAs' dots of the own rows
//   res[rows]          float pairs: residuals of all rows, zero past the batch
//   ring[slots]: codes [2][rows][pitch], labels of the own rows
template <int BITS>
__global__ void __launch_bounds__(kSliceThreads + 32, 1) sgd_table_kernel(const TableArgs a, const __grid_constant__ CUtensorMap tm1,
                                                                          const __grid_constant__ CUtensorMap tm2) {
    constexpr int CB = BITS == 2 ? 2 : 4, FPW = 32 / CB, UF = 4 * FPW, L = 1 << BITS;
    constexpr int WL = BITS == 4 ? 2 : 4, HW = 4 / WL, REGION = FPW * L * WL * 4;
    constexpr int RPW = 32 / WL, ROWS = kSliceWarps * RPW;     // lanes per row, rows of a warp, of a pass
    extern __shared__ __align__(256) unsigned char s_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, bi = blockIdx.x;
    const int n = a.n, F = a.units * UF, B = ((int)a.batch + 1) & ~1;       // (rows travel in pairs)
    TableShared* sh = reinterpret_cast<TableShared*>(s_raw);
    float* tab = reinterpret_cast<float*>(s_raw + sizeof(TableShared));
    float* lev = tab + F * L;
    float* xown = lev + F * L;
    float* gsub = xown + F;
    float* gsum = gsub + F;
    float2* dsum = reinterpret_cast<float2*>(gsum + F * 16);
    const int dstride = a.rpo + 2;                       // (pairs of a CTA's dots: 16 CTAs' same row in different banks, two by two)
    float2* res = dsum + a.nb * dstride;
    const int rows_pad = (B + 31) / 32 * 32;
    unsigned char* ring = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(res + rows_pad) + 127) & ~(uintptr_t)127);
    const int own = max(0, min(a.rpo, B - bi * a.rpo));          // rows whose residuals this CTA forms

    auto feature = [&](int g) { return bi * F + g / (FPW * WL) * (FPW * WL) + g % WL * FPW + g / WL % FPW; };   // g-th in the tables' order

    if (tid < a.slots) {
        mbar_init(sh->full + tid, 33);                           // the tile's byte count and the 32 lanes that copy labels
        mbar_init(sh->empty + tid, kSliceWarps);
    } else if (tid == 32) {
        mbar_init(&sh->dot_bar, 1);
        mbar_arrive_expect_tx(&sh->dot_bar, 8u * a.nb * own);
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
        sh->gave_up = 0;
    } else if (tid >= 64 && tid < 80) {
        sh->nrm_g[tid - 64] = sh->nrm_x[tid - 64] = 0.0;
    }
    after_previous_kernel(a.num_steps);
#pragma unroll 1
    for (int i = tid; i < F * L; i += kSliceThreads + 32) {
        const int c = i / WL % L, f = feature(i / (L * WL) * WL + i % WL);
        lev[i] = f < n && c < a.real_levels ? a.levels[(size_t)f * a.real_levels + c] : 0.0f;
    }
#pragma unroll 1
    for (int g = tid; g < F; g += kSliceThreads + 32) xown[g] = feature(g) < n ? a.x[feature(g)] : 0.0f;
#pragma unroll 1
    for (int r = B + tid; r < rows_pad; r += kSliceThreads + 32) res[r] = make_float2(0.0f, 0.0f);
    mbar_fence_init();
    __syncthreads();
    slice_cluster_sync();                                // every CTA's barriers exist before anyone writes into it

    // steps are counted from the call's first one; a batch is named by its index
    const int steps = (int)a.num_steps, whole = a.whole;
    auto batch_at = [&](int k) { return k < steps ? (a.order ? a.order[a.first_step + k] : (int)a.first_step + k) : 0; };
    auto own_of = [&](int batch) { return max(0, min(own, (batch < whole ? (int)a.batch : a.rows_last) - bi * a.rpo)); };
    if (warp == kSliceWarps) {
        // -------------------------------------------------------------------- the copying warp
        int slot = 0;
        uint32_t parity = 1;                             // of the slots' emptiness: all are empty at first
#pragma unroll 1
        for (int k = 0; k < steps; ++k) {
            const int batch = batch_at(k);
            const int64_t r0 = batch * a.batch;
            unsigned char* dst = ring + slot * a.slot_bytes;
            slice_wait(sh, sh->empty + slot, parity, a.status, 84);
            if (lane == 0) {                             // (boxes that reach past the last row are filled up and count in full)
                mbar_arrive_expect_tx(sh->full + slot, 2u * (uint32_t)(a.boxes * a.box_rows * a.pitch));
#pragma unroll 1
                for (int i = 0; i < a.boxes; ++i) {
                    slice_tensor_copy(dst + i * a.box_rows * a.pitch, &tm1, 2 * bi * a.units, (int)r0 + i * a.box_rows, sh->full + slot);
                    slice_tensor_copy(dst + a.plane_bytes + i * a.box_rows * a.pitch, &tm2, 2 * bi * a.units, (int)r0 + i * a.box_rows, sh->full + slot);
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
    const int wl = lane & (WL - 1), rl = lane / WL;
    const uint32_t tab_addr = smem_u32(tab), lev_addr = smem_u32(lev), lane_offsets = 0x04040404u * (uint32_t)wl;
    const uint32_t res_addr = smem_u32(res);
    const int p4 = tid & 3, g4 = tid >> 2;               // four lanes per feature of the own units
    auto owner_of = [&](int r) { return (int)__umulhi(2u * (uint32_t)r + 1u, a.rpo_inv); };
    float2* const dot_row = dsum + bi * dstride;         // this CTA's dots at an owner
    // a lane's quarter of the levels times the model entry
    auto put = [&](int g, float xt) {
        const int at = g / WL * (L * WL) + g % WL + p4 * WL;
#pragma unroll
        for (int c = 0; c < L; c += 4) tab[at + c * WL] = lev[at + c * WL] * xt;
    };
    auto publishes = [&](int step, int g, float xt) {
        if (a.model_out && step + 2 == steps && p4 == 0 && feature(g) < n) a.model_out[feature(g)] = xt;
    };
    auto update = [&](int step, int g, float gr) {
        const float x = xown[g], y = fmaf(-a.lr, gr, x);
        const float xt = a.reg == ZIPML_REG_NONE ? y : slice_regularise(y, x, a.reg, a.reg_cst);
        __syncwarp();
        if (p4 == 0) xown[g] = xt;
        if (a.model_bits == 0) { put(g, xt); publishes(step, g, xt); }
    };
    const int marked = blockIdx.x == 0 && tid == 0 && a.trace ? a.trace_steps : -1;
    int batch = batch_at(0), batch_next = batch_at(1);
    int slot = 0;
    uint32_t parity = 0, step_parity = 0, gn_parity = 0, xn_parity = 0;
#pragma unroll 1
    for (int step = -1; step < steps; ++step) {
        const bool last = step == steps - 1;
        if (step >= 0) {
            const unsigned char* tile = ring + slot * a.slot_bytes;
            const uint32_t lane_addr = smem_u32(tile) + (uint32_t)(wl * 4);
            if (step < marked) slice_mark(a.trace, step, 0);
            slice_wait(sh, sh->full + slot, parity, a.status, 6);
            if (step < marked) slice_mark(a.trace, step, 1);
            // -------------------------------------------------------------- dots
            if (B >= kTableRowLanes) {
                // a lane takes a row's units whole: nothing to exchange
#pragma unroll 1
                for (int r = tid; r < rows_pad; r += kSliceThreads) {
                    uint32_t addr = smem_u32(tile) + (uint32_t)(r * a.pitch), t = tab_addr;
                    float s1 = 0.0f, s2 = 0.0f;
#pragma unroll 1
                    for (int u = 0; u < a.units; ++u, addr += 16u, t += HW * REGION) {
                        uint32_t w1[4], w2[4];
                        table_words(w1, addr);
                        table_words(w2, addr + (uint32_t)a.plane_bytes);
                        float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                        for (int w = 0; w < 4; ++w) {
                            const TableOffsets<BITS> c1(w1[w], 0x04040404u * (w % WL)), c2(w2[w], 0x04040404u * (w % WL));
#pragma unroll
                            for (int i = 0; i < FPW; ++i) {
                                v[w & 1] += table_load(c1.at(i, t + w / WL * REGION));
                                v[2 + (w & 1)] += table_load(c2.at(i, t + w / WL * REGION));
                            }
                        }
                        s1 += v[0] + v[1];
                        s2 += v[2] + v[3];
                    }
                    const float n1 = __shfl_down_sync(0xffffffffu, s1, 1), n2 = __shfl_down_sync(0xffffffffu, s2, 1);
                    if ((lane & 1) == 0 && r < B) {
                        const int owner = owner_of(r);
                        slice_store16(slice_peer(dot_row + r - owner * a.rpo, owner), table_four(s1, s2, n1, n2), slice_peer(&sh->dot_bar, owner));
                    }
                }
            } else {
#pragma unroll 1
                for (int r0 = warp * RPW; r0 < B; r0 += ROWS) {
                    uint32_t addr = lane_addr + (uint32_t)((r0 + rl) * a.pitch), t = tab_addr;
                    float s1 = 0.0f, s2 = 0.0f;
#pragma unroll 1
                    for (int wd = 0; wd < a.units * HW; ++wd, addr += 4u * WL, t += REGION) {    // units, and in each the words of the lane
                        const TableOffsets<BITS> c1(table_word(addr), lane_offsets), c2(table_word(addr + (uint32_t)a.plane_bytes), lane_offsets);
                        float v1 = 0.0f, v2 = 0.0f;
#pragma unroll
                        for (int i = 0; i < FPW; ++i) {
                            v1 += table_load(c1.at(i, t));
                            v2 += table_load(c2.at(i, t));
                        }
                        s1 += v1;
                        s2 += v2;
                    }
                    // even lanes end up with plane 1, odd ones with plane 2
                    float v = (lane & 1 ? s2 : s1) + __shfl_xor_sync(0xffffffffu, lane & 1 ? s1 : s2, 1);
#pragma unroll
                    for (int o = 2; o < WL; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                    const float other = __shfl_xor_sync(0xffffffffu, v, 1);
                    if (wl == 0 && r0 + rl < B) {
                        const int owner = owner_of(r0 + rl);
                        slice_store8(slice_peer(dot_row + r0 + rl - owner * a.rpo, owner), table_pair(v, other), slice_peer(&sh->dot_bar, owner));
                    }
                }
            }
            if (step < marked) slice_mark(a.trace, step, 2);
            // -------------------------------------------------------------- residuals of the own rows
            const bool batch_full = batch < whole;
            if (2 * warp < own) {
                slice_wait(sh, &sh->dot_bar, step_parity, a.status, 4);
                if (tid == 0 && !last) mbar_arrive_expect_tx(&sh->dot_bar, 8u * a.nb * own);
                const float* labels = reinterpret_cast<const float*>(tile + 2 * a.plane_bytes);
                const int rows = own_of(batch);
#pragma unroll 1
                for (int i0 = 2 * warp; i0 < own; i0 += 2 * kSliceWarps) {
                    const int i = i0 + (lane >> 4);
                    const int p16 = lane & 15;
                    const float2 d = i < own && p16 < a.nb ? dsum[p16 * dstride + i] : make_float2(0.0f, 0.0f);
                    double v = (double)(lane & 1 ? d.y : d.x) + __shfl_xor_sync(0xffffffffu, (double)(lane & 1 ? d.x : d.y), 1);
#pragma unroll
                    for (int o = 2; o < 16; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                    const float r = i < rows ? (float)(v - (double)labels[i]) : 0.0f;
                    // lane p < nb gets both rows' residuals for CTA p (the odd lanes of a row have plane 2)
                    const float other = __shfl_xor_sync(0xffffffffu, r, 1);
                    const float r1 = lane & 1 ? other : r, r2 = lane & 1 ? r : other;
                    const float n1 = __shfl_down_sync(0xffffffffu, r1, 16), n2 = __shfl_down_sync(0xffffffffu, r2, 16);
                    if (lane < a.nb) slice_store16(slice_peer(res + bi * a.rpo + i, lane), table_four(r1, r2, n1, n2), slice_peer(&sh->res_bar, lane));
                }
            }
            if (step < marked) slice_mark(a.trace, step, 3);
            slice_wait(sh, &sh->res_bar, step_parity, a.status, 5);
            if (tid == 0 && !last) mbar_arrive_expect_tx(&sh->res_bar, 8u * B);
            step_parity ^= 1u;
            if (step < marked) slice_mark(a.trace, step, 4);
            // -------------------------------------------------------------- gradient of the own features
#pragma unroll 1
            for (int wd = 0; wd < a.units * HW; ++wd) {
                const uint32_t region = lev_addr + (uint32_t)(wd * REGION);
                float acc[FPW];
#pragma unroll
                for (int i = 0; i < FPW; ++i) acc[i] = 0.0f;
#pragma unroll 1
                for (int r0 = warp * RPW; r0 < B; r0 += ROWS) {
                    const uint32_t addr = lane_addr + (uint32_t)((r0 + rl) * a.pitch + wd * 4 * WL);
                    const TableOffsets<BITS> c1(table_word(addr), lane_offsets), c2(table_word(addr + (uint32_t)a.plane_bytes), lane_offsets);
                    float r1, r2;
                    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(r1), "=f"(r2) : "r"(res_addr + 8u * (uint32_t)(r0 + rl)));
#pragma unroll
                    for (int i = 0; i < FPW; ++i) {
                        acc[i] = fmaf(table_load(c1.at(i, region)), r2, acc[i]);
                        acc[i] = fmaf(table_load(c2.at(i, region)), r1, acc[i]);
                    }
                }
                // over the warp's rows: each exchange halves what a lane keeps
                int first = 0, kept = FPW;
#pragma unroll
                for (int o = 16; o >= WL; o >>= 1) {
                    if (kept > 1) {
                        kept >>= 1;
#pragma unroll
                        for (int j = 0; j < FPW / 2; ++j)
                            if (j < kept) {
                                const float give = lane & o ? acc[j] : acc[j + kept];
                                acc[j] = (lane & o ? acc[j + kept] : acc[j]) + __shfl_xor_sync(0xffffffffu, give, o);
                            }
                        if (lane & o) first += kept;
                    } else {
                        acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
                    }
                }
#pragma unroll
                for (int j = 0; j < FPW / RPW || j < 1; ++j) {
                    const int g = (wd * FPW + first + j) * WL + wl;
                    gsum[g * 16 + ((warp ^ (g << 1)) & 12) + (warp & 3)] = acc[j];
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(sh->empty + slot);
            if (++slot == a.slots) { slot = 0; parity ^= 1u; }
            batch = batch_next;
            batch_next = batch_at(step + 2);
            if (step < marked) slice_mark(a.trace, step, 5);
            slice_bar();
            // -------------------------------------------------------------- sums over the warps, update
            double gsq = 0.0;
#pragma unroll 1
            for (int g = g4; g < F; g += kSliceThreads / 4) {
                const float4 v = *reinterpret_cast<const float4*>(gsum + g * 16 + p4 * 4);
                double t = ((double)v.x + (double)v.y) + ((double)v.z + (double)v.w);
                t += __shfl_xor_sync(0xffffffffu, t, 1);
                t += __shfl_xor_sync(0xffffffffu, t, 2);
                const float gr = (float)(t * (batch_full ? a.full_scale : a.last_scale));
                const bool writes = p4 == 0 && feature(g) < n;
                if (last && a.grad_out && writes) {
                    a.grad_out[feature(g)] = gr;
                    if (a.grad_bits == 0) a.grad_out[n + feature(g)] = gr;
                }
                if (a.grad_bits > 0) {
                    if (writes) gsq += (double)gr * (double)gr;
                    if (p4 == 0) gsub[g] = gr;
                } else {
                    update(step, g, gr);
                }
            }
            if (step < marked) slice_mark(a.trace, step, 6);
            if (a.grad_bits > 0) {
                const float M = slice_norm(gsq, 4, bi, sh->red[0], sh->nrm_g, &sh->gn_bar, gn_parity, a.nb, sh, a.status, 3);
                gn_parity ^= 1u;
#pragma unroll 1
                for (int g = g4; g < F; g += kSliceThreads / 4) {
                    const uint32_t draw = slice_draw(a.seed, a.epoch, (uint32_t)a.first_step + (uint32_t)step, (uint32_t)feature(g), 4u);
                    const float gr = slice_quantize(gsub[g], M, a.grad_bits, draw);
                    if (last && a.grad_out && p4 == 0 && feature(g) < n) a.grad_out[n + feature(g)] = gr;
                    update(step, g, gr);
                }
            }
        } else if (a.model_bits == 0) {
#pragma unroll 1
            for (int g = g4; g < F; g += kSliceThreads / 4) { put(g, xown[g]); publishes(step, g, xown[g]); }
        }
        if (last) break;

        // ------------------------------------------------------------------ Q3: what the next step sees
        if (a.model_bits > 0) {
            __syncwarp();
            double xsq = 0.0;
            if (p4 == 0)
#pragma unroll 1
                for (int g = g4; g < F; g += kSliceThreads / 4) xsq += (double)xown[g] * (double)xown[g];
            const float M = slice_norm(xsq, 4, bi, sh->red[1], sh->nrm_x, &sh->xn_bar, xn_parity, a.nb, sh, a.status, 8);
            xn_parity ^= 1u;
#pragma unroll 1
            for (int g = g4; g < F; g += kSliceThreads / 4) {
                const uint32_t draw = slice_draw(a.seed, a.epoch, (uint32_t)a.first_step + (uint32_t)step + 1u, (uint32_t)feature(g), 3u);
                const float xt = slice_quantize(xown[g], M, a.model_bits, draw);
                put(g, xt);
                publishes(step, g, xt);
            }
        }
        slice_bar();
        if (step >= 0 && step < marked) slice_mark(a.trace, step, 7);
    }
    if (p4 == 0)
#pragma unroll 1
        for (int g = g4; g < F; g += kSliceThreads / 4)
            if (feature(g) < n) a.x[feature(g)] = xown[g];
    __syncwarp();
    slice_cluster_sync();                                // nobody leaves while a store may still target it
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
int launch_sgd_table(zipml_ctx* ctx, const zipml_dataset* d, const float* b, float* x, const zipml_sgd_params* p, int64_t first_step,
                     int64_t num_steps, float* grad_out) {
    if (d->level_mode != ZIPML_LEVELS_TABLE || d->bits > 4) return ZIPML_ERR_WORKSPACE;
    const int cb = container_bits(d->bits), bits = d->bits < 2 ? 2 : d->bits;
    const int64_t B = p->batch < d->m ? p->batch : d->m;
    const int64_t all_units = (d->n * cb + 127) / 128;
    const int64_t T = (d->m + p->batch - 1) / p->batch;
    if (B > 8192 || all_units > 1024 || d->m >= (1ll << 31) - 16384 || T > 0x7ffffff0) return ZIPML_ERR_WORKSPACE;
    const int64_t most = p->grid_row_parts > 0 && p->grid_row_parts < kSliceMaxCtas ? p->grid_row_parts : kSliceMaxCtas;
    TableArgs a;
    memset(&a, 0, sizeof(a));
    a.units = (int)((all_units + most - 1) / most);
    a.nb = (int)((all_units + a.units - 1) / a.units);
    a.rpo = 2 * (int)((B + 2 * a.nb - 1) / (2 * a.nb));           // (even: rows travel in pairs)
    a.rpo_inv = (uint32_t)((1ull << 31) / (uint64_t)a.rpo);
    a.boxes = (int)((B + 255) / 256);
    a.box_rows = (int)((B + a.boxes - 1) / a.boxes);
    if (a.boxes > 1) a.box_rows = (a.box_rows + 7) / 8 * 8;      // (a copy starts on 128 bytes)
    const int features = a.units * 512 / cb / 4, rows = (int)((B + 31) / 32 * 32);
    const size_t fixed = sizeof(TableShared) + 4 * (size_t)features * (((size_t)2 << bits) + 2 + 16) + (size_t)a.nb * (a.rpo + 2) * 8 + 8 * (size_t)rows + 128;
    // rows lie an odd number of units apart, so that 8 of them meet all banks; closer where two tiles would not fit otherwise
    for (int pad = 1;; pad = 0) {
        a.pitch = 16 * (pad ? a.units | 1 : a.units);
        const int tile_rows = a.boxes * a.box_rows > rows ? a.boxes * a.box_rows : rows;
        a.plane_bytes = (tile_rows * a.pitch + 127) / 128 * 128;
        a.slot_bytes = 2 * a.plane_bytes + (4 * a.rpo + 127) / 128 * 128;
        a.slots = kSliceMaxSlots;
        while (a.slots > 1 && fixed + (size_t)a.slots * a.slot_bytes > (size_t)ctx->smem_optin) --a.slots;
        if (a.slots >= 2) break;
        if (!pad || a.units % 2 != 0) return ZIPML_ERR_WORKSPACE;
    }
    CUtensorMap tmaps[2];
    memset(tmaps, 0, sizeof(tmaps));
    int rc = encode_plane_maps(ctx, d, a.pitch / 4, a.box_rows, true, tmaps);
    if (rc != ZIPML_OK) return ZIPML_ERR_WORKSPACE;              // (also where a box would be wider than 256 elements)
    const size_t smem = fixed + (size_t)a.slots * a.slot_bytes;
    const void* kernel = bits == 2 ? (const void*)sgd_table_kernel<2> : bits == 3 ? (const void*)sgd_table_kernel<3> : (const void*)sgd_table_kernel<4>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess && a.nb > 8) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return cuda_status(e);
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)a.nb);
    cfg.blockDim = dim3(kSliceThreads + 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = ctx->stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)a.nb;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int fit = 0;
    e = cudaOccupancyMaxActiveClusters(&fit, kernel, &cfg);
    if (e != cudaSuccess) { (void)cudaGetLastError(); return ZIPML_ERR_WORKSPACE; }
    if (fit < 1) return ZIPML_ERR_WORKSPACE;
    if (early_start(ctx, num_steps, attr + 1)) cfg.numAttrs = 2;
    if (p->batch_order) {
        rc = ws_reserve(ctx, carve_size(sizeof(int32_t) * (size_t)T));
        if (rc != ZIPML_OK) return rc;
        e = cudaMemcpyAsync(ctx->ws, p->batch_order, sizeof(int32_t) * (size_t)T, cudaMemcpyHostToDevice, ctx->stream);
        if (e != cudaSuccess) return cuda_status(e);
        a.order = reinterpret_cast<const int32_t*>(ctx->ws);
    }
    a.levels = d->levels;
    a.b = b; a.x = x; a.grad_out = grad_out; a.model_out = p->model_out;
    a.trace = reinterpret_cast<unsigned long long*>(p->trace);
    a.trace_steps = p->trace ? p->trace_steps : 0;
    a.status = ctx->d_status;
    a.batch = B;
    a.first_step = first_step; a.num_steps = num_steps;
    a.whole = (int)(d->m / B); a.rows_last = (int)(d->m - a.whole * B);
    a.full_scale = 1.0 / (2.0 * (double)B); a.last_scale = 1.0 / (2.0 * (double)(a.rows_last > 0 ? a.rows_last : 1));
    a.seed = p->seed; a.epoch = (uint32_t)p->epoch; a.lr = p->lr; a.reg = p->reg; a.reg_cst = reg_constant(p);
    a.n = (int)d->n; a.real_levels = 1 << d->bits; a.model_bits = p->model_bits; a.grad_bits = p->grad_bits;
    void* params[] = {&a, &tmaps[0], &tmaps[1]};
    e = cudaLaunchKernelExC(&cfg, kernel, params);
    if (e != cudaSuccess) return cuda_status(e);
    ctx->launches += 1;
    ctx->ran(ZIPML_ENGINE_CLUSTER, "sgd_table_kernel");
    return ZIPML_OK;
}

}  // namespace zipml
