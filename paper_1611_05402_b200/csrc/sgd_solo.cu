// Solo engine of zipml_sgd_epoch: the whole minibatch chain on one thread block, for steps so small that handing a
// value to another SM costs more than the arithmetic of the step (Supplement "Double Sampling", footnote form;
// "End-to-end Quantization").
//
// A step of 16 rows x 64 features is 4,096 multiply-adds.  Split over the two SMs that the cluster engine gives it, it
// took 3.4 us, nearly all of it two exchanges (gradient parts out, model back) at some 1,200 cycles each.  Here the
// model never leaves the block and a step has two block barriers:
//   * dots: 2^a_shift lanes share a row and walk its words; fp32 FMA on unpacked codes against w = step * x~, a halving
//     butterfly leaves plane 1's dot in even lanes and plane 2's in odd ones; residuals to shared memory; barrier;
//   * gradient and update: 2^b_shift lanes share a word column and walk the rows; a halving butterfly over the word's
//     features leaves each lane with the sums of its own KEEP features, whose x, step and mid value it holds in
//     registers: it updates them and writes the next step's w; barrier.  A quantized gradient or model adds a sum over
//     the block each, for the norm; their random draws are made while the others still form residuals.
//   * the code tiles do not depend on the model: an extra warp runs a few steps ahead with cp.async copies into a ring
//     of slots.  Rows lie `pitch` words apart, chosen with the lane splits (make_solo_plan) so that lanes on
//     different rows meet different banks.
// Codes are centred per feature (value = mid + (code - centre) * step, the centre the code whose value is nearest zero): the
// dot's two parts, mid^T x~ and the codes', stay small instead of cancelling, and fp32 sums of a lane keep their
// precision -- on features of both signs as on rows that are mostly zeros, where one centre for all (half the top code) lost 10 to
// 20 times of it.  The lanes' sums of a dot meet in double.  Where a feature lies apart from zero by more than its step ("far", found out
// once per launch), mid^T x~ and the sum of the residuals are held in double too; elsewhere |mid| <= step and fp32 adds no
// more than the codes' own rounding.
// What bounds it: the latency of the chain load - unpack - FMA - butterfly - barrier, twice a step.
// Measured, us per step of 200, cluster engine split by rows -> here: 16 x 64 at 4 bits 3.75 -> 1.08 (1.00 with one centre for all and every
// sum in fp32), 64 x 64 at 8 bits 3.75 -> 1.45, 16 x 250 on 2-bit tables 4.27 -> 1.87; 64 x 64 at 4 bits with quantized model and
// gradient 6.23 -> 3.00.
#include <string.h>

#include <type_traits>

#include "sgd_common.cuh"

namespace zipml {

constexpr int kSoloMaxThreads = 512;             // without the copying warp
constexpr int kSoloMaxSlots = 8;

struct SoloArgs {
    const uint32_t* p1;
    const uint32_t* p2;
    const float* lo;
    const float* step;
    const float* levels;
    const float* b;
    float* x;
    float* grad_out;             // null or 2n
    float* model_out;            // null or n: the model the last executed step's gradient saw
    const int32_t* order;        // device copy of the batch order, or null
    DeviceStatus* status;
    int64_t m, batch, first_step, num_steps;
    uint64_t seed;
    uint32_t epoch;
    float lr;
    int reg;                     // ZIPML_REG_* and its fp32 constant
    float reg_cst;
    int n, bits, row_words, words;   // words = ceil(n / codes per word) <= row_words
    int model_bits, grad_bits;
    int rc;                      // rows of a full batch
    int pitch;                   // words between rows of a tile in shared memory
    int slots;                   // tiles in the ring
    int a_shift;                 // 2^a_shift lanes share a row's dots
    int b_shift;                 // 2^b_shift lanes share a word column's gradient
    int copy_shift;              // 2^copy_shift lanes share the copy of a row
};

struct SoloShared {
    double red[2][16];           // parts of the gradient's and the model's squared norm, one per warp
    uint64_t full[kSoloMaxSlots], empty[kSoloMaxSlots];
    int rows[kSoloMaxSlots];     // rows of the slot's tile
    int gave_up;
    int far;                     // a feature lies apart from zero by more than its step
};
constexpr size_t kSoloSharedBytes = (sizeof(SoloShared) + 15) & ~(size_t)15;

// Codes of a word as floats minus their centres (bias = 2^23 + centre).
template <int CB>
__device__ __forceinline__ void unpack_centred(uint32_t w, const float (&bias)[32 / CB], float (&c)[32 / CB]) {
    auto byte = [&](uint32_t bytes, int i, int f) { c[f] = __uint_as_float(__byte_perm(bytes, 0x4B000000u, 0x7650 + i)) - bias[f]; };
    if constexpr (CB == 8) {
#pragma unroll
        for (int i = 0; i < 4; ++i) byte(w, i, i);
    } else if constexpr (CB == 4) {
        const uint32_t even = w & 0x0F0F0F0Fu, odd = (w >> 4) & 0x0F0F0F0Fu;
#pragma unroll
        for (int i = 0; i < 4; ++i) { byte(even, i, 2 * i); byte(odd, i, 2 * i + 1); }
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t t = (w >> (2 * k)) & 0x03030303u;
#pragma unroll
            for (int i = 0; i < 4; ++i) byte(t, i, 4 * i + k);
        }
    }
}

// A word's entries of a quad array (see below).
template <int FPW>
__device__ __forceinline__ void solo_quads(float (&v)[FPW], const float4* quads, int nwq, int q) {
#pragma unroll
    for (int i = 0; i < FPW / 4; ++i) {
        const float4 t = quads[i * nwq + q];
        v[4 * i] = t.x; v[4 * i + 1] = t.y; v[4 * i + 2] = t.z; v[4 * i + 3] = t.w;
    }
}

// VecQuant::apply with its draw given.
__device__ __forceinline__ float solo_quantize(float v, float M, int bits, uint32_t u24) {
    if (!(M > 0.0f)) return 0.0f;
    const int sm = (1 << (bits - 1)) - 1;
    const float t = __fmul_rn(__fdiv_rn(fabsf(v), M), (float)sm);
    float fl = floorf(t);
    fl = fl > (float)(sm - 1) ? (float)(sm - 1) : fl;
    const float p = __fsub_rn(t, fl);
    const uint32_t mag = (uint32_t)fl + ((__fmul_rn((float)u24, 5.9604644775390625e-08f) < p) ? 1u : 0u);
    const float q = __fmul_rn(M, __fdiv_rn((float)mag, (float)sm));
    return v < 0.0f ? -q : q;
}

__device__ __forceinline__ void copy16(void* dst_smem, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst_smem)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy4(void* dst_smem, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst_smem)), "l"(src) : "memory");
}
// This thread's copies so far count as one arrival on `bar` once they have landed.
__device__ __forceinline__ void arrive_after_copies(uint64_t* bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Bounded wait on a phase; once one has given up, none of the block waits any more and the launch runs to its end.
__device__ __forceinline__ void solo_wait(SoloShared* sh, uint64_t* bar, uint32_t parity, DeviceStatus* status, int where) {
    if (mbar_try_wait(bar, parity)) return;
    for (long long spin = 0; spin < kCopySpinLimit; ++spin) {
        if (mbar_try_wait(bar, parity)) return;
        if (*reinterpret_cast<volatile int*>(&sh->gave_up)) return;
    }
    sh->gave_up = 1;
    set_status(status, ZIPML_ERR_TIMEOUT, where);
}

// Shared memory; nwq = words rounded up to 8, a "quad array" holds 4 FPW nwq bytes as float4 [FPW / 4][nwq], feature
// i of word q in component i & 3 of element [i >> 2][q] (lanes on neighbouring words read neighbouring 16 bytes):
//   SoloShared
//   quad arrays   ws (uniform: step * x~; table: x~) and for uniform grids centre (2^23 + the feature's centre)
//   uniform       mid^T x~: a quad array, or (far) doubles mx [FPW / KEEP][nwq], an owner's features' part each
//   table         lev [L][FPW][nwq]
//   float res[2 rc]        residuals (r1, r2) per row
//   ring[slots]: codes [2][rc][pitch], labels [rc]
template <int CB, bool TABLE, int KEEP>
__global__ void __launch_bounds__(kSoloMaxThreads + 32, 1) sgd_solo_kernel(const SoloArgs a) {
    constexpr int FPW = 32 / CB, LOGF = CB == 8 ? 2 : CB == 4 ? 3 : 4;
    extern __shared__ __align__(16) unsigned char s_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, threads = blockDim.x - 32, nwarps = threads >> 5;
    const int nw = a.words, nwq = (nw + 7) & ~7, n = a.n, L = 1 << a.bits, F = nwq * FPW;
    SoloShared* sh = reinterpret_cast<SoloShared*>(s_raw);
    float* ws = reinterpret_cast<float*>(s_raw + kSoloSharedBytes);
    float* centre = ws + F;
    double* mx = reinterpret_cast<double*>(centre + (TABLE ? 0 : F));
    float* lev = ws + F;
    float* res = TABLE ? lev + L * F : reinterpret_cast<float*>(mx + F / (KEEP < 2 ? KEEP : 2));
    uint32_t* ring = reinterpret_cast<uint32_t*>(res + ((2 * a.rc + 3) & ~3));
    const int plane_words = a.rc * a.pitch, slot_words = 2 * plane_words + ((a.rc + 3) & ~3);
    if (tid < a.slots) {
        mbar_init(sh->full + tid, 33);                             // the copying lanes, and their leader for rows[]
        mbar_init(sh->empty + tid, 1);
        sh->rows[tid] = a.rc;
    }
    if (tid == 0) sh->gave_up = sh->far = 0;
    // (a wait that has given up computes on whatever lies in its slot: no code may then point past the table)
    if (TABLE && L < (1 << CB))
        for (int i = tid; i < a.slots * slot_words; i += blockDim.x) ring[i] = 0u;
    mbar_fence_init();
    __syncthreads();

    if (warp == nwarps) {
        // ------------------------------------------------------------------ the copying warp
        int slot = 0;
        uint32_t parity = 1;                                       // of the slots' emptiness: all are empty at first
        for (int64_t k = 0; k < a.num_steps; ++k) {
            const int64_t it = a.first_step + k;
            const int64_t r0 = (a.order ? (int64_t)a.order[it] : it) * a.batch;
            const int rows = (int)min(a.batch, a.m - r0);
            uint32_t* dst = ring + slot * slot_words;
            const int c = lane & ((1 << a.copy_shift) - 1), pieces = a.row_words >> 2, stride = 32 >> a.copy_shift;
            const uint32_t* s1 = a.p1 + (r0 + (lane >> a.copy_shift)) * a.row_words;
            const uint32_t* s2 = a.p2 + (r0 + (lane >> a.copy_shift)) * a.row_words;
            solo_wait(sh, sh->empty + slot, parity, a.status, 81);
            for (int r = lane >> a.copy_shift; r < rows; r += stride, s1 += stride * a.row_words, s2 += stride * a.row_words)
                for (int p = c; p < pieces; p += 1 << a.copy_shift) {
                    copy16(dst + r * a.pitch + 4 * p, s1 + 4 * p);
                    copy16(dst + plane_words + r * a.pitch + 4 * p, s2 + 4 * p);
                }
            for (int r = lane; r < rows; r += 32) copy4(dst + 2 * plane_words + r, a.b + r0 + r);
            arrive_after_copies(sh->full + slot);
            if (lane == 0) { sh->rows[slot] = rows; mbar_arrive(sh->full + slot); }
            if (++slot == a.slots) { slot = 0; parity ^= 1u; }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        return;
    }

    // ---------------------------------------------------------------------- the computing warps
    // the features that the butterfly over a word column leaves in this lane: KEEP consecutive ones, from `first` on
    const int GA = 1 << a.a_shift, GB = 1 << a.b_shift;
    const int la = tid & (GA - 1), lb = tid & (GB - 1), row_first = tid >> a.a_shift, row_stride = threads >> a.a_shift;
    const int q = min(tid >> a.b_shift, nw - 1);
    int first = 0;
#pragma unroll
    for (int s = 0; s < LOGF; ++s)
        if (s < a.b_shift && (lb >> s & 1)) first += FPW >> (s + 1);
    const int f0 = q * FPW + first, at0 = ((first >> 2) * nwq + q) * 4 + (first & 3);
    const bool owner = (tid >> a.b_shift) < nw && (lb >> LOGF) == 0;
    float x[KEEP], st[KEEP];
    double mid[KEEP];
    for (int f = tid; f < F; f += threads) ws[f] = 0.0f;           // (slots past the last feature stay zero)
    if constexpr (TABLE) {
        for (int f = tid; f < F; f += threads)
            for (int c = 0; c < L; ++c) lev[(c * FPW + (f & (FPW - 1))) * nwq + (f >> LOGF)] = f < n ? __ldg(a.levels + (size_t)f * L + c) : 0.0f;
    } else {
        for (int f = tid; f < F; f += threads) { centre[f] = 8388608.0f; reinterpret_cast<float*>(mx)[f] = 0.0f; }
    }
    auto bar = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory"); };
    // l2 norm of the owners' values, summed in double in a fixed order
    auto norm = [&](const float (&v)[KEEP], int which) {
        double t = 0.0;
        if (owner)
#pragma unroll
            for (int k = 0; k < KEEP; ++k) t += f0 + k < n ? (double)v[k] * (double)v[k] : 0.0;
        t = warp_sum(t);
        if (lane == 0) sh->red[which][warp] = t;
        bar();
        t = 0.0;
        for (int w = 0; w < nwarps; ++w) t += sh->red[which][w];
        return (float)sqrt(t);
    };
    auto draws = [&](int64_t it, uint32_t stream, uint32_t (&u)[KEEP]) {
        const Philox4 b = philox4x32_10((uint32_t)f0 >> 2, (uint32_t)it, a.epoch, stream, (uint32_t)a.seed, (uint32_t)(a.seed >> 32));
#pragma unroll
        for (int k = 0; k < KEEP; ++k) {
            const int c = (f0 & 3) + k;
            u[k] = (c == 0 ? b.v[0] : c == 1 ? b.v[1] : c == 2 ? b.v[2] : b.v[3]) >> 8;
        }
    };
    // what the next step's dots see of the model
    auto publish = [&](auto far, const float (&v)[KEEP], bool seen_last) {
        if (!owner) return;
#pragma unroll
        for (int k = 0; k < KEEP; ++k)
            if (f0 + k < n) {
                if (seen_last && a.model_out) a.model_out[f0 + k] = v[k];
                if constexpr (TABLE) ws[at0 + k] = v[k];
                else {
                    ws[at0 + k] = st[k] * v[k];
                    if constexpr (!decltype(far)::value) reinterpret_cast<float*>(mx)[at0 + k] = (float)mid[k] * v[k];
                }
            }
        if constexpr (!TABLE && decltype(far)::value) {
            double base = 0.0;
#pragma unroll
            for (int k = 0; k < KEEP; ++k) base = fma(mid[k], (double)v[k], base);
            mx[first / KEEP * nwq + q] = base;
        }
    };
    bar();                                                         // the zeros are in place
    bool far_lane = false;
#pragma unroll
    for (int k = 0; k < KEEP; ++k) {
        const bool real = f0 + k < n;
        x[k] = real ? a.x[f0 + k] : 0.0f;
        if constexpr (!TABLE) {
            st[k] = real ? __ldg(a.step + f0 + k) : 0.0f;
            const float lo = real ? __ldg(a.lo + f0 + k) : 0.0f;
            // (any whole number would do: how the quotient is rounded does not matter)
            const float c = fminf(fmaxf(rintf(__fdividef(-lo, st[k])), 0.0f), (float)((1 << a.bits) - 1));
            mid[k] = fma((double)c, (double)st[k], (double)lo);
            far_lane = far_lane || fabs(mid[k]) > (double)st[k];
            if (owner) centre[at0 + k] = 8388608.0f + c;
        }
    }
    auto run = [&](auto far) {
    constexpr bool FAR = decltype(far)::value;
    if (a.model_bits > 0) {
        uint32_t u[KEEP];
        draws(a.first_step, 3u, u);
        const float M = norm(x, 1);
        float v[KEEP];
#pragma unroll
        for (int k = 0; k < KEEP; ++k) v[k] = solo_quantize(x[k], M, a.model_bits, u[k]);
        publish(far, v, a.num_steps == 1);
    } else {
        publish(far, x, a.num_steps == 1);
    }
    bar();

    const float full_scale = 1.0f / (2.0f * (float)a.rc);
    const bool single = nw <= GA;                                  // a lane has one word of w: it keeps it for all its rows
    const float4* w4 = reinterpret_cast<const float4*>(ws) + (single ? min(la, nw - 1) : 0);
    [[maybe_unused]] const float4* c4 = reinterpret_cast<const float4*>(centre);
    [[maybe_unused]] const float4* m4 = reinterpret_cast<const float4*>(mx);
    const int stride_shift = 31 - __clz(row_stride);               // (threads is a power of two)
    // of the lane's word in the dots (where it has one), in the gradient; of 16 codes to a word anew in every step: too many registers
    constexpr bool kKept = !TABLE && FPW <= 8;
    [[maybe_unused]] float bias_a[FPW], bias_b[FPW];
    if constexpr (kKept) {
        solo_quads<FPW>(bias_a, c4, nwq, min(la, nw - 1));
        solo_quads<FPW>(bias_b, c4, nwq, q);
    }
    int slot = 0;
    uint32_t parity = 0;
#pragma unroll 1
    for (int64_t left = a.num_steps, it = a.first_step; left > 0; --left, ++it) {
        const bool last = left == 1;
        const uint32_t* t1 = ring + slot * slot_words;
        const uint32_t* t2 = t1 + plane_words;
        const float* labels = reinterpret_cast<const float*>(t2 + plane_words);
        solo_wait(sh, sh->full + slot, parity, a.status, 82);
        const int rows = sh->rows[slot];

        // ---------------------------------------------------------------- dots and residuals
        auto add_word = [&](int at, int col, const float (&w)[FPW], const float (&bias)[FPW], float& a1, float& a2) {
            const uint32_t u1 = t1[at], u2 = t2[at];
            if constexpr (!TABLE) {
                float c1[FPW], c2[FPW];
                unpack_centred<CB>(u1, bias, c1);
                unpack_centred<CB>(u2, bias, c2);
#pragma unroll
                for (int i = 0; i < FPW; ++i) { a1 = fmaf(c1[i], w[i], a1); a2 = fmaf(c2[i], w[i], a2); }
            } else {
#pragma unroll
                for (int i = 0; i < FPW; ++i) {
                    a1 = fmaf(lev[(code_at<CB>(u1, i) * FPW + i) * nwq + col], w[i], a1);
                    a2 = fmaf(lev[(code_at<CB>(u2, i) * FPW + i) * nwq + col], w[i], a2);
                }
            }
        };
        // mid^T x~ over the lane's words
        float base = 0.0f;
        [[maybe_unused]] double base_far = 0.0;
        if constexpr (!TABLE) {
            for (int c = la; c < nw; c += GA)
                if constexpr (FAR) {
#pragma unroll
                    for (int i = 0; i < FPW / KEEP; ++i) base_far += mx[i * nwq + c];
                } else {
#pragma unroll
                    for (int i = 0; i < FPW / 4; ++i) { const float4 u = m4[i * nwq + c]; base += (u.x + u.y) + (u.z + u.w); }
                }
        }
        // the two dots of a row from the parts of its lanes: a residual each in its lanes 0 and 1
        auto finish_row = [&](int r, float label, float a1, float a2) {
            if (a.a_shift > 0) {
                const bool odd = lane & 1;
                double d = (double)(odd ? a2 : a1) + (double)__shfl_xor_sync(0xffffffffu, odd ? a1 : a2, 1);
                if constexpr (FAR) d += base_far + __shfl_xor_sync(0xffffffffu, base_far, 1);
#pragma unroll
                for (int o = 2; o < 32; o <<= 1)
                    if (o < GA) d += __shfl_xor_sync(0xffffffffu, d, o);
                if (la < 2 && r < rows) res[2 * r + la] = (float)(d - (double)label);
            } else if (r < rows) {
                const double rest = base_far - (double)label;
                *reinterpret_cast<float2*>(res + 2 * r) = make_float2((float)((double)a1 + rest), (float)((double)a2 + rest));
            }
        };
        const int row_turns = (rows + row_stride - 1) >> stride_shift;
        if (single) {
            float w[FPW];
            solo_quads<FPW>(w, w4, nwq, 0);
            if constexpr (!TABLE && !kKept) solo_quads<FPW>(bias_a, c4, nwq, min(la, nw - 1));
#pragma unroll 2
            for (int turn = 0; turn < row_turns; ++turn) {
                const int r = row_first + turn * row_stride, rr = min(r, rows - 1);     // (every lane takes part in the butterfly)
                const float label = labels[rr];
                float a1 = base, a2 = base;
                if (la < nw) add_word(rr * a.pitch + la, la, w, bias_a, a1, a2);
                finish_row(r, label, a1, a2);
            }
        } else {
#pragma unroll 1
            for (int turn = 0; turn < row_turns; ++turn) {
                const int r = row_first + turn * row_stride, rr = min(r, rows - 1);
                const float label = labels[rr];
                float a1 = base, a2 = base;
#pragma unroll 2
                for (int c = la; c < nw; c += GA) {
                    float w[FPW], bias[FPW];
                    solo_quads<FPW>(w, w4, nwq, c);
                    if constexpr (!TABLE) solo_quads<FPW>(bias, c4, nwq, c);
                    add_word(rr * a.pitch + c, c, w, bias, a1, a2);
                }
                finish_row(r, label, a1, a2);
            }
        }
        uint32_t u_g[KEEP], u_x[KEEP];
        if (a.grad_bits > 0) draws(it, 4u, u_g);
        if (a.model_bits > 0) draws(it + 1, 3u, u_x);
        if constexpr (!TABLE && !kKept) solo_quads<FPW>(bias_b, c4, nwq, q);
        bar();

        // ---------------------------------------------------------------- gradient and update
        float acc[FPW];
        std::conditional_t<FAR, double, float> sum = 0;
#pragma unroll
        for (int i = 0; i < FPW; ++i) acc[i] = 0.0f;
#pragma unroll 2
        for (int r = lb; r < rows; r += GB) {
            const uint32_t u1 = t1[r * a.pitch + q], u2 = t2[r * a.pitch + q];
            const float2 rv = *reinterpret_cast<const float2*>(res + 2 * r);
            if constexpr (!TABLE) {
                float c1[FPW], c2[FPW];
                unpack_centred<CB>(u1, bias_b, c1);
                unpack_centred<CB>(u2, bias_b, c2);
                sum += rv.x + rv.y;
#pragma unroll
                for (int i = 0; i < FPW; ++i) acc[i] = fmaf(c1[i], rv.y, fmaf(c2[i], rv.x, acc[i]));
            } else {
#pragma unroll
                for (int i = 0; i < FPW; ++i)
                    acc[i] = fmaf(lev[(code_at<CB>(u1, i) * FPW + i) * nwq + q], rv.y,
                                  fmaf(lev[(code_at<CB>(u2, i) * FPW + i) * nwq + q], rv.x, acc[i]));
            }
        }
        // halving butterfly: step s leaves a lane with the upper or lower half of its features by bit s of its index
#pragma unroll
        for (int s = 0; s < 5; ++s) {
            if (s < a.b_shift) {
                const int o = 1 << s;
                if constexpr (!TABLE) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                if (s < LOGF) {
                    const int half = FPW >> (s + 1);
                    const bool up = lane & o;
#pragma unroll
                    for (int i = 0; i < FPW / 2; ++i)
                        if (i < half) acc[i] = (up ? acc[i + half] : acc[i]) + __shfl_xor_sync(0xffffffffu, up ? acc[i] : acc[i + half], o);
                } else {
                    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
                }
            }
        }
        const float scale = rows == a.rc ? full_scale : 1.0f / (2.0f * (float)rows);
        float g[KEEP];
#pragma unroll
        for (int k = 0; k < KEEP; ++k) {
            if constexpr (!TABLE) g[k] = fmaf(st[k], acc[k], FAR ? (float)(mid[k] * sum) : (float)mid[k] * (float)sum) * scale;
            else g[k] = acc[k] * scale;
        }
        if (last && a.grad_out && owner)
#pragma unroll
            for (int k = 0; k < KEEP; ++k)
                if (f0 + k < n) a.grad_out[f0 + k] = g[k];
        if (a.grad_bits > 0) {
            const float M = norm(g, 0);
#pragma unroll
            for (int k = 0; k < KEEP; ++k) g[k] = solo_quantize(g[k], M, a.grad_bits, u_g[k]);
        }
        if (last && a.grad_out && owner)
#pragma unroll
            for (int k = 0; k < KEEP; ++k)
                if (f0 + k < n) a.grad_out[n + f0 + k] = g[k];
#pragma unroll
        for (int k = 0; k < KEEP; ++k) {
            const float y = fmaf(-a.lr, g[k], x[k]);
            x[k] = a.reg == ZIPML_REG_NONE ? y : regularise(y, x[k], a.reg, a.reg_cst);
        }
        if (a.model_bits > 0) {
            const float M = norm(x, 1);
            float v[KEEP];
#pragma unroll
            for (int k = 0; k < KEEP; ++k) v[k] = solo_quantize(x[k], M, a.model_bits, u_x[k]);
            publish(far, v, left == 2);
        } else {
            publish(far, x, left == 2);
        }
        bar();
        if (tid == 0) mbar_arrive(sh->empty + slot);
        if (++slot == a.slots) { slot = 0; parity ^= 1u; }
    }
    };
    bool far = false;
    if constexpr (!TABLE) {
        if (far_lane) sh->far = 1;
        bar();
        far = *reinterpret_cast<volatile int*>(&sh->far) != 0;
    }
    if (far) run(std::integral_constant<bool, !TABLE>{});
    else run(std::false_type{});
    if (owner)
#pragma unroll
        for (int k = 0; k < KEEP; ++k)
            if (f0 + k < n) a.x[f0 + k] = x[k];
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
struct SoloPlan {
    int threads, keep, a_shift, b_shift, copy_shift, pitch, slots;
    size_t smem;
    double cycles;               // estimate of a step
};

static size_t solo_smem_bytes(int cb, bool table, int bits, int words, int rc, int pitch, int slots) {
    const size_t F = (size_t)((words + 7) & ~7) * (32 / cb);
    return kSoloSharedBytes + sizeof(float) * (F * (table ? 1 + ((size_t)1 << bits) : 4) + (size_t)((2 * rc + 3) & ~3) +
                                               (size_t)slots * (2 * (size_t)rc * pitch + (size_t)((rc + 3) & ~3)));
}

// The fullest bank's share of a warp's 32 loads: 32 / run rows of `run` consecutive words each, rows pitch = 4 u words
// apart, by [u % 8][log2 run].  (A table because a plan is made on every call: counted out there it cost 10 us of host time.)
struct BankTable {
    int degree[8][6];
    constexpr BankTable() : degree() {
        for (int u = 0; u < 8; ++u)
            for (int s = 0; s <= 5; ++s) {
                int load[32] = {0}, worst = 0;
                for (int l = 0; l < 32; ++l) {
                    const int bank = ((l >> s) * 4 * u + (l & ((1 << s) - 1))) & 31;
                    ++load[bank];
                    if (load[bank] > worst) worst = load[bank];
                }
                degree[u][s] = worst;
            }
    }
};
static constexpr BankTable kBanks;

template <int CB, bool TABLE>
static const void* solo_kernel(int keep) {
    return keep == 1 ? (const void*)sgd_solo_kernel<CB, TABLE, 1> : keep == 2 ? (const void*)sgd_solo_kernel<CB, TABLE, 2> : (const void*)sgd_solo_kernel<CB, TABLE, 4>;
}

// Threads, lane splits and pitch by a count of what a step issues and waits for (cycles; four schedulers that take an
// instruction of a lone warp every other cycle, a shared memory pipe of one wavefront a cycle, butterflies of 28
// cycles a stage).
static int make_solo_plan(const zipml_ctx* ctx, const zipml_dataset* d, const zipml_sgd_params* p, SoloPlan* best) {
    const int cb = container_bits(d->bits), fpw = 32 / cb, logf = cb == 8 ? 2 : cb == 4 ? 3 : 4;
    const bool table = d->level_mode == ZIPML_LEVELS_TABLE;
    const int64_t B64 = p->batch < d->m ? p->batch : d->m;
    if (B64 > 4096 || d->n > 4 * kSoloMaxThreads || d->row_bytes > 8192 || B64 * d->row_bytes > 48 * 1024) return ZIPML_ERR_WORKSPACE;
    const int B = (int)B64, row_words = (int)(d->row_bytes / 4), nw = (int)((d->n + fpw - 1) / fpw);
    const double unit = (table ? 7.0 : 4.2) * fpw + 6;              // instructions per word of both planes
    best->threads = 0;
    for (const int pad : {0, 4, 8, 16}) {
        const int pitch = row_words + pad;
        // two tiles at least; one where the tallest tiles of the narrowest rows leave no more (they fit beside half the quad arrays)
        int slots = kSoloMaxSlots;
        while (slots >= 1 && solo_smem_bytes(cb, table, d->bits, nw, B, pitch, slots) > (size_t)ctx->smem_optin) --slots;
        if (slots < 2 && (pad > 0 || table || solo_smem_bytes(cb, table, d->bits, nw, B, pitch, 2) - 8 * (size_t)((nw + 7) & ~7) * fpw > (size_t)ctx->smem_optin)) break;
        for (int threads = 32; threads <= kSoloMaxThreads; threads *= 2) {
            const int warps = threads / 32;
            const double issue = warps <= 4 ? 2.0 : warps == 8 ? 2.4 : 4.0;    // cycles per instruction of a warp
            double best_a = 1e30, best_b = 1e30;
            int sa = 0, sb = -1;
            for (int s = 0; s <= 5; ++s) {
                const int g = 1 << s;
                if (threads / g >= 1) {
                    const int turns = (B + threads / g - 1) / (threads / g), per = (nw + g - 1) / g;
                    const double instr = turns * (per * unit + (nw > g ? per * fpw * 0.5 : 0) + 5.0 * s + 14) + (table ? 0 : per * fpw * 1.5);
                    const double lds = (double)turns * per * warps * (2.0 * kBanks.degree[(pitch / 4) % 8][s] + (table ? 2.0 * fpw * 2 : fpw / 4));
                    const double c = (instr * issue > lds ? instr * issue : lds) + 28.0 * s + 80;
                    if (c < best_a) { best_a = c; sa = s; }
                }
                // a word column's lanes: enough threads for all columns at once, at most four features left to a lane
                if (nw * g <= threads && (fpw >> (s < logf ? s : logf)) <= 4) {
                    const int per = (B + g - 1) / g, kept = fpw >> (s < logf ? s : logf);
                    const double instr = per * (unit + 4) + 3.0 * (fpw - kept) + 4.0 * s + kept * 12 + 20;
                    const double lds = (double)per * warps * (2.0 * kBanks.degree[(pitch / 4) % 8][5 - s] + 2 + (table ? 2.0 * fpw * 2 : 0));
                    const double c = (instr * issue > lds ? instr * issue : lds) + 28.0 * s + 100;
                    if (c < best_b) { best_b = c; sb = s; }
                }
            }
            if (sb < 0) continue;
            const double cycles = best_a + best_b + 2 * (25 + 2.0 * warps);
            if (!best->threads || cycles < best->cycles) {
                best->threads = threads; best->a_shift = sa; best->b_shift = sb; best->pitch = pitch; best->slots = slots; best->cycles = cycles;
                best->keep = fpw >> (sb < logf ? sb : logf);
            }
        }
    }
    if (!best->threads) return ZIPML_ERR_WORKSPACE;
    best->copy_shift = 0;
    while ((1 << best->copy_shift) < row_words / 4 && best->copy_shift < 5) ++best->copy_shift;
    best->smem = solo_smem_bytes(cb, table, d->bits, nw, B, best->pitch, best->slots);
    return ZIPML_OK;
}

// Whether AUTO takes this engine: by what a step has one SM get through, batch x (features + 8).  Measured, us per step here / cluster
// engine, on both sides of the lines: 8 bits 512 x 16 1.94 / 2.28, 64 x 128 2.0 / 2.4, 333 x 32 3.9 / 2.6, 700 x 16 3.1 / 2.3; 4 bits 64 x 128
// 1.9 / 2.4, 333 x 32 2.6 / 2.6, 200 x 64 2.7 / 2.5; 2 bits 333 x 32 2.5 / 2.6, 120 x 128 2.8 / 2.6; tables (3 bits) 120 x 16 1.6 / 2.0, 250
// x 16 2.1 / 2.0, (2 bits) 64 x 64 2.3 / 2.6, 400 x 16 2.8 / 2.2.  A quantized model or gradient costs the others an exchange more each: 8 bits
// 512 x 32 4.8 / 5.1, 333 x 64 7.7 / 5.5, 4 bits 64 x 256 4.4 / 5.0, 333 x 64 6.5 / 5.5, 700 x 16 5.8 / 5.2, tables 250 x 16 4.0 / 5.0, 250 x 64
// 7.2 / 5.2.
static bool solo_pays(const zipml_dataset* d, const zipml_sgd_params* p) {
    const int64_t B = p->batch < d->m ? p->batch : d->m, work = B * (d->n + 8);
    const int cb = container_bits(d->bits);
    const bool quantized = p->model_bits > 0 || p->grad_bits > 0;
    if (d->level_mode == ZIPML_LEVELS_TABLE) return work <= (quantized ? 8000 : cb == 2 ? 5000 : 4000);
    if (quantized) return d->n <= 640 && work <= (cb == 8 ? 17000 : 18500);
    return d->n <= 1024 && work <= (cb == 8 ? 9500 : 11000);
}

int launch_sgd_solo(zipml_ctx* ctx, const zipml_dataset* d, const float* b, float* x, const zipml_sgd_params* p,
                    int64_t first_step, int64_t num_steps, float* grad_out, bool only_if_profitable) {
    const int cb = container_bits(d->bits);
    const bool table = d->level_mode == ZIPML_LEVELS_TABLE;
    if (only_if_profitable && !solo_pays(d, p)) return ZIPML_ERR_WORKSPACE;
    SoloPlan plan;
    int rc = make_solo_plan(ctx, d, p, &plan);
    if (rc != ZIPML_OK) return rc;
    const void* kernel = cb == 2 ? (table ? solo_kernel<2, true>(plan.keep) : solo_kernel<2, false>(plan.keep))
                       : cb == 4 ? (table ? solo_kernel<4, true>(plan.keep) : solo_kernel<4, false>(plan.keep))
                                 : solo_kernel<8, false>(plan.keep);
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plan.smem);
    if (e != cudaSuccess) return cuda_status(e);
    const int64_t T = (d->m + p->batch - 1) / p->batch;
    SoloArgs a;
    memset(&a, 0, sizeof(a));
    if (p->batch_order) {
        rc = ws_reserve(ctx, carve_size(sizeof(int32_t) * (size_t)T));
        if (rc != ZIPML_OK) return rc;
        e = cudaMemcpyAsync(ctx->ws, p->batch_order, sizeof(int32_t) * (size_t)T, cudaMemcpyHostToDevice, ctx->stream);
        if (e != cudaSuccess) return cuda_status(e);
        a.order = reinterpret_cast<const int32_t*>(ctx->ws);
    }
    a.p1 = reinterpret_cast<const uint32_t*>(d->plane1);
    a.p2 = reinterpret_cast<const uint32_t*>(d->plane2);
    a.lo = d->feat_lo; a.step = d->feat_step; a.levels = d->levels;
    a.b = b; a.x = x; a.grad_out = grad_out; a.model_out = p->model_out;
    a.status = ctx->d_status;
    a.m = d->m; a.batch = p->batch < d->m ? p->batch : d->m;
    a.first_step = first_step; a.num_steps = num_steps;
    a.seed = p->seed; a.epoch = (uint32_t)p->epoch; a.lr = p->lr; a.reg = p->reg; a.reg_cst = reg_constant(p);
    a.n = (int)d->n; a.bits = d->bits; a.row_words = (int)(d->row_bytes / 4);
    a.words = (int)((d->n + 32 / cb - 1) / (32 / cb));
    a.model_bits = p->model_bits; a.grad_bits = p->grad_bits;
    a.rc = (int)a.batch; a.pitch = plan.pitch; a.slots = plan.slots;
    a.a_shift = plan.a_shift; a.b_shift = plan.b_shift; a.copy_shift = plan.copy_shift;
    void* params[] = {&a};
    e = cudaLaunchKernel(kernel, dim3(1), dim3((unsigned)plan.threads + 32u), params, plan.smem, ctx->stream);
    if (e != cudaSuccess) return cuda_status(e);
    ctx->launches += 1;
    ctx->ran(ZIPML_ENGINE_SOLO, "sgd_solo_kernel");
    return ZIPML_OK;
}

}  // namespace zipml
