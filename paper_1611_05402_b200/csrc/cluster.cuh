// Pieces shared by the kernels that run as thread-block clusters (sgd_slice.cu, sgd_feature.cu, sgd_table.cu): stores and copies into another CTA's
// shared memory that complete on its mbarrier, bounded waits, the vector quantizer out of line, norms over the owners, fixed point and
// codes as the int8 contractions take them, and the hand-over of sums between clusters.  A kernel's
// block of shared memory has a member `gave_up`.
#pragma once

#include "sgd_common.cuh"

namespace zipml {

constexpr int kSliceWarps = 16;
constexpr int kSliceThreads = 32 * kSliceWarps;   // without the copying warp
constexpr int kSliceMaxSlots = 8;
constexpr int kSliceMaxCtas = 16;
constexpr int kSliceMaxClusters = 8;

__device__ __forceinline__ uint32_t slice_peer(const void* local_smem, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(local_smem)), "r"(rank));
    return r;
}
__device__ __forceinline__ void slice_store16(uint32_t dst, uint4 v, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1,%2,%3,%4}, [%5];"
                 ::"r"(dst), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar) : "memory");
}
__device__ __forceinline__ void slice_store8(uint32_t dst, double v, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];"
                 ::"r"(dst), "l"(__double_as_longlong(v)), "r"(bar) : "memory");
}
__device__ __forceinline__ void slice_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "r"(smem_u32(src)), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void slice_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The compute warps; and all, the copying warp included.
__device__ __forceinline__ void slice_bar() { asm volatile("bar.sync 1, %0;" ::"n"(kSliceThreads) : "memory"); }
__device__ __forceinline__ void slice_bar_all() { asm volatile("bar.sync 3, %0;" ::"n"(kSliceThreads + 32) : "memory"); }

// Sixteen doubles in a fixed order, four chains.
__device__ __forceinline__ double slice_sum16(const double* v) {
    double s[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
    for (int i = 4; i < 16; i += 4)
#pragma unroll
        for (int j = 0; j < 4; ++j) s[j] += v[i + j];
    return (s[0] + s[1]) + (s[2] + s[3]);
}

// Bounded wait on a local phase; after the first failure of this CTA every wait is skipped.
template <class Shared>
__device__ __noinline__ void slice_wait_long(Shared* sh, uint64_t* bar, uint32_t parity, DeviceStatus* status, int where) {
#pragma unroll 1
    for (long long spin = 0; spin < kCopySpinLimit; ++spin) {
        if (mbar_try_wait(bar, parity)) return;
        if (*reinterpret_cast<volatile int*>(&sh->gave_up)) return;
    }
    sh->gave_up = 1;
    set_status(status, ZIPML_ERR_TIMEOUT, where);
}
template <class Shared>
__device__ __forceinline__ void slice_wait(Shared* sh, uint64_t* bar, uint32_t parity, DeviceStatus* status, int where) {
    if (!mbar_try_wait(bar, parity)) slice_wait_long(sh, bar, parity, status, where);
}

static __device__ __noinline__ float slice_regularise(float y, float x_old, int reg, float cst) { return regularise(y, x_old, reg, cst); }
static __device__ __noinline__ uint32_t slice_draw(uint64_t seed, uint32_t epoch, uint32_t step, uint32_t coord, uint32_t stream) {
    return vector_u24(seed, epoch, step, coord, stream);
}
// VecQuant::apply with its draw given.
static __device__ __noinline__ float slice_quantize(float v, float M, int bits, uint32_t u24) {
    if (!(M > 0.0f)) return 0.0f;
    const float sm = (float)((1 << (bits - 1)) - 1);
    const float t = __fmul_rn(__fdiv_rn(fabsf(v), M), sm);
    float fl = floorf(t);
    fl = fl > sm - 1.0f ? sm - 1.0f : fl;
    const float p = __fsub_rn(t, fl);
    const float mag = fl + ((__fmul_rn((float)u24, 5.9604644775390625e-08f) < p) ? 1.0f : 0.0f);
    const float q = __fmul_rn(M, __fdiv_rn(mag, sm));
    return v < 0.0f ? -q : q;
}

// l2 norm of a vector spread over the owners (v: this thread's share of the squares, in every `every`-th lane): per-CTA sums, one store to
// every owner, added in CTA order.
template <class Shared>
__device__ __noinline__ float slice_norm(double v, int every, int rank, double* red, double* table, uint64_t* bar, uint32_t parity, int owners, Shared* sh,
                                         DeviceStatus* status, int where) {
#pragma unroll 1
    for (int o = 16; o >= every; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    slice_bar();
    if ((int)threadIdx.x < owners) {
        slice_store8(slice_peer(table + rank, threadIdx.x), slice_sum16(red), slice_peer(bar, threadIdx.x));
    }
    slice_wait(sh, bar, parity, status, where);
    if (threadIdx.x == 0) mbar_arrive_expect_tx(bar, 8u * (uint32_t)owners);     // the next one's
    return (float)sqrt(slice_sum16(table));          // (entries past the owners stay zero)
}

static __device__ __noinline__ void slice_mark(unsigned long long* trace, int step, int id) {
    unsigned long long t;
    asm volatile("mov.u64 %0, %clock64;" : "=l"(t));
    trace[step * 8 + id] = t;
}

__device__ __forceinline__ void slice_tensor_copy(void* dst_smem, const CUtensorMap* tm, int x, int y, uint64_t* bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(smem_u32(dst_smem)), "l"(tm), "r"(x), "r"(y), "r"(smem_u32(bar)) : "memory");
}

// Power of two 2^k by which values up to `top` become integers within the range of four balanced base-256 digits
// (2^31 - 2^31/128), `spare` bits kept back.  top = 0: 0.
__device__ __forceinline__ int slice_exponent(float top, int spare) {
    const int e = (int)(__float_as_uint(top * 1.01f) >> 23) - 127;
    return min(126, 30 - spare - e);
}
__device__ __forceinline__ float slice_pow2(int k) { return k >= -126 ? __uint_as_float((uint32_t)(k + 127) << 23) : 0.0f; }
// Codes of group g of a fragment register, where they lie in their bytes ...
template <int CB>
__device__ __forceinline__ uint32_t slice_codes(uint32_t u, int g) {
    if constexpr (CB == 8) return u;
    else return u & ((CB == 4 ? 0x0F0F0F0Fu : 0x03030303u) << (CB * g));
}
// ... and, for the dots, at most 4 bits up (2-bit codes: the upper pair is shifted down first).
template <int CB>
__device__ __forceinline__ uint32_t slice_dot_codes(uint32_t u, int g) {
    if constexpr (CB == 2) return slice_codes<2>(g & 2 ? u >> 4 : u, g & 1);
    else return slice_codes<CB>(u, g);
}
template <int CB>
struct SliceShift {                                       // bits that a group's digits are shifted up by, against the lowest group
    static constexpr int kMost = CB == 8 ? 0 : CB == 4 ? 4 : 2;
    __device__ static constexpr int of(int g) { return CB == 8 ? 0 : CB == 4 ? (g == 0 ? 4 : 0) : (g & 1 ? 0 : 2); }
};
// low + 65536 high: the integer's bits behind those of 1.5 x 2^52 (conversions to double run at a sixteenth of the FMA rate).
__device__ __forceinline__ double slice_double(int low, int high) {
    return __longlong_as_double(low + 65536ll * high + 0x4338000000000000ll) - 6755399441055744.0;
}
// D = A B + C with C's two columns given.
__device__ __forceinline__ void slice_mma_from(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1, int c0, int c1) {
    asm("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%10,%11};"
        : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "r"(c0), "r"(c1));
}

// A double, as the sum of two floats, handed over through L2: each 8-byte word carries the step's tag and is valid by itself.
__device__ __forceinline__ void slice_post(unsigned long long* box, float hi, float low, uint32_t tag) {
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(box), "l"(t | __float_as_uint(hi)), "l"(t | __float_as_uint(low)) : "memory");
}
template <class Shared>
__device__ __noinline__ double slice_collect(Shared* sh, const unsigned long long* box, uint32_t tag, DeviceStatus* status) {
    unsigned long long u, v;
#pragma unroll 1
    for (long long spin = 0; spin < kBarrierSpinLimit; ++spin) {
        asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(u), "=l"(v) : "l"(box) : "memory");
        if ((uint32_t)(u >> 32) == tag && (uint32_t)(v >> 32) == tag) return (double)__uint_as_float((uint32_t)u) + (double)__uint_as_float((uint32_t)v);
        if ((spin & 255) == 255 && *reinterpret_cast<volatile int*>(&sh->gave_up)) return 0.0;
    }
    sh->gave_up = 1;
    set_status(status, ZIPML_ERR_TIMEOUT, 85);
    return 0.0;
}

}  // namespace zipml
