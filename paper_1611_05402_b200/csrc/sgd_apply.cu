// zipml_sgd_apply_gradient: the owner stage of a step on its own -- Q4 of a gradient that the caller holds (paper
// "End-to-end Quantization": g -> Q4(g), the l2-scaled sign-magnitude quantizer of Supplement Eq. (quant2)) and the
// update x <- R(x - lr * Q4(g)) (Eq. (proxupdate); LS-SVM term of the Supplement) -- for callers that form the
// gradient of a minibatch from several devices' rows: every device applies the same sum with the same random draws
// (keyed by seed, epoch, step and coordinate), so the replicas of x stay identical.
#include <cstring>

#include "cluster.cuh"

namespace zipml {

constexpr int kApplyThreads = 1024;
constexpr int kApplyCtas = 8;

struct ApplyArgs {
    float* x;
    const float* g;
    float* applied_out;          // null or n
    int64_t n;
    float lr;
    int grad_bits, vector_norm, reg;
    float reg_cst;
    uint64_t seed;
    uint32_t epoch, step;
    int ctas, warps;             // of the cluster; of a CTA
    int wide;                    // all three on 16 bytes
};

// Four coordinates from j, zeros past n.
__device__ __forceinline__ float4 apply_read(const float* v, int64_t j, const ApplyArgs& a) {
    if (a.wide && j + 4 <= a.n) return *reinterpret_cast<const float4*>(v + j);
    return make_float4(j < a.n ? v[j] : 0.0f, j + 1 < a.n ? v[j + 1] : 0.0f, j + 2 < a.n ? v[j + 2] : 0.0f, j + 3 < a.n ? v[j + 3] : 0.0f);
}
__device__ __forceinline__ void apply_write(float* v, int64_t j, float4 y, const ApplyArgs& a) {
    if (a.wide && j + 4 <= a.n) {
        *reinterpret_cast<float4*>(v + j) = y;
        return;
    }
    if (j < a.n) v[j] = y.x;
    if (j + 1 < a.n) v[j + 1] = y.y;
    if (j + 2 < a.n) v[j + 2] = y.z;
    if (j + 3 < a.n) v[j + 3] = y.w;
}
__device__ __forceinline__ double apply_norm(double acc, float4 g, bool linf) {
    if (linf) return fmax(fmax(fmax(acc, (double)fabsf(g.x)), (double)fabsf(g.y)), fmax((double)fabsf(g.z), (double)fabsf(g.w)));
    return acc + (((double)g.x * (double)g.x + (double)g.y * (double)g.y) + ((double)g.z * (double)g.z + (double)g.w * (double)g.w));
}
__device__ __forceinline__ double apply_lanes(double v, bool linf) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double other = __shfl_xor_sync(0xffffffffu, v, o);
        v = linf ? fmax(v, other) : v + other;
    }
    return v;
}

// One cluster: the norm of g in a fixed order (double), then every coordinate.  The payload is n floats once per step beside a collective:
// latency, not bandwidth, is what it costs.  A thread keeps four neighbouring coordinates -- one generator call draws for all four, before g is
// looked at -- and the warps' parts of the norm go to every CTA, whose warps all add them up by shuffles: one barrier.
__global__ void __launch_bounds__(kApplyThreads) sgd_apply_kernel(const ApplyArgs a) {
    __shared__ double parts[kApplyCtas * 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool linf = a.vector_norm == ZIPML_NORM_LINF;
    const int64_t j0 = 4 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x), stride = 4 * (int64_t)gridDim.x * blockDim.x;
    if (a.ctas > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    VecQuant q4{0.0f, 1, a.seed, a.epoch, a.step, 4u};
    auto draws = [&](int64_t j) { return philox4x32_10((uint32_t)j >> 2, a.step, a.epoch, 4u, (uint32_t)a.seed, (uint32_t)(a.seed >> 32)); };
    Philox4 u = {};
    if (a.grad_bits > 0) u = draws(j0);
    after_previous_kernel(1);
    const float4 g0 = apply_read(a.g, j0, a), x0 = apply_read(a.x, j0, a);
    if (a.ctas > 1) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");          // (every CTA has started)
    if (a.grad_bits > 0) {
        double acc = apply_norm(0.0, g0, linf);
        for (int64_t j = j0 + stride; j < a.n; j += stride) acc = apply_norm(acc, apply_read(a.g, j, a), linf);
        acc = apply_lanes(acc, linf);
        if (a.ctas > 1) {
            if (lane < a.ctas) {
                const uint32_t dst = slice_peer(parts + blockIdx.x * a.warps + warp, lane);
                asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(dst), "d"(acc) : "memory");
            }
            slice_cluster_sync();
        } else {
            if (lane == 0) parts[warp] = acc;
            __syncthreads();
        }
        double all = 0.0;
        for (int k = lane; k < a.ctas * a.warps; k += 32) all = linf ? fmax(all, parts[k]) : all + parts[k];
        all = apply_lanes(all, linf);
        q4.M = linf ? (float)all : (float)sqrt(all);
        q4.sm = (1 << (a.grad_bits - 1)) - 1;
    }
    auto finish = [&](int64_t j, float4 g, float4 x, const Philox4& d) {
        if (a.grad_bits > 0)
            g = make_float4(q4.apply_drawn(g.x, d.v[0] >> 8), q4.apply_drawn(g.y, d.v[1] >> 8), q4.apply_drawn(g.z, d.v[2] >> 8), q4.apply_drawn(g.w, d.v[3] >> 8));
        if (a.applied_out) apply_write(a.applied_out, j, g, a);
        apply_write(a.x, j,
                    make_float4(regularise(fmaf(-a.lr, g.x, x.x), x.x, a.reg, a.reg_cst), regularise(fmaf(-a.lr, g.y, x.y), x.y, a.reg, a.reg_cst),
                                regularise(fmaf(-a.lr, g.z, x.z), x.z, a.reg, a.reg_cst), regularise(fmaf(-a.lr, g.w, x.w), x.w, a.reg, a.reg_cst)), a);
    };
    finish(j0, g0, x0, u);
    for (int64_t j = j0 + stride; j < a.n; j += stride) {
        const float4 g = apply_read(a.g, j, a), x = apply_read(a.x, j, a);
        if (a.grad_bits > 0) u = draws(j);
        finish(j, g, x, u);
    }
}

int launch_sgd_apply(zipml_ctx* ctx, float* x, const float* g, int64_t n, const zipml_sgd_params* p, int64_t step,
                     float* applied_out) {
    ApplyArgs a = {x, g, applied_out, n, p->lr, p->grad_bits, p->vector_norm, p->reg, reg_constant(p), p->seed, (uint32_t)p->epoch, (uint32_t)step, 1, 1, 0};
    a.wide = ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(g) | reinterpret_cast<uintptr_t>(applied_out)) & 15) == 0;
    // One CTA up to 2,048 coordinates (512 threads), then another for each 2,048 up to a cluster of eight.  us a call, calls back to back (some 6 of
    // it the host's), one block of 1,024 threads a coordinate at a time -> one CTA / this: n 1,000 5.3 -> 4.6, 4,096 8.3 -> 6.2 / 6.2, 6,000 10.3 -> 8.2 / 6.2,
    // 16,384 20.6 -> 14.4 / 6.2, 32,768 39.0 -> 22.6 / 6.6, 100,000 115 -> 60 / 14.4.
    const int64_t quads = (n + 3) / 4, ctas = (n + 2047) / 2048;
    a.ctas = (int)(ctas < kApplyCtas ? ctas : kApplyCtas);
    const int64_t warps = (quads + 32 * a.ctas - 1) / (32 * a.ctas);
    a.warps = (int)(warps < 32 ? warps : 32);
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)a.ctas);
    cfg.blockDim = dim3(32u * (unsigned)a.warps);
    cfg.stream = ctx->stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)a.ctas;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (early_start(ctx, 1, attr + 1)) cfg.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, sgd_apply_kernel, a);
    if (e != cudaSuccess) return cuda_status(e);
    ++ctx->launches;
    return ZIPML_OK;
}

}  // namespace zipml
