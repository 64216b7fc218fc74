// C-ABI entry points: argument validation, workspace management and the order of kernel launches.
#include <new>

#include "common.cuh"
#include "internal.h"

namespace zipml {

int cuda_status(cudaError_t e) {
    if (e == cudaSuccess) return ZIPML_OK;
    (void)cudaGetLastError();
    return ZIPML_ERR_CUDA;
}

static int grow(unsigned char** buf, size_t* have, size_t want, cudaStream_t stream) {
    if (want <= *have) return ZIPML_OK;
    // earlier work on the stream may still use the old buffer
    cudaError_t e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) return cuda_status(e);
    if (*buf) { e = cudaFree(*buf); *buf = nullptr; *have = 0; if (e != cudaSuccess) return cuda_status(e); }
    const size_t bytes = (want + (1u << 20) - 1) >> 20 << 20;
    e = cudaMalloc(reinterpret_cast<void**>(buf), bytes);
    if (e != cudaSuccess) { *buf = nullptr; return cuda_status(e); }
    *have = bytes;
    return ZIPML_OK;
}

int ws_reserve(zipml_ctx* ctx, size_t bytes) { return grow(&ctx->ws, &ctx->ws_bytes, bytes, ctx->stream); }
int stage_reserve(zipml_ctx* ctx, size_t bytes) { return grow(&ctx->stage, &ctx->stage_bytes, bytes, ctx->stream); }

bool early_start(zipml_ctx* ctx, int64_t steps, cudaLaunchAttribute* attr) {
    if (steps > kEarlySteps) return false;
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(ctx->stream, &capture) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    attr->id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr->val.programmaticStreamSerializationAllowed = 1;
    return capture == cudaStreamCaptureStatusNone;
}

int exchange_tags(zipml_ctx* ctx, size_t bytes, int64_t steps, unsigned long long** buffer, uint32_t* tag) {
    if (bytes > kExchangeBytes) return ZIPML_ERR_WORKSPACE;
    // Tags go up from launch to launch, so the buffer is cleared only before they would wrap.  A launch that is recorded into a
    // graph keeps its tags from replay to replay: there the clearing is recorded with it.
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(ctx->stream, &capture) != cudaSuccess) (void)cudaGetLastError();
    const bool recorded = capture != cudaStreamCaptureStatusNone, wraps = ctx->exchange_tag > 0xffffffffu - (uint32_t)steps - 1u;
    if (recorded || wraps) {
        const cudaError_t e = cudaMemsetAsync(ctx->exchange, 0, kExchangeBytes, ctx->stream);
        if (e != cudaSuccess) return cuda_status(e);
    }
    *buffer = reinterpret_cast<unsigned long long*>(ctx->exchange);
    *tag = wraps ? 1u : ctx->exchange_tag;
    // (a recorded clearing has not happened yet: the next launch that runs at once clears too)
    ctx->exchange_tag = recorded && wraps ? 0xffffffffu : *tag + (uint32_t)steps;
    return ZIPML_OK;
}

static bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

struct DeviceGuard {
    int prev = -1;
    bool ok = false;
    explicit DeviceGuard(int device) {
        if (cudaGetDevice(&prev) != cudaSuccess) { (void)cudaGetLastError(); prev = -1; }
        ok = cudaSetDevice(device) == cudaSuccess;
        if (!ok) (void)cudaGetLastError();
    }
    ~DeviceGuard() { if (prev >= 0) (void)cudaSetDevice(prev); }
};

int check_dataset(const zipml_dataset* d) {
    if (!d || d->struct_size != sizeof(zipml_dataset)) return ZIPML_ERR_INVALID_ARG;
    const int cb = container_bits(d->bits);
    if (cb == 0) return ZIPML_ERR_UNSUPPORTED;
    if (d->level_mode != ZIPML_LEVELS_UNIFORM && d->level_mode != ZIPML_LEVELS_TABLE) return ZIPML_ERR_INVALID_ARG;
    if (d->layout != ZIPML_LAYOUT_ROWS && d->layout != ZIPML_LAYOUT_COLUMN_BLOCKS) return ZIPML_ERR_INVALID_ARG;
    if (d->level_mode == ZIPML_LEVELS_TABLE && d->bits > 4) return ZIPML_ERR_UNSUPPORTED;
    if (d->m <= 0 || d->n <= 0) return ZIPML_ERR_INVALID_ARG;
    if (d->n > 0x7fffffffLL / 8) return ZIPML_ERR_WORKSPACE;
    if (!d->plane1 || !d->plane2 || !aligned16(d->plane1) || !aligned16(d->plane2)) return ZIPML_ERR_INVALID_ARG;
    if (d->row_bytes % 16 != 0 || d->row_bytes < zipml_row_bytes(d->n, d->bits)) return ZIPML_ERR_INVALID_ARG;
    if (d->level_mode == ZIPML_LEVELS_UNIFORM && (!d->feat_lo || !d->feat_step)) return ZIPML_ERR_INVALID_ARG;
    if (d->level_mode == ZIPML_LEVELS_TABLE && !d->levels) return ZIPML_ERR_INVALID_ARG;
    return ZIPML_OK;
}

constexpr int kLossPartials = 4096;

}  // namespace zipml

using namespace zipml;

namespace zipml {
// A wait that cannot succeed, bounded like the engines' waits: lane 0 polls a zero flag `limit` times with an
// acquire load and a pause now and then, then records the time-out (see zipml_wait_probe).
__global__ void wait_probe_kernel(const unsigned* flag, long long limit, DeviceStatus* status) {
    if (threadIdx.x != 0) return;
    for (long long it = 0; it < limit; ++it) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
        if (v != 0) return;
        if ((it & 1023) == 1023) __nanosleep(200);
    }
    set_status(status, ZIPML_ERR_TIMEOUT, 90);
}
}  // namespace zipml

extern "C" {

const char* zipml_strerror(int status) {
    switch (status) {
        case ZIPML_OK: return "ok";
        case ZIPML_ERR_INVALID_ARG: return "invalid argument";
        case ZIPML_ERR_UNSUPPORTED: return "unsupported configuration";
        case ZIPML_ERR_NONFINITE: return "non-finite value in the input";
        case ZIPML_ERR_CUDA: return "CUDA runtime error (no device, out of memory or failed launch)";
        case ZIPML_ERR_TIMEOUT: return "a device-side wait gave up";
        case ZIPML_ERR_WORKSPACE: return "problem does not fit the kernels' shared memory or scratch limits";
        default: return "unknown status";
    }
}

int64_t zipml_column_blocks_bytes(int64_t m, int64_t row_bytes) {
    if (m <= 0 || row_bytes <= 0) return 0;
    return (row_bytes + 127) / 128 * m * 128;
}

int zipml_convert_layout(zipml_ctx* ctx, const zipml_dataset* data, int32_t to_layout, uint8_t* out1, uint8_t* out2) {
    if (!ctx) return ZIPML_ERR_INVALID_ARG;
    int rc = check_dataset(data);
    if (rc != ZIPML_OK) return rc;
    if (to_layout != ZIPML_LAYOUT_ROWS && to_layout != ZIPML_LAYOUT_COLUMN_BLOCKS) return ZIPML_ERR_INVALID_ARG;
    if (to_layout == data->layout) return ZIPML_ERR_INVALID_ARG;
    if (!out1 || !out2 || !aligned16(out1) || !aligned16(out2)) return ZIPML_ERR_INVALID_ARG;
    if (out1 == data->plane1 || out1 == data->plane2 || out2 == data->plane1 || out2 == data->plane2 || out1 == out2)
        return ZIPML_ERR_INVALID_ARG;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return ZIPML_ERR_CUDA;
    return launch_convert_layout(ctx, data, to_layout, out1, out2);
}

int64_t zipml_row_bytes(int64_t n, int32_t bits) {
    const int cb = container_bits(bits);
    if (cb == 0 || n <= 0) return 0;
    return ((n * cb + 7) / 8 + 15) / 16 * 16;
}

int zipml_create(zipml_ctx** ctx_out, int device, void* cuda_stream) {
    if (!ctx_out) return ZIPML_ERR_INVALID_ARG;
    *ctx_out = nullptr;
    int count = 0;
    if (cudaGetDeviceCount(&count) != cudaSuccess || device < 0 || device >= count) {
        (void)cudaGetLastError();
        return ZIPML_ERR_CUDA;
    }
    DeviceGuard guard(device);
    if (!guard.ok) return ZIPML_ERR_CUDA;
    zipml_ctx* ctx = new (std::nothrow) zipml_ctx();
    if (!ctx) return ZIPML_ERR_CUDA;
    ctx->device = device;
    ctx->stream = reinterpret_cast<cudaStream_t>(cuda_stream);
    cudaError_t e = cudaDeviceGetAttribute(&ctx->sm_count, cudaDevAttrMultiProcessorCount, device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&ctx->smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&ctx->cooperative, cudaDevAttrCooperativeLaunch, device);
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&ctx->d_status), sizeof(DeviceStatus));
    if (e == cudaSuccess) e = cudaMemsetAsync(ctx->d_status, 0, sizeof(DeviceStatus), ctx->stream);
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&ctx->exchange), kExchangeBytes);
    if (e == cudaSuccess) e = cudaMemsetAsync(ctx->exchange, 0, kExchangeBytes, ctx->stream);
    constexpr size_t kRangeBytes = sizeof(uint32_t) * (2 * kRangeColumns + kRangeTiles);
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&ctx->range_keys), kRangeBytes);
    if (e == cudaSuccess) e = cudaMemsetAsync(ctx->range_keys, 0, kRangeBytes, ctx->stream);
    if (e != cudaSuccess) {
        if (ctx->d_status) (void)cudaFree(ctx->d_status);
        if (ctx->exchange) (void)cudaFree(ctx->exchange);
        if (ctx->range_keys) (void)cudaFree(ctx->range_keys);
        delete ctx;
        return cuda_status(e);
    }
    *ctx_out = ctx;
    return ZIPML_OK;
}

int zipml_destroy(zipml_ctx* ctx) {
    if (!ctx) return ZIPML_OK;
    DeviceGuard guard(ctx->device);
    (void)cudaStreamSynchronize(ctx->stream);
    if (ctx->ws) (void)cudaFree(ctx->ws);
    if (ctx->stage) (void)cudaFree(ctx->stage);
    if (ctx->exchange) (void)cudaFree(ctx->exchange);
    if (ctx->range_keys) (void)cudaFree(ctx->range_keys);
    if (ctx->d_status) (void)cudaFree(ctx->d_status);
    (void)cudaGetLastError();
    delete ctx;
    return ZIPML_OK;
}

int64_t zipml_kernel_launches(const zipml_ctx* ctx) { return ctx ? ctx->launches : 0; }

int32_t zipml_last_engine(const zipml_ctx* ctx) { return ctx ? ctx->last_engine : 0; }

const char* zipml_last_kernel(const zipml_ctx* ctx) { return ctx ? ctx->last_kernel : ""; }

int zipml_sync(zipml_ctx* ctx) {
    if (!ctx) return ZIPML_ERR_INVALID_ARG;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return ZIPML_ERR_CUDA;
    DeviceStatus host{0, 0};
    cudaError_t e = cudaMemcpyAsync(&host, ctx->d_status, sizeof(host), cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    if (e != cudaSuccess) return cuda_status(e);
    if (host.code != 0) {
        e = cudaMemsetAsync(ctx->d_status, 0, sizeof(DeviceStatus), ctx->stream);
        if (e != cudaSuccess) return cuda_status(e);
    }
    return host.code;
}

int zipml_quantize(zipml_ctx* ctx, const float* A, int64_t m, int64_t n, int64_t lda, int32_t bits,
                   int32_t level_mode, const float* levels, uint64_t seed, uint8_t* plane1, uint8_t* plane2,
                   int64_t row_bytes, float* feat_lo, float* feat_step) {
    return zipml_quantize_draw(ctx, A, m, n, lda, bits, level_mode, levels, seed, 0u, ZIPML_GRID_RANGE, plane1, plane2, row_bytes, feat_lo,
                               feat_step);
}

int zipml_quantize_draw(zipml_ctx* ctx, const float* A, int64_t m, int64_t n, int64_t lda, int32_t bits,
                        int32_t level_mode, const float* levels, uint64_t seed, uint32_t draw, int32_t grid, uint8_t* plane1,
                        uint8_t* plane2, int64_t row_bytes, float* feat_lo, float* feat_step) {
    if (!ctx) return ZIPML_ERR_INVALID_ARG;
    if (grid != ZIPML_GRID_RANGE && grid != ZIPML_GRID_SYMMETRIC) return ZIPML_ERR_INVALID_ARG;
    if (grid == ZIPML_GRID_SYMMETRIC && level_mode != ZIPML_LEVELS_UNIFORM) return ZIPML_ERR_INVALID_ARG;
    const int cb = container_bits(bits);
    if (cb == 0) return ZIPML_ERR_UNSUPPORTED;
    if (level_mode != ZIPML_LEVELS_UNIFORM && level_mode != ZIPML_LEVELS_TABLE) return ZIPML_ERR_INVALID_ARG;
    if (level_mode == ZIPML_LEVELS_TABLE && bits > 4) return ZIPML_ERR_UNSUPPORTED;
    if (!A || !plane1 || !plane2 || !feat_lo || m <= 0 || n <= 0 || lda < n) return ZIPML_ERR_INVALID_ARG;
    if (level_mode == ZIPML_LEVELS_TABLE && !levels) return ZIPML_ERR_INVALID_ARG;
    if (level_mode == ZIPML_LEVELS_UNIFORM && !feat_step) return ZIPML_ERR_INVALID_ARG;
    if (row_bytes % 16 != 0 || row_bytes < zipml_row_bytes(n, bits)) return ZIPML_ERR_INVALID_ARG;
    if (!aligned16(plane1) || !aligned16(plane2)) return ZIPML_ERR_INVALID_ARG;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return ZIPML_ERR_CUDA;
    const int s = (1 << bits) - 1;
    float* inv = nullptr;
    if (level_mode == ZIPML_LEVELS_UNIFORM) {
        int rc = ws_reserve(ctx, carve_size(sizeof(float) * (size_t)n));
        if (rc != ZIPML_OK) return rc;
        inv = reinterpret_cast<float*>(ctx->ws);
        rc = launch_column_range(ctx, A, m, n, lda, s, grid == ZIPML_GRID_SYMMETRIC, feat_lo, nullptr, inv, feat_step);
        if (rc != ZIPML_OK) return rc;
    }
    return launch_quantize(ctx, A, m, n, lda, bits, level_mode, feat_lo, inv, levels, seed, draw, plane1, plane2, row_bytes, feat_lo, feat_step);
}

int zipml_optimal_levels(zipml_ctx* ctx, const float* A, int64_t m, int64_t n, int64_t lda, int32_t bits,
                         int32_t hist_bins, float* levels_out, uint64_t* objective_out) {
    if (!ctx) return ZIPML_ERR_INVALID_ARG;
    if (bits != 2 && bits != 3 && bits != 4) return ZIPML_ERR_UNSUPPORTED;
    const int s = (1 << bits) - 1;
    if (!A || !levels_out || m <= 0 || n <= 0 || lda < n) return ZIPML_ERR_INVALID_ARG;
    if (hist_bins < s || hist_bins > 1024 || m > 1000000000LL) return ZIPML_ERR_UNSUPPORTED;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return ZIPML_ERR_CUDA;
    int rc = ws_reserve(ctx, 3 * carve_size(sizeof(float) * (size_t)n) + carve_size(sizeof(uint32_t) * histogram_count(n, hist_bins)));
    if (rc != ZIPML_OK) return rc;
    Carver cv(ctx->ws);
    float* lo = cv.take<float>((size_t)n);
    float* hi = cv.take<float>((size_t)n);
    float* inv = cv.take<float>((size_t)n);
    uint32_t* counts = cv.take<uint32_t>(histogram_count(n, hist_bins));
    rc = launch_column_range(ctx, A, m, n, lda, hist_bins, false, lo, hi, inv, nullptr);
    if (rc != ZIPML_OK) return rc;
    rc = launch_histogram(ctx, A, m, n, lda, hist_bins, lo, inv, counts);
    if (rc != ZIPML_OK) return rc;
    return launch_levels_dp(ctx, counts, n, hist_bins, s, lo, hi, levels_out, objective_out);
}

// ---- AUTO's rules, measured in us per step: C column, S stream, R ring, K cluster (fp32 form), L lean, G the persistent grid ----

// The engine for rows that no cluster takes (uniform grids, fp32 model and gradient), 0 for other data and quantized vectors.  Lean and ring
// take 20 to 80 there (4 bits n 6,747 batch 64 L 22.3 R 19.0 C 8.2; 2 bits n 13,499 L 52.9 R 22.2 S 10.8).
static int wide_rows_engine(const zipml_ctx* ctx, const zipml_dataset* d, const zipml_sgd_params* p, int64_t B) {
    if (d->level_mode != ZIPML_LEVELS_UNIFORM || p->model_bits != 0 || p->grad_bits != 0 || p->model_out) return 0;
    const int cb = container_bits(d->bits);
    // Many rows of a few KB: the ring engine streams them.  4 bits 2.4 KB x 3,000 S 31.9 R 34.1, x 6,000 S 57 R 43; 3.3 KB x 6,000
    // S 51 R 49; 4.5 KB x 6,000 S 44 R 50; 2 bits 3.3 KB x 3,000 S 38.5 R 42, x 6,000 S 65 R 59.  8 bits, of which it makes
    // half the work per byte: 3.3 KB x 2,000 S 19.2 R 18.9, x 3,000 S 26.8 R 22.8; 6 KB x 2,000 S 18.9 R 22.7, x 6,000 S 41 R 37.
    if (cb == 8 ? 4 * B > 3 * d->row_bytes : 3 * B > 4 * d->row_bytes) return ZIPML_ENGINE_RING;
    const int64_t blocks = (d->row_bytes + 127) / 128;                 // CTAs of the column engine
    if (2 * blocks >= ctx->sm_count) {
        // At least half the device.  At 32 to 255 rows of 4-bit codes the choice of the stream engine for short steps is a pinned one,
        // not the faster: 10 KB x 32 C 8.2 S 10.4, x 128 8.9 / 10.8, x 224 9.3 / 11.7; 16 KB x 128 9.7 / 11.3.  (Rows that the column
        // engine declines, 32 KB x 128 S 14.3, go to the stream engine anyway.)
        if (B >= 256 || cb == 8 || B < 32) return ZIPML_ENGINE_COLUMN;
        return ZIPML_ENGINE_STREAM;
    }
    // 2 bits: C 10.4 S 11.0 at 2.3 KB x 64, 12.4 / 12.3 x 200, 27 / 22 x 1,200.  Else the column engine, whose CTAs are few but exchange
    // less, up to many rows: 8 bits 7 KB x 1,200 C 12.5 S 15.7, x 3,000 24.5 / 25.5, x 4,500 35.2 / 33.5; 9 KB x 2,000 21.6 / 23.3, x 3,000
    // 31.1 / 31.6; but rows of an odd multiple of 16 bytes, whose pieces begin in the middle of a sector, 6,512 bytes x 1,300 0.90 times S, x 2,200
    // 24.4 / 23.4, x 2,900 30.5 / 27.8, 8,016 x 1,300 0.98, x 1,700 22.4 / 20.6, x 2,900 34.8 / 29.3.  (At 4 bits the line at 1,200 rows is a pinned one: 4.1 KB x 1,200 C 13.7 S 16.0, x 2,000 19.3 / 19.4.)
    return cb == 2 || B >= (cb == 8 ? (d->row_bytes % 32 == 0 ? 3000 : 1500) : 1200) ? ZIPML_ENGINE_STREAM : ZIPML_ENGINE_COLUMN;
}

// The same rows with a quantized model or gradient: column or ring engine.  Q0/8 (fp32 model, gradient of 8 bits): 2 bits 2.2 KB x 1,200
// C 29.4 R 34.5, x 2,000 41 / 36; 4 KB x 2,000 42 / 41; 6 KB x 3,000 56 / 56; 8 KB x 4,500 87 / 93.  4 bits 4.1 KB x 64 C 9.1 R 22, x 1,200
// 16.5 / 33, x 3,600 39 / 40, x 4,500 46 / 44, 5 KB x 4,500 47 / 48; 9 KB x 8,192 86 / 85; 16 KB x 64 10.7 / 31, x 8,192 92 / 145.  8 bits 9 KB x 64
// 9.4 / 21; rows of an odd multiple of 16 bytes, whose pieces begin in the middle of a sector: 4,112 bytes x 2,400 26 / 28, x 3,000 32 / 30, 6,512 x 3,000 35 / 34,
// 8,016 x 2,700 1.07 times R, 9,008 x 3,000 37 / 36; others: 4,160 bytes x 3,000 0.95 times R, x 3,500 1.05, 6,528 x 4,000 0.99, x 4,500 1.04, 8,000 x 4,000
// 37 / 38, 9,024 x 4,500 0.88; 12 KB x 6,000 49 / 68.  (With a quantized model too C takes some 3 more, R 6; single steps cost C some 7 more, R 5: at
// the lines 0.07 to 0.15 of a step.)
static bool column_pays_quantized(const zipml_dataset* d, const zipml_sgd_params* p, int64_t B, int64_t T) {
    if (d->level_mode != ZIPML_LEVELS_UNIFORM || (p->model_bits == 0 && p->grad_bits == 0)) return false;
    // (a quantized gradient alone on data of up to three batches: the choice of the ring engine is a pinned one, not the faster.  The batches
    // of the data count, not the steps of the call: a range of an epoch's steps runs on the engine of the whole epoch)
    if (p->model_bits == 0 && T <= 3) return false;
    const int cb = container_bits(d->bits);
    if (cb == 2) return B <= 1500 || 2 * B <= d->row_bytes;
    if (cb == 4) return B <= 4000 || 10 * B <= (d->row_bytes >= 8000 ? 9 : 7) * d->row_bytes;
    if (d->row_bytes >= 11000) return true;
    if (d->row_bytes % 32 != 0) return B <= (d->row_bytes < 9000 ? 2500 : 3200);
    return B <= (d->row_bytes < 6000 ? 3200 : d->row_bytes < 9000 ? 4000 : 4500);
}

// Small steps that the cluster engine declined: row parts that meet through L2 (lean), or the ring's or grid's 148 CTAs.
//   tables: 3 bits n 600 x 1,207 L 13.7 G 21.2, x 2,414 L 21.5 G 23.8, x 3,276 L 27 G 25; n 512 x 2,867 L 18.5 G 20.1, x 3,891 L 22.9 G 21.5;
//   n 300 x 3,276 L 19.1 G 20.7, x 4,587 L 24.3 G 22.9; n 700 x 1,489 L 15.8 G 16.6, x 2,084 L 20.0 G 19.0; n 1,000 x 1,024 L 15.4 G 16.6, x 1,433
//   L 18.5 G 18.2; n 1,400 x 521 L 16.0 G 14.0.  4 bits n 600 x 2,414 L 23.0 G 26.2; n 850 x 1,213 L 17.6 G 17.9, x 1,698 L 21.7 G 19.7; n 1,000 x
//   716 L 17.6 G 15.6.  2 bits n 600 x 3,276 L 25.2 G 27.9, x 4,587 L 32.6 G 30.2; n 1,000 x 2,048 L 20.1 G 22.3, x 2,867 L 25.2 G 24.3; n 1,400 x
//   1,042 L 18.9 G 19.3, x 1,489 L 22.6 G 21.2; n 2,000 x 716 L 18.5 G 19.2, x 1,024 L 22.4 G 21.0; n 4,091 x 64 L 22 G 24, x 256 L 26 G 18.
//   One row of n 4,091 L 27 G 16.  With a quantized vector the grid is seldom better (3 bits n 600 x 1,207 L 17.6 G 24.8).
static bool lean_pays(const zipml_dataset* d, const zipml_sgd_params* p, int64_t B) {
    if (d->level_mode == ZIPML_LEVELS_UNIFORM) return false;
    if (p->model_bits != 0 || p->grad_bits != 0) return true;
    if (d->n >= 3000) return B * d->n <= 700000 && B >= 32;
    const int64_t most = container_bits(d->bits) == 2 ? (d->n <= 1000 ? 2300000 : 1500000)
                         : d->n < 400 ? 1200000 : d->n <= 600 ? 1700000 : d->n > 1000 ? 700000 : d->bits == 3 ? 1250000 : d->n <= 900 ? 1000000 : 700000;
    return B * d->n <= most;
}

// Level tables of up to 3,000 features, past what the cluster engine takes by features: its form by rows, whose sixteen CTAs walk
// through the batch, row parts that meet through L2 (lean), the persistent grid with 148 CTAs, or the ring engine.
//   2 bits, fp32 vectors: n 16 to 256 x 1,024 K 11.4 L 9.9 G 18, x 4,096 28.6 / 20.4 / 25, x 8,192 51.5 / 34.5 / 31.5 (R 41), x 16,384 97.5 / 62 / 43
//   (R 69); n 512 x 4,096 28.8 / 22.1 / 24, x 16,384 G 37.6 R 69; n 1,400 x 2,048 L 28.6 G 24.7; n 2,000 x 8,192 G 53 R 120.
//   3 and 4 bits: n 16 to 40 x 1,024 K 9.1 L 8.7 G 17, x 4,096 20.5 / 16.6 / 22 (R 18), x 8,192 35.5 / 27 / 26, x 16,384 65.5 / 48 / 36 (R 43); 3 bits
//   n 256 x 4,096 20.3 / 18.1 / 20.5; n 512 x 16,384 (8 MB) G 35 R 67; n 1,400 x 8,192 (11 MB) G 46 R 61; n 1,024 x 16,384 (16 MB) G 81 R 66; 4 bits n
//   512 x 16,384 (8 MB) G 37.5 R 69; n 700 x 8,192 (6 MB) 37 / 41; n 1,400 x 4,096 (6 MB) 32 / 28.  Past 4 MB and
//   500 features the lean engine again, where it holds the rows: 3 bits n 700 x 16,384 L 38 G 51, n 1,400 x 6,000 31 / 39; 4 bits n 512 x 16,384 31 / 37;
//   2 bits n 2,000 x 8,192 39 / 53.
//   Both vectors of 8 bits (a norm is dear on the lean engine beyond 64 features): 2 bits n 16 x 1,024 K 13.9 L 13.5 G 22, x 4,096 31 / 24 / 29, x
//   8,192 54 / 38.5 / 35.6; n 256 x 2,048 19.8 / 22.5 / 24.6, x 4,096 31.4 / 30 / 27.7, x 16,384 L 73 G 46 R 75; n 1,024 x 16,384 L 67 G 55 R 132;
//   n 2,000 x 4,096 L 47.5 G 57.6 R 77; just above 2 MB a step up to n 2,560 x 2,048 the ring engine still: n 2,200 L 48.9 R 46.5, x 2,200 52.8 / 53.2, n
//   2,550 x 1,900 52.5 / 47.2, x 2,400 48.3 / 53.5, n 2,600 x 2,048 46.9 / 51.4.  3 bits n 40 x 2,048 K 15.3 L 15.2, x 4,096 22.6 / 20.7 / 23.2, x 6,000 30 / 29.6 / 25.5; n 256 x 4,096 K 23 G 22.5; n 700 x 2,048 L 24.4 G 27.4
//   R 28, x 8,192 46 / 39 / 64; n 1,024 x 8,192 58 / 40 / 73; n 1,400 x 4,096 49 / 48 / 46.  4 bits n 700 x 8,192 45 / 42 / 49; n 1,400 x 1,024 31 / 41 / 29.
// `lean_fits`: false once the lean engine has declined.
static int table_engine(const zipml_dataset* d, const zipml_sgd_params* p, int64_t B, int64_t step_bytes, bool lean_fits) {
    const bool quantized = p->model_bits != 0 || p->grad_bits != 0, two = container_bits(d->bits) == 2;
    const int64_t n = d->n;
    constexpr int64_t MB = 1 << 20;
    if (!quantized) {
        if (B < (two ? 800 : n <= 64 ? 1100 : 1600)) return ZIPML_ENGINE_CLUSTER;
        if (lean_fits && B <= (two ? 7000 : 6500) && lean_pays(d, p, B)) return ZIPML_ENGINE_LEAN;
        if (lean_fits && (two ? n >= 1000 && step_bytes > 5 * MB : n >= 500 && step_bytes > 4 * MB)) return ZIPML_ENGINE_LEAN;
        return step_bytes <= (two ? 10 : d->bits == 3 ? 11 : n <= 800 ? 8 : 3) * MB ? ZIPML_ENGINE_PERSISTENT : ZIPML_ENGINE_RING;
    }
    if (n <= 64) {
        if (B < (two ? 1000 : 3500)) return ZIPML_ENGINE_CLUSTER;
        if (B > 5000) return ZIPML_ENGINE_PERSISTENT;
        if (lean_fits) return ZIPML_ENGINE_LEAN;
        // (rows that lie far apart: the stride sizes what the lean engine stages.  2 bits n 16 x 1,200 G 24.7 R 24.5, n 40 x 3,000 25.5 / 30.0, n 64 x 4,900
        // 28.0 / 37.3; 3 bits n 40 x 3,600 22.6 / 22.0; 4 bits n 16 x 3,600 24.4 / 23.3, n 64 x 4,900 24.1 / 25.9)
        if (step_bytes <= 2 * MB) return ZIPML_ENGINE_CLUSTER;
        return two || B > 4000 ? ZIPML_ENGINE_PERSISTENT : ZIPML_ENGINE_RING;
    }
    if (B <= (two || n >= 400 ? 2500 : 4096) && step_bytes <= 2 * MB) return ZIPML_ENGINE_CLUSTER;
    if (n <= (two || d->bits == 3 ? 1100 : 800) && step_bytes <= (d->bits == 4 ? 8 : 10) * MB) return ZIPML_ENGINE_PERSISTENT;
    return lean_fits && two && step_bytes <= 10 * MB && (B > 2100 || n > 2560) ? ZIPML_ENGINE_LEAN : ZIPML_ENGINE_RING;
}

// Uniform rows too wide for the column and stream engines: the persistent grid up to 16 MB a step, 4 bits n 100,000 x 64 G 23 R 42, x 300
// (30 MB) 107 / 53; 8 bits n 150,000 x 64 (19 MB) 60 / 71, x 300 243 / 138.
// Level tables wider than a cluster holds: the persistent grid too, whose CTAs take row parts of a few columns and so build few of the
// tables, until the ring engine's asynchronous tiles win.  2 bits n 13,499 x 64 G 17 R 27, x 600 (4 MB) 37 / 45, x 1,500 (10 MB) 75 / 76;
// 3 bits n 6,747 x 600 (4 MB) 26 / 29, n 12,283 x 1,500 (18 MB) 91 / 64; 4 bits n 4,891 x 600 (2.9 MB) 29 / 32, n 20,475 x 256 (5 MB) 37 / 33.
static bool grid_pays(const zipml_dataset* d, const zipml_sgd_params* p, int64_t step_bytes, int wide) {
    if (p->model_bits != 0 || p->grad_bits != 0) return false;
    if (d->level_mode == ZIPML_LEVELS_UNIFORM) return (wide == ZIPML_ENGINE_COLUMN || wide == ZIPML_ENGINE_STREAM) && step_bytes <= (16ll << 20);
    return step_bytes <= (d->bits == 2 ? 10ll << 20 : d->bits == 3 ? 5ll << 20 : 3ll << 20);
}

int zipml_sgd_epoch(zipml_ctx* ctx, const zipml_dataset* data, const float* b, float* x,
                    const zipml_sgd_params* params, float* grad_out) {
    if (!ctx || !params || params->struct_size != sizeof(zipml_sgd_params)) return ZIPML_ERR_INVALID_ARG;
    int rc = check_dataset(data);
    if (rc != ZIPML_OK) return rc;
    if (!b || !x || params->batch <= 0) return ZIPML_ERR_INVALID_ARG;
    if (params->model_bits != 0 && (params->model_bits < 2 || params->model_bits > 8)) return ZIPML_ERR_UNSUPPORTED;
    if (params->grad_bits != 0 && (params->grad_bits < 2 || params->grad_bits > 8)) return ZIPML_ERR_UNSUPPORTED;
    if (params->engine < ZIPML_ENGINE_AUTO || params->engine > ZIPML_ENGINE_SOLO) return ZIPML_ERR_INVALID_ARG;
    if (params->epoch < 0 || params->epoch > 0xffffffffLL) return ZIPML_ERR_INVALID_ARG;
    if (params->reg < ZIPML_REG_NONE || params->reg > ZIPML_REG_LSSVM) return ZIPML_ERR_INVALID_ARG;
    if (params->reg != ZIPML_REG_NONE && params->reg != ZIPML_REG_NONNEG && !(params->reg_param >= 0.0f)) return ZIPML_ERR_INVALID_ARG;
    if (params->cluster_contraction < 0 || params->cluster_contraction > 4) return ZIPML_ERR_INVALID_ARG;
    if (params->stream_prefetch < 0 || params->stream_prefetch > 9) return ZIPML_ERR_INVALID_ARG;
    if (params->column_chunk_rows < 0 || params->column_chunk_rows > 256 || params->column_chunk_rows % 32 != 0) return ZIPML_ERR_INVALID_ARG;
    if (params->vector_norm != ZIPML_NORM_L2 && params->vector_norm != ZIPML_NORM_LINF) return ZIPML_ERR_INVALID_ARG;
    // the other scaling of Q3/Q4 lives in the first-generation engine only
    const bool linf = params->vector_norm == ZIPML_NORM_LINF && (params->model_bits > 0 || params->grad_bits > 0);
    if (linf && params->engine != ZIPML_ENGINE_AUTO && params->engine != ZIPML_ENGINE_STEPWISE && params->engine != ZIPML_ENGINE_PERSISTENT)
        return ZIPML_ERR_UNSUPPORTED;
    const int64_t T = (data->m + params->batch - 1) / params->batch;
    const int64_t first = params->first_step;
    const int64_t count = params->num_steps < 0 ? T - first : params->num_steps;
    if (first < 0 || first > T || count < 0 || first + count > T) return ZIPML_ERR_INVALID_ARG;
    if (params->batch_order)
        for (int64_t i = 0; i < T; ++i)
            if (params->batch_order[i] < 0 || params->batch_order[i] >= T) return ZIPML_ERR_INVALID_ARG;
    if (count == 0) return ZIPML_OK;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return ZIPML_ERR_CUDA;
    if (linf && data->layout == ZIPML_LAYOUT_COLUMN_BLOCKS) return ZIPML_ERR_UNSUPPORTED;
    if (data->layout == ZIPML_LAYOUT_COLUMN_BLOCKS) {                 // the column engine's own layout
        if (params->engine != ZIPML_ENGINE_AUTO && params->engine != ZIPML_ENGINE_COLUMN) return ZIPML_ERR_UNSUPPORTED;
        rc = launch_sgd_column(ctx, data, b, x, params, first, count, grad_out, false);
        return rc == ZIPML_ERR_WORKSPACE ? ZIPML_ERR_UNSUPPORTED : rc;
    }
    if (params->engine == ZIPML_ENGINE_RING) return launch_sgd_ring(ctx, data, b, x, params, first, count, grad_out, false);
    if (params->engine == ZIPML_ENGINE_LEAN) return launch_sgd_lean(ctx, data, b, x, params, first, count, grad_out);
    if (params->engine == ZIPML_ENGINE_CLUSTER) return launch_sgd_cluster(ctx, data, b, x, params, first, count, grad_out);
    if (params->engine == ZIPML_ENGINE_STREAM) return launch_sgd_stream(ctx, data, b, x, params, first, count, grad_out);
    if (params->engine == ZIPML_ENGINE_COLUMN) return launch_sgd_column(ctx, data, b, x, params, first, count, grad_out, false);
    if (params->engine == ZIPML_ENGINE_SOLO) return launch_sgd_solo(ctx, data, b, x, params, first, count, grad_out, false);
    if (params->engine == ZIPML_ENGINE_AUTO && !linf) {
        // Small minibatch tiles are bound by the step-to-step chain, not by HBM: the smallest stay on one SM, then
        // clusters whose CTAs exchange through shared memory.  What no cluster holds goes to the column engine
        // (codes read once per step), the stream engine or the ring engine, whatever the step's size.  Each engine
        // answers ZIPML_ERR_WORKSPACE when the shape does not fit it.
        const int64_t B = params->batch < data->m ? params->batch : data->m;
        const int64_t step_bytes = 2 * B * data->row_bytes;
        const bool small = step_bytes <= (2ll << 20);
        const int wide = wide_rows_engine(ctx, data, params, B);
        if (small) {
            rc = launch_sgd_solo(ctx, data, b, x, params, first, count, grad_out, true);
            if (rc != ZIPML_ERR_WORKSPACE) return rc;
        }
        int table = 0;
        if (data->level_mode == ZIPML_LEVELS_TABLE && data->n < 3000 && params->cluster_contraction == 0) {
            if (small && table_form_pays(data, params)) {
                rc = launch_sgd_table(ctx, data, b, x, params, first, count, grad_out);
                if (rc != ZIPML_ERR_WORKSPACE) return rc;
            }
            table = table_engine(data, params, B, step_bytes, true);
            if (table == ZIPML_ENGINE_LEAN) {
                rc = launch_sgd_lean(ctx, data, b, x, params, first, count, grad_out);
                if (rc != ZIPML_ERR_WORKSPACE) return rc;
                table = table_engine(data, params, B, step_bytes, false);
            }
        }
        if (data->level_mode == ZIPML_LEVELS_UNIFORM && params->cluster_contraction != 1) {
            rc = launch_sgd_int8(ctx, data, b, x, params, first, count, grad_out);
            if (rc != ZIPML_ERR_WORKSPACE) return rc;
        } else if (small && (table == 0 || table == ZIPML_ENGINE_CLUSTER)) {
            rc = launch_sgd_cluster(ctx, data, b, x, params, first, count, grad_out);
            if (rc != ZIPML_ERR_WORKSPACE) return rc;
        }
        if (small && (table == 0 || table == ZIPML_ENGINE_CLUSTER) && lean_pays(data, params, B)) {
            rc = launch_sgd_lean(ctx, data, b, x, params, first, count, grad_out);
            if (rc != ZIPML_ERR_WORKSPACE) return rc;
        }
        if (column_pays_quantized(data, params, B, T)) {
            rc = launch_sgd_column(ctx, data, b, x, params, first, count, grad_out, true);
            if (rc != ZIPML_ERR_WORKSPACE) return rc;
        }
        if (wide == ZIPML_ENGINE_COLUMN) {
            rc = launch_sgd_column(ctx, data, b, x, params, first, count, grad_out, false);
            if (rc != ZIPML_ERR_WORKSPACE) return rc;
        }
        if (wide == ZIPML_ENGINE_COLUMN || wide == ZIPML_ENGINE_STREAM) {
            rc = launch_sgd_stream(ctx, data, b, x, params, first, count, grad_out);
            if (rc != ZIPML_ERR_WORKSPACE) return rc;
        }
        if (table == ZIPML_ENGINE_PERSISTENT || (table != ZIPML_ENGINE_RING && grid_pays(data, params, step_bytes, wide))) {
            zipml_sgd_params grid = *params;
            grid.engine = ZIPML_ENGINE_PERSISTENT;
            rc = launch_sgd_epoch(ctx, data, b, x, &grid, first, count, grad_out);
            if (rc != ZIPML_ERR_WORKSPACE) return rc;
        }
        rc = launch_sgd_ring(ctx, data, b, x, params, first, count, grad_out, false);
        if (rc != ZIPML_ERR_WORKSPACE) return rc;
    }
    return launch_sgd_epoch(ctx, data, b, x, params, first, count, grad_out);
}

int zipml_sgd_apply_gradient(zipml_ctx* ctx, float* x, const float* g, int64_t n, const zipml_sgd_params* params,
                             int64_t step, float* applied_out) {
    if (!ctx || !params || params->struct_size != sizeof(zipml_sgd_params)) return ZIPML_ERR_INVALID_ARG;
    if (!x || !g || n <= 0 || n > 0x7fffffffLL || step < 0 || step > 0xffffffffLL) return ZIPML_ERR_INVALID_ARG;
    if (params->grad_bits != 0 && (params->grad_bits < 2 || params->grad_bits > 8)) return ZIPML_ERR_UNSUPPORTED;
    if (params->epoch < 0 || params->epoch > 0xffffffffLL) return ZIPML_ERR_INVALID_ARG;
    if (params->reg < ZIPML_REG_NONE || params->reg > ZIPML_REG_LSSVM) return ZIPML_ERR_INVALID_ARG;
    if (params->reg != ZIPML_REG_NONE && params->reg != ZIPML_REG_NONNEG && !(params->reg_param >= 0.0f)) return ZIPML_ERR_INVALID_ARG;
    if (params->vector_norm != ZIPML_NORM_L2 && params->vector_norm != ZIPML_NORM_LINF) return ZIPML_ERR_INVALID_ARG;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return ZIPML_ERR_CUDA;
    return launch_sgd_apply(ctx, x, g, n, params, step, applied_out);
}

int zipml_barrier_latency(zipml_ctx* ctx, int32_t ctas, int32_t floats_per_cta, int32_t iterations, uint64_t* ns_out) {
    if (!ctx || !ns_out || ctas < 1 || floats_per_cta < 0 || floats_per_cta % 4 != 0 || iterations < 1 || iterations > (1 << 20))
        return ZIPML_ERR_INVALID_ARG;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return ZIPML_ERR_CUDA;
    return launch_barrier_latency(ctx, ctas, floats_per_cta, iterations, reinterpret_cast<unsigned long long*>(ns_out));
}

int zipml_poly_rows(zipml_ctx* ctx, const zipml_dataset* grid, const uint8_t* const* planes, int32_t degree,
                    const double* coef, const float* x, const float* scale, double* rows_out) {
    if (!ctx || !coef || !x || !rows_out || degree < 0 || degree > ZIPML_POLY_MAX_DEGREE) return ZIPML_ERR_INVALID_ARG;
    int rc = check_dataset(grid);
    if (rc != ZIPML_OK) return rc;
    if (grid->layout != ZIPML_LAYOUT_ROWS) return ZIPML_ERR_UNSUPPORTED;
    if (degree > 0 && !planes) return ZIPML_ERR_INVALID_ARG;
    for (int i = 0; i < degree; ++i)
        if (!planes[i] || !aligned16(planes[i])) return ZIPML_ERR_INVALID_ARG;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return ZIPML_ERR_CUDA;
    const bool table = grid->level_mode == ZIPML_LEVELS_TABLE;
    const size_t wcount = (size_t)grid->n * (table ? ((size_t)1 << grid->bits) : 1);
    rc = ws_reserve(ctx, carve_size(sizeof(float) * wcount) + carve_size(sizeof(double)));
    if (rc != ZIPML_OK) return rc;
    Carver cv(ctx->ws);
    float* wtab = cv.take<float>(wcount);
    double* base = cv.take<double>(1);
    rc = launch_code_weights(ctx, grid, x, wtab, base);
    if (rc != ZIPML_OK) return rc;
    return launch_poly_rows(ctx, grid, planes, degree, coef, wtab, base, scale, rows_out);
}

int zipml_weighted_plane_mean(zipml_ctx* ctx, const zipml_dataset* grid, const uint8_t* plane, const double* c, float* g_out) {
    if (!ctx || !plane || !c || !g_out || !aligned16(plane)) return ZIPML_ERR_INVALID_ARG;
    int rc = check_dataset(grid);
    if (rc != ZIPML_OK) return rc;
    if (grid->layout != ZIPML_LAYOUT_ROWS) return ZIPML_ERR_UNSUPPORTED;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return ZIPML_ERR_CUDA;
    const size_t count = (size_t)plane_mean_chunks(ctx, grid->m) * ((size_t)grid->n + 1);
    rc = ws_reserve(ctx, carve_size(sizeof(double) * count));
    if (rc != ZIPML_OK) return rc;
    return launch_plane_mean(ctx, grid, plane, c, reinterpret_cast<double*>(ctx->ws), g_out);
}

int zipml_wait_probe(zipml_ctx* ctx, int64_t spin_limit) {
    if (!ctx || spin_limit < 1 || spin_limit > (1 << 24)) return ZIPML_ERR_INVALID_ARG;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return ZIPML_ERR_CUDA;
    int rc = ws_reserve(ctx, 256);
    if (rc != ZIPML_OK) return rc;
    cudaError_t e = cudaMemsetAsync(ctx->ws, 0, 256, ctx->stream);
    if (e != cudaSuccess) return cuda_status(e);
    wait_probe_kernel<<<1, 32, 0, ctx->stream>>>(reinterpret_cast<const unsigned*>(ctx->ws), spin_limit, ctx->d_status);
    ctx->launches += 1;
    return cuda_status(cudaGetLastError());
}

int zipml_loss(zipml_ctx* ctx, int32_t mode, const float* A, int64_t m, int64_t n, int64_t lda,
               const zipml_dataset* data, const float* b, const float* x, double* loss_out) {
    if (!ctx || !b || !x || !loss_out) return ZIPML_ERR_INVALID_ARG;
    if (mode != ZIPML_LOSS_DENSE && mode != ZIPML_LOSS_CODES) return ZIPML_ERR_INVALID_ARG;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return ZIPML_ERR_CUDA;
    if (mode == ZIPML_LOSS_DENSE) {
        if (!A || m <= 0 || n <= 0 || lda < n) return ZIPML_ERR_INVALID_ARG;
        int rc = ws_reserve(ctx, carve_size(sizeof(double) * kLossPartials));
        if (rc != ZIPML_OK) return rc;
        return launch_loss_dense(ctx, A, m, n, lda, b, x, reinterpret_cast<double*>(ctx->ws), kLossPartials, loss_out);
    }
    int rc = check_dataset(data);
    if (rc != ZIPML_OK) return rc;
    if (data->layout != ZIPML_LAYOUT_ROWS) return ZIPML_ERR_UNSUPPORTED;
    // behind the partials: the level * x table, or (uniform grids) the digit vectors of step * x, which follow the
    // packed row byte for byte and so take their size from the stride, not from n
    const size_t tab = data->level_mode == ZIPML_LEVELS_TABLE
                           ? sizeof(float) * ((size_t)1 << data->bits) * (size_t)data->n
                           : (size_t)(8 / container_bits(data->bits)) * 4 * (((size_t)data->row_bytes + 63) / 64 * 64);
    rc = ws_reserve(ctx, carve_size(sizeof(double) * (kLossPartials + 2) + tab + 256));
    if (rc != ZIPML_OK) return rc;
    return launch_loss_codes(ctx, data, b, x, reinterpret_cast<double*>(ctx->ws), kLossPartials, loss_out);
}

int zipml_train_host(zipml_ctx* ctx, const float* A_host, int64_t m, int64_t n, int64_t lda, const float* b_host,
                     float* x_host, int32_t bits, int32_t optimal_levels, int32_t hist_bins, uint64_t quantize_seed,
                     const zipml_sgd_params* params, int32_t epochs, int32_t lr_decay, double* loss_out_host) {
    if (!ctx || !params || params->struct_size != sizeof(zipml_sgd_params)) return ZIPML_ERR_INVALID_ARG;
    if (!A_host || !b_host || !x_host || !loss_out_host || m <= 0 || n <= 0 || lda < n || epochs < 0)
        return ZIPML_ERR_INVALID_ARG;
    const int64_t rb = zipml_row_bytes(n, bits);
    if (rb == 0) return ZIPML_ERR_UNSUPPORTED;
    if (optimal_levels && (bits < 2 || bits > 4)) return ZIPML_ERR_UNSUPPORTED;
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return ZIPML_ERR_CUDA;
    const size_t L = (size_t)1 << bits;
    size_t total = 0;
    auto piece = [&](size_t bytes) { const size_t off = total; total += carve_size(bytes); return off; };
    const size_t oA = piece(sizeof(float) * (size_t)m * n), ob = piece(sizeof(float) * (size_t)m);
    const size_t ox = piece(sizeof(float) * (size_t)n), op1 = piece((size_t)m * rb), op2 = piece((size_t)m * rb);
    const size_t olo = piece(sizeof(float) * (size_t)n), ostep = piece(sizeof(float) * (size_t)n);
    const size_t olev = piece(sizeof(float) * (size_t)n * L), oloss = piece(sizeof(double));
    int rc = stage_reserve(ctx, total);
    if (rc != ZIPML_OK) return rc;
    unsigned char* s = ctx->stage;
    float* dA = reinterpret_cast<float*>(s + oA);
    float* db = reinterpret_cast<float*>(s + ob);
    float* dx = reinterpret_cast<float*>(s + ox);
    float* dlev = reinterpret_cast<float*>(s + olev);
    double* dloss = reinterpret_cast<double*>(s + oloss);
    // (contiguous rows travel as one linear copy: a pitched copy of many short rows is much slower)
    cudaError_t e = lda == n ? cudaMemcpyAsync(dA, A_host, sizeof(float) * (size_t)m * n, cudaMemcpyHostToDevice, ctx->stream)
                             : cudaMemcpy2DAsync(dA, sizeof(float) * n, A_host, sizeof(float) * lda, sizeof(float) * n, (size_t)m,
                                                 cudaMemcpyHostToDevice, ctx->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(db, b_host, sizeof(float) * m, cudaMemcpyHostToDevice, ctx->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dx, x_host, sizeof(float) * n, cudaMemcpyHostToDevice, ctx->stream);
    if (e != cudaSuccess) return cuda_status(e);

    zipml_dataset d{};
    d.struct_size = sizeof(zipml_dataset);
    d.bits = bits; d.m = m; d.n = n; d.row_bytes = rb;
    d.plane1 = s + op1; d.plane2 = s + op2;
    d.feat_lo = reinterpret_cast<float*>(s + olo);
    d.feat_step = reinterpret_cast<float*>(s + ostep);
    d.levels = nullptr;
    d.level_mode = optimal_levels ? ZIPML_LEVELS_TABLE : ZIPML_LEVELS_UNIFORM;
    if (optimal_levels) {
        rc = zipml_optimal_levels(ctx, dA, m, n, n, bits, hist_bins, dlev, nullptr);
        if (rc != ZIPML_OK) return rc;
        d.levels = dlev;
    }
    rc = zipml_quantize(ctx, dA, m, n, n, bits, d.level_mode, d.levels, quantize_seed, s + op1, s + op2, rb,
                        reinterpret_cast<float*>(s + olo), reinterpret_cast<float*>(s + ostep));
    if (rc != ZIPML_OK) return rc;
    zipml_sgd_params p = *params;
    for (int32_t ep = 0; ep < epochs; ++ep) {
        p.epoch = ep; p.first_step = 0; p.num_steps = -1;
        p.lr = lr_decay ? params->lr / (float)(ep + 1) : params->lr;
        rc = zipml_sgd_epoch(ctx, &d, db, dx, &p, nullptr);
        if (rc != ZIPML_OK) return rc;
    }
    rc = zipml_loss(ctx, ZIPML_LOSS_DENSE, dA, m, n, n, nullptr, db, dx, dloss);
    if (rc != ZIPML_OK) return rc;
    e = cudaMemcpyAsync(x_host, dx, sizeof(float) * n, cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(loss_out_host, dloss, sizeof(double), cudaMemcpyDeviceToHost, ctx->stream);
    if (e != cudaSuccess) return cuda_status(e);
    return zipml_sync(ctx);
}

}  // extern "C"
