// Cluster engine of zipml_sgd_epoch, split by rows and in fp32 (level tables with few features and long batches, and what its other
// forms do not hold; sgd_feature.cu, sgd_slice.cu and sgd_table.cu have those): one persistent launch of a single thread-block cluster, built
// for steps whose code tile is small (Supplement "Double Sampling", footnote form; "End-to-end
// Quantization").
//
// A small step is bound by the chain  dots -> residuals -> partial gradients -> sum over the CTAs ->
// update -> new model at every CTA.  Measured on B200, a value handed from one SM to another through
// L2 (store, poll) takes about 1000 cycles; a bulk copy from shared memory into the shared memory
// of another CTA of the cluster that completes a transaction count on the receiver's mbarrier
// takes about 320 cycles for 256 bytes (st.async: 230), and the receiver waits on local shared
// memory.  So here the minibatch is cut into nb <= 16 row parts, one CTA each, all in one cluster:
//   * phase A: a warp takes rows, its lanes the words of a row; fp32 FMA on unpacked codes against
//     w = step * x~ (or a level-times-model table), the two dots of a row summed across the warp
//     in double; residuals stay in the CTA;
//   * phase B: a thread takes a word column, adds code * residual over the CTA's rows; the CTA's
//     part of the gradient (for uniform grids lo * sum(r) + step * sum(code * r)) lands in
//     shared memory;
//   * reduce-scatter: CTA o owns features [o * sub, (o + 1) * sub); every CTA bulk-copies slice o of
//     its part into owner o's receive buffer (one copy instruction per owner); the owner waits on
//     its mbarrier, adds the nb parts in a fixed order, applies the optional gradient quantizer and
//     the update to its master copy and writes what the next step sees (Q3 of it when the model
//     quantizer is on) into a staging buffer;
//   * all-gather: the owner bulk-copies the staging buffer to every CTA's model vector; every CTA
//     waits on its mbarrier and builds w.  The first model takes the same route: the loop starts
//     with a publish-only round.
//   * the code tiles do not depend on the model: bulk copies from global memory run several steps
//     ahead in a ring of shared-memory slots (one contiguous copy per plane and step).
// Buffer reuse: a CTA overwrites its part (and sends the next one) only after it has received the
// model of the step from every owner, and an owner publishes only after all parts of the step have
// landed in its buffer; an owner overwrites its staging buffer only after the parts of the next
// step have arrived, which their senders issued after the model had landed everywhere.  So single
// buffers suffice and no copy can still be reading a buffer that is being rewritten.
// Every wait is a bounded wait on a local mbarrier: when one gives up the CTA records
// ZIPML_ERR_TIMEOUT, skips its later waits and still issues every copy, so the launch ends; all CTAs
// meet at a cluster barrier before they exit (nobody's shared memory goes away under a copy).
#include <stdlib.h>
#include <string.h>

#include "sgd_common.cuh"

namespace zipml {

constexpr int kCluThreads = 512;
constexpr int kCluWarps = kCluThreads / 32;
constexpr int kCluMaxSlots = 8;
constexpr int kCluMaxCtas = 16;                   // one bulk copy per warp and destination: at most kCluWarps CTAs
static_assert(kCluMaxCtas <= kCluWarps, "a warp per destination CTA");

struct ClusterArgs {
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
    unsigned long long* trace;
    DeviceStatus* status;
    int64_t m, batch, first_step, num_steps;
    uint64_t seed;
    uint32_t epoch;
    float lr;
    int reg;                     // ZIPML_REG_* and its fp32 constant
    float reg_cst;
    int n, bits, row_words, words;   // words = ceil(n / codes per word) <= row_words
    int model_bits, grad_bits;
    int pitch;                       // words between the rows of a tile in shared memory: row_words (as an argument of its own: addressed through
                                     // row_words the kernel on 2-bit tables took 0.4 us a step longer, 5.3 -> 5.7 at 300 rows x 64)
    int nb, rc, slots;
    int sub;                     // a CTA owns `sub` consecutive features (a multiple of 4)
    int p_shift;                 // 2^p_shift lanes share the sum of one owned feature
    int trace_steps;
};

struct ClusterShared {
    double red[kCluWarps];       // block sums
    double wbase[kCluWarps];     // per-warp parts of lo^T x~
    double ssum[kCluWarps];      // per-warp sums of the residuals
    double nrm_g[kCluMaxCtas];   // partial squared gradient norms, one per CTA
    double nrm_x[kCluMaxCtas];   // partial squared model norms
    unsigned long long full[kCluMaxSlots];
    unsigned long long rs_bar, ag_bar, gn_bar, xn_bar;
    int abort_flag;
    int pad;
};

__device__ __forceinline__ uint32_t cluster_addr(const void* local_smem, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(local_smem)), "r"(rank));
    return r;
}
// shared::cta -> shared::cluster bulk copy; completes `bytes` on the mbarrier at the destination CTA.
__device__ __forceinline__ void bulk_copy_s2c(uint32_t dst_cluster, const void* src_smem, uint32_t bytes, uint32_t bar_cluster) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst_cluster), "r"(smem_u32(src_smem)), "r"(bytes), "r"(bar_cluster) : "memory");
}
__device__ __forceinline__ void store_async_f64(uint32_t dst_cluster, double v, uint32_t bar_cluster) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];"
                 ::"r"(dst_cluster), "l"(__double_as_longlong(v)), "r"(bar_cluster) : "memory");
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Bounded wait on a local mbarrier phase; after the first failure of this CTA every wait is skipped.
__device__ __forceinline__ void clu_wait(unsigned long long* bar, uint32_t parity, ClusterShared* sh, DeviceStatus* status, int where) {
    if (*reinterpret_cast<volatile int*>(&sh->abort_flag)) return;
    // (a phase that is complete already -- a tile copied steps ahead -- answers the non-blocking test at once)
    {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done) : "r"(smem_u32(bar)), "r"(parity) : "memory");
        if (done) return;
    }
#pragma unroll 1
    for (long long spin = 0; spin < kCopySpinLimit; ++spin)
        if (mbar_try_wait(reinterpret_cast<uint64_t*>(bar), parity)) return;
    sh->abort_flag = 1;
    set_status(status, ZIPML_ERR_TIMEOUT, where);
}

// l2 norm of a vector whose squared entries are spread over the threads of all CTAs: block sum, one
// double per CTA stored into every CTA's table, added there in CTA order.
__device__ __noinline__ float clu_norm(double v, double* table, unsigned long long* bar, uint32_t parity, int nb,
                                       ClusterShared* sh, DeviceStatus* status, int where) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) sh->red[warp] = v;
    if (threadIdx.x == 0) mbar_arrive_expect_tx(reinterpret_cast<uint64_t*>(bar), 8u * (uint32_t)nb);
    __syncthreads();
    if ((int)threadIdx.x < nb) {
        double t = 0.0;
        for (int w = 0; w < kCluWarps; ++w) t += sh->red[w];
        store_async_f64(cluster_addr(table + blockIdx.x, threadIdx.x), t, cluster_addr(bar, threadIdx.x));
    }
    clu_wait(bar, parity, sh, status, where);
    double t = 0.0;
    for (int c = 0; c < nb; ++c) t += table[c];
    return (float)sqrt(t);
}

__device__ __noinline__ float clu_quant(float v, float M, int sm, uint64_t seed, uint32_t epoch, uint32_t step,
                                        uint32_t stream, uint32_t coord) {
    VecQuant q{M, sm, seed, epoch, step, stream};
    return q.apply(v, coord);
}

__device__ __forceinline__ void clu_mark(const ClusterArgs& a, int64_t it, int id) {
    if (a.trace && blockIdx.x == 0 && threadIdx.x == 0 && it >= a.first_step && it - a.first_step < a.trace_steps) {
        unsigned long long t;
        asm volatile("mov.u64 %0, %clock64;" : "=l"(t));
        a.trace[(it - a.first_step) * 8 + id] = t;
    }
}

// Shared memory after ClusterShared; Fp = row_words * FPW feature slots of a row (padding included),
// Fs = nb * sub >= n features as the owners cut them:
//   uniform: wv[Fp]  w = step * x~ by feature;  los[Fp], steps[Fp]  lo and step by feature
//   table:   tab[L*Fp] level * x~ and lev[L*Fp] levels, both [code][slot i][word q]
//   xs[Fs]           the model this step sees (all-gather destination)
//   gpart[Fs]        this CTA's part of the gradient (reduce-scatter source)
//   gbuf[nb][sub]    the nb parts of the owned features (reduce-scatter destination)
//   xpub[sub], xown[sub], gsub[sub]   staging of the published slice, master model, gradient of the step
//   res[2*rc]        residuals (r1, r2) per row;   bsm[rc]  labels of the step's rows
//   gred[512*FPW]    cross-group sums of phase B (parts narrower than the CTA)
//   ring[slots][2][rc][row_words]  code tiles
template <int CB, bool TABLE>
__global__ void __launch_bounds__(kCluThreads, 1) sgd_cluster_kernel(const ClusterArgs a) {
    constexpr int FPW = 32 / CB;
    constexpr int LOGF = (CB == 8) ? 2 : (CB == 4) ? 3 : 4;
    extern __shared__ __align__(16) unsigned char s_raw[];
    ClusterShared* sh = reinterpret_cast<ClusterShared*>(s_raw);
    const int rw = a.row_words, nw = a.words, n = a.n;
    const int Fp = rw * FPW;
    const int L = 1 << a.bits;
    const int sub = a.sub;
    const int nb = a.nb;
    const int Fs = nb * sub;
    float* tab = reinterpret_cast<float*>(s_raw + ((sizeof(ClusterShared) + 15) & ~(size_t)15));
    float* wv = tab;                                     // uniform
    float* los = tab + Fp;
    float* steps = los + Fp;
    float* lev = tab + (size_t)L * Fp;                   // table
    float* gred = TABLE ? lev + (size_t)L * Fp : steps + Fp;
    const int lanes_q = min(kCluThreads, ((nw + 31) / 32) * 32), ngroups = kCluThreads / lanes_q;
    float* xs = gred + (ngroups > 1 ? kCluThreads * FPW : 0);
    float* gpart = xs + Fs;
    float* gbuf = gpart + Fs;
    float* xpub = gbuf + Fs;
    float* xown = xpub + sub;
    float* gsub = xown + sub;
    float* res = gsub + sub;
    float* bsm = res + ((2 * a.rc + 3) & ~3);
    uint32_t* ring = reinterpret_cast<uint32_t*>(
        (reinterpret_cast<uintptr_t>(bsm + ((a.rc + 3) & ~3)) + 127) & ~(uintptr_t)127);
    const int pitch = a.pitch;
    const size_t slot_words = (size_t)2 * a.rc * pitch;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int bi = blockIdx.x;                           // the grid is one cluster: block index = rank
    const int k0 = bi * a.rc;
    const int64_t step_end = a.first_step + a.num_steps;

    auto step_rows = [&](int64_t it, int64_t& r0, int& bt, int& rcnt) {
        const int64_t t = a.order ? (int64_t)a.order[it] : it;
        r0 = t * a.batch;
        bt = (int)min(a.batch, a.m - r0);
        rcnt = max(0, min(a.rc, bt - k0));
    };
    // the tile of step `it` into `slot`, issued by one whole warp: one contiguous piece per plane
    auto issue_tile = [&](int64_t it, int slot) {
        int64_t r0; int bt, rcnt;
        step_rows(it, r0, bt, rcnt);
        uint64_t* full = reinterpret_cast<uint64_t*>(sh->full + slot);
        const uint32_t bytes = (uint32_t)rcnt * (uint32_t)rw * 4u;
        if (lane == 0) mbar_arrive_expect_tx(full, 2u * bytes);
        __syncwarp();
        uint32_t* dst = ring + (size_t)slot * slot_words;
        const size_t src = (size_t)(r0 + k0) * rw;
        if (lane < 2 && rcnt > 0) bulk_copy_g2s(dst + (size_t)lane * a.rc * rw, (lane ? a.p2 : a.p1) + src, bytes, full);
    };

    if (tid == 0) {
        for (int s = 0; s < a.slots; ++s) mbar_init(reinterpret_cast<uint64_t*>(sh->full + s), 1);
        mbar_init(reinterpret_cast<uint64_t*>(&sh->rs_bar), 1);
        mbar_init(reinterpret_cast<uint64_t*>(&sh->ag_bar), 1);
        mbar_init(reinterpret_cast<uint64_t*>(&sh->gn_bar), 1);
        mbar_init(reinterpret_cast<uint64_t*>(&sh->xn_bar), 1);
        sh->abort_flag = 0;
        mbar_fence_init();
    }
    for (int f = tid; f < Fp; f += kCluThreads) {
        const int q = f >> LOGF, i = f & (FPW - 1);
        if constexpr (TABLE) {
            for (int c = 0; c < L; ++c) lev[(c * FPW + i) * rw + q] = (f < n) ? __ldg(a.levels + (size_t)f * L + c) : 0.0f;
        } else {
            los[f] = (f < n) ? __ldg(a.lo + f) : 0.0f;
            steps[f] = (f < n) ? __ldg(a.step + f) : 0.0f;
        }
    }
    for (int f = tid; f < Fs; f += kCluThreads) gpart[f] = 0.0f;       // features past n stay zero
    for (int k = tid; k < sub; k += kCluThreads) xown[k] = (bi * sub + k < n) ? a.x[bi * sub + k] : 0.0f;
    __syncthreads();
    if (warp == 0)
        for (int s = 0; s < a.slots && a.first_step + s < step_end; ++s) issue_tile(a.first_step + s, s);
    cluster_sync_all();                                  // every CTA's barriers exist before anyone copies into it

    // thread roles: owner group of P lanes per owned feature; word column and row group of phase B
    const int P = 1 << a.p_shift;
    const int pp = tid & (P - 1);
    const int kpt = kCluThreads >> a.p_shift;                      // owned features handled per pass
    const int group = tid / lanes_q, ql = tid - group * lanes_q;
    const uint32_t slice_bytes = (uint32_t)sub * 4u;

    int slot = 0;                                                  // slot and mbarrier parity of the current step's tile
    uint32_t parity = 0;
    uint32_t ag_parity = 0, rs_parity = 0, gn_parity = 0, xn_parity = 0;
    // rows of the current step (set at the end of the previous round) and the batch index one step further on
    int64_t r0 = 0;
    int bt = 1, rcnt = 0;
    int64_t t_ahead = a.order ? (int64_t)a.order[a.first_step] : a.first_step;
    for (int64_t it = a.first_step - 1; it < step_end; ++it) {
        const bool last = (it == step_end - 1);
        // arm this round's receive barriers (tx counts may arrive earlier; the phase cannot complete before this)
        if (tid == 0) {
            if (it >= a.first_step) mbar_arrive_expect_tx(reinterpret_cast<uint64_t*>(&sh->rs_bar), (uint32_t)Fs * 4u);
            if (!last) mbar_arrive_expect_tx(reinterpret_cast<uint64_t*>(&sh->ag_bar), (uint32_t)Fs * 4u);
        }
        float gq_M = 0.0f;                                         // Q4 scale of this step
        if (it >= a.first_step) {
            clu_mark(a, it, 0);
            clu_wait(sh->full + slot, parity, sh, a.status, 6);
            const uint32_t* t1 = ring + (size_t)slot * slot_words;
            const uint32_t* t2 = t1 + (size_t)a.rc * pitch;
            clu_mark(a, it, 1);

            // ---------------------------------------------------------- phase A: dots and residuals
            double base = 0.0;                                     // lo^T x~ (uniform grids)
            if constexpr (!TABLE) {
#pragma unroll
                for (int w = 0; w < kCluWarps; ++w) base += sh->wbase[w];
            }
            double srow = 0.0;
#pragma unroll 1
            for (int r = warp; r < rcnt; r += kCluWarps) {
                const uint32_t* row1 = t1 + (size_t)r * pitch;
                const uint32_t* row2 = t2 + (size_t)r * pitch;
                float acc1 = 0.0f, acc2 = 0.0f;
#pragma unroll 2
                for (int q = lane; q < nw; q += 32) {
                    const uint32_t u1 = row1[q], u2 = row2[q];
                    if constexpr (!TABLE) {
                        float c1[FPW], c2[FPW];
                        unpack_word<CB>(u1, c1);
                        unpack_word<CB>(u2, c2);
                        // the word's FPW entries of w lie together: 16-byte loads, a quarter of the load instructions
                        const float4* wq = reinterpret_cast<const float4*>(wv) + (size_t)q * (FPW / 4);
#pragma unroll
                        for (int i4 = 0; i4 < FPW / 4; ++i4) {
                            const float4 w4 = wq[i4];
                            acc1 = fmaf(c1[4 * i4], w4.x, acc1); acc2 = fmaf(c2[4 * i4], w4.x, acc2);
                            acc1 = fmaf(c1[4 * i4 + 1], w4.y, acc1); acc2 = fmaf(c2[4 * i4 + 1], w4.y, acc2);
                            acc1 = fmaf(c1[4 * i4 + 2], w4.z, acc1); acc2 = fmaf(c2[4 * i4 + 2], w4.z, acc2);
                            acc1 = fmaf(c1[4 * i4 + 3], w4.w, acc1); acc2 = fmaf(c2[4 * i4 + 3], w4.w, acc2);
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < FPW; ++i) {
                            acc1 += tab[(code_at<CB>(u1, i) * FPW + i) * rw + q];
                            acc2 += tab[(code_at<CB>(u2, i) * FPW + i) * rw + q];
                        }
                    }
                }
                // both sums with one butterfly: the upper half-warp ends up with plane 2, the lower with plane 1
                const bool up = (lane & 16) != 0;
                double d = (double)(up ? acc2 : acc1) + __shfl_xor_sync(0xffffffffu, (double)(up ? acc1 : acc2), 16);
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
                if ((lane & 15) == 0) {
                    const float rv = (float)(d + base - (double)bsm[r]);
                    res[2 * r + (up ? 1 : 0)] = rv;
                    srow += (double)rv;
                }
            }
            srow += __shfl_xor_sync(0xffffffffu, srow, 16);
            if (lane == 0) sh->ssum[warp] = srow;
            __syncthreads();
            clu_mark(a, it, 2);

            // ---------------------------------------------------------- phase B: the rows' part of the gradient
            double S = 0.0;                                        // sum of r1 + r2 over the CTA's rows
            if constexpr (!TABLE) {
#pragma unroll
                for (int w = 0; w < kCluWarps; ++w) S += sh->ssum[w];
            }
            const float Sf = (float)S;
#pragma unroll 1
            for (int q0 = 0; q0 < nw; q0 += lanes_q) {
                const int q = q0 + ql;
                const bool active = group < ngroups && q < nw;
                float acc[FPW];
#pragma unroll
                for (int i = 0; i < FPW; ++i) acc[i] = 0.0f;
                if (active) {
#pragma unroll 2
                    for (int r = group; r < rcnt; r += ngroups) {
                        const uint32_t u1 = t1[(size_t)r * pitch + q], u2 = t2[(size_t)r * pitch + q];
                        const float2 rv = *reinterpret_cast<const float2*>(res + 2 * r);
                        if constexpr (!TABLE) {
                            float c1[FPW], c2[FPW];
                            unpack_word<CB>(u1, c1);
                            unpack_word<CB>(u2, c2);
#pragma unroll
                            for (int i = 0; i < FPW; ++i) acc[i] = fmaf(c1[i], rv.y, fmaf(c2[i], rv.x, acc[i]));
                        } else {
#pragma unroll
                            for (int i = 0; i < FPW; ++i) {
                                const float l1 = lev[(code_at<CB>(u1, i) * FPW + i) * rw + q];
                                const float l2 = lev[(code_at<CB>(u2, i) * FPW + i) * rw + q];
                                acc[i] = fmaf(l1, rv.y, fmaf(l2, rv.x, acc[i]));
                            }
                        }
                    }
                }
                if (ngroups == 1) {                          // (wide rows: a thread has its columns' sums to itself)
                    if (active)
#pragma unroll
                        for (int i = 0; i < FPW; ++i)
                            if (q * FPW + i < n) gpart[q * FPW + i] = TABLE ? acc[i] : fmaf(steps[q * FPW + i], acc[i], los[q * FPW + i] * Sf);
                    continue;
                }
                // the groups' sums meet in shared memory ([group][feature of the pass]); then one thread per
                // feature adds them in order and writes the feature's entry of the CTA's part
                if (q0 > 0) __syncthreads();
                if (active) {
#pragma unroll
                    for (int i = 0; i < FPW; ++i) gred[(group * lanes_q + ql) * FPW + i] = acc[i];
                }
                __syncthreads();
#pragma unroll 1
                for (int fl = tid; fl < lanes_q * FPW; fl += kCluThreads) {
                    const int f = q0 * FPW + fl;
                    if (f < n) {
                        float v = gred[fl];
                        for (int g = 1; g < ngroups; ++g) v += gred[g * lanes_q * FPW + fl];
                        if constexpr (!TABLE) v = fmaf(steps[f], v, los[f] * Sf);      // (fp32: conversions are slow)
                        gpart[f] = v;
                    }
                }
            }
            // reduce-scatter: slice o of the part goes to owner o
            fence_async_smem();
            __syncthreads();
            // (one copy per warp: the copies of one warp's lanes would be issued one after the other)
            if (lane == 0 && warp < nb)
                bulk_copy_s2c(cluster_addr(gbuf + (size_t)bi * sub, warp), gpart + (size_t)warp * sub, slice_bytes,
                              cluster_addr(&sh->rs_bar, warp));
            // the tile is consumed: refill its slot while the parts travel
            if (it + a.slots < step_end && warp == kCluWarps - 1) issue_tile(it + a.slots, slot);
            if (++slot == a.slots) { slot = 0; parity ^= 1u; }
            clu_mark(a, it, 3);

            // ---------------------------------------------------------- owners: sum the parts, update
            clu_wait(&sh->rs_bar, rs_parity, sh, a.status, 2);
            rs_parity ^= 1u;
            const double scale = 1.0 / (2.0 * (double)bt);
            double gsq = 0.0;
#pragma unroll 1
            for (int kb = 0; kb < sub; kb += kpt) {
                const int k = kb + (tid >> a.p_shift);
                const int f = bi * sub + k;
                const bool mine = k < sub && f < n;
                double t = 0.0;
                if (mine)
                    for (int w = pp; w < nb; w += P) t += (double)gbuf[w * sub + k];
                for (int o = 1; o < P; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                if (mine && pp == 0) {
                    const float g = (float)(t * scale);
                    if (last && a.grad_out) a.grad_out[f] = g;
                    gsub[k] = g;
                    gsq += (double)g * (double)g;
                }
            }
            clu_mark(a, it, 4);
            if (a.grad_bits > 0) {
                gq_M = clu_norm(gsq, sh->nrm_g, &sh->gn_bar, gn_parity, nb, sh, a.status, 3);
                gn_parity ^= 1u;
            }
#pragma unroll 1
            for (int kb = 0; kb < sub; kb += kpt) {
                const int k = kb + (tid >> a.p_shift);
                const int f = bi * sub + k;
                if (k < sub && f < n && pp == 0) {
                    float g = gsub[k];
                    if (a.grad_bits > 0)
                        g = clu_quant(g, gq_M, (1 << (a.grad_bits - 1)) - 1, a.seed, a.epoch, (uint32_t)it, 4u, (uint32_t)f);
                    if (last && a.grad_out) a.grad_out[n + f] = g;
                    xown[k] = regularise(fmaf(-a.lr, g, xown[k]), xown[k], a.reg, a.reg_cst);
                }
            }
        }
        if (last) break;

        // -------------------------------------------------------------- publish what the next step sees
        float xq_M = 0.0f;
        if (a.model_bits > 0) {
            double xsq = 0.0;
            for (int kb = 0; kb < sub; kb += kpt) {
                const int k = kb + (tid >> a.p_shift);
                if (k < sub && bi * sub + k < n && pp == 0) xsq += (double)xown[k] * (double)xown[k];
            }
            xq_M = clu_norm(xsq, sh->nrm_x, &sh->xn_bar, xn_parity, nb, sh, a.status, 8);
            xn_parity ^= 1u;
        }
#pragma unroll 1
        for (int kb = 0; kb < sub; kb += kpt) {
            const int k = kb + (tid >> a.p_shift);
            const int f = bi * sub + k;
            if (k < sub && pp == 0) {
                float xt = (f < n) ? xown[k] : 0.0f;
                if (a.model_bits > 0 && f < n)
                    xt = clu_quant(xt, xq_M, (1 << (a.model_bits - 1)) - 1, a.seed, a.epoch, (uint32_t)(it + 1), 3u, (uint32_t)f);
                if (a.model_out && it + 2 == step_end && f < n) a.model_out[f] = xt;
                xpub[k] = xt;
            }
        }
        // labels of the next step's rows: requested now, parked in shared memory after the model has arrived
        r0 = t_ahead * a.batch;
        bt = (int)min(a.batch, a.m - r0);
        rcnt = max(0, min(a.rc, bt - k0));
        if (it + 2 < step_end) t_ahead = a.order ? (int64_t)a.order[it + 2] : it + 2;
        float breg = 0.0f;
        if (tid < rcnt) breg = __ldg(a.b + r0 + k0 + tid);
        fence_async_smem();
        __syncthreads();
        if (lane == 0 && warp < nb)
            bulk_copy_s2c(cluster_addr(xs + (size_t)bi * sub, warp), xpub, slice_bytes, cluster_addr(&sh->ag_bar, warp));
        clu_mark(a, it, 5);

        // -------------------------------------------------------------- the model arrives; build w
        clu_wait(&sh->ag_bar, ag_parity, sh, a.status, 4);
        ag_parity ^= 1u;
        double bpart = 0.0;
#pragma unroll 1
        for (int idx = tid; idx < Fp; idx += kCluThreads) {
            // level tables: consecutive threads take consecutive word columns of one feature slot, so that the L
            // table rows they read and write are contiguous (feature-major threads hit one bank eight times when
            // the row has a multiple of 32 words: 2 k cycles per step on 64-word rows)
            const int q = TABLE ? idx % rw : idx >> LOGF, i = TABLE ? idx / rw : idx & (FPW - 1);
            const int f = TABLE ? q * FPW + i : idx;
            const float xt = (f < n) ? xs[f] : 0.0f;
            if constexpr (!TABLE) {
                wv[f] = steps[f] * xt;
                bpart += (double)los[f] * (double)xt;
            } else {
                for (int c = 0; c < L; ++c) tab[(c * FPW + i) * rw + q] = lev[(c * FPW + i) * rw + q] * xt;
            }
        }
        if constexpr (!TABLE) {
            bpart = warp_sum(bpart);
            if (lane == 0) sh->wbase[warp] = bpart;
        }
        if (tid < rcnt) bsm[tid] = breg;
        for (int r = tid + kCluThreads; r < rcnt; r += kCluThreads) bsm[r] = __ldg(a.b + r0 + k0 + r);
        clu_mark(a, it, 6);
        __syncthreads();
        clu_mark(a, it, 7);
    }
    // owners return the master model
    for (int kb = 0; kb < sub; kb += kpt) {
        const int k = kb + (tid >> a.p_shift);
        if (k < sub && bi * sub + k < n && pp == 0) a.x[bi * sub + k] = xown[k];
    }
    cluster_sync_all();                                  // nobody leaves while a copy may still target it
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
struct ClusterPlan {
    int nb, rc, slots, sub, p_shift;
    size_t smem;
};

static size_t cluster_smem_bytes(int cb, bool table, int row_words, int words, int bits, int nb, int sub, int rc, int slots) {
    const size_t fpw = 32 / cb, Fp = (size_t)row_words * fpw, L = (size_t)1 << bits, Fs = (size_t)nb * sub;
    size_t bytes = (sizeof(ClusterShared) + 15) & ~(size_t)15;
    const int lanes_q = (words + 31) / 32 * 32;                     // one group of threads: no meeting of groups
    bytes += sizeof(float) * ((table ? 2 * L * Fp : 3 * Fp) + (2 * lanes_q <= kCluThreads ? (size_t)kCluThreads * fpw : 0));
    bytes += sizeof(float) * (3 * Fs + 3 * (size_t)sub + (size_t)((2 * rc + 3) & ~3) + (size_t)((rc + 3) & ~3));
    bytes += 128 + 64;                                              // slack to align the ring, and past its last row
    bytes += sizeof(uint32_t) * (size_t)slots * 2 * rc * row_words;
    return bytes;
}

static const void* cluster_kernel_ptr(int cb, bool table) {
    if (cb == 2) return table ? (const void*)sgd_cluster_kernel<2, true> : (const void*)sgd_cluster_kernel<2, false>;
    if (cb == 4) return table ? (const void*)sgd_cluster_kernel<4, true> : (const void*)sgd_cluster_kernel<4, false>;
    return (const void*)sgd_cluster_kernel<8, false>;
}

static int make_cluster_plan(const zipml_ctx* ctx, const zipml_dataset* d, const zipml_sgd_params* p, ClusterPlan* plan) {
    const int cb = container_bits(d->bits);
    const bool table = d->level_mode == ZIPML_LEVELS_TABLE;
    const int64_t B = p->batch < d->m ? p->batch : d->m;
    const int64_t row_words = d->row_bytes / 4;
    if (d->n > (1 << 18) || row_words > (1 << 16)) return ZIPML_ERR_WORKSPACE;
    int64_t nb = p->grid_row_parts > 0 ? p->grid_row_parts : kCluMaxCtas;
    if (p->grid_row_parts <= 0 && nb * 8 > B) nb = B / 8;           // automatic: at least 8 rows per CTA
    if (nb > kCluMaxCtas) nb = kCluMaxCtas;
    if (nb > B) nb = B;
    if (nb < 1) nb = 1;
    const size_t cap = (size_t)ctx->smem_optin;
    const int64_t nb_max = B < kCluMaxCtas ? B : kCluMaxCtas;
    const int words = (int)((d->n * cb + 31) / 32);
    // the requested number of row parts is a hint: more parts are used when a tile does not fit
    for (;; ++nb) {
        if (nb > nb_max) return ZIPML_ERR_WORKSPACE;
        ClusterPlan r;
        r.rc = (int)((B + nb - 1) / nb);
        r.nb = (int)((B + r.rc - 1) / r.rc);                        // no CTA without rows in a full batch
        const int64_t per = (d->n + r.nb - 1) / r.nb;
        r.sub = (int)((per + 3) & ~(int64_t)3);                     // slices are copied in 16-byte units
        r.p_shift = 0;
        while (r.p_shift < 5 && ((int64_t)r.sub << (r.p_shift + 1)) <= kCluThreads && (1 << r.p_shift) < r.nb) ++r.p_shift;
        if ((uint64_t)2 * r.rc * row_words * 4 >= (1u << 20)) continue;                     // mbarrier tx-count range
        if ((uint64_t)r.nb * r.sub * 4 >= (1u << 20)) continue;
        int slots = kCluMaxSlots;
        while (slots >= 2 && cluster_smem_bytes(cb, table, (int)row_words, words, d->bits, r.nb, r.sub, r.rc, slots) > cap) --slots;
        if (slots < 2) continue;
        r.slots = slots;
        r.smem = cluster_smem_bytes(cb, table, (int)row_words, words, d->bits, r.nb, r.sub, r.rc, slots);
        *plan = r;
        return ZIPML_OK;
    }
}

// Level tables: split by features, or by rows where the features make too few 16-byte units for the CTAs.  us per step by features / by
// rows: 3 bits n 17 to 32 (1 unit) x 180 3.72 / 3.86, x 240 4.33 / 4.02, n 64 (2) x 420 4.49 / 4.82, x 500 4.86 / 5.02, x 600 5.89 / 5.65, n 96 (3) x
// 800 6.11 / 6.50, n 120 (4) x 1,024 6.5 / 7.2, x 2,048 11.5 / 11.3, n 512 (16) x 2,048 8.7 / 15.3; 4 bits n 32 x 180 3.90 / 4.01, x 240 4.55 /
// 4.18, n 64 x 420 4.85 / 4.98, x 500 5.25 / 5.18, n 96 x 800 6.59 / 6.67; 2 bits n 33 to 64 (1) x 180 4.23 / 4.29, x 240 4.98 / 4.55, n 100 (2) x 500
// 6.04 / 6.11, x 600 7.40 / 7.00, n 190 (3) x 800 8.10 / 8.34; n 1,019 (16) x 1,024 7.5 / 14.3.  With a quantized vector the features do a little
// longer: 3 bits n 64 x 600 8.30 / 8.43, 4 bits x 500 7.35 / 7.57.
bool table_form_pays(const zipml_dataset* d, const zipml_sgd_params* p) {
    const int64_t B = p->batch < d->m ? p->batch : d->m, units = (d->n * container_bits(d->bits) + 127) / 128;
    if (container_bits(d->bits) == 2) return B <= 240 * units - (units == 1 ? 55 : 0);
    return B <= 300 * units - (units == 1 || (units <= 3 && p->model_bits == 0 && p->grad_bits == 0) ? 100 : 0);
}

// Uniform grids: split by features, or by rows where the features make too little work for the CTAs, or a batch is so long that it goes
// through in chunks.  us per step by features / by rows: 8 bits n 250 x 16 2.55 / 2.64, x 256 3.11 / 2.78, n 512 x 64 2.59 / 2.99, x 256 3.11 /
// 3.10, x 1,024 4.12 / 4.41, n 1,000 x 256 3.15 / 3.56, n 2,000 x 2,048 6.6 / 9.5; 4 bits n 250 x 256 3.19 / 2.92, n 512 x 2,048 5.15 / 5.27, x 4,096
// 7.06 / 5.99; 2 bits n 256 x 128 3.04 / 2.83, n 1,000 x 64 2.82 / 3.33, x 512 4.05 / 4.58, x 4,096 8.04 / 7.66.
static bool features_pay(const zipml_dataset* d, const zipml_sgd_params* p) {
    const int64_t B = p->batch < d->m ? p->batch : d->m, T = (d->m + p->batch - 1) / p->batch;
    // (From 2^24 entries a step a quantized vector on data of up to three batches leaves this form, and wide rows then go to the ring
    // engine: a pinned choice, not the faster.  2 bits 4,096 x 4,096 features 13.8, rows 22.9, ring 43.5.  Whether the model is asked
    // for makes no difference.)
    if ((p->model_bits > 0 || p->grad_bits > 0) && T <= 3 && B * d->n >= 1 << 24) return false;
    return d->n >= (container_bits(d->bits) == 2 ? 900 : 480) && B <= 5 * d->n;
}
int launch_sgd_int8(zipml_ctx* ctx, const zipml_dataset* d, const float* b, float* x, const zipml_sgd_params* p, int64_t first_step,
                    int64_t num_steps, float* grad_out) {
    // (the caller may fix the form by its tuning hint: 3 = by rows, 4 = by features)
    const bool features = p->cluster_contraction == 4 || (p->cluster_contraction != 3 && features_pay(d, p));
    int rc = features ? launch_sgd_feature(ctx, d, b, x, p, first_step, num_steps, grad_out) : launch_sgd_slice(ctx, d, b, x, p, first_step, num_steps, grad_out);
    if (rc != ZIPML_ERR_WORKSPACE) return rc;
    if (features) return launch_sgd_slice(ctx, d, b, x, p, first_step, num_steps, grad_out);
    // (few features, or one of few rows, that the other form does not hold)
    const int64_t B = p->batch < d->m ? p->batch : d->m;
    return p->cluster_contraction == 3 || B * d->n >= 1 << 24 ? ZIPML_ERR_WORKSPACE : launch_sgd_feature(ctx, d, b, x, p, first_step, num_steps, grad_out);
}

int launch_sgd_cluster(zipml_ctx* ctx, const zipml_dataset* d, const float* b, float* x, const zipml_sgd_params* p,
                       int64_t first_step, int64_t num_steps, float* grad_out) {
    const int cb = container_bits(d->bits);
    const bool table = d->level_mode == ZIPML_LEVELS_TABLE;
    const int fpw = 32 / cb;
    const int64_t T = (d->m + p->batch - 1) / p->batch;
    if (p->cluster_contraction != 1) {
        int rc = ZIPML_ERR_WORKSPACE;
        if (!table) rc = launch_sgd_int8(ctx, d, b, x, p, first_step, num_steps, grad_out);
        else if (p->cluster_contraction >= 2 || table_form_pays(d, p)) rc = launch_sgd_table(ctx, d, b, x, p, first_step, num_steps, grad_out);
        if (rc != ZIPML_ERR_WORKSPACE) return rc;
    }
    ClusterPlan plan;
    int rc = make_cluster_plan(ctx, d, p, &plan);
    if (rc != ZIPML_OK) return rc;
    const void* kernel = cluster_kernel_ptr(cb, table);
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plan.smem);
    if (e != cudaSuccess) return cuda_status(e);
    if (plan.nb > 8) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return cuda_status(e);
    }
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)plan.nb);
    cfg.blockDim = dim3(kCluThreads);
    cfg.dynamicSmemBytes = plan.smem;
    cfg.stream = ctx->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)plan.nb;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    e = cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg);
    if (e != cudaSuccess) { (void)cudaGetLastError(); return ZIPML_ERR_WORKSPACE; }
    if (clusters < 1) return ZIPML_ERR_WORKSPACE;

    size_t off = 0;
    auto piece = [&](size_t bytes) { const size_t o = off; off += carve_size(bytes); return o; };
    const size_t o_ord = piece(sizeof(int32_t) * (size_t)(p->batch_order ? T : 0));
    rc = ws_reserve(ctx, off > 0 ? off : 256);
    if (rc != ZIPML_OK) return rc;

    ClusterArgs a;
    memset(&a, 0, sizeof(a));
    a.p1 = reinterpret_cast<const uint32_t*>(d->plane1);
    a.p2 = reinterpret_cast<const uint32_t*>(d->plane2);
    a.lo = d->feat_lo; a.step = d->feat_step; a.levels = d->levels;
    a.b = b; a.x = x; a.grad_out = grad_out; a.model_out = p->model_out;
    a.trace = reinterpret_cast<unsigned long long*>(p->trace);
    a.trace_steps = p->trace ? p->trace_steps : 0;
    a.status = ctx->d_status;
    a.m = d->m; a.batch = p->batch < d->m ? p->batch : d->m;
    a.first_step = first_step; a.num_steps = num_steps;
    a.seed = p->seed; a.epoch = (uint32_t)p->epoch; a.lr = p->lr; a.reg = p->reg; a.reg_cst = reg_constant(p);
    a.n = (int)d->n; a.bits = d->bits; a.row_words = (int)(d->row_bytes / 4);
    a.words = (int)((d->n + fpw - 1) / fpw);
    a.model_bits = p->model_bits; a.grad_bits = p->grad_bits;
    a.nb = plan.nb; a.rc = plan.rc; a.slots = plan.slots;
    a.pitch = a.row_words; a.sub = plan.sub; a.p_shift = plan.p_shift;
    if (p->batch_order) {
        int32_t* dev_order = reinterpret_cast<int32_t*>(ctx->ws + o_ord);
        e = cudaMemcpyAsync(dev_order, p->batch_order, sizeof(int32_t) * (size_t)T, cudaMemcpyHostToDevice, ctx->stream);
        if (e != cudaSuccess) return cuda_status(e);
        a.order = dev_order;
    }
    void* params[] = {&a};
    e = cudaLaunchKernelExC(&cfg, kernel, params);
    if (e != cudaSuccess) return cuda_status(e);
    ctx->launches += 1;
    ctx->ran(ZIPML_ENGINE_CLUSTER, "sgd_cluster_kernel");
    return ZIPML_OK;
}

}  // namespace zipml
