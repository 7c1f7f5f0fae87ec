// C ABI of the Kernel K-means engine: argument checks, workspace, and the
// stream-ordered driver of Alg. 2 (K once, then assignment passes whose loop
// control lives on the device).
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "popcorn.h"
#include "popcorn_internal.cuh"

using namespace popcorn;

namespace {

thread_local std::string g_err;

popcorn_status fail(popcorn_status s, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return s;
}

#define POPCORN_CUDA(call)                                                                    \
    do {                                                                                      \
        cudaError_t e_ = (call);                                                              \
        if (e_ != cudaSuccess) {                                                              \
            cudaGetLastError();                                                               \
            return fail(e_ == cudaErrorMemoryAllocation ? POPCORN_ERR_NOMEM : POPCORN_ERR_CUDA, \
                        "%s failed: %s", #call, cudaGetErrorString(e_));                     \
        }                                                                                     \
    } while (0)

#define POPCORN_TRY(expr)                      \
    do {                                       \
        popcorn_status s_ = (expr);            \
        if (s_ != POPCORN_OK) return s_;       \
    } while (0)

struct DeviceInfo {
    int sms = 0;
    int smem_optin = 0;
    int reduce_smem = 0;   // dynamic shared memory usable by the reduction kernel
    int recompute_smem = 0;
    int batched_smem = 0;
    bool coop = false;   // cooperative launches (all CTAs of a grid resident at once)
    cudaMemPool_t pool = nullptr;
    bool ready = false;
};

std::mutex g_dev_mu;
DeviceInfo g_dev[64];

// Per-device set-up, done once with that device current: SM count, shared
// memory opt-in, and a private stream-ordered pool that keeps freed blocks.
popcorn_status device_info(DeviceInfo** out) {
    int dev = 0;
    POPCORN_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(POPCORN_ERR_UNSUPPORTED, "device ordinal %d >= 64", dev);
    std::lock_guard<std::mutex> lk(g_dev_mu);
    DeviceInfo& d = g_dev[dev];
    if (!d.ready) {
        POPCORN_CUDA(cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev));
        POPCORN_CUDA(cudaDeviceGetAttribute(&d.smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
        cudaMemPoolProps props;
        memset(&props, 0, sizeof props);
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        POPCORN_CUDA(cudaMemPoolCreate(&d.pool, &props));
        uint64_t thr = UINT64_MAX;
        POPCORN_CUDA(cudaMemPoolSetAttribute(d.pool, cudaMemPoolAttrReleaseThreshold, &thr));
        POPCORN_CUDA(configure_reduce_smem(d.smem_optin, &d.reduce_smem));
        POPCORN_CUDA(configure_kbuild_tc());
        POPCORN_CUDA(configure_recompute(d.smem_optin, &d.recompute_smem));
        POPCORN_CUDA(configure_batched(d.smem_optin));
        POPCORN_CUDA(configure_batched_mma(d.smem_optin));
        POPCORN_CUDA(configure_reduce_tiles(d.smem_optin));
        POPCORN_CUDA(configure_reduce_sym(d.smem_optin));
        POPCORN_CUDA(configure_pack_half());
        POPCORN_CUDA(configure_sym_mma(d.smem_optin));
        POPCORN_CUDA(configure_fused_fit(d.smem_optin));
        POPCORN_CUDA(configure_kmeanspp(d.smem_optin));
        int coop = 0;
        POPCORN_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
        d.coop = coop != 0;
        d.batched_smem = d.smem_optin - 1024;
        d.ready = true;
    }
    *out = &d;
    return POPCORN_OK;
}

// Allocations the library has made (workspace blocks and pinned host staging), for
// popcorn_allocation_count.
std::atomic<int64_t> g_alloc_count{0};

// Stream-ordered workspace: every block is returned to the pool (on the
// stream) when the object goes out of scope, on success and on error paths.
class Workspace {
  public:
    Workspace(cudaMemPool_t pool, cudaStream_t s) : pool_(pool), s_(s) {}
    ~Workspace() {
        for (void* p : blocks_) cudaFreeAsync(p, s_);
    }
    template <class T>
    popcorn_status alloc(T** out, size_t count, const char* what) {
        void* p = nullptr;
        size_t bytes = count * sizeof(T);
        if (bytes == 0) bytes = 16;
        bytes = (bytes + 255) & ~(size_t)255;
        cudaError_t e = cudaMallocFromPoolAsync(&p, bytes, pool_, s_);
        if (e != cudaSuccess) {
            cudaGetLastError();
            // a failed request can leave the pool holding what it reserved while trying;
            // hand every unused byte back to the device
            cudaMemPoolTrimTo(pool_, 0);
            cudaGetLastError();
            return fail(e == cudaErrorMemoryAllocation ? POPCORN_ERR_NOMEM : POPCORN_ERR_CUDA,
                        "workspace for %s (%zu bytes): %s", what, bytes, cudaGetErrorString(e));
        }
        blocks_.push_back(p);
        g_alloc_count.fetch_add(1, std::memory_order_relaxed);
        *out = static_cast<T*>(p);
        return POPCORN_OK;
    }
    // returns one block to the pool now (stream-ordered) instead of at the end
    void release(void* p) {
        for (size_t i = 0; i < blocks_.size(); ++i)
            if (blocks_[i] == p) {
                cudaFreeAsync(p, s_);
                blocks_.erase(blocks_.begin() + (long)i);
                return;
            }
    }

  private:
    cudaMemPool_t pool_;
    cudaStream_t s_;
    std::vector<void*> blocks_;
};

// Pinned host staging for small device->host reads, grown on demand.
struct PinnedScratch {
    void* p = nullptr;
    size_t bytes = 0;
};
thread_local PinnedScratch g_pinned;

popcorn_status pinned(size_t bytes, void** out) {
    if (g_pinned.bytes < bytes) {
        if (g_pinned.p) cudaFreeHost(g_pinned.p);
        g_pinned.p = nullptr;
        g_pinned.bytes = 0;
        POPCORN_CUDA(cudaMallocHost(&g_pinned.p, bytes));
        g_alloc_count.fetch_add(1, std::memory_order_relaxed);
        g_pinned.bytes = bytes;
    }
    *out = g_pinned.p;
    return POPCORN_OK;
}

bool is_device_pointer(const void* p) {
    cudaPointerAttributes at;
    cudaError_t e = cudaPointerGetAttributes(&at, p);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

popcorn_status check_kernel(const popcorn_kernel& kern, KernParams* kp) {
    kp->kind = kern.kind;
    kp->degree = kern.degree;
    kp->gamma = (float)kern.gamma;
    kp->coef0 = (float)kern.coef0;
    kp->neg_gamma_over_sigma2 = 0.f;
    switch (kern.kind) {
        case POPCORN_LINEAR:
            return POPCORN_OK;
        case POPCORN_POLYNOMIAL:
            if (kern.degree < 1 || kern.degree > 64)
                return fail(POPCORN_ERR_INVALID, "polynomial degree %d outside [1, 64]", kern.degree);
            if (!std::isfinite(kern.gamma) || !std::isfinite(kern.coef0))
                return fail(POPCORN_ERR_INVALID, "polynomial gamma/coef0 must be finite");
            return POPCORN_OK;
        case POPCORN_GAUSSIAN:
            if (!(kern.sigma > 0) || !std::isfinite(kern.sigma))
                return fail(POPCORN_ERR_INVALID, "Gaussian sigma must be > 0 (got %g)", kern.sigma);
            if (!(kern.gamma > 0) || !std::isfinite(kern.gamma))
                return fail(POPCORN_ERR_INVALID, "Gaussian gamma must be > 0 (got %g)", kern.gamma);
            kp->neg_gamma_over_sigma2 = (float)(-kern.gamma / (kern.sigma * kern.sigma));
            return POPCORN_OK;
        default:
            return fail(POPCORN_ERR_INVALID, "unknown kernel kind %d", kern.kind);
    }
}

// K = kappa(P P^T) on stream s.  FP32: CUDA-core tiles, or tcgen05 tiles of the points split
// into two FP16 parts where their values are close enough together (decided on the device).  BF16 / BF16X3: tcgen05
// tiles.  Operand copies come from `ws`, and *err (device) reports a timed-out wait inside a
// kernel.
// packed: the build writes the block-packed upper triangle (symmetric pass only).
popcorn_status build_kernel_matrix(const float* P, int n, int d, int64_t ldp, const KernParams& kp,
                                   int precision, void* K, int64_t ldk, int k_storage, float* kdiag, Workspace* ws,
                                   int* err, int num_sms, cudaStream_t s, int* launches, int packed = 0,
                                   int full = 0) {
    if (precision == POPCORN_FP32) {
        float* rn = nullptr;
        unsigned* maxr = nullptr;
        if (kp.kind == POPCORN_GAUSSIAN && ws) {
            POPCORN_TRY(ws->alloc(&rn, (size_t)n, "row norms"));
            POPCORN_TRY(ws->alloc(&maxr, 1, "largest row norm"));
        }
        // The tensor-core split build's operands (kbuild_tc.cu).  Without room for them the
        // CUDA-core build runs alone.
        unsigned char* split = nullptr;
        if (ws && err && k_storage == POPCORN_K_FP32 && kbuild_split_applies(n, d, kp.kind != POPCORN_GAUSSIAN) &&
            ws->alloc(&split, kbuild_split_workspace(n, d), "split operands") != POPCORN_OK) {
            split = nullptr;
            g_err.clear();
        }
        POPCORN_CUDA(launch_kbuild_simt(P, n, d, ldp, kp, K, ldk, k_storage, kdiag, s, launches, packed, full, rn,
                                        maxr, split, err, num_sms));
        if (split) ws->release(split);
        return POPCORN_OK;
    }
    if (k_storage != POPCORN_K_FP32 && packed != kPackedSw128H)
        return fail(POPCORN_ERR_UNSUPPORTED,
                    "an FP16/BF16 K from a BF16/BF16X3 build is written as half tiles (not inside a caller's "
                    "stream capture when read as the full square)");
    if (precision != POPCORN_BF16 && precision != POPCORN_BF16X3)
        return fail(POPCORN_ERR_UNSUPPORTED, "precision %d is not available for a stored K", precision);
    unsigned char* w;
    POPCORN_TRY(ws->alloc(&w, kbuild_tc_workspace(n, d, precision), "BF16 operands"));
    cudaError_t e = launch_kbuild_tc(P, n, d, ldp, kp, precision, static_cast<float*>(K), ldk, kdiag, w, err, num_sms,
                                     s, launches, packed, full, k_storage);
    if (e == cudaErrorInvalidValue)
        return fail(POPCORN_ERR_CUDA, "tensor map creation failed (cuTensorMapEncodeTiled unavailable or rejected)");
    POPCORN_CUDA(e);
    return POPCORN_OK;
}

struct EventPool {
    std::vector<cudaEvent_t> ev;
    size_t used = 0;
    popcorn_status get(cudaEvent_t* out) {
        if (used == ev.size()) {
            cudaEvent_t e;
            POPCORN_CUDA(cudaEventCreate(&e));
            ev.push_back(e);
        }
        *out = ev[used++];
        return POPCORN_OK;
    }
};
thread_local EventPool g_events;

float elapsed(cudaEvent_t a, cudaEvent_t b) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, a, b) != cudaSuccess) {
        cudaGetLastError();
        return 0.f;
    }
    return ms;
}

}  // namespace

void popcorn::set_error_message(const char* msg) { g_err = msg; }


namespace {

// Kernel K-means without a stored K: operand rows once, then every pass
// recomputes the tiles it needs (recompute.cu), reduces z and assigns.
popcorn_status fit_recompute(const float* P, int64_t n, int32_t d, int64_t ldp, int32_t k, const KernParams& kp,
                             const int32_t* init_labels, int32_t max_iter, double tol, const popcorn_options& opt,
                             int32_t* labels_out, double* objective_out, int32_t* iterations_out,
                             popcorn_fit_info* info, cudaStream_t s, DeviceInfo* dev) {
    const int ni = (int)n;
    RecomputePlan rp = plan_recompute(ni, d, k, opt.precision, dev->sms, dev->recompute_smem);
    // schedules the autotuner may time: row blocks per tile x units per SM
    std::vector<RecomputePlan> cands;
    int max_nslot = rp.nslot;
    if (opt.autotune && rp.ok) {
        for (int rbp : {2, 1})
            for (int upsm : {8, 16, 32}) {
                const RecomputePlan c = plan_recompute(ni, d, k, opt.precision, dev->sms, dev->recompute_smem, rbp, upsm);
                if (!c.ok) continue;
                cands.push_back(c);
                max_nslot = c.nslot > max_nslot ? c.nslot : max_nslot;
            }
    }
    if (!rp.ok)
        return fail(POPCORN_ERR_UNSUPPORTED, "the recompute path needs d <= %d (%s) and k <= 255",
                    opt.precision == POPCORN_FP8 ? 512 : 256, opt.precision == POPCORN_FP8 ? "FP8" : "BF16");
    const bool timing = opt.timing != 0;
    int launches = 0;
    int64_t h2d = 0, d2h = 0;
    Workspace ws(dev->pool, s);
    const float* Pd = P;
    int64_t ldpd = ldp;
    if (!is_device_pointer(P)) {
        float* tmp;
        POPCORN_TRY(ws.alloc(&tmp, (size_t)ni * d, "points"));
        POPCORN_CUDA(cudaMemcpy2DAsync(tmp, (size_t)d * sizeof(float), P, (size_t)ldp * sizeof(float),
                                       (size_t)d * sizeof(float), (size_t)ni, cudaMemcpyHostToDevice, s));
        h2d += (int64_t)ni * d * sizeof(float);
        Pd = tmp;
        ldpd = d;
    }
    const int32_t* Ld = init_labels;
    if (!is_device_pointer(init_labels)) {
        int32_t* tmp;
        POPCORN_TRY(ws.alloc(&tmp, (size_t)ni, "initial labels"));
        POPCORN_CUDA(cudaMemcpyAsync(tmp, init_labels, (size_t)ni * sizeof(int32_t), cudaMemcpyHostToDevice, s));
        h2d += (int64_t)ni * sizeof(int32_t);
        Ld = tmp;
    }
    RecomputeBuffers rb{};
    const int nb = recompute_sort_blocks(ni);
    POPCORN_TRY(ws.alloc(&rb.Q, (size_t)ni * rp.row_bytes, "operand rows"));
    POPCORN_TRY(ws.alloc(&rb.norms, (size_t)ni, "row norms"));
    POPCORN_TRY(ws.alloc(&rb.knorms, (size_t)ni, "epilogue row norms"));
    POPCORN_TRY(ws.alloc(&rb.scales, (size_t)ni, "row scales"));
    POPCORN_TRY(ws.alloc(&rb.Qs, (size_t)rp.ncols * rp.row_bytes, "sorted operand rows"));
    POPCORN_TRY(ws.alloc(&rb.snorm, (size_t)rp.ncols, "sorted norms"));
    POPCORN_TRY(ws.alloc(&rb.sscale, (size_t)rp.ncols, "sorted scales"));
    POPCORN_TRY(ws.alloc(&rb.slab, (size_t)rp.ncols, "sorted labels"));
    POPCORN_TRY(ws.alloc(&rb.blockhist, (size_t)nb * k, "sort histograms"));
    POPCORN_TRY(ws.alloc(&rb.blockoff, (size_t)nb * k, "sort offsets"));
    POPCORN_TRY(ws.alloc(&rb.maxkn, 1, "largest row exponent"));
    POPCORN_TRY(ws.alloc(&rb.crange, (size_t)k, "cluster slots"));
    PassBuffers b{};
    b.crange = rb.crange;
    float* kdiag;
    POPCORN_TRY(ws.alloc(&kdiag, (size_t)ni, "diag(K)"));
    const size_t nlab = ((size_t)ni + 15) & ~(size_t)15;
    const int hist_len = max_iter > 0 ? max_iter : 1;
    const int zblocks = (ni + kZReduceRows - 1) / kZReduceRows;
    b.K = nullptr;
    b.ldk = 0;
    b.kdiag = kdiag;
    b.n = ni;
    b.k = k;
    POPCORN_TRY(ws.alloc(&b.lab32, ni, "labels"));
    POPCORN_TRY(ws.alloc(&b.lab8, nlab, "label bytes"));
    POPCORN_TRY(ws.alloc(&b.counts, 2 * (size_t)k, "counts"));
    POPCORN_TRY(ws.alloc(&b.Spart, (size_t)max_nslot * ni * k, "segment sums"));
    POPCORN_TRY(ws.alloc(&b.zpart, (size_t)zblocks * k, "block partials"));
    POPCORN_TRY(ws.alloc(&b.zsum, (size_t)k, "z sums"));
    POPCORN_TRY(ws.alloc(&b.cnorm, (size_t)k, "centroid norms"));
    POPCORN_TRY(ws.alloc(&b.invm, (size_t)k, "inverse cluster sizes"));
    POPCORN_TRY(ws.alloc(&b.st, 1, "loop state"));
    POPCORN_TRY(ws.alloc(&b.J_hist, (size_t)hist_len, "objective history"));
    POPCORN_TRY(ws.alloc(&b.changed_hist, (size_t)hist_len, "change history"));
    b.E_out = nullptr;

    g_events.used = 0;
    cudaEvent_t ev_b0 = nullptr, ev_b1 = nullptr, ev_l1 = nullptr, ev_e1 = nullptr;
    std::vector<cudaEvent_t> ev_r, ev_a;
    if (timing) {
        POPCORN_TRY(g_events.get(&ev_b0));
        POPCORN_CUDA(cudaEventRecord(ev_b0, s));
    }
    POPCORN_CUDA(cudaMemsetAsync(b.counts, 0, 2 * (size_t)k * sizeof(int32_t), s));
    // padding rows of the sorted copy are read by the MMAs (their results are skipped):
    // keep them finite
    POPCORN_CUDA(cudaMemsetAsync(rb.Qs, 0, (size_t)rp.ncols * rp.row_bytes, s));
    POPCORN_CUDA(cudaMemsetAsync(rb.snorm, 0, (size_t)rp.ncols * sizeof(float), s));
    POPCORN_CUDA(cudaMemsetAsync(rb.sscale, 0, (size_t)rp.ncols * sizeof(float), s));
    POPCORN_CUDA(cudaMemsetAsync(rb.maxkn, 0, sizeof(int), s));
    POPCORN_CUDA(launch_init_state(b.st, max_iter, opt.check_convergence ? 1 : 0, tol, s));
    POPCORN_CUDA(launch_quantize(Pd, ni, d, ldpd, kp, rp, rb, kdiag, s));
    POPCORN_CUDA(launch_trace(kdiag, ni, b.st, s));
    POPCORN_CUDA(launch_init_labels(Ld, ni, k, b.lab32, b.lab8, b.counts, b.st, s));
    launches += 4;
    int tune_hit = 0, tune_cands = 0;
    double tune_ms = 0.0;
    if (opt.autotune && !cands.empty()) {
        const TuneKey key{2, opt.precision, log2_bucket((double)ni), d, k, kp.kind, 0, dev->sms};
        TuneValue best{};
        if (tune_lookup(key, &best)) {
            tune_hit = 1;
        } else {
            // time one pass of every candidate on the initial labels (a pass only
            // rewrites its scratch: the sorted copies and the segment sums)
            const auto w0 = std::chrono::steady_clock::now();
            cudaEvent_t t0, t1;
            POPCORN_TRY(g_events.get(&t0));
            POPCORN_TRY(g_events.get(&t1));
            best.ms = 3.0e38f;
            for (const RecomputePlan& c : cands) {
                float ms = 3.0e38f;
                for (int rep = 0; rep < 3; ++rep) {
                    POPCORN_CUDA(cudaEventRecord(t0, s));
                    cudaError_t e = launch_recompute_pass(b, kp, c, rb, &b.st->wait_err, 0, s);
                    if (e == cudaErrorInvalidValue) return fail(POPCORN_ERR_CUDA, "tensor map creation failed");
                    POPCORN_CUDA(e);
                    POPCORN_CUDA(cudaEventRecord(t1, s));
                    POPCORN_CUDA(cudaEventSynchronize(t1));
                    float el = 0.f;
                    POPCORN_CUDA(cudaEventElapsedTime(&el, t0, t1));
                    if (rep > 0 && el < ms) ms = el;   // rep 0 warms up
                }
                ++tune_cands;
                if (ms < best.ms) {
                    best.ms = ms;
                    best.p[0] = c.rbp;
                    best.p[1] = c.units_per_sm;
                    best.p[2] = 0;
                    best.p[3] = 0;
                }
            }
            tune_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - w0).count();
            tune_store(key, best);
        }
        for (const RecomputePlan& c : cands)
            if (c.rbp == best.p[0] && c.units_per_sm == best.p[1]) rp = c;
    }
    if (timing) {
        POPCORN_TRY(g_events.get(&ev_b1));
        POPCORN_CUDA(cudaEventRecord(ev_b1, s));
    }
    const int chunk = 4;
    void* hpin;
    POPCORN_TRY(pinned(2 * sizeof(int32_t) + sizeof(LoopState), &hpin));
    volatile int32_t* hflag = static_cast<int32_t*>(hpin);
    cudaEvent_t poll_ev[2] = {nullptr, nullptr};
    if (opt.check_convergence) {
        POPCORN_TRY(g_events.get(&poll_ev[0]));
        POPCORN_TRY(g_events.get(&poll_ev[1]));
    }
    int launched = 0, pending = -1, slot = 0;
    while (launched < max_iter) {
        const int m = (max_iter - launched < chunk) ? (max_iter - launched) : chunk;
        for (int t = 0; t < m; ++t) {
            cudaEvent_t e0 = nullptr, e1 = nullptr, e2 = nullptr;
            if (timing) {
                POPCORN_TRY(g_events.get(&e0));
                POPCORN_TRY(g_events.get(&e1));
                POPCORN_TRY(g_events.get(&e2));
                POPCORN_CUDA(cudaEventRecord(e0, s));
            }
            cudaError_t e = launch_recompute_pass(b, kp, rp, rb, &b.st->wait_err, 0, s);
            if (e == cudaErrorInvalidValue) return fail(POPCORN_ERR_CUDA, "tensor map creation failed");
            POPCORN_CUDA(e);
            POPCORN_CUDA(launch_zreduce(b, rp.nslot, 0, s));
            if (timing) POPCORN_CUDA(cudaEventRecord(e1, s));
            POPCORN_CUDA(launch_assign_nseg(b, rp.nslot, s));
            if (timing) {
                POPCORN_CUDA(cudaEventRecord(e2, s));
                ev_r.push_back(e0);
                ev_r.push_back(e1);
                ev_a.push_back(e1);
                ev_a.push_back(e2);
            }
            launches += 6;
        }
        launched += m;
        if (opt.check_convergence && launched < max_iter) {
            POPCORN_CUDA(cudaMemcpyAsync((void*)(hflag + slot), &b.st->done, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
            POPCORN_CUDA(cudaEventRecord(poll_ev[slot], s));
            if (pending >= 0) {
                POPCORN_CUDA(cudaEventSynchronize(poll_ev[pending]));
                if (hflag[pending]) break;
            }
            pending = slot;
            slot ^= 1;
        }
    }
    if (timing) {
        POPCORN_TRY(g_events.get(&ev_l1));
        POPCORN_CUDA(cudaEventRecord(ev_l1, s));
    }
    {
        cudaError_t e = launch_recompute_pass(b, kp, rp, rb, &b.st->wait_err, 1, s);
        if (e == cudaErrorInvalidValue) return fail(POPCORN_ERR_CUDA, "tensor map creation failed");
        POPCORN_CUDA(e);
        POPCORN_CUDA(launch_zreduce(b, rp.nslot, 1, s));
        launches += 5;
    }
    if (timing) {
        POPCORN_TRY(g_events.get(&ev_e1));
        POPCORN_CUDA(cudaEventRecord(ev_e1, s));
    }
    LoopState* hs_pin = reinterpret_cast<LoopState*>(static_cast<char*>(hpin) + 2 * sizeof(int32_t));
    POPCORN_CUDA(cudaMemcpyAsync(hs_pin, b.st, sizeof(LoopState), cudaMemcpyDeviceToHost, s));
    d2h += sizeof(LoopState);
    if (is_device_pointer(labels_out)) {
        POPCORN_CUDA(cudaMemcpyAsync(labels_out, b.lab32, (size_t)ni * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
    } else {
        POPCORN_CUDA(cudaMemcpyAsync(labels_out, b.lab32, (size_t)ni * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
        d2h += (int64_t)ni * sizeof(int32_t);
    }
    POPCORN_CUDA(cudaStreamSynchronize(s));
    LoopState hs;
    memcpy(&hs, hs_pin, sizeof hs);
    if (hs.bad_label) return fail(POPCORN_ERR_INVALID, "an initial label is outside [0, %d)", k);
    if (hs.wait_err) return fail(POPCORN_ERR_TIMEOUT, "a bounded wait in the recompute kernel ran out");
    *objective_out = hs.J_eval;
    *iterations_out = hs.iter;
    if (info) {
        const int iters = hs.iter;
        if (iters > 0 && info->J_history)
            POPCORN_CUDA(cudaMemcpy(info->J_history, b.J_hist, (size_t)iters * sizeof(double), cudaMemcpyDeviceToHost));
        if (iters > 0 && info->changed_history)
            POPCORN_CUDA(cudaMemcpy(info->changed_history, b.changed_hist, (size_t)iters * sizeof(int32_t),
                                    cudaMemcpyDeviceToHost));
        const bool eval_ran = !(hs.iter > 0 && hs.last_changed == 0);
        info->converged = hs.converged;
        info->kernel_launches = launches;
        info->reduce_launches = iters + (eval_ran ? 1 : 0);
        info->assign_launches = iters;
        info->h2d_bytes = h2d;
        info->d2h_bytes = d2h;
        info->tune_cache_hit = tune_hit;
        info->tune_candidates = tune_cands;
        info->tune_ms = tune_ms;
        info->fold_ms = 0.0;
        info->k_pass_used = 0;
        info->sym_form = 0;
        info->schedule[0] = rp.rbp;
        info->schedule[1] = rp.nseg;
        info->schedule[2] = rp.units_per_sm;
        info->schedule[3] = 0;
        info->kbuild_ms = info->loop_ms = info->reduce_ms = info->assign_ms = info->eval_ms = 0.0;
        if (timing) {
            info->kbuild_ms = elapsed(ev_b0, ev_b1);
            info->loop_ms = elapsed(ev_b1, ev_l1);
            info->eval_ms = elapsed(ev_l1, ev_e1);
            double r = 0, a2 = 0;
            for (size_t t = 0; t + 1 < ev_r.size() && t < 2 * (size_t)iters; t += 2) r += elapsed(ev_r[t], ev_r[t + 1]);
            for (size_t t = 0; t + 1 < ev_a.size() && t < 2 * (size_t)iters; t += 2) a2 += elapsed(ev_a[t], ev_a[t + 1]);
            info->reduce_ms = r;
            info->assign_ms = a2;
        }
    }
    return POPCORN_OK;
}

}  // namespace

extern "C" {

const char* popcorn_status_string(popcorn_status status) {
    switch (status) {
        case POPCORN_OK: return "POPCORN_OK";
        case POPCORN_ERR_INVALID: return "POPCORN_ERR_INVALID";
        case POPCORN_ERR_NOMEM: return "POPCORN_ERR_NOMEM";
        case POPCORN_ERR_CUDA: return "POPCORN_ERR_CUDA";
        case POPCORN_ERR_TIMEOUT: return "POPCORN_ERR_TIMEOUT";
        case POPCORN_ERR_UNSUPPORTED: return "POPCORN_ERR_UNSUPPORTED";
    }
    return "POPCORN_ERR_UNKNOWN";
}

const char* popcorn_last_error_message(void) { return g_err.c_str(); }

int32_t popcorn_version(void) { return 100; }

int64_t popcorn_allocation_count(void) { return g_alloc_count.load(std::memory_order_relaxed); }

popcorn_status popcorn_kernel_matrix_ex(const float* P, int64_t n, int32_t d, int64_t ldp, popcorn_kernel kern,
                                        int32_t precision, int32_t schedule, float* K, int64_t ldk, float* kdiag,
                                        popcorn_stream_t stream) {
    g_err.clear();
    if (!P || !K || !kdiag) return fail(POPCORN_ERR_INVALID, "null pointer argument");
    if (n < 1 || n >= (1LL << 31)) return fail(POPCORN_ERR_INVALID, "n = %lld outside [1, 2^31)", (long long)n);
    if (d < 1) return fail(POPCORN_ERR_INVALID, "d = %d < 1", d);
    if (ldp < d) return fail(POPCORN_ERR_INVALID, "ldp = %lld < d = %d", (long long)ldp, d);
    if (ldk < n || ldk % 4 != 0)
        return fail(POPCORN_ERR_INVALID, "ldk = %lld must be >= n and a multiple of 4", (long long)ldk);
    if (reinterpret_cast<uintptr_t>(K) % 16 != 0) return fail(POPCORN_ERR_INVALID, "K must be 16-byte aligned");
    if (schedule < POPCORN_SCHEDULE_AUTO || schedule > POPCORN_SCHEDULE_TUNE)
        return fail(POPCORN_ERR_INVALID, "unknown K-build schedule %d", schedule);
    if (precision != POPCORN_FP32 && precision != POPCORN_BF16 && precision != POPCORN_BF16X3)
        return fail(POPCORN_ERR_UNSUPPORTED, "precision %d is not available for a stored K", precision);
    KernParams kp;
    POPCORN_TRY(check_kernel(kern, &kp));
    DeviceInfo* dev;
    POPCORN_TRY(device_info(&dev));
    int launches = 0;
    cudaStream_t s = (cudaStream_t)stream;
    Workspace ws(dev->pool, s);
    int* err;
    POPCORN_TRY(ws.alloc(&err, 1, "error flag"));
    POPCORN_CUDA(cudaMemsetAsync(err, 0, sizeof(int), s));
    // AUTO takes the tuned schedule of this workload signature if one is cached, else the
    // symmetric one; TUNE times both once per signature (best of two after a warm-up), caches
    // the faster and leaves its K in place
    const TuneKey key{3, precision, log2_bucket((double)n), log2_bucket((double)d), kp.kind, 0, 0, dev->sms};
    int use = schedule;
    if (schedule == POPCORN_SCHEDULE_AUTO || schedule == POPCORN_SCHEDULE_TUNE) {
        TuneValue tv{};
        if (tune_lookup(key, &tv)) {
            use = tv.p[0];
        } else if (schedule == POPCORN_SCHEDULE_TUNE) {
            cudaEvent_t t0, t1;
            g_events.used = 0;
            POPCORN_TRY(g_events.get(&t0));
            POPCORN_TRY(g_events.get(&t1));
            TuneValue best{};
            best.ms = 3.0e38f;
            for (int cand : {POPCORN_SCHEDULE_SYMMETRIC, POPCORN_SCHEDULE_FULL}) {
                float ms = 3.0e38f;
                for (int rep = 0; rep < 3; ++rep) {
                    POPCORN_CUDA(cudaEventRecord(t0, s));
                    POPCORN_TRY(build_kernel_matrix(P, (int)n, d, ldp, kp, precision, K, ldk, POPCORN_K_FP32, kdiag,
                                                    &ws, err, dev->sms, s, &launches, 0,
                                                    cand == POPCORN_SCHEDULE_FULL ? 1 : 0));
                    POPCORN_CUDA(cudaEventRecord(t1, s));
                    POPCORN_CUDA(cudaEventSynchronize(t1));
                    float el = 0.f;
                    POPCORN_CUDA(cudaEventElapsedTime(&el, t0, t1));
                    if (rep > 0 && el < ms) ms = el;
                }
                if (ms < best.ms) {
                    best.ms = ms;
                    best.p[0] = cand;
                }
            }
            tune_store(key, best);
            use = best.p[0];
        } else {
            use = POPCORN_SCHEDULE_SYMMETRIC;
        }
    }
    POPCORN_TRY(build_kernel_matrix(P, (int)n, d, ldp, kp, precision, K, ldk, POPCORN_K_FP32, kdiag, &ws, err,
                                    dev->sms, s, &launches, 0, use == POPCORN_SCHEDULE_FULL ? 1 : 0));
    int herr = 0;
    POPCORN_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s));
    POPCORN_CUDA(cudaStreamSynchronize(s));
    if (herr) return fail(POPCORN_ERR_TIMEOUT, "a bounded wait in the tensor-core K build ran out");
    return POPCORN_OK;
}

popcorn_status popcorn_kernel_matrix(const float* P, int64_t n, int32_t d, int64_t ldp, popcorn_kernel kern,
                                     int32_t precision, float* K, int64_t ldk, float* kdiag, popcorn_stream_t stream) {
    return popcorn_kernel_matrix_ex(P, n, d, ldp, kern, precision, POPCORN_SCHEDULE_AUTO, K, ldk, kdiag, stream);
}

popcorn_status popcorn_assign_step(const float* K, int64_t ldk, const float* kdiag, int64_t n, int32_t k,
                                   const int32_t* labels, int32_t* new_labels, int32_t* counts, float* E,
                                   double* cnorm, double* objective, int32_t* changed,
                                   popcorn_stream_t stream) {
    g_err.clear();
    cudaStream_t s = (cudaStream_t)stream;
    if (!K || !kdiag || !labels || !new_labels) return fail(POPCORN_ERR_INVALID, "null pointer argument");
    if (n < 2 || n >= (1LL << 31)) return fail(POPCORN_ERR_INVALID, "n = %lld outside [2, 2^31)", (long long)n);
    if (k < 1 || k > n || k > kMaxClusters)
        return fail(POPCORN_ERR_INVALID, "k = %d outside [1, min(n, %d)]", k, kMaxClusters);
    if (ldk < n || ldk % 4 != 0)
        return fail(POPCORN_ERR_INVALID, "ldk = %lld must be >= n and a multiple of 4", (long long)ldk);
    if (reinterpret_cast<uintptr_t>(K) % 16 != 0) return fail(POPCORN_ERR_INVALID, "K must be 16-byte aligned");
    DeviceInfo* dev;
    POPCORN_TRY(device_info(&dev));
    const int ni = (int)n;
    ReducePlan plan = plan_reduce(ni, k, dev->sms, dev->reduce_smem);
    if (plan.grid == 0) return fail(POPCORN_ERR_UNSUPPORTED, "n = %d is too large for the materialized path", ni);

    Workspace ws(dev->pool, s);
    PassBuffers b{};
    b.K = K;
    b.ldk = ldk;
    b.kdiag = kdiag;
    b.n = ni;
    b.k = k;
    const size_t nlab = ((size_t)ni + 15) & ~(size_t)15;
    POPCORN_TRY(ws.alloc(&b.lab32, ni, "labels"));
    POPCORN_TRY(ws.alloc(&b.lab8, nlab, "label bytes"));
    POPCORN_TRY(ws.alloc(&b.counts, 2 * (size_t)k, "counts"));
    POPCORN_TRY(ws.alloc(&b.Spart, (size_t)plan.nseg * ni * k, "segment sums"));
    POPCORN_TRY(ws.alloc(&b.zpart, (size_t)plan.grid * k, "block partials"));
    POPCORN_TRY(ws.alloc(&b.zsum, (size_t)k, "z sums"));
    POPCORN_TRY(ws.alloc(&b.cnorm, (size_t)k, "centroid norms"));
    POPCORN_TRY(ws.alloc(&b.invm, (size_t)k, "inverse cluster sizes"));
    POPCORN_TRY(ws.alloc(&b.st, 1, "loop state"));
    POPCORN_TRY(ws.alloc(&b.J_hist, 1, "objective history"));
    POPCORN_TRY(ws.alloc(&b.changed_hist, 1, "change history"));
    b.E_out = E;

    POPCORN_CUDA(cudaMemsetAsync(b.counts, 0, 2 * (size_t)k * sizeof(int32_t), s));
    POPCORN_CUDA(launch_init_state(b.st, 1, 0, 0.0, s));
    POPCORN_CUDA(launch_init_labels(labels, ni, k, b.lab32, b.lab8, b.counts, b.st, s));
    POPCORN_CUDA(launch_trace(kdiag, ni, b.st, s));
    POPCORN_CUDA(launch_reduce(b, plan, 0, s));
    if (cnorm) POPCORN_CUDA(cudaMemcpyAsync(cnorm, b.cnorm, (size_t)k * sizeof(double), cudaMemcpyDeviceToDevice, s));
    POPCORN_CUDA(launch_assign(b, plan, s));
    POPCORN_CUDA(cudaMemcpyAsync(new_labels, b.lab32, (size_t)ni * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
    if (counts) POPCORN_CUDA(cudaMemcpyAsync(counts, b.counts + k, (size_t)k * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
    void* host;
    POPCORN_TRY(pinned(sizeof(LoopState), &host));
    POPCORN_CUDA(cudaMemcpyAsync(host, b.st, sizeof(LoopState), cudaMemcpyDeviceToHost, s));
    POPCORN_CUDA(cudaStreamSynchronize(s));
    LoopState hs;
    memcpy(&hs, host, sizeof hs);
    if (hs.bad_label) return fail(POPCORN_ERR_INVALID, "a label is outside [0, %d)", k);
    if (objective) *objective = hs.J_last;
    if (changed) *changed = hs.last_changed;
    return POPCORN_OK;
}

popcorn_status popcorn_fit(const float* P, int64_t n, int32_t d, int64_t ldp, int32_t k, popcorn_kernel kern,
                           const int32_t* init_labels, int32_t max_iter, double tol,
                           const popcorn_options* opt_in, int32_t* labels_out, double* objective_out,
                           int32_t* iterations_out, popcorn_fit_info* info, popcorn_stream_t stream) {
    g_err.clear();
    cudaStream_t s = (cudaStream_t)stream;
    popcorn_options opt;
    memset(&opt, 0, sizeof opt);
    opt.precision = POPCORN_FP32;
    opt.store_k = 1;
    opt.check_convergence = 1;
    if (opt_in) opt = *opt_in;
    if (!P || !init_labels || !labels_out || !objective_out || !iterations_out)
        return fail(POPCORN_ERR_INVALID, "null pointer argument");
    if (n < 2 || n >= (1LL << 31)) return fail(POPCORN_ERR_INVALID, "n = %lld outside [2, 2^31)", (long long)n);
    if (d < 1) return fail(POPCORN_ERR_INVALID, "d = %d < 1", d);
    if (ldp < d) return fail(POPCORN_ERR_INVALID, "ldp = %lld < d = %d", (long long)ldp, d);
    if (k < 1 || k >= n || k > kMaxClusters)
        return fail(POPCORN_ERR_INVALID, "k = %d outside [1, min(n - 1, %d)]", k, kMaxClusters);
    if (max_iter < 0) return fail(POPCORN_ERR_INVALID, "max_iter = %d < 0", max_iter);
    if (!(tol >= 0) || !std::isfinite(tol)) return fail(POPCORN_ERR_INVALID, "tol must be finite and >= 0");
    if (opt.autotune != 0 && opt.autotune != 1) return fail(POPCORN_ERR_INVALID, "options.autotune must be 0 or 1");
    if (opt.k_pass < 0 || opt.k_pass > 2) return fail(POPCORN_ERR_INVALID, "options.k_pass must be 0, 1 or 2");
    if (opt.sym_tile < 0 || opt.sym_tile > 8)
        return fail(POPCORN_ERR_INVALID, "options.sym_tile must be in [0, 8]");
    for (int r = 0; r < 4; ++r)
        if (opt.reserved[r] != 0) return fail(POPCORN_ERR_INVALID, "options.reserved[%d] must be 0", r);
    if (opt.k_storage < POPCORN_K_FP32 || opt.k_storage > POPCORN_K_BF16)
        return fail(POPCORN_ERR_INVALID, "unknown k_storage %d", opt.k_storage);
    if (opt.timing < 0 || opt.timing > 2) return fail(POPCORN_ERR_INVALID, "options.timing must be 0, 1 or 2");
    if (opt.store_k != 0 && opt.store_k != 1) return fail(POPCORN_ERR_INVALID, "store_k must be 0 or 1");
    if (opt.store_k == 0 && opt.precision != POPCORN_BF16 && opt.precision != POPCORN_FP8)
        return fail(POPCORN_ERR_UNSUPPORTED, "the recompute path (store_k = 0) runs in POPCORN_BF16 or POPCORN_FP8");
    if (opt.store_k == 1 && opt.precision == POPCORN_FP8)
        return fail(POPCORN_ERR_UNSUPPORTED, "POPCORN_FP8 is available on the recompute path (store_k = 0) only");
    KernParams kp;
    POPCORN_TRY(check_kernel(kern, &kp));
    DeviceInfo* dev;
    POPCORN_TRY(device_info(&dev));
    if (opt.store_k == 0)
        return fit_recompute(P, n, d, ldp, k, kp, init_labels, max_iter, tol, opt, labels_out, objective_out,
                             iterations_out, info, s, dev);
    const int ni = (int)n;
    const int ks = opt.k_storage;
    const size_t kelem = ks == POPCORN_K_FP32 ? 4 : 2;
    const int64_t ldk = ks == POPCORN_K_FP32 ? (n + 3) / 4 * 4 : (n + 7) / 8 * 8;   // 16-byte rows
    ReducePlan plan = plan_reduce(ni, k, dev->sms, dev->reduce_smem, ks);
    if (plan.grid == 0) return fail(POPCORN_ERR_UNSUPPORTED, "n = %d is too large for the materialized path", ni);
    // symmetric pass (k <= kSymMaxK; k_pass 0 or 1): the blocks on and above the diagonal,
    // row and column sums into slots, folded into slot 0.  An FP16 / BF16 K takes the
    // tensor-core form (2 bytes an entry).
    SymPlan sym{};
    // automatic choice, from measurements on GB300: the symmetric pass (sorted form) once K
    // outgrows L2, where a pass streams it from HBM and reading half of it pays (images,
    // n = 70,000, k = 10: 1.67 ms a stream plus 0.09 ms of fold against 3.05 ms for the
    // full square; rings, n = 20,000, k = 4: 0.152 + 0.014 against 0.275).  Below that a
    // pass is a few microseconds of launches and the full square's two kernels win.
    // A half K from a tensor-core build exists only as the packed triangle (its epilogue
    // writes FP16 / BF16 boxes for the symmetric pass), so that pairing takes it at every n.
    const bool sym_auto = ni >= kSymAutoMinN || (ks != POPCORN_K_FP32 && opt.precision != POPCORN_FP32);
    if (opt.k_pass == 1 || (opt.k_pass == 0 && sym_auto))
        sym = plan_reduce_sym(ni, k, dev->sms, dev->smem_optin, opt.sym_tile, 0, (int)kelem);
    const bool use_sym = sym.ok;
    // more clusters than the symmetric pass takes, FP32 K: the packed triangle all the same, read
    // by block rows (each tile twice, the second time from L2).  k_pass = 2 keeps the row-by-row
    // read of a row-major K.
    const bool use_tiles = !use_sym && ks == POPCORN_K_FP32 && opt.k_pass != 2 && k > kSymMaxK && ni >= kTilesMinN &&
                           plan_reduce_tiles(ni, k, dev->sms, &plan);
    const int64_t tri_tiles = (int64_t)((ni + 127) / 128) * ((ni + 127) / 128 + 1) / 2;
    // A half K read as the full square (k > kSymMaxK, or k_pass = 2) goes through the tensor
    // cores, as batched mode's one-instance form: the packed triangle of half tiles, each
    // 128-row block's tiles (those below the diagonal transposed) MMA'd against the one-hot label operands with the
    // row sums in TMEM, one segment, then the z reduction.  Taken when the K build runs on
    // the tensor cores (they write no row-major half K) or K outgrows L2; below that the
    // CUDA-core full-square pass reads the row-major half K.
    // (It uploads a descriptor and its units from the host, so not inside a caller's stream
    // capture, where a copy would read host memory at replay.)
    cudaStreamCaptureStatus cap_status = cudaStreamCaptureStatusNone;
    POPCORN_CUDA(cudaStreamIsCapturing(s, &cap_status));
    const bool capturing = cap_status != cudaStreamCaptureStatusNone;
    const bool mma_full = !use_sym && ks != POPCORN_K_FP32 && !capturing &&
                          (opt.precision != POPCORN_FP32 || ni >= kSymAutoMinN);
    const int Tf = (ni + 127) / 128;
    // With the symmetric pass, K is stored block-packed: the upper triangle of 128 x 128
    // tiles only (half the memory; each value written once), by the FP32 build and by the
    // tensor-core builds alike.
    sym.packed = use_sym;
    const size_t k_bytes = sym.packed ? (size_t)sym.items * 128 * 128 * kelem
                           : use_tiles ? (size_t)tri_tiles * 128 * 128 * kelem
                           : mma_full ? (size_t)tri_tiles * 32768
                                      : (size_t)ni * (size_t)ldk * kelem;
    const int nslots = use_sym ? sym.nslots : mma_full ? 1 : plan.nseg;
    if (use_sym || mma_full) plan.nseg = 1;   // the assignment reads one (folded) segment
    BatchPlan bpf{};
    if (mma_full) {
        bpf.count = 1;
        bpf.half = ks;
        bpf.vblocks = Tf;
        bpf.nunits = Tf;
        bpf.Nmax = (k + 15) / 16 * 16;
        if (!plan_batched_mma(&bpf, dev->sms, dev->smem_optin))
            return fail(POPCORN_ERR_UNSUPPORTED, "the tensor-core full-square stream does not fit this device");
    }
    const bool timing = opt.timing != 0;          // phase events (K build, passes)
    const bool kernel_events = opt.timing == 1;   // and events around every kernel of every pass
    int launches = 0;
    int64_t h2d = 0, d2h = 0;

    Workspace ws(dev->pool, s);
    const float* Pd = P;
    int64_t ldpd = ldp;
    if (!is_device_pointer(P)) {
        float* tmp;
        POPCORN_TRY(ws.alloc(&tmp, (size_t)ni * d, "points"));
        POPCORN_CUDA(cudaMemcpy2DAsync(tmp, (size_t)d * sizeof(float), P, (size_t)ldp * sizeof(float),
                                       (size_t)d * sizeof(float), (size_t)ni, cudaMemcpyHostToDevice, s));
        h2d += (int64_t)ni * d * sizeof(float);
        Pd = tmp;
        ldpd = d;
    }
    const int32_t* Ld = init_labels;
    if (!is_device_pointer(init_labels)) {
        int32_t* tmp;
        POPCORN_TRY(ws.alloc(&tmp, (size_t)ni, "initial labels"));
        POPCORN_CUDA(cudaMemcpyAsync(tmp, init_labels, (size_t)ni * sizeof(int32_t), cudaMemcpyHostToDevice, s));
        h2d += (int64_t)ni * sizeof(int32_t);
        Ld = tmp;
    }

    PassBuffers b{};
    unsigned char* K;
    float* kdiag;
    POPCORN_TRY(ws.alloc(&K, k_bytes, "kernel matrix"));
    POPCORN_TRY(ws.alloc(&kdiag, (size_t)ni, "diag(K)"));
    const size_t nlab = ((size_t)ni + 15) & ~(size_t)15;
    const int hist_len = max_iter > 0 ? max_iter : 1;
    b.K = K;
    b.ldk = ldk;
    b.k_storage = ks;
    b.kdiag = kdiag;
    b.n = ni;
    b.k = k;
    POPCORN_TRY(ws.alloc(&b.lab32, ni, "labels"));
    POPCORN_TRY(ws.alloc(&b.lab8, nlab, "label bytes"));
    POPCORN_TRY(ws.alloc(&b.counts, 2 * (size_t)k, "counts"));
    POPCORN_TRY(ws.alloc(&b.Spart, (size_t)nslots * ni * k, "segment sums"));
    const int zblocks_f = (ni + kZReduceRows - 1) / kZReduceRows;
    POPCORN_TRY(ws.alloc(&b.zpart,
                         (size_t)(use_sym ? sym.fold_blocks : mma_full ? std::max(plan.grid, zblocks_f) : plan.grid) * k,
                         "block partials"));
    b.sym_meta = nullptr;
    b.sym_order = nullptr;
    if (use_sym && sym.meta_bytes) POPCORN_TRY(ws.alloc(&b.sym_meta, sym.meta_bytes, "block label metadata"));
    if (use_tiles) {
        POPCORN_TRY(ws.alloc(&b.sym_meta, tiles_record_bytes(ni), "label records"));
        POPCORN_TRY(ws.alloc(&b.Srun, (size_t)nslots * ni * k, "running segment sums"));
    }
    std::vector<int> sym_order;
    if (use_sym && sym.units > 1 && !capturing) {   // (the natural order inside a caller's capture)
        sym_unit_order(sym, &sym_order);
        int* d_order;
        POPCORN_TRY(ws.alloc(&d_order, sym_order.size(), "super-tile order"));
        POPCORN_CUDA(cudaMemcpyAsync(d_order, sym_order.data(), sym_order.size() * sizeof(int),
                                     cudaMemcpyHostToDevice, s));
        b.sym_order = d_order;
    }
    // one pass's reduction: the K stream (for the symmetric pass: stream, then fold with z)
    // kernels of one pass's reduction: the full-square stream; or the symmetric stream and its
    // fold (the sorted form first sorts every block's labels)
    const int red_launches = use_sym ? (sym.sorted || sym.mma ? 3 : 2) : mma_full ? 3 : use_tiles ? 2 : 1;
    // Error-path test hook: with POPCORN_TEST_SYM_STALL_MS=<ms> in the environment, the
    // first symmetric stream launch of this fit (either form) leaves one block's copies out
    // and bounds its waits by <ms>, so the fit reports POPCORN_ERR_TIMEOUT (nothing faults
    // or hangs; the context stays usable).  Unset in every ordinary run.
    // The same hook makes CTA 0 of the one-launch fit leave before its first grid barrier.
    int stall_ms = 0;
    {
        const char* env = getenv("POPCORN_TEST_SYM_STALL_MS");
        if (env && *env) stall_ms = atoi(env);
        if (stall_ms < 0 || stall_ms > 10000) stall_ms = 0;
    }
    // the tensor-core full square: a one-instance batch descriptor and its units (0, row block)
    BatchInst* dIf = nullptr;
    int2* unitsf = nullptr;
    unsigned char* Vf = nullptr;
    auto reduce_pass = [&](int eval, cudaEvent_t mid, cudaStream_t st) -> cudaError_t {
        const int stall = stall_ms;
        if (mma_full) {
            stall_ms = 0;
            cudaError_t e = launch_batched_mma_stream(dIf, unitsf, bpf, &b.st->wait_err, eval, st, stall);
            if (e == cudaSuccess && mid) e = cudaEventRecord(mid, st);
            return e != cudaSuccess ? e : launch_zreduce(b, 1, eval, st);
        }
        if (!use_sym && !use_tiles) return launch_reduce(b, plan, eval, st);
        stall_ms = 0;
        if (use_tiles) return launch_reduce_tiles(b, plan, &b.st->wait_err, eval, st, stall);
        return launch_reduce_sym(b, sym, &b.st->wait_err, eval, st, mid, stall);
    };
    POPCORN_TRY(ws.alloc(&b.zsum, (size_t)k, "z sums"));
    POPCORN_TRY(ws.alloc(&b.cnorm, (size_t)k, "centroid norms"));
    POPCORN_TRY(ws.alloc(&b.invm, (size_t)k, "inverse cluster sizes"));
    POPCORN_TRY(ws.alloc(&b.st, 1, "loop state"));
    POPCORN_TRY(ws.alloc(&b.J_hist, (size_t)hist_len, "objective history"));
    POPCORN_TRY(ws.alloc(&b.changed_hist, (size_t)hist_len, "change history"));
    b.E_out = info ? info->E_out : nullptr;   // written by every assignment pass; the last one stays

    g_events.used = 0;
    cudaEvent_t ev_b0 = nullptr, ev_b1 = nullptr, ev_l1 = nullptr, ev_e1 = nullptr;
    std::vector<cudaEvent_t> ev_r, ev_a;   // before/after each reduction and assignment launch
    std::vector<cudaEvent_t> ev_f;         // symmetric pass: between stream and fold, after the fold
    if (timing) {
        POPCORN_TRY(g_events.get(&ev_b0));
        POPCORN_CUDA(cudaEventRecord(ev_b0, s));
    }
    POPCORN_CUDA(cudaMemsetAsync(b.counts, 0, 2 * (size_t)k * sizeof(int32_t), s));
    POPCORN_CUDA(launch_init_state(b.st, max_iter, opt.check_convergence ? 1 : 0, tol, s));
    if (((sym.packed && sym.ebytes == 2) || mma_full) && opt.precision != POPCORN_FP32) {
        // half layout from the tensor-core build: its epilogue rounds and stores the tiles
        POPCORN_TRY(build_kernel_matrix(Pd, ni, d, ldpd, kp, opt.precision, K, ldk, ks, kdiag, &ws,
                                        &b.st->wait_err, dev->sms, s, &launches, kPackedSw128H));
    } else if ((sym.packed && sym.ebytes == 2) || mma_full) {
        // half layout from the FP32 build: it writes the FP32 triangle into a temporary, one
        // pack launch rounds it into K (and rounds diag K with it), and the temporary goes back
        float* kf;
        POPCORN_TRY(ws.alloc(&kf, (size_t)tri_tiles * 128 * 128, "FP32 kernel matrix"));
        POPCORN_TRY(build_kernel_matrix(Pd, ni, d, ldpd, kp, opt.precision, kf, ldk, POPCORN_K_FP32, kdiag, &ws,
                                        &b.st->wait_err, dev->sms, s, &launches, kPackedSw4));
        POPCORN_CUDA(launch_pack_half(kf, K, ks, ni, kdiag, s));
        ++launches;
        ws.release(kf);
    } else {
        POPCORN_TRY(build_kernel_matrix(Pd, ni, d, ldpd, kp, opt.precision, K, ldk, ks, kdiag, &ws,
                                        &b.st->wait_err, dev->sms, s, &launches,
                                        sym.packed ? sym.layout : use_tiles ? kPackedSw4 : 0));
    }
    if (mma_full) {
        POPCORN_TRY(ws.alloc(&Vf, (size_t)Tf * bpf.Nmax * 256, "one-hot operands"));
        BatchInst hf;
        memset(&hf, 0, sizeof hf);
        hf.T = Tf;
        hf.kdiag = kdiag;
        hf.n = ni;
        hf.k = k;
        hf.nseg = 1;
        hf.seglen = ni;
        hf.lab8 = b.lab8;
        hf.lab32 = b.lab32;
        hf.Spart = b.Spart;
        hf.st = b.st;
        hf.Kh = K;
        hf.V = Vf;
        hf.N = bpf.Nmax;
        std::vector<int2> hu((size_t)Tf);
        for (int r = 0; r < Tf; ++r) hu[(size_t)r] = make_int2(0, r);
        POPCORN_TRY(ws.alloc(&dIf, 1, "batch descriptor"));
        POPCORN_TRY(ws.alloc(&unitsf, (size_t)Tf, "row-block units"));
        POPCORN_CUDA(cudaMemcpyAsync(dIf, &hf, sizeof hf, cudaMemcpyHostToDevice, s));
        POPCORN_CUDA(cudaMemcpyAsync(unitsf, hu.data(), sizeof(int2) * hu.size(), cudaMemcpyHostToDevice, s));
    }
    POPCORN_CUDA(launch_trace(kdiag, ni, b.st, s));
    POPCORN_CUDA(launch_init_labels(Ld, ni, k, b.lab32, b.lab8, b.counts, b.st, s));
    launches += 3;
    if (timing) {
        POPCORN_TRY(g_events.get(&ev_b1));
        POPCORN_CUDA(cudaEventRecord(ev_b1, s));
    }

    // Fixed-iteration mode (no convergence checking, no per-kernel events): every pass
    // and the final objective pass are captured once into a CUDA graph on a private
    // stream and launched on s as one unit, so the passes run back to back without a
    // host launch between kernels (this matters when K sits in L2 and a pass takes
    // microseconds).  A caller that is itself capturing s gets the plain launches.
    // An FP32 K that sits in L2 (the automatic choice only): the whole fit -- every pass and
    // the final objective -- in one cooperative launch, with grid barriers between the
    // phases of a pass instead of three launches a pass.
    bool fused = !use_sym && opt.k_pass == 0 && ks == POPCORN_K_FP32 && dev->coop &&
                 cap_status == cudaStreamCaptureStatusNone && fused_fit_applies(ni, k, dev->sms, dev->smem_optin);
    if (fused) {
        double* fz;
        unsigned* fbar;
        POPCORN_TRY(ws.alloc(&fz, (size_t)dev->sms * k, "fused-fit partials"));
        POPCORN_TRY(ws.alloc(&fbar, fused_xchg_words(dev->sms, k), "exchange slots"));
        const cudaError_t fe = launch_fused_fit(b, fz, fbar, dev->sms, dev->smem_optin, s, stall_ms);
        if (fe == cudaErrorCooperativeLaunchTooLarge) {
            // not every SM can hold a CTA now (a shared device): the launched passes instead
            cudaGetLastError();
            fused = false;
        } else {
            POPCORN_CUDA(fe);
            launches += 1;
        }
    }
    const bool use_graph = !fused && !opt.check_convergence && !kernel_events && max_iter > 0 &&
                           cap_status == cudaStreamCaptureStatusNone;
    cudaGraphExec_t pass_exec = nullptr;
    struct ExecGuard {
        cudaGraphExec_t* e;
        ~ExecGuard() {
            if (*e) cudaGraphExecDestroy(*e);
        }
    } pass_exec_guard{&pass_exec};
    if (use_graph) {
        cudaStream_t cs;
        POPCORN_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
        struct StreamGuard {
            cudaStream_t s;
            ~StreamGuard() { cudaStreamDestroy(s); }
        } sg{cs};
        POPCORN_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
        cudaError_t ce = cudaSuccess;
        for (int t = 0; t < max_iter && ce == cudaSuccess; ++t) {
            ce = reduce_pass(0, nullptr, cs);
            if (ce == cudaSuccess) ce = launch_assign(b, plan, cs);
            launches += red_launches + 1;
        }
        if (ce == cudaSuccess) ce = reduce_pass(1, nullptr, cs);
        launches += red_launches;
        cudaGraph_t graph = nullptr;
        const cudaError_t ee = cudaStreamEndCapture(cs, &graph);
        if (ce == cudaSuccess) ce = ee;
        if (ce == cudaSuccess) ce = cudaGraphInstantiate(&pass_exec, graph, 0);
        if (graph) cudaGraphDestroy(graph);
        POPCORN_CUDA(ce);
        POPCORN_CUDA(cudaGraphLaunch(pass_exec, s));
    }

    // Assignment passes.  With convergence checking, the host polls the
    // device "done" flag one chunk behind, so at most one chunk of passes is
    // launched after convergence (those return at once on the device).
    const int chunk = 4;
    void* hpin;
    POPCORN_TRY(pinned(2 * sizeof(int32_t) + sizeof(LoopState), &hpin));
    volatile int32_t* hflag = static_cast<int32_t*>(hpin);
    cudaEvent_t poll_ev[2] = {nullptr, nullptr};
    if (opt.check_convergence) {
        POPCORN_TRY(g_events.get(&poll_ev[0]));
        POPCORN_TRY(g_events.get(&poll_ev[1]));
    }
    int launched = (use_graph || fused) ? max_iter : 0, pending = -1, slot = 0;
    while (launched < max_iter) {
        const int m = (max_iter - launched < chunk) ? (max_iter - launched) : chunk;
        for (int t = 0; t < m; ++t) {
            cudaEvent_t e0 = nullptr, e1 = nullptr, e2 = nullptr, em = nullptr;
            if (kernel_events) {
                POPCORN_TRY(g_events.get(&e0));
                POPCORN_TRY(g_events.get(&e1));
                POPCORN_TRY(g_events.get(&e2));
                if (use_sym || mma_full) POPCORN_TRY(g_events.get(&em));
                POPCORN_CUDA(cudaEventRecord(e0, s));
            }
            POPCORN_CUDA(reduce_pass(0, em, s));
            if (kernel_events) POPCORN_CUDA(cudaEventRecord(e1, s));
            POPCORN_CUDA(launch_assign(b, plan, s));
            if (kernel_events) {
                POPCORN_CUDA(cudaEventRecord(e2, s));
                ev_r.push_back(e0);
                ev_r.push_back(e1);
                ev_a.push_back(e1);
                ev_a.push_back(e2);
                if (use_sym || mma_full) {
                    ev_f.push_back(em);
                    ev_f.push_back(e1);
                }
            }
            launches += red_launches + 1;
        }
        launched += m;
        if (opt.check_convergence && launched < max_iter) {
            POPCORN_CUDA(cudaMemcpyAsync((void*)(hflag + slot), &b.st->done, sizeof(int32_t),
                                         cudaMemcpyDeviceToHost, s));
            POPCORN_CUDA(cudaEventRecord(poll_ev[slot], s));
            if (pending >= 0) {
                POPCORN_CUDA(cudaEventSynchronize(poll_ev[pending]));
                if (hflag[pending]) break;
            }
            pending = slot;
            slot ^= 1;
        }
    }
    if (timing) {
        POPCORN_TRY(g_events.get(&ev_l1));
        POPCORN_CUDA(cudaEventRecord(ev_l1, s));
    }
    // J(labels_out): reuses J of the last pass when it changed nothing (in the graph above
    // when there is one)
    if (!use_graph && !fused) {
        POPCORN_CUDA(reduce_pass(1, nullptr, s));
        launches += red_launches;
    }
    if (timing) {
        POPCORN_TRY(g_events.get(&ev_e1));
        POPCORN_CUDA(cudaEventRecord(ev_e1, s));
    }

    LoopState* hs_pin = reinterpret_cast<LoopState*>(static_cast<char*>(hpin) + 2 * sizeof(int32_t));
    POPCORN_CUDA(cudaMemcpyAsync(hs_pin, b.st, sizeof(LoopState), cudaMemcpyDeviceToHost, s));
    d2h += sizeof(LoopState);
    if (is_device_pointer(labels_out)) {
        POPCORN_CUDA(cudaMemcpyAsync(labels_out, b.lab32, (size_t)ni * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
    } else {
        POPCORN_CUDA(cudaMemcpyAsync(labels_out, b.lab32, (size_t)ni * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
        d2h += (int64_t)ni * sizeof(int32_t);
    }
    POPCORN_CUDA(cudaStreamSynchronize(s));
    LoopState hs;
    memcpy(&hs, hs_pin, sizeof hs);
    if (hs.bad_label) return fail(POPCORN_ERR_INVALID, "an initial label is outside [0, %d)", k);
    if (hs.wait_err)
        return fail(POPCORN_ERR_TIMEOUT,
                    "a bounded wait in the tensor-core K build, the symmetric pass or a grid barrier ran out");
    *objective_out = hs.J_eval;
    *iterations_out = hs.iter;

    if (info) {
        const int iters = hs.iter;
        if (iters > 0 && (info->J_history || info->changed_history)) {
            if (info->J_history)
                POPCORN_CUDA(cudaMemcpy(info->J_history, b.J_hist, (size_t)iters * sizeof(double), cudaMemcpyDeviceToHost));
            if (info->changed_history)
                POPCORN_CUDA(cudaMemcpy(info->changed_history, b.changed_hist, (size_t)iters * sizeof(int32_t),
                                        cudaMemcpyDeviceToHost));
        }
        info->converged = hs.converged;
        info->kernel_launches = launches;
        info->tune_cache_hit = info->tune_candidates = 0;
        info->tune_ms = 0.0;
        info->fold_ms = 0.0;
        info->k_pass_used = 0;
        info->sym_form = 0;
        for (int q = 0; q < 4; ++q) info->schedule[q] = 0;
        if (use_sym) {
            info->schedule[0] = sym.a;
            info->schedule[1] = sym.stages;
            info->schedule[2] = sym.nslots;
            info->schedule[3] = sym.kb;
            info->sym_form = sym.mma ? 3 : sym.sorted ? 2 : 1;
        } else if (mma_full) {
            info->schedule[1] = bpf.mstages;
            info->schedule[3] = bpf.Nmax;
        }
        // passes that did work (launches after convergence return at once)
        const bool eval_ran = !(hs.iter > 0 && hs.last_changed == 0);
        info->reduce_launches = iters + (eval_ran ? 1 : 0);
        info->assign_launches = iters;
        info->h2d_bytes = h2d;
        info->d2h_bytes = d2h;
        info->kbuild_ms = info->loop_ms = info->reduce_ms = info->assign_ms = info->eval_ms = 0.0;
        if (timing) {
            info->kbuild_ms = elapsed(ev_b0, ev_b1);
            info->loop_ms = elapsed(ev_b1, ev_l1);
            info->eval_ms = elapsed(ev_l1, ev_e1);
            double r = 0, a = 0;
            for (size_t t = 0; t + 1 < ev_r.size() && t < 2 * (size_t)iters; t += 2) r += elapsed(ev_r[t], ev_r[t + 1]);
            for (size_t t = 0; t + 1 < ev_a.size() && t < 2 * (size_t)iters; t += 2) a += elapsed(ev_a[t], ev_a[t + 1]);
            info->reduce_ms = r;
            info->assign_ms = a;
            double f = 0;
            for (size_t t = 0; t + 1 < ev_f.size() && t < 2 * (size_t)iters; t += 2) f += elapsed(ev_f[t], ev_f[t + 1]);
            info->fold_ms = f;
        }
        info->k_pass_used = fused ? 3 : use_sym ? 1 : 2;
    }
    return POPCORN_OK;
}


popcorn_status popcorn_kmeanspp(const float* P, int64_t n, int32_t d, int64_t ldp, int32_t k, popcorn_kernel kern,
                                const double* u, int32_t* labels_out, int32_t* centers_out, popcorn_stream_t stream) {
    g_err.clear();
    cudaStream_t s = (cudaStream_t)stream;
    if (!P || !u || !labels_out) return fail(POPCORN_ERR_INVALID, "null pointer argument");
    if (n < 1 || n >= (1LL << 31)) return fail(POPCORN_ERR_INVALID, "n = %lld outside [1, 2^31)", (long long)n);
    if (d < 1) return fail(POPCORN_ERR_INVALID, "d = %d < 1", d);
    if (ldp < d) return fail(POPCORN_ERR_INVALID, "ldp = %lld < d = %d", (long long)ldp, d);
    if (k < 1 || k > n || k > kMaxClusters)
        return fail(POPCORN_ERR_INVALID, "k = %d outside [1, min(n, %d)]", k, kMaxClusters);
    KernParams kp;
    POPCORN_TRY(check_kernel(kern, &kp));
    const bool u_dev = is_device_pointer(u);
    if (!u_dev)
        for (int t = 0; t < k; ++t)
            if (!(u[t] >= 0.0 && u[t] < 1.0)) return fail(POPCORN_ERR_INVALID, "u[%d] = %g outside [0, 1)", t, u[t]);
    DeviceInfo* dev;
    POPCORN_TRY(device_info(&dev));
    if (!dev->coop) return fail(POPCORN_ERR_UNSUPPORTED, "the device has no cooperative launches");
    const int ni = (int)n;
    if (!kmeanspp_fits(ni, d, dev->sms, dev->smem_optin))
        return fail(POPCORN_ERR_UNSUPPORTED, "n = %d, d = %d: the seeding's per-SM state exceeds shared memory", ni,
                    d);
    Workspace ws(dev->pool, s);
    const float* Pd = P;
    int64_t ldpd = ldp;
    if (!is_device_pointer(P)) {
        float* tmp;
        POPCORN_TRY(ws.alloc(&tmp, (size_t)ni * d, "points"));
        POPCORN_CUDA(cudaMemcpy2DAsync(tmp, (size_t)d * sizeof(float), P, (size_t)ldp * sizeof(float),
                                       (size_t)d * sizeof(float), (size_t)ni, cudaMemcpyHostToDevice, s));
        Pd = tmp;
        ldpd = d;
    }
    const double* ud = u;
    if (!u_dev) {
        double* tmp;
        POPCORN_TRY(ws.alloc(&tmp, (size_t)k, "draws"));
        POPCORN_CUDA(cudaMemcpyAsync(tmp, u, (size_t)k * sizeof(double), cudaMemcpyHostToDevice, s));
        ud = tmp;
    }
    const bool lab_dev = is_device_pointer(labels_out);
    const bool cen_dev = centers_out && is_device_pointer(centers_out);
    int32_t* labd = labels_out;
    if (!lab_dev) POPCORN_TRY(ws.alloc(&labd, (size_t)ni, "labels"));
    int32_t* cend = cen_dev ? centers_out : nullptr;
    if (!cend) POPCORN_TRY(ws.alloc(&cend, (size_t)k, "centers"));
    double *part, *Dg;
    int* err;
    unsigned* bar;
    POPCORN_TRY(ws.alloc(&part, 2 * (size_t)dev->sms, "seeding partial sums"));
    POPCORN_TRY(ws.alloc(&Dg, 2 * (size_t)ni, "seeding distances"));
    POPCORN_TRY(ws.alloc(&err, 1, "error word"));
    POPCORN_TRY(ws.alloc(&bar, 32, "grid barrier"));
    POPCORN_CUDA(cudaMemsetAsync(err, 0, sizeof(int), s));
    POPCORN_CUDA(launch_kmeanspp(Pd, ni, d, ldpd, k, kern, ud, labd, cend, part, Dg, bar, err, dev->sms, s));
    void* hpin;
    POPCORN_TRY(pinned(sizeof(int), &hpin));
    int* herr = static_cast<int*>(hpin);
    POPCORN_CUDA(cudaMemcpyAsync(herr, err, sizeof(int), cudaMemcpyDeviceToHost, s));
    if (!lab_dev)
        POPCORN_CUDA(cudaMemcpyAsync(labels_out, labd, (size_t)ni * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    if (centers_out && !cen_dev)
        POPCORN_CUDA(cudaMemcpyAsync(centers_out, cend, (size_t)k * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    POPCORN_CUDA(cudaStreamSynchronize(s));
    if (*herr) return fail(POPCORN_ERR_TIMEOUT, "a bounded grid-barrier wait in the seeding ran out");
    return POPCORN_OK;
}

popcorn_status popcorn_fit_batched(int32_t count, const popcorn_instance* inst, int32_t max_iter, double tol,
                                   const popcorn_options* opt_in, double* objectives_out, int32_t* iterations_out,
                                   popcorn_fit_info* info, popcorn_stream_t stream) {
    g_err.clear();
    cudaStream_t s = (cudaStream_t)stream;
    popcorn_options opt;
    memset(&opt, 0, sizeof opt);
    opt.precision = POPCORN_FP32;
    opt.store_k = 1;
    opt.check_convergence = 1;
    if (opt_in) opt = *opt_in;
    if (count < 1 || !inst || !objectives_out || !iterations_out)
        return fail(POPCORN_ERR_INVALID, "count must be >= 1 and the output arrays non-null");
    if (max_iter < 0) return fail(POPCORN_ERR_INVALID, "max_iter = %d < 0", max_iter);
    if (!(tol >= 0) || !std::isfinite(tol)) return fail(POPCORN_ERR_INVALID, "tol must be finite and >= 0");
    if (opt.autotune != 0 && opt.autotune != 1) return fail(POPCORN_ERR_INVALID, "options.autotune must be 0 or 1");
    if (opt.k_pass < 0 || opt.k_pass > 2) return fail(POPCORN_ERR_INVALID, "options.k_pass must be 0, 1 or 2");
    if (opt.sym_tile < 0 || opt.sym_tile > 8)
        return fail(POPCORN_ERR_INVALID, "options.sym_tile must be in [0, 8]");
    for (int r = 0; r < 4; ++r)
        if (opt.reserved[r] != 0) return fail(POPCORN_ERR_INVALID, "options.reserved[%d] must be 0", r);
    if (opt.k_storage < POPCORN_K_FP32 || opt.k_storage > POPCORN_K_BF16)
        return fail(POPCORN_ERR_INVALID, "unknown k_storage %d", opt.k_storage);
    if (opt.store_k != 1) return fail(POPCORN_ERR_UNSUPPORTED, "batched mode stores K (store_k = 1)");
    if (opt.precision != POPCORN_FP32 && opt.precision != POPCORN_BF16 && opt.precision != POPCORN_BF16X3)
        return fail(POPCORN_ERR_UNSUPPORTED, "batched mode runs in FP32, BF16 or BF16X3");
    DeviceInfo* dev;
    POPCORN_TRY(device_info(&dev));

    // ---- layout of every instance, flattened work prefixes
    std::vector<BatchInst> h(count);
    std::vector<size_t> off(count);
    BatchPlan bp{};
    bp.count = count;
    size_t bytes = 0;
    size_t tc_ws = 0;
    auto take = [&](size_t nbytes) {
        const size_t o = bytes;
        bytes += (nbytes + 255) & ~(size_t)255;
        return o;
    };
    struct Offs {
        size_t K, kdiag, lab32, lab8, counts, Spart, Srun, zpart, zsum, cnorm, invm, st, J, ch;
    };
    std::vector<Offs> o(count);
    // FP16 / BF16 K: every instance's square as half tiles read by the tensor-core stream
    const int half = opt.k_storage != POPCORN_K_FP32 ? opt.k_storage : 0;
    bp.half = half;
    std::vector<size_t> o_kh(count), o_v(count);
    const int hist_len = max_iter > 0 ? max_iter : 1;
    // K-stream unit lengths the autotuner may pick (Spart is sized for the shortest)
    static const int kSegCand[] = {2048, 4096, 8192, 16384};
    const int min_seglen = opt.autotune ? kSegCand[0] : kBatchSeg;
    // FP32 K by block rows, or row by row where there are fewer 128-row blocks than the block rows' stream
    // has CTAs (or 4 an SM: with few clusters 5 fit, but 600 blocks are enough).  Whole calls of 20 passes,
    // by block rows and row by row: one instance of n = 2,000 1,877 and 900 us, 8 of n = 300 to 600 1,256 and
    // 882, 8 of 4,000 to 7,000 (344 blocks for 456 CTAs) 6,252 and 5,636; 256 of 128 to 400 (about 640 for 760)
    // 4,904 and 5,532, 64 of 1,000 to 4,000 (1,250 for 456) 9,466 and 12,206.
    bool rows = false;
    if (!half) {
        long long blocks = 0;
        BatchPlan probe{};
        for (int t = 0; t < count; ++t) {   // (what is not valid is reported below)
            blocks += inst[t].n > 0 ? (inst[t].n + 127) / 128 : 0;
            probe.kmax = std::max(probe.kmax, std::min(std::max(inst[t].k, 1), kMaxClusters));
        }
        rows = blocks < dev->sms;   // (a CTA an SM at least: no need to ask what fits)
        if (!rows && !plan_batched_tiles(&probe, dev->sms))
            return fail(POPCORN_ERR_UNSUPPORTED, "the batched K stream does not fit this device");
        rows = rows || blocks < std::min(probe.grid, 4 * dev->sms);
    }
    bp.rows = rows ? 1 : 0;
    // FP32 K: columns a unit (and a sum) takes
    auto set_segments = [rows](BatchInst* b, int seglen) {
        if (rows) {
            b->seglen = seglen;
            b->nseg = (b->n + seglen - 1) / seglen;
            return;
        }
        const int blocks = std::min(seglen / 128, b->T);
        b->seglen = 128 * blocks;
        b->nseg = (b->T + blocks - 1) / blocks;
    };
    for (int t = 0; t < count; ++t) {
        const popcorn_instance& x = inst[t];
        if (!x.P || !x.init_labels || !x.labels_out) return fail(POPCORN_ERR_INVALID, "instance %d: null pointer", t);
        if (x.n < 2 || x.n >= (1LL << 31)) return fail(POPCORN_ERR_INVALID, "instance %d: n = %lld", t, (long long)x.n);
        if (x.d < 1 || x.ldp < x.d) return fail(POPCORN_ERR_INVALID, "instance %d: d = %d, ldp = %lld", t, x.d, (long long)x.ldp);
        if (x.k < 1 || x.k >= x.n || x.k > kMaxClusters)
            return fail(POPCORN_ERR_INVALID, "instance %d: k = %d outside [1, min(n - 1, %d)]", t, x.k, kMaxClusters);
        if (!is_device_pointer(x.P) || !is_device_pointer(x.init_labels) || !is_device_pointer(x.labels_out))
            return fail(POPCORN_ERR_INVALID, "instance %d: batched mode takes device pointers", t);
        KernParams kp;
        popcorn_status ks = check_kernel(x.kern, &kp);
        if (ks != POPCORN_OK) return fail(ks, "instance %d: %s", t, g_err.c_str());
        const int n = (int)x.n, k = x.k;
        BatchInst& b = h[t];
        memset(&b, 0, sizeof b);
        b.P = x.P;
        b.ldp = x.ldp;
        b.d = x.d;
        b.kp = kp;
        b.T = (n + 127) / 128;
        b.tile0 = bp.tiles;
        bp.tiles += (long long)b.T * (b.T + 1) / 2;
        b.ldk = (n + 3) / 4 * 4;
        b.n = n;
        b.k = k;
        if (half) {   // S written once a row
            b.seglen = n;
            b.nseg = 1;
        } else {
            set_segments(&b, min_seglen);
        }
        b.init_labels = x.init_labels;
        b.labels_out = x.labels_out;
        b.unit0 = bp.units;
        bp.units += (rows ? n : b.T) * b.nseg;
        b.zblock0 = bp.zblocks;
        bp.zblocks += (n + kZReduceRows - 1) / kZReduceRows;
        b.ablock0 = bp.ablocks;
        bp.ablocks += (n + kAssignThreads - 1) / kAssignThreads;
        b.lblock0 = bp.lblocks;
        bp.lblocks += (n + kBatchLabelThreads - 1) / kBatchLabelThreads;
        if (k > bp.kmax) bp.kmax = k;
        const int zb = (n + kZReduceRows - 1) / kZReduceRows;
        // the packed triangle the K stream reads, FP32 or half tiles, or the square by rows
        const size_t tiles = (size_t)b.T * (b.T + 1) / 2;
        o[t].K = half ? 0 : rows ? take((size_t)n * b.ldk * 4) : take(tiles * 65536);
        if (half) {
            b.N = (k + 15) / 16 * 16;
            bp.nunits += b.T;
            if (b.N > bp.Nmax) bp.Nmax = b.N;
            o_kh[t] = take(tiles * 32768);
        }
        b.vblock0 = bp.vblocks;
        bp.vblocks += b.T;
        o_v[t] = rows ? 0 : take(half ? (size_t)b.T * b.N * 256 : tiles_record_bytes(n));
        o[t].kdiag = take((size_t)n * 4);
        o[t].lab32 = take((size_t)n * 4);
        o[t].lab8 = take(((size_t)n + 15) & ~(size_t)15);
        o[t].counts = take(2 * (size_t)k * 4);
        o[t].Spart = take((size_t)n * b.nseg * k * 4);
        o[t].Srun = half || rows ? 0 : take((size_t)n * b.nseg * k * 8);
        o[t].zpart = take((size_t)zb * k * 8);
        o[t].zsum = take((size_t)k * 8);
        o[t].cnorm = take((size_t)k * 8);
        o[t].invm = take((size_t)k * 8);
        o[t].st = take(sizeof(LoopState));
        o[t].J = take((size_t)hist_len * 8);
        o[t].ch = take((size_t)hist_len * 4);
        if (opt.precision != POPCORN_FP32) {
            const size_t w = kbuild_tc_workspace(n, x.d, opt.precision);
            if (w > tc_ws) tc_ws = w;
        }
    }
    if (bp.units <= 0 || bp.units >= (1 << 30)) return fail(POPCORN_ERR_UNSUPPORTED, "batch too large");
    // the units of the K stream -- half K: (instance, row block); FP32 K: (instance, segment x T +
    // row block) -- the larger instances first (their units take longer), so that the static
    // round-robin of the stream ends near balance; an instance's units stay together (its block
    // rows share tiles in L2)
    std::vector<int2> hunits;
    std::vector<int> order(count);
    for (int t = 0; t < count; ++t) order[t] = t;
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return h[x].T > h[y].T; });
    auto list_units = [&]() {
        hunits.clear();
        if (rows) return;   // (the kernel finds a row's instance by itself)
        for (int t : order)
            for (int r = 0; r < h[t].T * (half ? 1 : h[t].nseg); ++r) hunits.push_back(make_int2(t, r));
    };
    if (rows)
        plan_batched_reduce(&bp, dev->sms, dev->batched_smem);
    else if (half ? !plan_batched_mma(&bp, dev->sms, dev->smem_optin) : !plan_batched_tiles(&bp, dev->sms))
        return fail(POPCORN_ERR_UNSUPPORTED, "the batched K stream does not fit this device");
    list_units();
    const size_t units_off = take(sizeof(int2) * hunits.size());   // (the most units of any schedule)
    const size_t inst_off = take(sizeof(BatchInst) * (size_t)count);
    const size_t tc_off = tc_ws ? take(tc_ws) : 0;
    const size_t err_off = take(sizeof(int));

    Workspace ws(dev->pool, s);
    unsigned char* base;
    POPCORN_TRY(ws.alloc(&base, bytes, "batch workspace"));
    for (int t = 0; t < count; ++t) {
        BatchInst& b = h[t];
        b.K = !half ? reinterpret_cast<float*>(base + o[t].K) : nullptr;
        b.kdiag = reinterpret_cast<float*>(base + o[t].kdiag);
        b.lab32 = reinterpret_cast<int32_t*>(base + o[t].lab32);
        b.lab8 = base + o[t].lab8;
        b.counts = reinterpret_cast<int32_t*>(base + o[t].counts);
        b.Spart = reinterpret_cast<float*>(base + o[t].Spart);
        b.Srun = half || rows ? nullptr : reinterpret_cast<float2*>(base + o[t].Srun);
        b.zpart = reinterpret_cast<double*>(base + o[t].zpart);
        b.zsum = reinterpret_cast<double*>(base + o[t].zsum);
        b.cnorm = reinterpret_cast<double*>(base + o[t].cnorm);
        b.invm = reinterpret_cast<double*>(base + o[t].invm);
        b.st = reinterpret_cast<LoopState*>(base + o[t].st);
        b.J_hist = reinterpret_cast<double*>(base + o[t].J);
        b.changed_hist = reinterpret_cast<int32_t*>(base + o[t].ch);
        if (half) b.Kh = base + o_kh[t];
        b.V = rows ? nullptr : base + o_v[t];
    }
    const int2* dunits = reinterpret_cast<const int2*>(base + units_off);
    auto upload_units = [&]() {
        return cudaMemcpyAsync(base + units_off, hunits.data(), sizeof(int2) * hunits.size(), cudaMemcpyHostToDevice, s);
    };
    if (half) POPCORN_CUDA(upload_units());   // (FP32 K: once the schedule is known)
    BatchInst* dI = reinterpret_cast<BatchInst*>(base + inst_off);
    POPCORN_CUDA(cudaMemcpyAsync(dI, h.data(), sizeof(BatchInst) * (size_t)count, cudaMemcpyHostToDevice, s));
    int* err = reinterpret_cast<int*>(base + err_off);
    POPCORN_CUDA(cudaMemsetAsync(err, 0, sizeof(int), s));

    // ---- schedule of the batched K stream: unit length, blocks per SM (4 consumer warps a block).
    // A tuned schedule says 1, or 2 for as many as fit: two where three fit took 178 ms for a batch
    // that takes 142 ms so (256 instances of
    // n = 500 .. 8,000, 30 passes).
    auto set_seglen = [&](int seglen) {
        bp.units = 0;
        for (int t = 0; t < count; ++t) {
            set_segments(&h[t], seglen);
            h[t].unit0 = bp.units;
            bp.units += (rows ? h[t].n : h[t].T) * h[t].nseg;
        }
        list_units();
    };
    int sched[3] = {kBatchSeg, 0, 0};
    int tune_hit = 0, tune_cands = 0;
    double tune_ms = 0.0;
    if (opt.autotune && !half) {   // the half-K stream has no tuned schedule
        double sum_n2 = 0.0, max_n = 0.0;
        for (int t = 0; t < count; ++t) {
            sum_n2 += (double)h[t].n * h[t].n;
            max_n = h[t].n > max_n ? h[t].n : max_n;
        }
        const TuneKey key{rows ? 1 : 4, opt.precision, count, bp.kmax, log2_bucket(sum_n2), log2_bucket(max_n),
                          opt.k_storage, dev->sms};
        TuneValue best{};
        if (tune_lookup(key, &best)) {
            tune_hit = 1;
        } else {
            // K and the initial labels are needed to time the stream: build them now
            // (the captured graph below builds them again for the real run)
            const auto w0 = std::chrono::steady_clock::now();
            POPCORN_CUDA(launch_batched_init(dI, bp, max_iter, opt.check_convergence ? 1 : 0, tol, s));
            if (opt.precision == POPCORN_FP32) {
                POPCORN_CUDA(launch_batched_kbuild_simt(dI, bp, s));
            } else {
                for (int t = 0; t < count; ++t)
                    POPCORN_CUDA(launch_kbuild_tc(h[t].P, h[t].n, h[t].d, h[t].ldp, h[t].kp, opt.precision, h[t].K,
                                                  rows ? h[t].ldk : 0, h[t].kdiag, base + tc_off, err, dev->sms, s, nullptr,
                                                  rows ? 0 : kPackedSw4));
            }
            cudaEvent_t t0, t1;
            g_events.used = 0;
            POPCORN_TRY(g_events.get(&t0));
            POPCORN_TRY(g_events.get(&t1));
            best.ms = 3.0e38f;
            const std::vector<int> warp_cand = rows ? std::vector<int>{4, 8, 16} : std::vector<int>{4};
            auto stream = [&](const BatchPlan& p) {
                return rows ? launch_batched_reduce(dI, p, 0, s) : launch_batched_tiles(dI, dunits, p, err, 0, s);
            };
            for (int seglen : kSegCand)
                for (int w : warp_cand)
                    for (int ps : {1, 2}) {
                        BatchPlan cand = bp;
                        set_seglen(seglen);
                        cand.units = bp.units;
                        if (rows) {
                            plan_batched_reduce(&cand, dev->sms, dev->batched_smem, w, ps);
                            if (cand.warps != w || cand.per_sm != ps) continue;   // does not fit
                        } else if (!plan_batched_tiles(&cand, dev->sms, ps == 2 ? 0 : ps) || cand.per_sm < ps) {
                            continue;
                        }
                        POPCORN_CUDA(cudaMemcpyAsync(dI, h.data(), sizeof(BatchInst) * (size_t)count,
                                                     cudaMemcpyHostToDevice, s));
                        if (!rows) POPCORN_CUDA(upload_units());
                        POPCORN_CUDA(stream(cand));   // warm-up
                        float ms = 3.0e38f;
                        for (int rep = 0; rep < 2; ++rep) {
                            POPCORN_CUDA(cudaEventRecord(t0, s));
                            POPCORN_CUDA(stream(cand));
                            POPCORN_CUDA(cudaEventRecord(t1, s));
                            POPCORN_CUDA(cudaEventSynchronize(t1));
                            float e = 0.f;
                            POPCORN_CUDA(cudaEventElapsedTime(&e, t0, t1));
                            ms = e < ms ? e : ms;
                        }
                        // the argmin and the z reduction read every segment's slot, at about 1 TB/s (shorter
                        // units alone stream up to a tenth faster, and lost more than that there)
                        for (int t = 0; t < count; ++t) ms += (float)(4.0 * h[t].nseg * h[t].k * h[t].n / 1e9);
                        ++tune_cands;
                        if (ms < best.ms) {
                            best.ms = ms;
                            best.p[0] = seglen;
                            best.p[1] = cand.warps;
                            best.p[2] = ps;
                            best.p[3] = 0;
                        }
                    }
            int herr = 0;
            POPCORN_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s));
            POPCORN_CUDA(cudaStreamSynchronize(s));
            if (herr) return fail(POPCORN_ERR_TIMEOUT, "a bounded wait in the tensor-core K build ran out");
            if (tune_cands == 0) return fail(POPCORN_ERR_UNSUPPORTED, "no batched schedule fits this device");
            tune_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - w0).count();
            tune_store(key, best);
        }
        sched[0] = std::max(best.p[0], min_seglen);   // (units and Spart are sized for min_seglen)
        sched[1] = best.p[1];
        sched[2] = best.p[2];
    }
    if (!half) {
        set_seglen(sched[0]);
        const bool tuned = sched[2] != 0;
        if (rows) {
            plan_batched_reduce(&bp, dev->sms, dev->batched_smem, sched[1], sched[2]);
        } else {
            POPCORN_CUDA(upload_units());
            if (!plan_batched_tiles(&bp, dev->sms, sched[2] == 1 ? 1 : 0))
                return fail(POPCORN_ERR_UNSUPPORTED, "the batched K stream does not fit this device");
        }
        sched[1] = bp.warps;
        sched[2] = tuned ? std::min(bp.per_sm, 2) : bp.per_sm;
    } else {
        sched[0] = 0;            // whole 128-row blocks a unit
        sched[1] = bp.mstages;   // ring depth of the tensor-core stream
        sched[2] = 1;            // one block an SM
    }
    if (bp.units <= 0 || bp.units >= (1 << 30)) return fail(POPCORN_ERR_UNSUPPORTED, "batch too large");
    POPCORN_CUDA(cudaMemcpyAsync(dI, h.data(), sizeof(BatchInst) * (size_t)count, cudaMemcpyHostToDevice, s));

    // ---- capture the whole batch once
    cudaStream_t cs;
    POPCORN_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    struct StreamGuard {
        cudaStream_t s;
        ~StreamGuard() { cudaStreamDestroy(s); }
    } sg{cs};
    int launches = 0;
    popcorn_status cap = POPCORN_OK;
    POPCORN_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
    auto step = [&](cudaError_t e, const char* what) {
        if (cap == POPCORN_OK && e != cudaSuccess) {
            cudaGetLastError();
            cap = fail(POPCORN_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
        }
    };
    step(launch_batched_init(dI, bp, max_iter, opt.check_convergence ? 1 : 0, tol, cs), "batched init");
    launches += 2;
    if (opt.precision == POPCORN_FP32) {
        step(launch_batched_kbuild_simt(dI, bp, cs), "batched K build");
        launches += 1;
    } else {
        for (int t = 0; t < count && cap == POPCORN_OK; ++t) {
            const BatchInst& b = h[t];
            step(launch_kbuild_tc(b.P, b.n, b.d, b.ldp, b.kp, opt.precision,
                                  half ? reinterpret_cast<float*>(b.Kh) : b.K, rows ? b.ldk : 0, b.kdiag, base + tc_off, err,
                                  dev->sms, cs, &launches, half ? kPackedSw128H : rows ? 0 : kPackedSw4, 0, half),
                 "tensor-core K build");
        }
    }
    step(launch_batched_trace(dI, bp, cs), "batched trace");
    launches += 1;
    // Error-path test hook: with POPCORN_TEST_SYM_STALL_MS=<ms> in the environment, the first
    // K stream of the graph leaves one tile's copies out and bounds its
    // waits by <ms>, so the fit reports POPCORN_ERR_TIMEOUT.  Unset in every ordinary run.
    int stall_ms = 0;
    {
        const char* env = getenv("POPCORN_TEST_SYM_STALL_MS");
        if (env && *env) stall_ms = atoi(env);
        if (stall_ms < 0 || stall_ms > 10000) stall_ms = 0;
    }
    auto pass = [&](int eval) -> cudaError_t {
        const cudaError_t e = half   ? launch_batched_mma_stream(dI, dunits, bp, err, eval, cs, stall_ms)
                              : rows ? launch_batched_reduce(dI, bp, eval, cs)
                                     : launch_batched_tiles(dI, dunits, bp, err, eval, cs, stall_ms);
        stall_ms = 0;
        return e != cudaSuccess ? e : launch_batched_finish(dI, bp, eval, cs);
    };
    for (int it = 0; it < max_iter && cap == POPCORN_OK; ++it) {
        step(pass(0), "batched pass");
        launches += rows ? 3 : 4;
    }
    step(pass(1), "batched objective pass");
    step(launch_batched_copy_labels(dI, bp, cs), "batched label copy");
    launches += rows ? 3 : 4;
    cudaGraph_t graph = nullptr;
    cudaError_t ec = cudaStreamEndCapture(cs, &graph);
    if (cap != POPCORN_OK) {
        if (graph) cudaGraphDestroy(graph);
        return cap;
    }
    POPCORN_CUDA(ec);
    cudaGraphExec_t exec = nullptr;
    cudaError_t ei = cudaGraphInstantiate(&exec, graph, 0);
    cudaGraphDestroy(graph);
    POPCORN_CUDA(ei);
    struct ExecGuard {
        cudaGraphExec_t e;
        ~ExecGuard() { cudaGraphExecDestroy(e); }
    } eg{exec};

    cudaEvent_t e0 = nullptr, e1 = nullptr;
    const bool timing = opt.timing != 0;
    g_events.used = 0;
    if (timing) {
        POPCORN_TRY(g_events.get(&e0));
        POPCORN_TRY(g_events.get(&e1));
        POPCORN_CUDA(cudaEventRecord(e0, s));
    }
    POPCORN_CUDA(cudaGraphLaunch(exec, s));
    if (timing) POPCORN_CUDA(cudaEventRecord(e1, s));
    std::vector<LoopState> hs(count);
    int herr = 0;
    for (int t = 0; t < count; ++t)
        POPCORN_CUDA(cudaMemcpyAsync(&hs[t], h[t].st, sizeof(LoopState), cudaMemcpyDeviceToHost, s));
    POPCORN_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s));
    POPCORN_CUDA(cudaStreamSynchronize(s));
    for (int t = 0; t < count; ++t) {
        if (hs[t].bad_label) return fail(POPCORN_ERR_INVALID, "instance %d: an initial label is outside [0, %d)", t, h[t].k);
        objectives_out[t] = hs[t].J_eval;
        iterations_out[t] = hs[t].iter;
    }
    if (herr) return fail(POPCORN_ERR_TIMEOUT, "a bounded wait in the tensor-core K build or K stream ran out");
    if (info) {
        int conv = 1;
        for (int t = 0; t < count; ++t) conv &= hs[t].converged;
        info->converged = conv;
        info->kernel_launches = launches;
        info->reduce_launches = info->assign_launches = max_iter;
        info->h2d_bytes = info->d2h_bytes = 0;
        info->kbuild_ms = info->reduce_ms = info->assign_ms = info->eval_ms = 0.0;
        info->loop_ms = timing ? elapsed(e0, e1) : 0.0;
        info->tune_cache_hit = tune_hit;
        info->tune_candidates = tune_cands;
        info->tune_ms = tune_ms;
        info->fold_ms = 0.0;
        info->k_pass_used = 0;
        info->sym_form = 0;
        info->schedule[0] = sched[0];
        info->schedule[1] = sched[1];
        info->schedule[2] = sched[2];
        info->schedule[3] = half ? bp.Nmax : 0;
    }
    return POPCORN_OK;
}

}  // extern "C"
