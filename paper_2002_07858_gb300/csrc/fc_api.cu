// fc_api.cu -- host runtime behind the C ABI of include/fc.h.
//
// A context owns one CUDA stream, a device-memory budget, the resident grids
// (spectra, centred BF16 screen image, covariance cache) and a serving worker.
// fc_run_points drives the per-universe procedure of §2 over a batch of true
// points: fake data (step 2), then scans (steps 3-4) with the covariance
// rebuilt at each universe's current best fit (step 5) until it repeats, and
// finally dchi2 (step 6) in residual form.  All arithmetic runs in the
// kernels of fc_kernels.cu / fc_screen.cu; the host only sizes buffers,
// assigns covariance-cache slots and reads back counts between scans.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstddef>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <thread>
#include <unordered_map>
#include <vector>

#include "fc.h"
#include "fc_internal.cuh"

using namespace fcdev;

std::atomic<long long> fcdev::g_launches{0};

namespace {
thread_local std::string t_last_error;
}  // namespace

void fcdev::record_error(const char* msg) { t_last_error = msg ? msg : ""; }

namespace {

fc_status fail(fc_status st, const std::string& msg) {
    t_last_error = msg;
    return st;
}

#define FC_CUDA(call)                                                                           \
    do {                                                                                        \
        cudaError_t e_ = (call);                                                                \
        if (e_ != cudaSuccess)                                                                  \
            return fail(FC_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_));       \
    } while (0)

#define FC_TRY(expr)                  \
    do {                              \
        fc_status s_ = (expr);        \
        if (s_ != FC_OK) return s_;   \
    } while (0)

bool is_device_ptr(const void* p) {
    if (!p) return false;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

// ----------------------------------------------------------------- context --

struct Grid {
    int32_t id = -1;
    int64_t G = 0, G_pad = 0;
    int nf = 0, nfit = 0, K = 0;
    bool has_F = false;
    bool identity_collapse = true;
    double* S_full = nullptr;   // [G][nf]
    double* S_fit = nullptr;    // [G][nfit]
    double* centre = nullptr;   // [nfit]
    double* Sc = nullptr;       // [G][nfit] centred
    float2* Sdf = nullptr;      // [G][nfit] S_fit as double-float (mixed-path residuals)
    float2* centre_df = nullptr;  // [nfit]
    float* Sc32 = nullptr;      // [G][nfit]
    float4* gnorm = nullptr;    // [G] |s~|, |S_lo|, |r_S|
    uint16_t* Bt = nullptr;     // screen B image [G_pad/BN][2K/8][BN/8][8][8]
    int32_t* collapse = nullptr;
    double* F = nullptr;
    // shape-model grids: the model on the device (int and double arrays, sine
    // table included); recompute = no spectra are stored, every row is evaluated
    // where it is read (S_full, S_fit, Sc, Sdf, Sc32 stay null)
    bool recompute = false;
    int32_t* model_i = nullptr;
    double* model_d = nullptr;
    SpecModel model;
    // where kernels read the grid's rows
    GridSpec spec() const {
        GridSpec s;
        s.S_fit = S_fit;
        s.Sc = Sc;
        s.Sc32 = Sc32;
        s.Sdf = Sdf;
        s.centre = centre;
        s.nfit = nfit;
        s.m = model;
        return s;
    }
    FullSrc full() const {
        FullSrc f;
        f.S = S_full;
        f.m = model;
        return f;
    }
    // covariance cache: one slot per grid index used as a fit covariance (plus
    // one for A = I).  Grows by doubling up to max_cap; when full, the slots
    // least recently used by a scan are handed to new indices.
    int64_t cap = 0;                 // slots allocated
    int64_t max_cap = 0;             // memory-derived limit
    int32_t n_slots = 0;             // slot ids handed out so far (high-water mark)
    int64_t epoch = 0;               // ensure_slots calls
    std::vector<int32_t> slot_host;  // [G] grid index -> slot or -1
    std::vector<int32_t> slot_q;     // [cap] slot -> grid index (-2 identity)
    std::vector<int64_t> slot_used;  // [cap] epoch of last use
    int32_t ident_slot = -1;
    int32_t* slot_of = nullptr;      // device [G]
    double* A64 = nullptr;           // [cap][nfit][nfit]
    double* W64 = nullptr;           // [cap][nfit][nfit]  A = W^T W, W lower triangular
    float* Wdf = nullptr;            // [cap][wdf_bytes / 4]  W as double-float, blocked rows
    float* A32 = nullptr;
    float* rho = nullptr;
    uint16_t* Wimg = nullptr;        // [cap][2K][K] bf16 hi/lo image of W (tensor-core q-vectors)
    float4* wnorm = nullptr;         // [cap] Frobenius norms of W, W_lo, r_W, W_hi + W_lo
    float* Qc = nullptr;             // [cap][G_pad] (mixed)
    float* Qb = nullptr;
    uint16_t* Qb3 = nullptr;         // [cap][G_pad][8] bf16 q-step rows of the screen
    double* Q64 = nullptr;           // [cap][G]   (plain)
    std::vector<uint8_t> q32_ready, q64_ready;
    bool unread = false;             // covariances or q-vectors launched whose status the host has not read yet
    fc_tuning tune{};                // kernel choices (all zero: built-in)
    int busy = 0;                    // queued jobs referencing the grid
};

struct Scratch {
    void* p = nullptr;
    size_t bytes = 0;
    bool spare = false;  // only makes a call faster: given up where something it needs finds no room
};

// What the host reads between launches, in one block on the device and one
// pinned mirror, so that a decision costs one small copy and one wait: the
// counts of a scan, its counters, and the status word the kernels raise.
struct Ctrl {
    int32_t cnts[8];                  // [1] failed rows, [2] continuing, [3] finishing, [4] failed again, [5] tiles, [6] rows,
                                      // [7] universes of a wave
    unsigned long long counters[16];  // see scan_once
    int status;                       // kDev* flags, sticky until reported
    int32_t sync_left;                // universes of a synchronous call that have not finished (its lane's job_left)
};
constexpr int32_t kListHost = 4096;   // entries of a device list fetched along with its count
constexpr size_t kStageHost = 256 * 1024;  // bytes of small host lists on their way to the device

// Served job: a copy of the caller's arguments and its completion state.
struct JobRec {
    fc_job job;
    size_t need = 0;  // device bytes the job may take while it runs (admission estimate)
    std::vector<int64_t> ps;
    std::atomic<int> state{FC_PENDING};
    std::atomic<bool> cancelled{false};
    std::chrono::steady_clock::time_point t_submit, t_done;
    std::string error;  // message of a failed job (set before state)
};

// A lane holds the per-universe state of every job that runs with the same
// grid and scan options (precision, top-k bucket, identity or data
// covariance).  Jobs own contiguous universe ranges of the lane; one call of
// scan_once advances every active universe of every job by one scan, whatever
// scan each is on, so a job admitted between two scans joins the next one
// (continuous batching).  A job is complete when its last universe finishes.

constexpr int kLaneJobs = 1024;  // jobs resident in one lane at a time

// Where a job's results go when it completes.
struct LaneJob {
    std::shared_ptr<JobRec> jr;  // null for synchronous calls
    int32_t slot = -1;
    int64_t base = 0, n = 0;
    double* dchi2 = nullptr;     // caller outputs (host or device), nullable
    int64_t* best = nullptr;
    int8_t* nscans = nullptr;
    double* chi2min = nullptr;
    bool done = false;
    fc_status status = FC_OK;
};

struct Lane {
    Grid* g = nullptr;
    fc_opts o{};           // precision, top_k and cov; max_iter and fluct are per job
    int64_t cap = 0;       // universes
    int nfit = 0;
    float* d = nullptr;    // [cap][nfit] data
    int32_t *cur = nullptr, *pt = nullptr, *best = nullptr, *job_of = nullptr;
    int8_t *nscan = nullptr, *maxit = nullptr;
    uint8_t* rmask = nullptr;     // [cap] rounds that decided the universe's scans (FC_DECIDED_*)
    double *dchi2 = nullptr, *chi2min = nullptr;
    float* thr = nullptr;
    int32_t *active = nullptr, *next = nullptr, *fin = nullptr, *uslot = nullptr;
    int32_t *fb = nullptr, *fb2 = nullptr, *fbslot = nullptr;
    int32_t* job_left = nullptr;  // [kLaneJobs]; of the synchronous lane, which holds one job: [1], in the control block
    uint8_t* job_dead = nullptr;  // [kLaneJobs]
    int64_t n_active = 0;
    int64_t n_first = 0;          // universes admitted since the last scan
    std::map<int64_t, int64_t> free_ranges;  // start -> length
    std::vector<int32_t> free_jobs;
    std::vector<std::shared_ptr<LaneJob>> jobs;  // indexed by job slot
};

struct fc_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    size_t budget = 0;
    size_t used = 0;
    int n_sm = 148;
    std::string dev_name;
    std::unordered_map<void*, size_t> allocs;
    std::map<int32_t, std::unique_ptr<Grid>> grids;
    int32_t next_grid = 1;
    std::map<std::string, Scratch> scratch;
    Ctrl* ctrl = nullptr;            // device
    Ctrl* ctrl_host = nullptr;       // pinned; the device's values as of the last read_ctrl
    bool ctrl_read = false;          // nothing that changes the counts was launched since then
    int32_t* list_host = nullptr;    // pinned [kListHost]
    char* stage_host = nullptr;      // pinned [kStageHost]: sources of the copies launched since the last wait
    size_t stage_used = 0;
    int* status_dev = nullptr;       // &ctrl->status
    unsigned long long* counters_dev = nullptr;  // ctrl->counters
    // stage timers: event pairs around the stages since the last flush_stages, and where each one counts
    std::vector<std::pair<cudaEvent_t, cudaEvent_t>> stage_ev;
    std::vector<double*> stage_acc;
    cudaEvent_t run_ev[3] = {nullptr, nullptr, nullptr};
    fc_stats stats{};              // last synchronous call
    fc_stats serve_stats{};        // everything the serving worker ran
    fc_stats* acc = &stats;        // where the running work counts
    Lane sync_lane;                // synchronous calls
    int64_t last_base = 0, last_n = -1;  // universes of the last synchronous fit in sync_lane
    WaitTest wait_test{0, -1};     // test hook of the screen's bounded waits (fc_set_wait_test)
    size_t reserved = 0;           // serving: admission estimates of the running jobs (worker only)
    std::vector<std::unique_ptr<Lane>> lanes;  // serving (worker thread only)
    std::mutex api_mu;  // serialises device work of this context
    // serving
    std::mutex q_mu;
    std::condition_variable q_cv;
    std::deque<std::shared_ptr<JobRec>> queue;
    std::unordered_map<uint64_t, std::shared_ptr<JobRec>> jobs;
    uint64_t next_ticket = 1;
    std::thread worker;
    bool stop = false;
    bool worker_started = false;
};

namespace {

void dfree(fc_ctx* c, void* p);

// Gives up the spare scratch (its users are launched by the time anything else is allocated, and freeing waits
// for them); false: there was none.
bool drop_spare(fc_ctx* c) {
    bool any = false;
    for (auto& kv : c->scratch) {
        Scratch& s = kv.second;
        if (!s.spare || !s.p) continue;
        dfree(c, s.p);
        s.p = nullptr;
        s.bytes = 0;
        any = true;
    }
    return any;
}

fc_status dalloc(fc_ctx* c, void** p, size_t bytes, bool spare = false) {
    *p = nullptr;
    if (bytes == 0) bytes = 16;
    bytes = (bytes + 255) & ~(size_t)255;
    if (!spare && c->budget && c->used + bytes > c->budget) drop_spare(c);
    if (c->budget && c->used + bytes > c->budget)
        return fail(FC_ERR_BUDGET, "device-memory budget exceeded (" + std::to_string(c->used + bytes) + " > " +
                                       std::to_string(c->budget) + " bytes)");
    cudaError_t e = cudaMalloc(p, bytes);
    if (e != cudaSuccess && !spare && drop_spare(c)) {
        cudaGetLastError();
        e = cudaMalloc(p, bytes);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return fail(FC_ERR_BUDGET, std::string("cudaMalloc failed: ") + cudaGetErrorString(e));
    }
    c->used += bytes;
    c->allocs[*p] = bytes;
    return FC_OK;
}

template <class T>
fc_status dalloc_t(fc_ctx* c, T** p, size_t count) {
    void* v = nullptr;
    fc_status s = dalloc(c, &v, count * sizeof(T));
    *p = (T*)v;
    return s;
}

void dfree(fc_ctx* c, void* p) {
    if (!p) return;
    auto it = c->allocs.find(p);
    if (it != c->allocs.end()) {
        c->used -= it->second;
        c->allocs.erase(it);
    }
    cudaFree(p);
}

// grow-only named scratch buffer
template <class T>
fc_status scratch(fc_ctx* c, const char* name, size_t count, T** out, bool spare = false) {
    Scratch& s = c->scratch[name];
    s.spare = spare;
    const size_t bytes = std::max<size_t>(count * sizeof(T), 16);
    if (s.bytes < bytes) {
        dfree(c, s.p);
        s.p = nullptr;
        s.bytes = 0;
        const size_t want = bytes + bytes / 4;
        void* p = nullptr;
        FC_TRY(dalloc(c, &p, want, spare));
        s.p = p;
        s.bytes = want;
    }
    *out = (T*)s.p;
    return FC_OK;
}

void drop_scratch(fc_ctx* c, const char* name) {
    Scratch& s = c->scratch[name];
    dfree(c, s.p);
    s.p = nullptr;
    s.bytes = 0;
}

size_t spare_bytes(const fc_ctx* c) {
    size_t n = 0;
    for (const auto& kv : c->scratch) n += kv.second.spare ? kv.second.bytes : 0;
    return n;
}

// The caller's array where a kernel can read it in place: memory of this context's device, aligned for
// its elements (a misaligned or foreign array is copied instead).
template <class T>
bool readable_in_place(fc_ctx* c, const T* p) {
    cudaPointerAttributes a;
    if (((uintptr_t)p % alignof(T)) != 0 || cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice && a.device == c->device;
}

fc_status copy_in(fc_ctx* c, void* dst, const void* src, size_t bytes) {
    const cudaMemcpyKind k = is_device_ptr(src) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    FC_CUDA(cudaMemcpyAsync(dst, src, bytes, k, c->stream));
    return FC_OK;
}

fc_status copy_out(fc_ctx* c, void* dst, const void* src, size_t bytes) {
    const cudaMemcpyKind k = is_device_ptr(dst) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    FC_CUDA(cudaMemcpyAsync(dst, src, bytes, k, c->stream));
    return FC_OK;
}

// host data to a caller buffer that may be host or device memory
fc_status put_out(fc_ctx* c, void* dst, const void* host_src, size_t bytes) {
    if (is_device_ptr(dst)) {
        FC_CUDA(cudaMemcpyAsync(dst, host_src, bytes, cudaMemcpyHostToDevice, c->stream));
        FC_CUDA(cudaStreamSynchronize(c->stream));
    } else {
        memcpy(dst, host_src, bytes);
    }
    return FC_OK;
}

fc_status sync(fc_ctx* c) {
    FC_CUDA(cudaStreamSynchronize(c->stream));
    c->stage_used = 0;
    FC_CUDA(cudaGetLastError());
    return FC_OK;
}

// Host data of this call to the device, for launches that nothing waits for: a
// copy from pageable memory may still be reading it when the call returns (it
// "might" be synchronous), so the bytes go through the context's pinned block
// and the source may end as soon as this returns.  The block fills up until
// the next wait; what does not fit is copied and waited for.
fc_status to_device(fc_ctx* c, void* dst, const void* src, size_t bytes) {
    if (bytes == 0) return FC_OK;
    const size_t room = (bytes + 15) & ~(size_t)15;
    if (room > kStageHost) {
        FC_CUDA(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, c->stream));
        return sync(c);
    }
    if (c->stage_used + room > kStageHost) FC_TRY(sync(c));
    char* at = c->stage_host + c->stage_used;
    memcpy(at, src, bytes);
    c->stage_used += room;
    FC_CUDA(cudaMemcpyAsync(dst, at, bytes, cudaMemcpyHostToDevice, c->stream));
    return FC_OK;
}

void reset_cache(fc_ctx* c, Grid* g);

// The control block as of now (waits for the stream), and the errors the kernels raised.  With an error the
// grids whose covariances or q-vectors were launched since the last read forget them: one that is not
// positive definite was never written, and the next call has to build it and fail again, not use it.
fc_status read_ctrl(fc_ctx* c) {
    FC_CUDA(cudaMemcpyAsync(c->ctrl_host, c->ctrl, sizeof(Ctrl), cudaMemcpyDeviceToHost, c->stream));
    FC_TRY(sync(c));
    c->ctrl_read = true;
    const int st = c->ctrl_host->status;
    for (auto& kv : c->grids) {
        if (st && kv.second->unread) reset_cache(c, kv.second.get());
        kv.second->unread = false;
    }
    if (st) {
        FC_CUDA(cudaMemsetAsync(c->status_dev, 0, sizeof(int), c->stream));
        if (st & kDevTimeout) return fail(FC_ERR_TIMEOUT, "a device-side wait timed out");
        if (st & kDevNotSpd) return fail(FC_ERR_NOT_SPD, "covariance matrix is not positive definite");
        return fail(FC_ERR_CUDA, "device reported error flags " + std::to_string(st));
    }
    return FC_OK;
}

// After a call that failed half-way: waits for what it launched (its sources may end with it) and takes the
// status it left, which is not the next call's.  The error and its message stay the call's own.
void settle(fc_ctx* c) {
    const std::string msg = t_last_error;
    read_ctrl(c);
    t_last_error = msg;
}

// Stage timing: an event pair on the context stream around a stage's kernels.
// The pairs are read together once the stream has been waited for anyway.
fc_status flush_stages(fc_ctx* c, bool waited) {
    if (!waited) FC_TRY(sync(c));
    for (size_t i = 0; i < c->stage_acc.size(); ++i) {
        float ms = 0.0f;
        FC_CUDA(cudaEventElapsedTime(&ms, c->stage_ev[i].first, c->stage_ev[i].second));
        *c->stage_acc[i] += ms;
    }
    c->stage_acc.clear();
    return FC_OK;
}

fc_status stage_begin(fc_ctx* c) {
    constexpr size_t kMaxStages = 64;
    if (c->stage_acc.size() >= kMaxStages) FC_TRY(flush_stages(c, false));
    if (c->stage_acc.size() == c->stage_ev.size()) {
        cudaEvent_t a = nullptr, b = nullptr;
        FC_CUDA(cudaEventCreate(&a));
        c->stage_ev.emplace_back(a, b);
        FC_CUDA(cudaEventCreate(&b));
        c->stage_ev.back().second = b;
    }
    FC_CUDA(cudaEventRecord(c->stage_ev[c->stage_acc.size()].first, c->stream));
    return FC_OK;
}

fc_status stage_end(fc_ctx* c, double* acc_ms) {
    FC_CUDA(cudaEventRecord(c->stage_ev[c->stage_acc.size()].second, c->stream));
    c->stage_acc.push_back(acc_ms);
    return FC_OK;
}

// x where launch_quantiles can read it: in place, or copied to scratch
fc_status quantile_input(fc_ctx* c, const double* x, size_t count, const double** out) {
    if (readable_in_place(c, x)) {
        *out = x;
        return FC_OK;
    }
    double* dx = nullptr;
    FC_TRY(scratch(c, "qx", count, &dx));
    FC_TRY(copy_in(c, dx, x, count * 8));
    *out = dx;
    return FC_OK;
}

Grid* find_grid(fc_ctx* c, int32_t id) {
    auto it = c->grids.find(id);
    return it == c->grids.end() ? nullptr : it->second.get();
}

void free_cache(fc_ctx* c, Grid* g) {
    dfree(c, g->slot_of); g->slot_of = nullptr;
    dfree(c, g->A64); g->A64 = nullptr;
    dfree(c, g->W64); g->W64 = nullptr;
    dfree(c, g->Wdf); g->Wdf = nullptr;
    dfree(c, g->A32); g->A32 = nullptr;
    dfree(c, g->rho); g->rho = nullptr;
    dfree(c, g->Wimg); g->Wimg = nullptr;
    dfree(c, g->wnorm); g->wnorm = nullptr;
    dfree(c, g->Qc); g->Qc = nullptr;
    dfree(c, g->Qb); g->Qb = nullptr;
    dfree(c, g->Qb3); g->Qb3 = nullptr;
    dfree(c, g->Q64); g->Q64 = nullptr;
    g->cap = 0;
    g->max_cap = 0;
    g->n_slots = 0;
    g->ident_slot = -1;
    g->slot_host.clear();
    g->slot_q.clear();
    g->slot_used.clear();
    g->q32_ready.clear();
    g->q64_ready.clear();
}

// Forget every cached covariance (a new F); storage is kept.
void reset_cache(fc_ctx* c, Grid* g) {
    if (!g->cap) return;
    g->n_slots = 0;
    g->ident_slot = -1;
    std::fill(g->slot_host.begin(), g->slot_host.end(), -1);
    std::fill(g->slot_q.begin(), g->slot_q.end(), -1);
    std::fill(g->slot_used.begin(), g->slot_used.end(), 0);
    std::fill(g->q32_ready.begin(), g->q32_ready.end(), 0);
    std::fill(g->q64_ready.begin(), g->q64_ready.end(), 0);
    launch_fill_i32(g->slot_of, g->G, -1, c->stream);
}

// Device bytes one cache slot costs (covariance, W image, binary32 q-vectors,
// binary64 q-vectors).
size_t slot_bytes(const Grid* g) {
    return (size_t)g->nfit * g->nfit * (8 + 8 + 4) + wdf_bytes(g->nfit) + 4 + (size_t)4 * g->K * g->K + 16 + (size_t)g->G_pad * 24 +
           (size_t)g->G * 8;
}

// Resize one per-slot array from `old_cap` to `new_cap` slots, keeping contents.
template <class T>
fc_status regrow(fc_ctx* c, T** p, size_t per_slot, int64_t old_cap, int64_t new_cap) {
    T* q = nullptr;
    FC_TRY(dalloc_t(c, &q, (size_t)new_cap * per_slot));
    if (*p) {
        FC_CUDA(cudaMemcpyAsync(q, *p, (size_t)old_cap * per_slot * sizeof(T), cudaMemcpyDeviceToDevice, c->stream));
        FC_CUDA(cudaStreamSynchronize(c->stream));
        dfree(c, *p);
    }
    *p = q;
    return FC_OK;
}

// Device memory the covariance caches leave free for scratch, lanes and other
// grids: a tenth of the budget (of the device when there is none), at least
// 2 GiB or a quarter of a budget below 8 GiB.
size_t cache_reserve(fc_ctx* c) {
    size_t free_b = 0, total_b = 0;
    cudaMemGetInfo(&free_b, &total_b);
    const size_t base = c->budget ? c->budget : total_b;
    return std::max<size_t>(base / 10, std::min<size_t>(size_t(2) << 30, base / 4));
}

// Bytes a cache may still take: what the budget (or the device) has left
// above the reserve, with the spare scratch, which gives way.
size_t cache_headroom(fc_ctx* c) {
    size_t free_b = 0, total_b = 0;
    cudaMemGetInfo(&free_b, &total_b);
    const size_t spare = spare_bytes(c);
    size_t room = free_b + spare;
    if (c->budget) room = std::min(room, c->budget + spare > c->used ? c->budget + spare - c->used : 0);
    const size_t res = cache_reserve(c);
    return room > res ? room - res : 0;
}

fc_status grow_cache(fc_ctx* c, Grid* g, int64_t new_cap) {
    const int64_t old = g->cap;
    // the copy needs old and new arrays at once
    if ((size_t)(new_cap - old) * slot_bytes(g) + (size_t)old * slot_bytes(g) > cache_headroom(c) && old > 0)
        return fail(FC_ERR_BUDGET, "covariance cache at its memory limit");
    const size_t n2 = (size_t)g->nfit * g->nfit;
    FC_TRY(regrow(c, &g->A64, n2, old, new_cap));
    FC_TRY(regrow(c, &g->W64, n2, old, new_cap));
    FC_TRY(regrow(c, &g->Wdf, wdf_bytes(g->nfit) / sizeof(float), old, new_cap));
    FC_TRY(regrow(c, &g->A32, n2, old, new_cap));
    FC_TRY(regrow(c, &g->rho, 1, old, new_cap));
    if (g->Wimg) FC_TRY(regrow(c, &g->Wimg, (size_t)2 * g->K * g->K, old, new_cap));
    if (g->wnorm) FC_TRY(regrow(c, &g->wnorm, 1, old, new_cap));
    if (g->Qc) {
        FC_TRY(regrow(c, &g->Qc, (size_t)g->G_pad, old, new_cap));
        FC_TRY(regrow(c, &g->Qb, (size_t)g->G_pad, old, new_cap));
        FC_TRY(regrow(c, &g->Qb3, (size_t)g->G_pad * 8, old, new_cap));
    }
    if (g->Q64) FC_TRY(regrow(c, &g->Q64, (size_t)g->G, old, new_cap));
    g->cap = new_cap;
    g->slot_q.resize(new_cap, -1);
    g->slot_used.resize(new_cap, 0);
    g->q32_ready.resize(new_cap, 0);
    g->q64_ready.resize(new_cap, 0);
    return FC_OK;
}

// Grow the cache towards `need` slots (doubling), as far as `lim` and memory allow.
void grow_for(fc_ctx* c, Grid* g, int64_t need, int64_t lim) {
    if (g->cap >= std::min(need, lim)) return;
    int64_t target = std::min<int64_t>(lim, std::max<int64_t>(2 * g->cap, need));
    target = std::min<int64_t>(target, (int64_t)(cache_headroom(c) / slot_bytes(g)));
    if (target > g->cap && grow_cache(c, g, target) != FC_OK) cudaGetLastError();
}

// Covariance cache of a grid: at most one slot per grid index (plus A = I);
// it grows while cache_headroom allows and evicts beyond that.
fc_status ensure_cache(fc_ctx* c, Grid* g) {
    if (g->cap) return FC_OK;
    // the slot count is bounded by the grid; memory decides at each growth step
    g->max_cap = g->G + 1;
    if ((int64_t)(cache_headroom(c) / slot_bytes(g)) < 2) return fail(FC_ERR_BUDGET, "no room for the covariance cache");
    g->slot_host.assign(g->G, -1);
    FC_TRY(dalloc_t(c, &g->slot_of, g->G));
    launch_fill_i32(g->slot_of, g->G, -1, c->stream);
    return grow_cache(c, g, std::min<int64_t>(g->max_cap, 32));
}

fc_status ensure_q32_storage(fc_ctx* c, Grid* g) {
    // each by itself: an earlier call may have had room for some of them only
    if (!g->Qc) FC_TRY(dalloc_t(c, &g->Qc, (size_t)g->cap * g->G_pad));
    if (!g->Qb) FC_TRY(dalloc_t(c, &g->Qb, (size_t)g->cap * g->G_pad));
    if (!g->Qb3) FC_TRY(dalloc_t(c, &g->Qb3, (size_t)g->cap * g->G_pad * 8));
    return FC_OK;
}

fc_status ensure_q64_storage(fc_ctx* c, Grid* g) {
    if (g->Q64) return FC_OK;
    FC_TRY(dalloc_t(c, &g->Q64, (size_t)g->cap * g->G));
    return FC_OK;
}

// q-vector kernel of a grid: the tensor-core form unless the grid's tuning asks
// for the binary32 one (measured faster at every K, including N_fit = 45).
bool use_qvec_tc(const Grid* g) {
    if (!qvec_tc_supported(g->K)) return false;
    return g->tune.qvec != FC_QVEC_SIMT;
}

// Make sure every grid index in `qs` has a covariance slot (build + invert the
// missing ones) and, for the given path, its q-vector.  The slots of `qs` are
// all resident when this returns: they are marked as used by this call, so a
// full cache hands out only slots that this call does not need.  The kernels
// are launched, not waited for: a covariance that is not positive definite
// raises the status word, which the next read_ctrl reports.
fc_status fill_slots(fc_ctx* c, Grid* g, const std::vector<int32_t>& qs, int cov_mode, bool need_q32,
                       bool need_q64, std::vector<int32_t>* slots_out) {
    FC_TRY(ensure_cache(c, g));
    const int64_t ep = ++g->epoch;
    std::vector<int32_t> new_q, new_s, q32_list, q64_list, evicted_q;
    if (slots_out) slots_out->clear();
    // a slot for one more grid index: unused id, else grow, else the least recently used
    std::vector<int32_t> lru;  // candidates for eviction, oldest first (built on first need)
    size_t lru_pos = 0;
    const int64_t lim = g->tune.cache_slots > 0 ? std::min<int64_t>(g->tune.cache_slots, g->max_cap) : g->max_cap;
    auto take_slot = [&](int32_t* out) -> fc_status {
        if (g->n_slots >= g->cap) grow_for(c, g, g->n_slots + 1, lim);
        if (g->n_slots < std::min<int64_t>(g->cap, lim)) {
            *out = g->n_slots++;
            return FC_OK;
        }
        if (lru.empty()) {
            for (int32_t s = 0; s < g->n_slots; ++s)
                if (g->slot_used[s] < ep && s != g->ident_slot) lru.push_back(s);
            std::sort(lru.begin(), lru.end(),
                      [&](int32_t a, int32_t b) { return g->slot_used[a] < g->slot_used[b]; });
        }
        while (lru_pos < lru.size() && g->slot_used[lru[lru_pos]] >= ep) ++lru_pos;
        if (lru_pos >= lru.size())
            return fail(FC_ERR_BUDGET, "covariance cache (" + std::to_string(g->cap) +
                                           " slots) cannot hold the covariances of one scan");
        const int32_t s = lru[lru_pos++];
        const int32_t q_old = g->slot_q[s];
        if (q_old >= 0) {
            g->slot_host[q_old] = -1;
            evicted_q.push_back(q_old);
        }
        g->q32_ready[s] = 0;
        g->q64_ready[s] = 0;
        *out = s;
        return FC_OK;
    };
    if (cov_mode == FC_COV_IDENTITY) {
        if (g->ident_slot < 0) {
            int32_t s = -1;
            FC_TRY(take_slot(&s));
            g->ident_slot = s;
            g->slot_q[s] = -2;
            new_q.push_back(0);
            new_s.push_back(s);
        }
        g->slot_used[g->ident_slot] = ep;
        if (slots_out) slots_out->push_back(g->ident_slot);
    } else {
        for (int32_t q : qs) {
            const int32_t s = g->slot_host[q];
            if (s >= 0) g->slot_used[s] = ep;
        }
        for (int32_t q : qs) {
            int32_t s = g->slot_host[q];
            if (s < 0) {
                FC_TRY(take_slot(&s));
                g->slot_host[q] = s;
                g->slot_q[s] = q;
                g->slot_used[s] = ep;
                new_q.push_back(q);
                new_s.push_back(s);
            }
            if (slots_out) slots_out->push_back(s);
        }
    }
    auto want_q = [&](int32_t s) {
        if (need_q32 && !g->q32_ready[s]) { q32_list.push_back(s); g->q32_ready[s] = 1; }
        if (need_q64 && !g->q64_ready[s]) { q64_list.push_back(s); g->q64_ready[s] = 1; }
    };
    if (cov_mode == FC_COV_IDENTITY) {
        want_q(g->ident_slot);
    } else {
        for (int32_t q : qs) want_q(g->slot_host[q]);
    }
    int32_t *dq = nullptr, *ds = nullptr;
    const size_t nn = std::max(std::max(new_q.size(), evicted_q.size()), std::max(q32_list.size(), q64_list.size()));
    FC_TRY(scratch(c, "slot_q", nn + 1, &dq));
    FC_TRY(scratch(c, "slot_s", nn + 1, &ds));
    if (!evicted_q.empty()) {
        // evicted grid indices lose their slot on the device too
        std::vector<int32_t> minus(evicted_q.size(), -1);
        FC_TRY(to_device(c, dq, evicted_q.data(), evicted_q.size() * 4));
        FC_TRY(to_device(c, ds, minus.data(), minus.size() * 4));
        launch_set_slots(dq, ds, (int)evicted_q.size(), g->slot_of, c->stream);
        c->acc->evicted += (int64_t)evicted_q.size();
    }
    if (!new_q.empty() || !q32_list.empty() || !q64_list.empty()) g->unread = true;
    if (!new_q.empty()) {
        FC_TRY(to_device(c, dq, new_q.data(), new_q.size() * 4));
        FC_TRY(to_device(c, ds, new_s.data(), new_s.size() * 4));
        launch_build_cov(g->full(), g->nf, g->nfit, g->identity_collapse ? nullptr : g->collapse, g->F, dq, ds,
                         (int)new_q.size(), cov_mode == FC_COV_IDENTITY ? 2 : 0, g->A64, g->W64, g->A32, g->rho,
                         c->n_sm, c->status_dev, c->stream);
        launch_wdf(g->W64, ds, (int)new_q.size(), g->nfit, g->Wdf, c->stream);
        if (cov_mode != FC_COV_IDENTITY) launch_set_slots(dq, ds, (int)new_q.size(), g->slot_of, c->stream);
        c->acc->distinct_cov += (int64_t)new_q.size();
    }
    if (!q32_list.empty()) {
        FC_TRY(ensure_q32_storage(c, g));
        FC_TRY(to_device(c, ds, q32_list.data(), q32_list.size() * 4));
        if (use_qvec_tc(g)) {
            if (!g->Wimg) FC_TRY(dalloc_t(c, &g->Wimg, (size_t)g->cap * 2 * g->K * g->K));
            if (!g->wnorm) FC_TRY(dalloc_t(c, &g->wnorm, (size_t)g->cap));
            launch_wimage(g->W64, ds, (int)q32_list.size(), g->nfit, g->K, g->Wimg, g->wnorm, c->stream);
            launch_qvec_tc(g->Bt, g->Wimg, g->wnorm, g->gnorm, ds, (int)q32_list.size(), g->G, g->G_pad, g->nfit,
                           g->K, g->Qc, g->Qb, g->Qb3, c->status_dev, c->n_sm, c->stream);
        } else {
            launch_qvec32(g->spec(), g->gnorm, g->G, g->G_pad, g->nfit, g->A32, g->rho, ds, (int)q32_list.size(),
                          g->Qc, g->Qb, g->Qb3, c->stream);
        }
    }
    if (!q64_list.empty()) {
        FC_TRY(ensure_q64_storage(c, g));
        FC_TRY(to_device(c, ds, q64_list.data(), q64_list.size() * 4));
        launch_qvec64(g->spec(), g->G, g->nfit, g->W64, ds, (int)q64_list.size(), g->G, g->Q64, c->stream);
    }
    return FC_OK;
}

fc_status ensure_slots(fc_ctx* c, Grid* g, const std::vector<int32_t>& qs, int cov_mode, bool need_q32,
                       bool need_q64, std::vector<int32_t>* slots_out) {
    const fc_status st = fill_slots(c, g, qs, cov_mode, need_q32, need_q64, slots_out);
    // slots are handed out before they are filled: after an error none of them can be told from a filled one
    if (st != FC_OK) reset_cache(c, g);
    return st;
}

fc_status validate_opts(const fc_opts* o, const Grid* g) {
    if (o->max_iter < 1 || o->max_iter > 127) return fail(FC_ERR_ARG, "max_iter must be in [1, 127]");
    if (o->precision != FC_PREC_FP64 && o->precision != FC_PREC_MIXED) return fail(FC_ERR_ARG, "bad precision");
    if (o->top_k < 1 || o->top_k > kMaxTopK) return fail(FC_ERR_ARG, "top_k must be in [1, 16]");
    if (o->fluct != FC_FLUCT_POISSON_SYS && o->fluct != FC_FLUCT_GAUSS) return fail(FC_ERR_ARG, "bad fluct");
    if (o->cov < FC_COV_ITERATE || o->cov > FC_COV_IDENTITY) return fail(FC_ERR_ARG, "bad cov mode");
    if (o->precision == FC_PREC_MIXED && g->K > kMaxScreenK)
        return fail(FC_ERR_ARG, "no tensor-core screen for this N_fit (use FC_PREC_FP64)");
    return FC_OK;
}

__global__ void k_widen(const int32_t* __restrict__ a, int64_t n, int64_t* __restrict__ b) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) b[i] = a[i];
}

__global__ void k_gather_cur(const int32_t* __restrict__ list, int n, const int32_t* __restrict__ cur,
                             int32_t* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = cur[list[i]];
}

// State of a newly admitted job's universes base .. base+n-1: universe i of
// the job belongs to true point ps[i / U]; its first covariance is that point's
// (§2 step 3 starts from M at the true point).  The universes are appended to
// the lane's active list at `tail`.
__global__ void k_lane_admit(const int64_t* __restrict__ ps, int64_t n, int U, int64_t base, int8_t max_iter,
                             int32_t job, int32_t* __restrict__ cur, int32_t* __restrict__ pt,
                             int8_t* __restrict__ nscan, int8_t* __restrict__ maxit, uint8_t* __restrict__ rmask,
                             int32_t* __restrict__ job_of, int32_t* __restrict__ tail) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t u = base + i;
    const int32_t p = (int32_t)ps[i / U];
    cur[u] = p;
    pt[u] = p;
    nscan[u] = 0;
    maxit[u] = max_iter;
    rmask[u] = 0;
    job_of[u] = job;
    tail[i] = (int32_t)u;
}

// Drop the universes of cancelled jobs from an active list.
__global__ void k_drop_jobs(const int32_t* __restrict__ active, int64_t n, const int32_t* __restrict__ job_of,
                            const uint8_t* __restrict__ dead, int32_t* __restrict__ out, int32_t* __restrict__ n_out) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int32_t u = active[i];
    if (!dead[job_of[u]]) out[atomicAdd(n_out, 1)] = u;
}

__global__ void k_flag_list(const int32_t* __restrict__ q, int n, uint8_t* __restrict__ flag) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) flag[q[i]] = 1;
}

// The universes of `active` whose covariance index at the start of the scan
// (cur0, by list position) is flagged, in any order.
__global__ void k_select_cur(const int32_t* __restrict__ active, int64_t n, const int32_t* __restrict__ cur0,
                             const uint8_t* __restrict__ flag, int32_t* __restrict__ out, int32_t* __restrict__ n_out) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (flag[cur0[i]]) out[atomicAdd(n_out, 1)] = active[i];
}

__global__ void k_gather_int2(const int32_t* __restrict__ list, int n, const int2* __restrict__ src,
                              int2* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = src[list[i]];
}

__global__ void k_scatter_lists(const int32_t* __restrict__ u, int n, const int64_t* __restrict__ off,
                                const int2* __restrict__ cnt, int64_t* __restrict__ loff, int2* __restrict__ lnum) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        loff[u[i]] = off[i];
        lnum[u[i]] = cnt[i];
    }
}

// Longest candidate list (both half rows) rescored from a fourth screen round;
// longer ones take the exact scan.
constexpr int64_t kBigList = 1 << 16;

inline unsigned nb(int64_t n, int t = 256) { return (unsigned)std::max<int64_t>(1, (n + t - 1) / t); }

// Distinct grid indices currently used as fit covariances by the active set.
fc_status distinct_cur(fc_ctx* c, Grid* g, const int32_t* active, int64_t n_active, const int32_t* cur,
                       std::vector<int32_t>& out) {
    uint8_t* flag = nullptr;
    int32_t* list = nullptr;  // [0]: count, then the indices
    const size_t room = (size_t)std::min<int64_t>(g->G, n_active) + 1;
    FC_TRY(scratch(c, "flag", (size_t)g->G, &flag));
    FC_TRY(scratch(c, "dlist", room, &list));
    FC_CUDA(cudaMemsetAsync(flag, 0, (size_t)g->G, c->stream));
    FC_CUDA(cudaMemsetAsync(list, 0, 4, c->stream));
    launch_mark_used(active, n_active, cur, flag, c->stream);
    launch_compact_flags(flag, g->G, list + 1, list, c->stream);
    const size_t first = std::min<size_t>(room, kListHost);
    FC_CUDA(cudaMemcpyAsync(c->list_host, list, first * 4, cudaMemcpyDeviceToHost, c->stream));
    FC_TRY(read_ctrl(c));
    const size_t h = (size_t)c->list_host[0];
    out.assign(c->list_host + 1, c->list_host + std::min(h + 1, first));
    if (h + 1 > first) {
        out.resize(h);
        FC_CUDA(cudaMemcpyAsync(out.data() + (first - 1), list + first, (h + 1 - first) * 4, cudaMemcpyDeviceToHost,
                                c->stream));
        FC_TRY(sync(c));
    }
    std::sort(out.begin(), out.end());
    return FC_OK;
}

// ------------------------------------------------------------------ lanes ---

void lane_free(fc_ctx* c, Lane* L) {
    if (c->ctrl && L->job_left == &c->ctrl->sync_left) L->job_left = nullptr;
    for (void* p : {(void*)L->d, (void*)L->cur, (void*)L->pt, (void*)L->best, (void*)L->job_of, (void*)L->nscan,
                    (void*)L->maxit, (void*)L->rmask, (void*)L->dchi2, (void*)L->chi2min, (void*)L->thr, (void*)L->active,
                    (void*)L->next, (void*)L->fin, (void*)L->uslot, (void*)L->fb, (void*)L->fb2, (void*)L->fbslot,
                    (void*)L->job_left, (void*)L->job_dead})
        dfree(c, p);
    *L = Lane{};
}

void lane_reset(Lane* L) {
    L->n_active = 0;
    L->n_first = 0;
    L->free_ranges.clear();
    L->free_ranges[0] = L->cap;
    L->free_jobs.clear();
    for (int j = kLaneJobs - 1; j >= 0; --j) L->free_jobs.push_back(j);
    L->jobs.assign(kLaneJobs, nullptr);
}

fc_status lane_alloc(fc_ctx* c, Lane* L, Grid* g, const fc_opts& o, int64_t cap) {
    lane_free(c, L);
    L->g = g;
    L->o = o;
    L->cap = cap;
    L->nfit = g->nfit;
    fc_status st = FC_OK;
    auto A = [&](auto** p, size_t count) {
        if (st == FC_OK) st = dalloc_t(c, p, count);
    };
    A(&L->d, (size_t)cap * g->nfit);
    A(&L->cur, cap);
    A(&L->pt, cap);
    A(&L->best, cap);
    A(&L->job_of, cap);
    A(&L->nscan, cap);
    A(&L->maxit, cap);
    A(&L->rmask, cap);
    A(&L->dchi2, cap);
    A(&L->chi2min, cap);
    A(&L->thr, cap);
    A(&L->active, cap);
    A(&L->next, cap);
    A(&L->fin, cap);
    A(&L->uslot, cap);
    A(&L->fb, cap);
    A(&L->fb2, cap);
    A(&L->fbslot, cap);
    if (L == &c->sync_lane)
        L->job_left = &c->ctrl->sync_left;
    else
        A(&L->job_left, kLaneJobs);
    A(&L->job_dead, kLaneJobs);
    if (st != FC_OK) {
        lane_free(c, L);
        return st;
    }
    FC_CUDA(cudaMemsetAsync(L->job_dead, 0, kLaneJobs, c->stream));
    lane_reset(L);
    return FC_OK;
}

bool lane_reserve(Lane* L, int64_t n, int64_t* base) {
    if (L->free_jobs.empty()) return false;
    for (auto it = L->free_ranges.begin(); it != L->free_ranges.end(); ++it) {
        if (it->second >= n) {
            *base = it->first;
            const int64_t rest = it->second - n;
            L->free_ranges.erase(it);
            if (rest) L->free_ranges[*base + n] = rest;
            return true;
        }
    }
    return false;
}

void lane_release(Lane* L, int64_t base, int64_t n) {
    auto it = L->free_ranges.emplace(base, n).first;
    auto nx = std::next(it);
    if (nx != L->free_ranges.end() && it->first + it->second == nx->first) {
        it->second += nx->second;
        L->free_ranges.erase(nx);
    }
    if (it != L->free_ranges.begin()) {
        auto pv = std::prev(it);
        if (pv->first + pv->second == it->first) {
            pv->second += it->second;
            L->free_ranges.erase(it);
        }
    }
}

// No job resident (an unallocated lane, cap 0, has none either).
bool lane_idle(const Lane* L) { return L->cap == 0 || L->free_jobs.size() == (size_t)kLaneJobs; }

// Admit a job into reserved range [base, base+n): data (fake, from the job's
// seed, or the caller's), per-universe state, active-list entries.  On error
// nothing of the job is left in the lane.
//   ps_dev  [P] true points (device)      d_in  caller data [n][nfit] or NULL
fc_status lane_admit(fc_ctx* c, Lane* L, const std::shared_ptr<LaneJob>& J, const int64_t* ps_host, int32_t P,
                     int32_t U, uint64_t seed, int fluct, int max_iter, const float* d_in) {
    Grid* g = L->g;
    const int64_t n = J->n;
    int64_t* ps_dev = nullptr;
    FC_TRY(scratch(c, "ps", (size_t)P, &ps_dev));
    FC_TRY(to_device(c, ps_dev, ps_host, (size_t)P * 8));
    float* dst = L->d + (size_t)J->base * g->nfit;
    if (d_in) {
        FC_TRY(copy_in(c, dst, d_in, (size_t)n * g->nfit * sizeof(float)));
    } else {
        double* L64 = nullptr;
        float *L32 = nullptr, *s32 = nullptr;
        FC_TRY(scratch(c, "L64", (size_t)P * g->nf * g->nf, &L64));
        FC_TRY(scratch(c, "L32", (size_t)P * g->nf * g->nf, &L32));
        FC_TRY(scratch(c, "s32", (size_t)P * g->nf, &s32));
        launch_chol_sys(g->full(), g->nf, g->F, ps_dev, P, fluct == FC_FLUCT_GAUSS, L64, L32, s32, c->n_sm,
                        c->status_dev, c->stream);
        // a served job's own factor must not fail the jobs it would join; a synchronous call reports it
        // with the first count it reads
        if (J->jr) FC_TRY(read_ctrl(c));
        launch_fake_data(L32, s32, g->nf, g->identity_collapse ? nullptr : g->collapse, g->nfit, ps_dev, P, U, seed,
                         fluct == FC_FLUCT_GAUSS, dst, c->n_sm, c->stream);
    }
    count_launch();
    k_lane_admit<<<nb(n), 256, 0, c->stream>>>(ps_dev, n, U, J->base, (int8_t)max_iter, J->slot, L->cur, L->pt,
                                               L->nscan, L->maxit, L->rmask, L->job_of,
                                               L->active + L->n_active);
    launch_fill_i32(L->job_left + J->slot, 1, (int32_t)n, c->stream);
    FC_CUDA(cudaGetLastError());
    L->jobs[J->slot] = J;
    L->n_active += n;
    L->n_first += n;
    return FC_OK;
}

// One scan (§2 steps 3-5) of every active universe of the lane: covariances
// at each universe's current index, the scan itself (plain binary64, or the
// tensor-core screen with certified binary64 resolution), and the advance /
// finish bookkeeping.  Universes that finish get dchi2 and leave the active
// list; the others continue from their new minimum in the next call.
fc_status scan_once(fc_ctx* c, Lane* L) {
    Grid* g = L->g;
    const fc_opts& o = L->o;
    fc_stats* S = c->acc;
    const int64_t n_active = L->n_active;
    if (n_active == 0) return FC_OK;
    const bool mixed = (o.precision == FC_PREC_MIXED);
    const int topk = o.top_k <= 4 ? 4 : (o.top_k <= 8 ? 8 : 16);
    // The probe at the true point is a loose first seed; when most universes
    // are on their first scan a min-only pass tightens the seeds first.
    const bool first_heavy = 2 * L->n_first >= n_active;
    L->n_first = 0;
    // round 1's failures go straight to the list round unless the top-16 round is asked for: the
    // failures are few per covariance, so each round costs its sparse tiles, and one round fewer was
    // faster on the 100x100 (N 90->45) and 64^3 (N 120) grids
    const bool skip16 = mixed && g->tune.first_round != FC_ROUND_TOPK;
    int32_t *active = L->active, *next = L->next, *fin = L->fin, *uslot = L->uslot, *cur = L->cur;
    const float* d = L->d;
    int32_t* cnts = c->ctrl->cnts;
    const int32_t* h_cnts = c->ctrl_host->cnts;  // valid after read_ctrl
    c->stage_acc.clear();                        // of a scan that ended in an error
    UniverseState us;
    us.cur = L->cur;
    us.pt = L->pt;
    us.nscan = L->nscan;
    us.maxit = L->maxit;
    us.job_of = L->job_of;
    us.job_left = L->job_left;
    us.status = c->status_dev;
    us.G = g->G;
    // counts ([2], the continuing universes, is the whole scan's) and counters; not the status
    FC_CUDA(cudaMemsetAsync(c->ctrl, 0, offsetof(Ctrl, status), c->stream));
    c->ctrl_read = false;
    // exact scan for `list`, then advance / finish them; lslot: their slots (null: looked up here)
    auto exact_scan = [&](const int32_t* list, int64_t cnt, const int32_t* lslot) -> fc_status {
        c->ctrl_read = false;
        if (!lslot) {
            int32_t* fslot = nullptr;
            FC_TRY(scratch(c, "fslot", (size_t)cnt, &fslot));
            if (o.cov == FC_COV_IDENTITY)
                launch_fill_i32(fslot, cnt, g->ident_slot, c->stream);
            else
                launch_lookup_slots(list, cnt, cur, g->slot_of, fslot, c->stream);
            lslot = fslot;
        }
        if (mixed) {
            // the mixed path's last resort: residual form for every g, no binary64 q-vectors.
            // enough CTAs to cover the GPU about four times, each at least 1024 grid points
            int nsp = (int)std::max<int64_t>(1, (4 * (int64_t)c->n_sm + cnt - 1) / cnt);
            nsp = (int)std::min<int64_t>(nsp, std::max<int64_t>(1, g->G / 1024));
            double* pv = nullptr;
            int32_t* pg = nullptr;
            FC_TRY(scratch(c, "fb_pv", (size_t)cnt * nsp, &pv));
            FC_TRY(scratch(c, "fb_pg", (size_t)cnt * nsp, &pg));
            FC_TRY(stage_begin(c));
            launch_scan_resid(list, cnt, lslot, d, g->spec(), g->G, g->nfit, g->Wdf, pv, pg, nsp, L->best,
                              c->stream);
            S->residuals += cnt * g->G;
            FC_TRY(stage_end(c, &S->ms_fallback));
        } else {
            int nsp = scan64_splits(cnt, g->G, c->n_sm);
            double *pv = nullptr, *py = nullptr;
            int32_t* pg = nullptr;
            if (nsp > 1 && (scratch(c, "s64_y", (size_t)cnt * g->nfit, &py, true) != FC_OK ||
                            scratch(c, "s64_pv", (size_t)cnt * nsp, &pv, true) != FC_OK ||
                            scratch(c, "s64_pg", (size_t)cnt * nsp, &pg, true) != FC_OK))
                nsp = 1;  // no room for the partial minima
            FC_TRY(stage_begin(c));
            launch_scan64(list, cnt, lslot, d, g->spec(), g->G, g->nfit, g->A64, g->Q64, g->G, L->best, nsp, py, pv,
                          pg, c->stream);
            FC_TRY(stage_end(c, &S->ms_scan64));
        }
        launch_or_mask(list, cnt, mixed ? kDecidedScan : kDecidedPlain, L->rmask, c->stream);
        // finishing universes keep cur (the covariance of this scan); others move to their minimum
        FC_CUDA(cudaMemsetAsync(cnts + 3, 0, 4, c->stream));
        launch_advance(list, cnt, L->best, us, next, cnts + 2, fin, cnts + 3, c->stream);
        // as many as finish, a count that stays on the device
        FC_TRY(stage_begin(c));
        launch_finish(fin, cnt, cnts + 3, o.cov == FC_COV_IDENTITY ? g->ident_slot : -1, g->slot_of, L->best, us, d,
                      g->spec(), g->nfit, g->W64, mixed ? g->Wdf : nullptr, L->dchi2, L->chi2min, c->stream);
        FC_TRY(stage_end(c, &S->ms_finish));
        if (mixed) {
            FC_TRY(read_ctrl(c));
            S->residuals += 2 * (int64_t)h_cnts[3];
        }
        return FC_OK;
    };
    bool first_list = true;
    // one scan of the universes in `list` (their covariance slots in lslot, by list position)
    auto scan_list = [&](const int32_t* sl_list, int64_t sl_n, const int32_t* sl_slot) -> fc_status {
        if (!first_list) {  // a later wave: the scan's first list finds the counts cleared
            FC_CUDA(cudaMemsetAsync(cnts + 3, 0, 12, c->stream));  // n_fin, n_fb2, n_tiles
            FC_CUDA(cudaMemsetAsync(cnts + 1, 0, 4, c->stream));   // n_fb
        }
        first_list = false;
        if (!mixed) {
            FC_TRY(exact_scan(sl_list, sl_n, sl_slot));
        } else {
            int32_t *fb = L->fb, *fb2 = L->fb2, *fslot = L->fbslot;
            float* thr = L->thr;
            int2* lcount = nullptr;
            FC_TRY(scratch(c, "lcount", (size_t)L->cap, &lcount));
            // one certified screen round over `list` (grouped into tiles by covariance slot)
            // rounds 2 and 3 list candidates; round 3 stores them in the exact-size regions
            // loff / lnum (u-indexed, list_total entries) sized by round 2's overflow counts
            // seeded: the rows carry an upper bound of their minimum from an earlier round (thr); else
            // the probe seeds them, tightened by a min-only pass when most rows are on their first scan
            auto screen_round = [&](int round, const int32_t* list, int64_t cnt, const int32_t* lslot, int rtopk,
                                    int32_t* fb_out, int32_t* n_fb_out, bool seeded,
                                    const int64_t* loff = nullptr, const int2* lnum = nullptr,
                                    int64_t list_total = 0) -> fc_status {
                const bool listing = (round >= 2);
                const int64_t n_slots = g->n_slots;
                const int64_t max_tiles = cnt / kBM + std::min<int64_t>(n_slots, cnt) + 1;
                const std::string sfx = round ? std::to_string(round + 1) : "";
                int32_t *tcnt = nullptr, *tbase = nullptr, *tfill = nullptr, *tslot = nullptr, *tuniv = nullptr,
                        *tj0 = nullptr, *cidx = nullptr;
                uint16_t* Yt = nullptr;
                float *cval = nullptr, *tau0 = nullptr;
                float4* alpha = nullptr;
                FC_TRY(scratch(c, "tcnt", (size_t)n_slots, &tcnt));
                FC_TRY(scratch(c, "tbase", (size_t)n_slots + 1, &tbase));
                FC_TRY(scratch(c, "tfill", (size_t)n_slots, &tfill));
                FC_TRY(scratch(c, ("tslot" + sfx).c_str(), (size_t)max_tiles * kQuads, &tslot));
                FC_TRY(scratch(c, ("tuniv" + sfx).c_str(), (size_t)max_tiles * kBM, &tuniv));
                FC_TRY(scratch(c, ("Yt" + sfx).c_str(), (size_t)max_tiles * kBM * 2 * g->K, &Yt));
                FC_TRY(scratch(c, ("alpha" + sfx).c_str(), (size_t)max_tiles * kBM, &alpha));
                FC_TRY(scratch(c, ("tau0" + sfx).c_str(), (size_t)max_tiles * kBM, &tau0));
                FC_TRY(scratch(c, ("tile_j0" + sfx).c_str(), (size_t)max_tiles, &tj0));
                const size_t per_row = listing ? 2 * kListCap : rtopk;
                const size_t n_cand = loff ? (size_t)list_total : (size_t)max_tiles * kBM * per_row;
                int32_t* ccount = nullptr;
                FC_TRY(scratch(c, ("cval" + sfx).c_str(), n_cand, &cval));
                FC_TRY(scratch(c, ("cidx" + sfx).c_str(), n_cand, &cidx));
                FC_TRY(scratch(c, "ccount", (size_t)max_tiles * kBM * 2, &ccount));
                FC_TRY(stage_begin(c));
                launch_group(list, cnt, lslot, (int)n_slots, tcnt, tbase, tfill, cnts + 5, tslot, tuniv, max_tiles,
                             g->tune.slot_rows ? g->tune.slot_rows : kQuadRows, c->stream);
                FC_TRY(read_ctrl(c));
                c->ctrl_read = false;
                const int32_t n_tiles = h_cnts[5];
                launch_yprep(tslot, tuniv, n_tiles, d, g->centre_df, g->nfit, g->K, g->A32, g->rho, cur, g->spec(),
                             g->gnorm, g->Qc, g->Qb, g->G_pad, Yt, alpha, tau0, tj0, c->stream);
                if (seeded) launch_min_tau(tuniv, n_tiles, thr, tau0, c->stream);
                FC_TRY(stage_end(c, &S->ms_prep));
                FC_TRY(stage_begin(c));
                // round 0: a min-only pass to tighten the seeds when most rows are on their first scan (the probe
                // at the true point is loose there; later scans probe at the previous minimum), then the top-k
                // pass.  Later rounds are seeded by the best binary64 value (round 1: top-k, round 2: list).
                const bool min_pass = (!seeded && first_heavy);
                ScreenSplit ss;
                ss.parts = screen_parts(n_tiles, g->G_pad, c->n_sm, &ss.len);
                if (ss.parts > 1) {
                    // a split that has no room for its storage runs unsplit
                    const size_t rows = (size_t)n_tiles * kBM, cand = listing ? 0 : rows * ss.parts * rtopk;
                    if ((min_pass && scratch(c, "split_key", rows, &ss.key, true) != FC_OK) ||
                        (cand && (scratch(c, "split_val", cand, &ss.val, true) != FC_OK ||
                                  scratch(c, "split_idx", cand, &ss.idx, true) != FC_OK)))
                        ss.parts = 1;
                }
                for (int pass = min_pass ? 0 : 1; pass < 2; ++pass) {
                    const int mode = pass == 0 ? kScreenMin : (listing ? kScreenList : kScreenTopK);
                    if (!launch_screen(g->K, rtopk, mode, g->tune.screen_stages, g->tune.screen_ybuf, Yt, g->Bt, g->Qb3,
                                       tslot, tau0, tj0, n_tiles, g->G, g->G_pad, cval, cidx, ccount, c->status_dev,
                                       g->Qc, g->Qb, g->gnorm, alpha, g->spec(), g->nfit, ListArgs{tuniv, loff, lnum},
                                       c->wait_test, ss, c->n_sm, c->stream))
                        return fail(FC_ERR_ARG, "no tensor-core screen instance for K = " + std::to_string(g->K));
                    S->screen_launches += 1;
                    S->screen_tiles += n_tiles;
                    S->screen_rows += cnt;
                }
                // a screen that gave up (a bounded wait ran out) leaves its candidates incomplete: the
                // resolution does nothing then, and the next read_ctrl reports it
                FC_TRY(stage_end(c, &S->ms_screen));
                S->screen_flops += 2.0 * g->nfit * (double)cnt * (double)g->G;
                ResolveArgs ra{};
                ra.quad_slot = tslot;
                ra.tile_univ = tuniv;
                ra.topk = rtopk;
                ra.cval = cval;
                ra.cidx = cidx;
                ra.alpha = alpha;
                ra.gnorm = g->gnorm;
                ra.Qc = g->Qc;
                ra.Qb = g->Qb;
                ra.G_pad = g->G_pad;
                ra.d = d;
                ra.centre = g->centre;
                ra.nfit = g->nfit;
                ra.W64 = g->W64;
                ra.Wdf = g->Wdf;
                ra.gs = g->spec();
                ra.centre_df = g->centre_df;
                ra.cur = cur;
                ra.pt = L->pt;
                ra.maxit = L->maxit;
                ra.job_of = L->job_of;
                ra.job_left = L->job_left;
                ra.best = L->best;
                ra.nscan = L->nscan;
                ra.dchi2 = L->dchi2;
                ra.chi2min = L->chi2min;
                ra.next = next;
                ra.n_next = cnts + 2;
                ra.fb = fb_out;
                ra.n_fb = n_fb_out;
                ra.counters = c->counters_dev + 3 * round;
                ra.n_resid = c->counters_dev + 12;
                ra.thr = thr;
                ra.lcount = (round == 2) ? lcount : nullptr;
                ra.list_off = loff;
                ra.list_n = lnum;
                ra.rmask = L->rmask;
                ra.round_bit = round == 0 ? 0 : (round == 1 ? kDecidedTop16 : (round == 2 ? kDecidedList
                                                                                          : kDecidedExactList));
                ra.n_sm = c->n_sm;
                ra.status = c->status_dev;
                FC_TRY(stage_begin(c));
                if (listing)
                {
                    int32_t* lrows = nullptr;
                    FC_TRY(scratch(c, "lrows", (size_t)n_tiles * kBM, &lrows));
                    // chunks: a complete list holds at most 2 kListCap points (round 2) or its exact
                    // size (round 3, list_total over the rows), and a row adds at most one partial chunk.
                    // Wide chunks take a quarter of the plan's storage: where it has no room for the others,
                    // or its 32-bit positions would not reach
                    ListPlan lp{};
                    FC_TRY(scratch(c, "lp_base", (size_t)cnt, &lp.row_base));
                    FC_TRY(scratch(c, "lp_nc", (size_t)cnt, &lp.row_nc));
                    FC_TRY(scratch(c, "lp_done", (size_t)cnt, &lp.row_done));
                    FC_TRY(scratch(c, "lp_n", 1, &lp.n_chunk));
                    auto plan = [&](int pts) -> fc_status {
                        lp.pts = pts;
                        lp.max_chunks = loff ? list_total / pts + cnt : cnt * ((2 * kListCap + pts - 1) / pts);
                        const bool spare = pts < kListChunkWide;
                        FC_TRY(scratch(c, "lp_chunk", (size_t)lp.max_chunks, &lp.chunk, spare));
                        FC_TRY(scratch(c, "lp_pv", (size_t)lp.max_chunks, &lp.pv, spare));
                        return scratch(c, "lp_pg", (size_t)lp.max_chunks, &lp.pg, spare);
                    };
                    const bool reach = (loff ? list_total : cnt * 2 * kListCap) / kListChunk + cnt < INT32_MAX;
                    if (!reach || plan(kListChunk) != FC_OK) {
                        for (const char* name : {"lp_chunk", "lp_pv", "lp_pg"}) drop_scratch(c, name);
                        FC_TRY(plan(kListChunkWide));
                    }
                    launch_resolve_list(ra, ccount, n_tiles, cnt, lrows, cnts + 6, lp, c->stream);
                }
                else {
                    // work lists of the flat resolution: up to topk + 1 residuals per row, and
                    // chi2_p of at most every row
                    const size_t rows = (size_t)n_tiles * kBM;
                    FC_TRY(scratch(c, "rs_items", rows * (rtopk + 1), &ra.items));
                    FC_TRY(scratch(c, "rs_res", rows * (rtopk + 1), &ra.res));
                    FC_TRY(scratch(c, "rs_base", rows, &ra.item_base));
                    FC_TRY(scratch(c, "rs_items2", rows, &ra.items2));
                    FC_TRY(scratch(c, "rs_res2", rows, &ra.res2));
                    FC_TRY(scratch(c, "rs_cmin2", rows, &ra.cmin2));
                    FC_TRY(scratch(c, "rs_counts", 2, &ra.counts));
                    FC_TRY(scratch(c, "rs_tiles", (size_t)n_tiles * kQuads, &ra.tile_items));
                    FC_TRY(scratch(c, "rs_tiles2", (size_t)n_tiles * kQuads, &ra.tile_items2));
                    launch_resolve(ra, n_tiles, cnt, c->stream);
                }
                return stage_end(c, &S->ms_rescore);
            };
            // fourth round for universes whose candidate lists overflowed: the same list screen
            // again with exact-size storage, then binary64 rescoring of every listed point;
            // lists above kBigList entries (or aborted ones) take the exact scan
            auto big_lists = [&](const int32_t* ov, int32_t n_ov, const int2* cnt2) -> fc_status {
                std::vector<int32_t> hu(n_ov);
                std::vector<int2> hn(n_ov);
                int2* dn = nullptr;
                FC_TRY(scratch(c, "big_n", (size_t)n_ov, &dn));
                count_launch();
                k_gather_int2<<<nb(n_ov), 256, 0, c->stream>>>(ov, n_ov, cnt2, dn);
                FC_CUDA(cudaMemcpyAsync(hu.data(), ov, (size_t)n_ov * 4, cudaMemcpyDeviceToHost, c->stream));
                FC_CUDA(cudaMemcpyAsync(hn.data(), dn, (size_t)n_ov * 8, cudaMemcpyDeviceToHost, c->stream));
                FC_TRY(sync(c));
                std::vector<int32_t> big_u, exact_u;
                std::vector<int64_t> big_off;
                std::vector<int2> big_n;
                int64_t total = 0;
                for (int32_t i = 0; i < n_ov; ++i) {
                    const int64_t m = (int64_t)hn[i].x + hn[i].y;
                    if (hn[i].x < 0 || hn[i].y < 0 || m > kBigList) {
                        exact_u.push_back(hu[i]);
                    } else {
                        big_u.push_back(hu[i]);
                        big_off.push_back(total);
                        big_n.push_back(hn[i]);
                        total += m;
                    }
                }
                S->fallback += (int64_t)exact_u.size();
                int32_t *d_u = nullptr, *d_x = nullptr, *n_x = nullptr;
                FC_TRY(scratch(c, "big_u", std::max<size_t>(big_u.size(), exact_u.size()) + 1, &d_u));
                if (!big_u.empty()) {
                    const int32_t nb4 = (int32_t)big_u.size();
                    int64_t* loff = nullptr;
                    int2* lnum = nullptr;
                    int64_t* d_off = nullptr;
                    FC_TRY(scratch(c, "big_loff", (size_t)L->cap, &loff));
                    FC_TRY(scratch(c, "big_lnum", (size_t)L->cap, &lnum));
                    FC_TRY(scratch(c, "big_off", (size_t)nb4, &d_off));
                    FC_TRY(scratch(c, "big_x", (size_t)nb4, &d_x));
                    FC_TRY(scratch(c, "big_nx", 1, &n_x));
                    FC_TRY(to_device(c, d_u, big_u.data(), (size_t)nb4 * 4));
                    FC_TRY(to_device(c, d_off, big_off.data(), (size_t)nb4 * 8));
                    FC_TRY(to_device(c, dn, big_n.data(), (size_t)nb4 * 8));
                    count_launch();
                    k_scatter_lists<<<nb(nb4), 256, 0, c->stream>>>(d_u, nb4, d_off, dn, loff, lnum);
                    if (o.cov == FC_COV_IDENTITY)
                        launch_fill_i32(fslot, nb4, g->ident_slot, c->stream);
                    else
                        launch_lookup_slots(d_u, nb4, cur, g->slot_of, fslot, c->stream);
                    FC_CUDA(cudaMemsetAsync(n_x, 0, 4, c->stream));
                    FC_TRY(screen_round(3, d_u, nb4, fslot, kMaxTopK, d_x, n_x, true, loff, lnum, total));
                    int32_t nx = 0;
                    FC_CUDA(cudaMemcpyAsync(&nx, n_x, 4, cudaMemcpyDeviceToHost, c->stream));
                    FC_TRY(read_ctrl(c));
                    S->fallback += nx;
                    if (nx > 0) FC_TRY(exact_scan(d_x, nx, nullptr));
                }
                if (!exact_u.empty()) {
                    FC_TRY(to_device(c, d_u, exact_u.data(), exact_u.size() * 4));
                    FC_TRY(exact_scan(d_u, (int64_t)exact_u.size(), nullptr));
                }
                return FC_OK;
            };
            FC_TRY(screen_round(0, sl_list, sl_n, sl_slot, topk, fb, cnts + 1, false));
            FC_TRY(read_ctrl(c));
            const int32_t n_fb = h_cnts[1];
            if (n_fb > 0 && skip16) {
                // straight to the list round, seeded by the binary64 value round 1 found
                if (o.cov == FC_COV_IDENTITY)
                    launch_fill_i32(fslot, n_fb, g->ident_slot, c->stream);
                else
                    launch_lookup_slots(fb, n_fb, cur, g->slot_of, fslot, c->stream);
                FC_TRY(screen_round(2, fb, n_fb, fslot, kMaxTopK, fb2, cnts + 4, true));
                FC_TRY(read_ctrl(c));
                const int32_t n_ov = h_cnts[4];
                if (n_ov > 0) FC_TRY(big_lists(fb2, n_ov, lcount));
            } else if (n_fb > 0) {
                // second certified round for the universes whose certificate failed
                if (o.cov == FC_COV_IDENTITY)
                    launch_fill_i32(fslot, n_fb, g->ident_slot, c->stream);
                else
                    launch_lookup_slots(fb, n_fb, cur, g->slot_of, fslot, c->stream);
                FC_TRY(screen_round(1, fb, n_fb, fslot, kMaxTopK, fb2, cnts + 4, true));
                FC_TRY(read_ctrl(c));
                const int32_t n_fb2 = h_cnts[4];
                if (n_fb2 > 0) {
                    // third round: list every point that can still be the minimum
                    if (o.cov == FC_COV_IDENTITY)
                        launch_fill_i32(fslot, n_fb2, g->ident_slot, c->stream);
                    else
                        launch_lookup_slots(fb2, n_fb2, cur, g->slot_of, fslot, c->stream);
                    FC_CUDA(cudaMemsetAsync(cnts + 1, 0, 4, c->stream));
                    FC_TRY(screen_round(2, fb2, n_fb2, fslot, kMaxTopK, fb, cnts + 1, true));
                    FC_TRY(read_ctrl(c));
                    const int32_t n_fb3 = h_cnts[1];
                    if (n_fb3 > 0) FC_TRY(big_lists(fb, n_fb3, lcount));
                }
            }
        }
        return FC_OK;
    };
    S->chi2_evals += n_active * g->G;
    S->scans += n_active;
    // ---- covariances for this scan, then the scan itself; a scan that needs more
    // distinct covariances than the cache holds runs in waves of cache-sized groups
    if (o.cov == FC_COV_IDENTITY) {
        std::vector<int32_t> qs, slots;
        FC_TRY(stage_begin(c));
        FC_TRY(ensure_slots(c, g, qs, o.cov, mixed, !mixed, &slots));
        launch_fill_i32(uslot, n_active, slots[0], c->stream);
        FC_TRY(stage_end(c, &S->ms_cov));
        FC_TRY(scan_list(active, n_active, uslot));
    } else {
        std::vector<int32_t> qs;
        FC_TRY(stage_begin(c));
        FC_TRY(distinct_cur(c, g, active, n_active, cur, qs));
        FC_TRY(ensure_cache(c, g));
        const int64_t lim =
            g->tune.cache_slots > 0 ? std::min<int64_t>(g->tune.cache_slots, g->max_cap) : g->max_cap;
        // room for this scan's covariances as far as memory allows; beyond that, waves
        grow_for(c, g, (int64_t)qs.size() + 2, lim);
        const int64_t wave = std::max<int64_t>(1, std::min(lim, g->cap) - 1 - (g->ident_slot >= 0 ? 1 : 0));
        S->max_distinct_cov = std::max<int64_t>(S->max_distinct_cov, (int64_t)qs.size());
        if ((int64_t)qs.size() <= wave) {
            FC_TRY(ensure_slots(c, g, qs, o.cov, mixed, !mixed, nullptr));
            launch_lookup_slots(active, n_active, cur, g->slot_of, uslot, c->stream);
            FC_TRY(stage_end(c, &S->ms_cov));
            FC_TRY(scan_list(active, n_active, uslot));
        } else {
            FC_TRY(stage_end(c, &S->ms_cov));
            uint8_t* flag = nullptr;
            int32_t *wq = nullptr, *wl = nullptr, *wn = cnts + 7, *cur0 = nullptr;
            FC_TRY(scratch(c, "wave_flag", (size_t)g->G, &flag));
            FC_TRY(scratch(c, "wave_q", (size_t)wave, &wq));
            FC_TRY(scratch(c, "wave_list", (size_t)n_active, &wl));
            FC_TRY(scratch(c, "wave_cur0", (size_t)n_active, &cur0));
            // the waves partition the universes by their covariance index before any of them
            // moves on (a universe advanced by one wave must not join a later one)
            count_launch();
            k_gather_cur<<<nb(n_active), 256, 0, c->stream>>>(active, (int)n_active, cur, cur0);
            for (size_t q0 = 0; q0 < qs.size(); q0 += (size_t)wave) {
                const std::vector<int32_t> part(qs.begin() + q0,
                                                qs.begin() + std::min(qs.size(), q0 + (size_t)wave));
                S->scan_waves += 1;
                FC_TRY(stage_begin(c));
                // the universes whose covariance index is in this part
                FC_CUDA(cudaMemsetAsync(flag, 0, (size_t)g->G, c->stream));
                FC_CUDA(cudaMemsetAsync(wn, 0, 4, c->stream));
                FC_TRY(to_device(c, wq, part.data(), part.size() * 4));
                count_launch(2);
                k_flag_list<<<nb((int64_t)part.size()), 256, 0, c->stream>>>(wq, (int)part.size(), flag);
                k_select_cur<<<nb(n_active), 256, 0, c->stream>>>(active, n_active, cur0, flag, wl, wn);
                FC_TRY(ensure_slots(c, g, part, o.cov, mixed, !mixed, nullptr));
                FC_TRY(read_ctrl(c));
                c->ctrl_read = false;
                const int32_t n_w = h_cnts[7];
                if (n_w <= 0) return fail(FC_ERR_STATE, "internal: a wave of no universes");
                launch_lookup_slots(wl, n_w, cur, g->slot_of, uslot, c->stream);
                FC_TRY(stage_end(c, &S->ms_cov));
                FC_TRY(scan_list(wl, n_w, uslot));
            }
        }
    }
    if (!c->ctrl_read) FC_TRY(read_ctrl(c));
    const int32_t n_next = h_cnts[2];
    // [0..2] round 1: screened, rescored, handed on; [3..5] round 2 likewise; [6] listed, [7] list
    // overflow; [9] resolved from exact-size lists, [10] their failures (counted with the fallback)
    // [12] residual chi2 evaluated by the certified rounds
    const unsigned long long* cn = c->ctrl_host->counters;
    std::swap(L->active, L->next);
    L->n_active = n_next;
    S->screened += (int64_t)(cn[0] + cn[3]);
    S->rescored += (int64_t)(cn[1] + cn[4] + cn[6] + cn[9]);
    S->rescreened += (int64_t)(cn[2] + cn[5]);
    S->big_listed += (int64_t)(cn[9] + cn[10]);
    S->residuals += (int64_t)cn[12];
    return flush_stages(c, true);
}

// Jobs of the lane whose universes have all finished: results to the
// caller's buffers, range and job slot back to the lane.  `done` receives
// them (in job-slot order).
fc_status lane_harvest(fc_ctx* c, Lane* L, std::vector<std::shared_ptr<LaneJob>>* done) {
    if (lane_idle(L)) return FC_OK;
    std::vector<int32_t> left(kLaneJobs, 0);
    if (L == &c->sync_lane) {  // job slot 0; it came with the scan's last read of the control block
        if (!c->ctrl_read) FC_TRY(read_ctrl(c));
        left[0] = c->ctrl_host->sync_left;
    } else {
        FC_CUDA(cudaMemcpyAsync(left.data(), L->job_left, kLaneJobs * 4, cudaMemcpyDeviceToHost, c->stream));
        FC_TRY(sync(c));
    }
    // the universes' own count against the scan's: a universe that left the active list unfinished is an error,
    // not a job that never completes
    for (int j = 0; j < kLaneJobs; ++j)
        if (L->jobs[j] && left[j] != 0 && L->n_active == 0)
            return fail(FC_ERR_STATE, "internal: universes left the scan unfinished");
    for (int j = 0; j < kLaneJobs; ++j) {
        std::shared_ptr<LaneJob> J = L->jobs[j];
        if (!J || left[j] != 0) continue;
        const bool cancelled = J->jr && J->jr->cancelled.load();
        if (!cancelled) {
            if (J->dchi2) FC_TRY(copy_out(c, J->dchi2, L->dchi2 + J->base, (size_t)J->n * 8));
            if (J->chi2min) FC_TRY(copy_out(c, J->chi2min, L->chi2min + J->base, (size_t)J->n * 8));
            if (J->nscans) FC_TRY(copy_out(c, J->nscans, L->nscan + J->base, (size_t)J->n));
            if (J->best) {
                int64_t* b64 = nullptr;
                if (is_device_ptr(J->best)) {
                    b64 = J->best;
                } else {
                    FC_TRY(scratch(c, "best64", (size_t)J->n, &b64));
                }
                count_launch();
                k_widen<<<nb(J->n), 256, 0, c->stream>>>(L->best + J->base, J->n, b64);
                if (b64 != J->best) FC_TRY(copy_out(c, J->best, b64, (size_t)J->n * 8));
            }
            FC_TRY(sync(c));
        }
        J->status = cancelled ? FC_ERR_CANCELLED : FC_OK;
        J->done = true;
        lane_release(L, J->base, J->n);
        L->jobs[j] = nullptr;
        L->free_jobs.push_back(j);
        done->push_back(J);
    }
    return FC_OK;
}

// Remove the universes of cancelled running jobs from the active list; they
// complete (with FC_ERR_CANCELLED) at the next harvest.
fc_status lane_drop_cancelled(fc_ctx* c, Lane* L) {
    std::vector<uint8_t> dead(kLaneJobs, 0);
    std::vector<int32_t> hit;
    for (int j = 0; j < kLaneJobs; ++j) {
        const auto& J = L->jobs[j];
        if (J && J->jr && J->jr->cancelled.load()) {
            dead[j] = 1;
            hit.push_back(j);
        }
    }
    if (hit.empty() || L->n_active == 0) return FC_OK;
    int32_t* cnt = nullptr;
    FC_TRY(scratch(c, "dropcnt", 1, &cnt));
    FC_TRY(to_device(c, L->job_dead, dead.data(), kLaneJobs));
    FC_CUDA(cudaMemsetAsync(cnt, 0, 4, c->stream));
    count_launch();
    k_drop_jobs<<<nb(L->n_active), 256, 0, c->stream>>>(L->active, L->n_active, L->job_of, L->job_dead, L->next, cnt);
    int32_t h = 0;
    FC_CUDA(cudaMemcpyAsync(&h, cnt, 4, cudaMemcpyDeviceToHost, c->stream));
    FC_CUDA(cudaMemsetAsync(L->job_dead, 0, kLaneJobs, c->stream));
    FC_TRY(sync(c));
    std::swap(L->active, L->next);
    L->n_active = h;
    for (int j : hit) launch_fill_i32(L->job_left + j, 1, 0, c->stream);
    return FC_OK;
}

// Every job of the lane fails with `st` (a device error mid-scan cannot be
// attributed to one job); the lane is emptied.
void lane_fail_all(Lane* L, fc_status st, std::vector<std::shared_ptr<LaneJob>>* done) {
    for (int j = 0; j < kLaneJobs; ++j) {
        if (!L->jobs[j]) continue;
        L->jobs[j]->status = st;
        L->jobs[j]->done = true;
        done->push_back(L->jobs[j]);
    }
    lane_reset(L);
}

fc_status check_points(const Grid* g, const int64_t* ps, int32_t P, std::vector<int64_t>* out) {
    out->resize(P);
    if (P == 0) return FC_OK;
    if (is_device_ptr(ps)) {
        FC_CUDA(cudaMemcpy(out->data(), ps, (size_t)P * 8, cudaMemcpyDeviceToHost));
    } else {
        memcpy(out->data(), ps, (size_t)P * 8);
    }
    for (int64_t p : *out)
        if (p < 0 || p >= g->G) return fail(FC_ERR_ARG, "grid index out of range");
    return FC_OK;
}

int effective_max_iter(const fc_opts& o) { return o.cov == FC_COV_ITERATE ? o.max_iter : 1; }

// The lane a synchronous call uses (kept by the context, grown on demand).
fc_status sync_lane(fc_ctx* c, Grid* g, const fc_opts& o, int64_t n, Lane** out) {
    Lane* L = &c->sync_lane;
    if (L->cap < n || L->nfit < g->nfit) FC_TRY(lane_alloc(c, L, g, o, n));
    L->g = g;
    L->o = o;
    lane_reset(L);
    *out = L;
    return FC_OK;
}

// Synchronous job through a lane of its own: admit, scan until every
// universe finished, harvest.
fc_status run_sync(fc_ctx* c, Grid* g, const fc_opts& o, const std::vector<int64_t>& ps, int32_t U, uint64_t seed,
                   const float* d_in, double* dchi2, int64_t* best, int8_t* nscans, double* chi2min,
                   cudaEvent_t ev_data) {
    const int64_t n = (int64_t)ps.size() * U;
    c->last_n = -1;
    Lane* L = nullptr;
    FC_TRY(sync_lane(c, g, o, n, &L));
    auto J = std::make_shared<LaneJob>();
    J->n = n;
    J->dchi2 = dchi2;
    J->best = best;
    J->nscans = nscans;
    J->chi2min = chi2min;
    J->slot = L->free_jobs.back();
    L->free_jobs.pop_back();
    if (!lane_reserve(L, n, &J->base)) return fail(FC_ERR_STATE, "synchronous lane has no room");
    fc_status st = lane_admit(c, L, J, ps.data(), (int32_t)ps.size(), U, seed, o.fluct, effective_max_iter(o), d_in);
    if (ev_data) cudaEventRecord(ev_data, c->stream);
    while (st == FC_OK && L->n_active > 0) st = scan_once(c, L);
    std::vector<std::shared_ptr<LaneJob>> done;
    if (st == FC_OK) st = lane_harvest(c, L, &done);
    if (st == FC_OK && (done.size() != 1 || !lane_idle(L)))
        st = fail(FC_ERR_STATE, "internal: synchronous job did not complete");
    if (st != FC_OK) {
        settle(c);
        lane_reset(L);
    }
    c->last_base = J->base;
    c->last_n = st == FC_OK ? n : -1;
    return st;
}

fc_status run_points_impl(fc_ctx* c, int32_t grid_id, const int64_t* ps, int32_t P, uint64_t seed, int32_t U,
                          const fc_opts* opts_in, double* dchi2, int64_t* bestfit, int8_t* nscans) {
    Grid* g = find_grid(c, grid_id);
    if (!g) return fail(FC_ERR_NOT_FOUND, "unknown grid id");
    if (!g->has_F) return fail(FC_ERR_STATE, "fractional covariance not set (fc_set_frac_cov)");
    if (P < 0 || U < 0 || (P > 0 && !ps)) return fail(FC_ERR_ARG, "bad P, U or ps");
    if (P > 0 && U > 0 && !dchi2) return fail(FC_ERR_ARG, "dchi2 output is required");
    fc_opts o;
    fc_default_opts(&o);
    if (opts_in) o = *opts_in;
    FC_TRY(validate_opts(&o, g));
    const int64_t n = (int64_t)P * U;
    if (n == 0) return FC_OK;
    if (n > (int64_t)INT32_MAX / 2) return fail(FC_ERR_ARG, "P * U too large");
    std::vector<int64_t> hps;
    FC_TRY(check_points(g, ps, P, &hps));
    c->stats = fc_stats{};
    c->acc = &c->stats;
    const long long launches0 = g_launches.load();
    cudaEvent_t e0 = c->run_ev[0], e1 = c->run_ev[1], e2 = c->run_ev[2];
    cudaEventRecord(e0, c->stream);
    fc_status st = run_sync(c, g, o, hps, U, seed, nullptr, dchi2, bestfit, nscans, nullptr, e1);
    if (st == FC_OK) {
        cudaEventRecord(e2, c->stream);
        st = sync(c);
    }
    if (st == FC_OK) {
        float t_fake = 0, t_all = 0;
        cudaEventElapsedTime(&t_fake, e0, e1);
        cudaEventElapsedTime(&t_all, e0, e2);
        c->stats.ms_fake = t_fake;
        c->stats.ms_total = t_all;
        c->stats.universes = n;
        c->stats.kernel_launches = g_launches.load() - launches0;
        c->stats.cache_slots = g->cap;
    }
    return st;
}

// Fake data only: the systematic factors of the points, then the draws
// straight into the caller's buffer when it is device memory.
fc_status fake_data_impl(fc_ctx* c, int32_t grid_id, const int64_t* ps, int32_t P, uint64_t seed, int32_t U,
                         int fluct, float* out) {
    Grid* g = find_grid(c, grid_id);
    if (!g) return fail(FC_ERR_NOT_FOUND, "unknown grid id");
    if (!g->has_F) return fail(FC_ERR_STATE, "fractional covariance not set (fc_set_frac_cov)");
    if (P < 0 || U < 0 || (P > 0 && !ps)) return fail(FC_ERR_ARG, "bad P, U or ps");
    const int64_t n = (int64_t)P * U;
    if (n == 0) return FC_OK;
    std::vector<int64_t> hps;
    FC_TRY(check_points(g, ps, P, &hps));
    int64_t* ps_dev = nullptr;
    double* L64 = nullptr;
    float *L32 = nullptr, *s32 = nullptr, *d = nullptr;
    FC_TRY(scratch(c, "ps", (size_t)P, &ps_dev));
    FC_TRY(to_device(c, ps_dev, hps.data(), (size_t)P * 8));
    FC_TRY(scratch(c, "L64", (size_t)P * g->nf * g->nf, &L64));
    FC_TRY(scratch(c, "L32", (size_t)P * g->nf * g->nf, &L32));
    FC_TRY(scratch(c, "s32", (size_t)P * g->nf, &s32));
    launch_chol_sys(g->full(), g->nf, g->F, ps_dev, P, fluct == FC_FLUCT_GAUSS, L64, L32, s32, c->n_sm,
                    c->status_dev, c->stream);
    FC_TRY(read_ctrl(c));
    if (is_device_ptr(out)) {
        d = out;
    } else {
        FC_TRY(scratch(c, "d", (size_t)n * g->nfit, &d));
    }
    launch_fake_data(L32, s32, g->nf, g->identity_collapse ? nullptr : g->collapse, g->nfit, ps_dev, P, U, seed,
                     fluct == FC_FLUCT_GAUSS, d, c->n_sm, c->stream);
    if (d != out) FC_TRY(copy_out(c, out, d, (size_t)n * g->nfit * sizeof(float)));
    return sync(c);
}

// --------------------------------------------------------------- serving ---

// Lane key of a served job: jobs that agree on it share scans.
bool same_key(int32_t grid_a, const fc_opts& a, int32_t grid_b, const fc_opts& b) {
    return grid_a == grid_b && a.precision == b.precision && (a.top_k <= 8) == (b.top_k <= 8) &&
           (a.cov == FC_COV_IDENTITY) == (b.cov == FC_COV_IDENTITY);
}

bool same_lane(const Lane* L, const fc_job& j) { return L->g && same_key(L->g->id, L->o, j.grid_id, j.opts); }

constexpr int64_t kServeLaneMin = int64_t(1) << 18;  // universes per serving lane at least

void complete(fc_ctx* c, const std::shared_ptr<JobRec>& jr, fc_status st) {
    std::lock_guard<std::mutex> lk(c->q_mu);
    auto it = c->grids.find(jr->job.grid_id);
    if (it != c->grids.end()) it->second->busy--;
    jr->t_done = std::chrono::steady_clock::now();
    if (st != FC_OK) jr->error = st == FC_ERR_CANCELLED ? "job cancelled" : t_last_error;
    jr->state.store(st);
}

// Try to admit a queued job.  Returns true when the job left the queue
// (admitted, or completed with an error); false when its lane has no room now.
bool serve_admit(fc_ctx* c, const std::shared_ptr<JobRec>& jr) {
    const fc_job& jb = jr->job;
    Grid* g = find_grid(c, jb.grid_id);
    if (!g) {
        complete(c, jr, FC_ERR_NOT_FOUND);
        return true;
    }
    const int64_t n = (int64_t)jb.P * jb.U;
    if (n == 0 || jr->cancelled.load()) {
        complete(c, jr, jr->cancelled.load() ? FC_ERR_CANCELLED : FC_OK);
        return true;
    }
    // admission by the memory budget: the running jobs' estimates plus this one's must fit;
    // otherwise the job waits for running jobs to finish (it fits alone: fc_submit checked)
    bool others_running = false;
    for (auto& l : c->lanes) others_running = others_running || !lane_idle(l.get());
    if (c->budget && others_running && c->reserved + jr->need > c->budget) {
        c->acc->deferred += 1;
        return false;
    }
    Lane* L = nullptr;
    for (auto& l : c->lanes)
        if (same_lane(l.get(), jb)) L = l.get();
    if (!L) {
        c->lanes.push_back(std::make_unique<Lane>());
        L = c->lanes.back().get();
    }
    int64_t base = 0;
    if (!L->cap || !lane_reserve(L, n, &base)) {
        if (L->cap && !lane_idle(L)) return false;  // wait for running jobs of the lane to finish
        // empty lane: (re)size it for this job, with headroom for later ones
        fc_status st = lane_alloc(c, L, g, jb.opts, std::max(n, kServeLaneMin));
        if (st != FC_OK) {
            cudaGetLastError();
            // give back the memory of idle lanes, then try the job's own size
            for (auto& l : c->lanes)
                if (l.get() != L && lane_idle(l.get())) lane_free(c, l.get());
            st = lane_alloc(c, L, g, jb.opts, n);
        }
        if (st != FC_OK) {
            cudaGetLastError();
            if (others_running) {
                // memory held by running jobs: retry when they finish
                c->acc->deferred += 1;
                return false;
            }
            complete(c, jr, st);
            return true;
        }
        lane_reserve(L, n, &base);
    }
    auto J = std::make_shared<LaneJob>();
    J->jr = jr;
    J->n = n;
    J->base = base;
    J->dchi2 = jb.dchi2;
    J->best = jb.bestfit;
    J->nscans = jb.nscans;
    J->slot = L->free_jobs.back();
    L->free_jobs.pop_back();
    const fc_status st =
        lane_admit(c, L, J, jr->ps.data(), jb.P, jb.U, jb.seed, jb.opts.fluct, effective_max_iter(jb.opts), nullptr);
    if (st != FC_OK) {
        lane_release(L, base, n);
        L->free_jobs.push_back(J->slot);
        complete(c, jr, st);
    } else {
        c->reserved += jr->need;
    }
    return true;
}

// The serving loop.  Each turn: admit queued jobs (FIFO per lane) into free
// universe ranges, run one scan of every non-empty lane, hand back the jobs
// that completed.  Jobs admitted in a turn join the scans of jobs that are
// mid-iteration; a job's latency is its own universes' scans, not the batch's.
void worker_main(fc_ctx* c) {
    cudaSetDevice(c->device);
    std::deque<std::shared_ptr<JobRec>> waiting;
    int64_t running = 0;  // jobs inside lanes
    for (;;) {
        {
            std::unique_lock<std::mutex> lk(c->q_mu);
            c->q_cv.wait(lk, [&] { return c->stop || !c->queue.empty() || running > 0 || !waiting.empty(); });
            while (!c->queue.empty()) {
                waiting.push_back(c->queue.front());
                c->queue.pop_front();
            }
            if (c->stop && waiting.empty() && running == 0) break;
        }
        std::lock_guard<std::mutex> lk(c->api_mu);
        c->acc = &c->serve_stats;
        // admission, FIFO within a lane key
        std::vector<const fc_job*> blocked;
        for (auto it = waiting.begin(); it != waiting.end();) {
            const fc_job& jb = (*it)->job;
            bool skip = false;
            for (const fc_job* b : blocked) skip = skip || same_key(b->grid_id, b->opts, jb.grid_id, jb.opts);
            const int64_t n = (int64_t)jb.P * jb.U;
            if (!skip && serve_admit(c, *it)) {
                if (n > 0 && (*it)->state.load() == FC_PENDING) running++;
                it = waiting.erase(it);
            } else {
                if (!skip) blocked.push_back(&jb);
                ++it;
            }
        }
        // one scan per lane, then completions
        for (auto& l : c->lanes) {
            Lane* L = l.get();
            if (lane_idle(L)) continue;
            std::vector<std::shared_ptr<LaneJob>> done;
            fc_status st = lane_drop_cancelled(c, L);
            if (st == FC_OK) st = scan_once(c, L);
            if (st == FC_OK) st = lane_harvest(c, L, &done);
            if (st != FC_OK) {
                settle(c);
                lane_fail_all(L, st, &done);
            }
            for (auto& J : done) {
                c->reserved -= std::min(c->reserved, J->jr->need);
                complete(c, J->jr, J->status);
                running--;
            }
        }
        // release the memory of empty lanes when nothing waits
        if (waiting.empty() && running == 0) {
            for (auto& l : c->lanes) lane_free(c, l.get());
            c->lanes.clear();
        }
        c->acc = &c->stats;
    }
}

}  // namespace

// ---------------------------------------------------------------- C ABI -----

extern "C" {

void fc_default_opts(fc_opts* o) {
    if (!o) return;
    o->max_iter = 5;
    o->precision = FC_PREC_MIXED;
    o->top_k = 8;
    o->fluct = FC_FLUCT_POISSON_SYS;
    o->cov = FC_COV_ITERATE;
}

fc_status fc_create(fc_ctx** out, int device, size_t hbm_budget_bytes, void* cuda_stream) {
    if (!out) return fail(FC_ERR_ARG, "out is NULL");
    *out = nullptr;
    int ndev = 0;
    FC_CUDA(cudaGetDeviceCount(&ndev));
    if (device < 0 || device >= ndev) return fail(FC_ERR_ARG, "no such CUDA device");
    FC_CUDA(cudaSetDevice(device));
    auto c = std::make_unique<fc_ctx>();
    c->device = device;
    c->budget = hbm_budget_bytes;
    cudaDeviceProp prop;
    FC_CUDA(cudaGetDeviceProperties(&prop, device));
    c->n_sm = prop.multiProcessorCount;
    c->dev_name = prop.name;
    for (char& ch : c->dev_name)
        if (ch == ' ' || ch == '\t') ch = '_';
    if (prop.major != 10) return fail(FC_ERR_ARG, "libfc is built for sm_103a (Blackwell Ultra); device is sm_" +
                                                      std::to_string(prop.major) + std::to_string(prop.minor));
    if (cuda_stream) {
        c->stream = (cudaStream_t)cuda_stream;
    } else {
        FC_CUDA(cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking));
        c->own_stream = true;
    }
    for (cudaEvent_t& e : c->run_ev) FC_CUDA(cudaEventCreate(&e));
    FC_TRY(dalloc_t(c.get(), &c->ctrl, 1));
    c->status_dev = &c->ctrl->status;
    c->counters_dev = c->ctrl->counters;
    FC_CUDA(cudaMallocHost((void**)&c->ctrl_host, sizeof(Ctrl)));
    FC_CUDA(cudaMallocHost((void**)&c->list_host, kListHost * sizeof(int32_t)));
    FC_CUDA(cudaMallocHost((void**)&c->stage_host, kStageHost));
    memset(c->ctrl_host, 0, sizeof(Ctrl));
    FC_CUDA(cudaMemsetAsync(c->ctrl, 0, sizeof(Ctrl), c->stream));
    FC_CUDA(cudaStreamSynchronize(c->stream));
    *out = c.release();
    return FC_OK;
}

fc_status fc_destroy(fc_ctx* c) {
    if (!c) return fail(FC_ERR_ARG, "ctx is NULL");
    {
        std::lock_guard<std::mutex> lk(c->q_mu);
        c->stop = true;
    }
    c->q_cv.notify_all();
    if (c->worker.joinable()) c->worker.join();
    cudaSetDevice(c->device);
    cudaStreamSynchronize(c->stream);
    for (auto& kv : c->allocs) cudaFree(kv.first);
    c->allocs.clear();
    if (c->own_stream) cudaStreamDestroy(c->stream);
    for (cudaEvent_t e : c->run_ev)
        if (e) cudaEventDestroy(e);
    for (auto& e : c->stage_ev) {
        cudaEventDestroy(e.first);
        if (e.second) cudaEventDestroy(e.second);
    }
    cudaFreeHost(c->ctrl_host);
    cudaFreeHost(c->list_host);
    cudaFreeHost(c->stage_host);
    delete c;
    return FC_OK;
}

}  // extern "C"

namespace {

// Validate the grid's sizes and collapse map (copied to the host in hcoll).
fc_status check_grid_args(int64_t G, int32_t nf, const int32_t* collapse, int32_t nfit, std::vector<int32_t>* hcoll) {
    if (G < 1 || G > (int64_t)INT32_MAX - 1) return fail(FC_ERR_ARG, "G out of range");
    if (nf < 1 || nf > kMaxBins || nfit < 1 || nfit > kMaxBins) return fail(FC_ERR_ARG, "bins out of range [1, 200]");
    if (!collapse && nfit != nf) return fail(FC_ERR_ARG, "N_fit must equal N_full without a collapse map");
    if (collapse) {
        hcoll->resize(nf);
        if (is_device_ptr(collapse))
            FC_CUDA(cudaMemcpy(hcoll->data(), collapse, (size_t)nf * 4, cudaMemcpyDeviceToHost));
        else
            memcpy(hcoll->data(), collapse, (size_t)nf * 4);
        std::vector<int> seen(nfit, 0);
        for (int32_t v : *hcoll) {
            if (v < 0 || v >= nfit) return fail(FC_ERR_ARG, "collapse map entry out of [0, N_fit)");
            seen[v] = 1;
        }
        for (int v : seen)
            if (!v) return fail(FC_ERR_ARG, "collapse map leaves a fit bin empty");
    }
    return FC_OK;
}

void free_grid_arrays(fc_ctx* c, Grid* g) {
    dfree(c, g->S_full); dfree(c, g->S_fit); dfree(c, g->centre); dfree(c, g->Sc); dfree(c, g->Sc32);
    dfree(c, g->gnorm); dfree(c, g->Bt); dfree(c, g->collapse); dfree(c, g->Sdf); dfree(c, g->centre_df);
    dfree(c, g->model_i); dfree(c, g->model_d);
}

// A new grid's sizes and its resident arrays (S_full still to be filled).  A
// recomputed grid keeps no spectra: only the centre, the screen's image and
// norms, and the collapse map.
fc_status alloc_grid(fc_ctx* c, Grid* g, int64_t G, int32_t nf, int32_t nfit, const std::vector<int32_t>& hcoll,
                     bool recompute = false) {
    g->G = G;
    g->G_pad = ((G + kBN - 1) / kBN) * kBN;
    g->nf = nf;
    g->nfit = nfit;
    g->K = screen_k(nfit);
    bool ident = true;
    if (!hcoll.empty())
        for (int i = 0; i < nf; ++i) ident = ident && (hcoll[i] == i) && (nf == nfit);
    g->identity_collapse = ident;
    g->recompute = recompute;
    if (!recompute) {
        FC_TRY(dalloc_t(c, &g->S_full, (size_t)G * nf));
        FC_TRY(dalloc_t(c, &g->S_fit, (size_t)G * nfit));
        FC_TRY(dalloc_t(c, &g->Sc, (size_t)G * nfit));
        FC_TRY(dalloc_t(c, &g->Sdf, (size_t)G * nfit));
        FC_TRY(dalloc_t(c, &g->Sc32, (size_t)G * nfit));
    }
    FC_TRY(dalloc_t(c, &g->centre, (size_t)nfit));
    FC_TRY(dalloc_t(c, &g->centre_df, (size_t)nfit));
    FC_TRY(dalloc_t(c, &g->gnorm, (size_t)G));
    FC_TRY(dalloc_t(c, &g->Bt, (size_t)g->G_pad * 2 * g->K));
    FC_TRY(dalloc_t(c, &g->collapse, (size_t)nf));
    if (!hcoll.empty())
        FC_CUDA(cudaMemcpyAsync(g->collapse, hcoll.data(), (size_t)nf * 4, cudaMemcpyHostToDevice, c->stream));
    return FC_OK;
}

// Derived arrays of a grid whose S_full is in place (fit-space spectra, centre, the screen's
// B image and norms, double-float copies), then the grid is registered under a new id.
fc_status finish_grid(fc_ctx* c, std::unique_ptr<Grid>& g, int32_t* grid_id) {
    const int64_t G = g->G;
    const int nf = g->nf, nfit = g->nfit;
    if (!g->recompute)
        launch_collapse(g->S_full, G, nf, g->identity_collapse ? nullptr : g->collapse, nfit, g->S_fit, c->stream);
    launch_centre(g->spec(), G, g->centre, c->stream);
    launch_centred(g->spec(), G, g->G_pad, g->K, g->Sc, g->Sc32, g->gnorm, g->Bt, c->stream);
    if (!g->recompute) launch_to_df(g->S_fit, G * nfit, g->Sdf, c->stream);
    launch_to_df(g->centre, nfit, g->centre_df, c->stream);
    FC_TRY(sync(c));
    std::lock_guard<std::mutex> lq(c->q_mu);
    g->id = c->next_grid++;
    *grid_id = g->id;
    c->grids[g->id] = std::move(g);
    return FC_OK;
}

}  // namespace

extern "C" {

fc_status fc_load_grid(fc_ctx* c, const double* S, int64_t G, int32_t nf, const int32_t* collapse, int32_t nfit,
                       int32_t* grid_id) {
    if (!c || !S || !grid_id) return fail(FC_ERR_ARG, "NULL argument");
    std::vector<int32_t> hcoll;
    FC_TRY(check_grid_args(G, nf, collapse, nfit, &hcoll));
    std::lock_guard<std::mutex> lk(c->api_mu);
    cudaSetDevice(c->device);
    auto g = std::make_unique<Grid>();
    fc_status st = alloc_grid(c, g.get(), G, nf, nfit, hcoll);
    if (st == FC_OK) st = copy_in(c, g->S_full, S, (size_t)G * nf * 8);
    // spectra must be finite and non-negative (checked on the host copy; a device S is read back)
    if (st == FC_OK) {
        std::vector<double> hs;
        const double* hv = S;
        if (is_device_ptr(S)) {
            hs.resize((size_t)G * nf);
            if (cudaMemcpy(hs.data(), S, hs.size() * 8, cudaMemcpyDeviceToHost) != cudaSuccess)
                st = fail(FC_ERR_CUDA, "reading the spectra back failed");
            hv = hs.data();
        }
        for (int64_t e = 0; st == FC_OK && e < G * nf; ++e)
            if (!(hv[e] >= 0.0) || !std::isfinite(hv[e])) st = fail(FC_ERR_ARG, "spectra must be finite and >= 0");
    }
    if (st == FC_OK) st = finish_grid(c, g, grid_id);
    if (st != FC_OK && g) free_grid_arrays(c, g.get());
    return st;
}

fc_status fc_load_grid_osc(fc_ctx* c, const fc_osc_model* m, int32_t nf, const int32_t* collapse, int32_t nfit,
                           int32_t* grid_id) {
    return fc_load_grid_osc_ex(c, m, nf, collapse, nfit, 0u, grid_id);
}

fc_status fc_load_grid_osc_ex(fc_ctx* c, const fc_osc_model* m, int32_t nf, const int32_t* collapse, int32_t nfit,
                              uint32_t flags, int32_t* grid_id) {
    if (!c || !m || !grid_id || !m->axis_len || !m->axis_values || !m->amp_axis || !m->dm2_axis || !m->b || !m->f ||
        !m->L || !m->E)
        return fail(FC_ERR_ARG, "NULL argument");
    if (flags & ~(uint32_t)FC_GRID_RECOMPUTE) return fail(FC_ERR_ARG, "unknown grid flag");
    const bool recompute = (flags & FC_GRID_RECOMPUTE) != 0;
    if (m->D < 1 || m->D > kMaxOscAxes) return fail(FC_ERR_ARG, "D out of range [1, 8]");
    if (m->n_terms < 1 || m->n_terms > kMaxOscTerms) return fail(FC_ERR_ARG, "n_terms out of range [1, 4]");
    int64_t G = 1;
    std::vector<int32_t> off(m->D);
    int32_t n_vals = 0;
    for (int a = 0; a < m->D; ++a) {
        if (m->axis_len[a] < 1) return fail(FC_ERR_ARG, "axis length < 1");
        off[a] = n_vals;
        n_vals += m->axis_len[a];
        G *= m->axis_len[a];
        if (G > (int64_t)INT32_MAX - 1) return fail(FC_ERR_ARG, "G out of range");
    }
    for (int t = 0; t < m->n_terms; ++t)
        if (m->amp_axis[t] < 0 || m->amp_axis[t] >= m->D || m->dm2_axis[t] < 0 || m->dm2_axis[t] >= m->D)
            return fail(FC_ERR_ARG, "term axis out of [0, D)");
    for (int i = 0; i < nf && i < kMaxBins; ++i)
        if (!(m->E[i] > 0.0) || !std::isfinite(m->L[i]) || !std::isfinite(m->E[i]))
            return fail(FC_ERR_ARG, "energies must be > 0 and baselines finite");
    std::vector<int32_t> hcoll;
    FC_TRY(check_grid_args(G, nf, collapse, nfit, &hcoll));
    bool ident = true;
    if (!hcoll.empty())
        for (int i = 0; i < nf; ++i) ident = ident && (hcoll[i] == i) && (nf == nfit);
    std::lock_guard<std::mutex> lk(c->api_mu);
    cudaSetDevice(c->device);
    // The model on the device, packed.  ints: axis lengths, axis offsets, term axes (amplitude, dm2),
    // each term's first sine-table row, the generator's error count, then (a collapse other than the
    // identity) each fit bin's first member and the members.  doubles: axis values, b, f, L, E, then
    // the sine table (one row per dm2 value of each term).
    const int D = m->D, T = m->n_terms;
    std::vector<int32_t> hi;
    hi.insert(hi.end(), m->axis_len, m->axis_len + D);
    hi.insert(hi.end(), off.begin(), off.end());
    hi.insert(hi.end(), m->amp_axis, m->amp_axis + T);
    hi.insert(hi.end(), m->dm2_axis, m->dm2_axis + T);
    int32_t rows = 0;
    for (int t = 0; t < T; ++t) {
        hi.push_back(rows);
        rows += m->axis_len[m->dm2_axis[t]];
    }
    const size_t o_bad = hi.size();
    hi.push_back(0);
    const size_t o_moff = hi.size();
    if (!ident) {
        std::vector<int32_t> moff(nfit + 1, 0), mem(nf), cur(nfit);
        for (int i = 0; i < nf; ++i) ++moff[hcoll[i] + 1];
        for (int j = 0; j < nfit; ++j) moff[j + 1] += moff[j];
        for (int j = 0; j < nfit; ++j) cur[j] = moff[j];
        for (int i = 0; i < nf; ++i) mem[cur[hcoll[i]]++] = i;  // increasing i within each fit bin
        hi.insert(hi.end(), moff.begin(), moff.end());
        hi.insert(hi.end(), mem.begin(), mem.end());
    }
    std::vector<double> hd;
    hd.insert(hd.end(), m->axis_values, m->axis_values + n_vals);
    const size_t o_b = hd.size();
    hd.insert(hd.end(), m->b, m->b + nf);
    const size_t o_f = hd.size();
    hd.insert(hd.end(), m->f, m->f + (size_t)T * nf);
    const size_t o_L = hd.size();
    hd.insert(hd.end(), m->L, m->L + nf);
    const size_t o_E = hd.size();
    hd.insert(hd.end(), m->E, m->E + nf);
    const size_t o_sin = hd.size();
    auto g = std::make_unique<Grid>();
    fc_status st = dalloc_t(c, &g->model_i, hi.size());
    if (st == FC_OK) st = dalloc_t(c, &g->model_d, o_sin + (size_t)rows * nf);
    if (st == FC_OK && cudaMemcpyAsync(g->model_i, hi.data(), hi.size() * 4, cudaMemcpyHostToDevice, c->stream))
        st = fail(FC_ERR_CUDA, "copying the model failed");
    if (st == FC_OK && cudaMemcpyAsync(g->model_d, hd.data(), hd.size() * 8, cudaMemcpyHostToDevice, c->stream))
        st = fail(FC_ERR_CUDA, "copying the model failed");
    if (st == FC_OK) st = alloc_grid(c, g.get(), G, nf, nfit, hcoll, recompute);
    int bad = 0;
    if (st == FC_OK) {
        SpecModel& sm = g->model;
        const int32_t* di = g->model_i;
        const double* dd = g->model_d;
        sm.D = D;
        sm.n_terms = T;
        sm.nf = nf;
        sm.nfit = nfit;
        sm.axis_len = di;
        sm.axis_off = di + D;
        sm.amp_ax = di + 2 * D;
        sm.dm2_ax = di + 2 * D + T;
        sm.sin_off = di + 2 * D + 2 * T;
        sm.axis_val = dd;
        sm.b = dd + o_b;
        sm.f = dd + o_f;
        sm.sinT = dd + o_sin;
        sm.mem_off = ident ? nullptr : di + o_moff;
        sm.mem = ident ? nullptr : di + o_moff + nfit + 1;
        int* dbad = g->model_i + o_bad;
        launch_osc_sin(sm, rows, dd + o_L, dd + o_E, g->model_d + o_sin, c->stream);
        // a stored grid is filled by the model's evaluation; a recomputed one is only checked
        launch_osc_spectra(sm, G, g->S_full, dbad, c->stream);
        if (cudaMemcpyAsync(&bad, dbad, 4, cudaMemcpyDeviceToHost, c->stream) != cudaSuccess)
            st = fail(FC_ERR_CUDA, "reading the generator's check back failed");
        if (st == FC_OK) st = sync(c);
        if (st == FC_OK && bad) st = fail(FC_ERR_ARG, "the model gives spectra that are not finite and >= 0");
        // a stored grid reads its rows from memory from now on
        if (!recompute) g->model = SpecModel{};
    }
    if (st == FC_OK) st = finish_grid(c, g, grid_id);
    if (st != FC_OK && g) free_grid_arrays(c, g.get());
    return st;
}

fc_status fc_set_frac_cov(fc_ctx* c, int32_t grid_id, const double* F, int32_t nf) {
    if (!c || !F) return fail(FC_ERR_ARG, "NULL argument");
    std::lock_guard<std::mutex> lk(c->api_mu);
    cudaSetDevice(c->device);
    Grid* g = find_grid(c, grid_id);
    if (!g) return fail(FC_ERR_NOT_FOUND, "unknown grid id");
    if (nf != g->nf) return fail(FC_ERR_ARG, "F must be N_full x N_full");
    std::vector<double> h((size_t)nf * nf);
    if (is_device_ptr(F))
        FC_CUDA(cudaMemcpy(h.data(), F, h.size() * 8, cudaMemcpyDeviceToHost));
    else
        memcpy(h.data(), F, h.size() * 8);
    for (int i = 0; i < nf; ++i)
        for (int j = 0; j < nf; ++j) {
            const double a = h[(size_t)i * nf + j], b = h[(size_t)j * nf + i];
            if (!std::isfinite(a)) return fail(FC_ERR_ARG, "F must be finite");
            if (std::fabs(a - b) > 1e-12 * (std::fabs(a) + std::fabs(b)) + 1e-300)
                return fail(FC_ERR_ARG, "F must be symmetric");
        }
    // a new F invalidates every cached covariance; keep the storage
    reset_cache(c, g);
    if (!g->F) FC_TRY(dalloc_t(c, &g->F, (size_t)nf * nf));
    FC_CUDA(cudaMemcpyAsync(g->F, h.data(), h.size() * 8, cudaMemcpyHostToDevice, c->stream));
    FC_TRY(sync(c));
    g->has_F = true;
    return FC_OK;
}

fc_status fc_unload_grid(fc_ctx* c, int32_t grid_id) {
    if (!c) return fail(FC_ERR_ARG, "ctx is NULL");
    std::lock_guard<std::mutex> lk(c->api_mu);
    Grid* g = find_grid(c, grid_id);
    if (!g) return fail(FC_ERR_NOT_FOUND, "unknown grid id");
    std::unique_ptr<Grid> owned;
    {
        std::lock_guard<std::mutex> lq(c->q_mu);
        if (g->busy > 0) return fail(FC_ERR_STATE, "grid is used by a queued job");
        owned = std::move(c->grids[grid_id]);
        c->grids.erase(grid_id);
    }
    cudaSetDevice(c->device);
    cudaStreamSynchronize(c->stream);
    if (c->sync_lane.g == g) c->sync_lane.g = nullptr;
    for (auto it = c->lanes.begin(); it != c->lanes.end();) {
        if ((*it)->g == g) {
            lane_free(c, it->get());
            it = c->lanes.erase(it);
        } else {
            ++it;
        }
    }
    free_cache(c, g);
    dfree(c, g->S_full); dfree(c, g->S_fit); dfree(c, g->centre); dfree(c, g->Sc); dfree(c, g->Sc32);
    dfree(c, g->gnorm); dfree(c, g->Bt); dfree(c, g->collapse); dfree(c, g->F); dfree(c, g->Sdf);
    dfree(c, g->centre_df); dfree(c, g->model_i); dfree(c, g->model_d);
    return FC_OK;
}

fc_status fc_run_points(fc_ctx* c, int32_t grid_id, const int64_t* ps, int32_t P, uint64_t seed, int32_t U,
                        const fc_opts* opts, double* dchi2, int64_t* bestfit, int8_t* nscans) {
    if (!c) return fail(FC_ERR_ARG, "ctx is NULL");
    std::lock_guard<std::mutex> lk(c->api_mu);
    cudaSetDevice(c->device);
    return run_points_impl(c, grid_id, ps, P, seed, U, opts, dchi2, bestfit, nscans);
}

fc_status fc_run_point(fc_ctx* c, int32_t grid_id, int64_t p, uint64_t seed, int32_t U, const fc_opts* opts,
                       double* dchi2, int64_t* bestfit, int8_t* nscans) {
    return fc_run_points(c, grid_id, &p, 1, seed, U, opts, dchi2, bestfit, nscans);
}

fc_status fc_fake_data(fc_ctx* c, int32_t grid_id, const int64_t* ps, int32_t P, uint64_t seed, int32_t U,
                       int32_t fluct, float* d) {
    if (!c || !d) return fail(FC_ERR_ARG, "NULL argument");
    if (fluct != FC_FLUCT_POISSON_SYS && fluct != FC_FLUCT_GAUSS) return fail(FC_ERR_ARG, "bad fluct");
    std::lock_guard<std::mutex> lk(c->api_mu);
    cudaSetDevice(c->device);
    return fake_data_impl(c, grid_id, ps, P, seed, U, fluct, d);
}

fc_status fc_covariance(fc_ctx* c, int32_t grid_id, int64_t q, double* A, double* L_sys) {
    if (!c) return fail(FC_ERR_ARG, "ctx is NULL");
    std::lock_guard<std::mutex> lk(c->api_mu);
    cudaSetDevice(c->device);
    Grid* g = find_grid(c, grid_id);
    if (!g) return fail(FC_ERR_NOT_FOUND, "unknown grid id");
    if (!g->has_F) return fail(FC_ERR_STATE, "fractional covariance not set");
    if (q < 0 || q >= g->G) return fail(FC_ERR_ARG, "grid index out of range");
    if (A) {
        std::vector<int32_t> qs{(int32_t)q}, slots;
        FC_TRY(ensure_slots(c, g, qs, FC_COV_ITERATE, false, false, &slots));
        FC_TRY(read_ctrl(c));
        FC_TRY(copy_out(c, A, g->A64 + (size_t)slots[0] * g->nfit * g->nfit, (size_t)g->nfit * g->nfit * 8));
    }
    if (L_sys) {
        int64_t* pd = nullptr;
        double* L64 = nullptr;
        float *L32 = nullptr, *s32 = nullptr;
        FC_TRY(scratch(c, "cov_ps", 1, &pd));
        FC_TRY(scratch(c, "cov_L64", (size_t)g->nf * g->nf, &L64));
        FC_TRY(scratch(c, "cov_L32", (size_t)g->nf * g->nf, &L32));
        FC_TRY(scratch(c, "cov_s32", (size_t)g->nf, &s32));
        FC_CUDA(cudaMemcpyAsync(pd, &q, 8, cudaMemcpyHostToDevice, c->stream));
        launch_chol_sys(g->full(), g->nf, g->F, pd, 1, 0, L64, L32, s32, c->n_sm, c->status_dev, c->stream);
        FC_TRY(read_ctrl(c));
        FC_TRY(copy_out(c, L_sys, L64, (size_t)g->nf * g->nf * 8));
    }
    return sync(c);
}

fc_status fc_scan(fc_ctx* c, int32_t grid_id, const float* d, const int64_t* q_cov, int32_t U, int32_t precision,
                  int32_t top_k, int64_t* best, double* chi2_min) {
    if (!c || !d || !q_cov || !best) return fail(FC_ERR_ARG, "NULL argument");
    if (U < 0) return fail(FC_ERR_ARG, "U < 0");
    std::lock_guard<std::mutex> lk(c->api_mu);
    cudaSetDevice(c->device);
    Grid* g = find_grid(c, grid_id);
    if (!g) return fail(FC_ERR_NOT_FOUND, "unknown grid id");
    if (!g->has_F) return fail(FC_ERR_STATE, "fractional covariance not set");
    fc_opts o;
    fc_default_opts(&o);
    o.precision = precision;
    o.top_k = top_k;
    o.max_iter = 1;
    FC_TRY(validate_opts(&o, g));
    if (U == 0) return FC_OK;
    std::vector<int64_t> hq;
    FC_TRY(check_points(g, q_cov, U, &hq));
    c->stats = fc_stats{};
    c->acc = &c->stats;
    // every universe is its own point: its true point and first covariance are q_cov[u]
    FC_TRY(run_sync(c, g, o, hq, 1, 0, d, nullptr, best, nullptr, chi2_min, nullptr));
    return sync(c);
}

fc_status fc_data_dchi2(fc_ctx* c, int32_t grid_id, const float* d, const int64_t* ps, int32_t P,
                        const fc_opts* opts, double* dchi2, int64_t* bestfit, int8_t* nscans) {
    if (!c || !d || (P > 0 && (!ps || !dchi2))) return fail(FC_ERR_ARG, "NULL argument");
    if (P < 0) return fail(FC_ERR_ARG, "P < 0");
    std::lock_guard<std::mutex> lk(c->api_mu);
    cudaSetDevice(c->device);
    Grid* g = find_grid(c, grid_id);
    if (!g) return fail(FC_ERR_NOT_FOUND, "unknown grid id");
    if (!g->has_F) return fail(FC_ERR_STATE, "fractional covariance not set (fc_set_frac_cov)");
    fc_opts o;
    fc_default_opts(&o);
    if (opts) o = *opts;
    FC_TRY(validate_opts(&o, g));
    if (P == 0) return FC_OK;
    std::vector<int64_t> hps;
    FC_TRY(check_points(g, ps, P, &hps));
    std::vector<float> hd(g->nfit);
    if (is_device_ptr(d)) {
        FC_CUDA(cudaMemcpy(hd.data(), d, (size_t)g->nfit * 4, cudaMemcpyDeviceToHost));
    } else {
        memcpy(hd.data(), d, (size_t)g->nfit * 4);
    }
    for (float v : hd)
        if (!std::isfinite(v)) return fail(FC_ERR_ARG, "data must be finite");
    // every point is one universe whose data is the observed vector
    std::vector<float> rep((size_t)P * g->nfit);
    for (int32_t i = 0; i < P; ++i) memcpy(rep.data() + (size_t)i * g->nfit, hd.data(), (size_t)g->nfit * 4);
    c->stats = fc_stats{};
    c->acc = &c->stats;
    FC_TRY(run_sync(c, g, o, hps, 1, 0, rep.data(), dchi2, bestfit, nscans, nullptr, nullptr));
    return sync(c);
}

fc_status fc_fc_region(fc_ctx* c, const double* dchi2_univ, int32_t P, int32_t U, const double* dchi2_data,
                       double cl, double* crit, uint8_t* accepted) {
    if (!c || (P > 0 && (!dchi2_univ || !dchi2_data || !accepted))) return fail(FC_ERR_ARG, "NULL argument");
    if (P < 0 || U < 1 || U > 16384) return fail(FC_ERR_ARG, "bad sizes (1 <= U <= 16384)");
    if (!(cl >= 0.0 && cl <= 1.0)) return fail(FC_ERR_ARG, "cl must be in [0, 1]");
    if (P == 0) return FC_OK;
    std::lock_guard<std::mutex> lk(c->api_mu);
    cudaSetDevice(c->device);
    double *dp = nullptr, *dout = nullptr;
    const double* dx = nullptr;
    FC_TRY(scratch(c, "qp", 1, &dp));
    FC_TRY(scratch(c, "qout", (size_t)P, &dout));
    FC_TRY(quantile_input(c, dchi2_univ, (size_t)P * U, &dx));
    FC_CUDA(cudaMemcpyAsync(dp, &cl, 8, cudaMemcpyHostToDevice, c->stream));
    launch_quantiles(dx, P, U, dp, 1, dout, c->n_sm, c->stream);
    std::vector<double> hc(P), hd(P);
    FC_CUDA(cudaMemcpyAsync(hc.data(), dout, (size_t)P * 8, cudaMemcpyDeviceToHost, c->stream));
    FC_TRY(sync(c));
    if (is_device_ptr(dchi2_data)) {
        FC_CUDA(cudaMemcpy(hd.data(), dchi2_data, (size_t)P * 8, cudaMemcpyDeviceToHost));
    } else {
        memcpy(hd.data(), dchi2_data, (size_t)P * 8);
    }
    std::vector<uint8_t> acc(P);
    for (int32_t i = 0; i < P; ++i) acc[i] = (hd[i] <= hc[i]) ? 1 : 0;
    if (crit) FC_TRY(put_out(c, crit, hc.data(), (size_t)P * 8));
    FC_TRY(put_out(c, accepted, acc.data(), (size_t)P));
    return FC_OK;
}

fc_status fc_fc_region_adaptive(fc_ctx* c, int32_t grid_id, const int64_t* ps, int32_t P, const double* dchi2_data,
                                double cl, int32_t U0, int32_t U_max, double z, uint64_t seed, const fc_opts* opts,
                                uint8_t* accepted, int32_t* U_used, double* frac) {
    if (!c || (P > 0 && (!ps || !dchi2_data || !accepted))) return fail(FC_ERR_ARG, "NULL argument");
    if (P < 0 || U0 < 1 || U_max < U0 || U_max > (1 << 20))
        return fail(FC_ERR_ARG, "bad sizes (1 <= U0 <= U_max <= 2^20)");
    if (!(cl >= 0.0 && cl <= 1.0)) return fail(FC_ERR_ARG, "cl must be in [0, 1]");
    if (!(z >= 0.0) || !std::isfinite(z)) return fail(FC_ERR_ARG, "z must be finite and >= 0");
    std::lock_guard<std::mutex> lk(c->api_mu);
    cudaSetDevice(c->device);
    Grid* g = find_grid(c, grid_id);
    if (!g) return fail(FC_ERR_NOT_FOUND, "unknown grid id");
    if (!g->has_F) return fail(FC_ERR_STATE, "fractional covariance not set (fc_set_frac_cov)");
    fc_opts o;
    fc_default_opts(&o);
    if (opts) o = *opts;
    FC_TRY(validate_opts(&o, g));
    if (P == 0) return FC_OK;
    std::vector<int64_t> hps;
    FC_TRY(check_points(g, ps, P, &hps));
    std::vector<double> hd(P);
    if (is_device_ptr(dchi2_data))
        FC_CUDA(cudaMemcpy(hd.data(), dchi2_data, (size_t)P * 8, cudaMemcpyDeviceToHost));
    else
        memcpy(hd.data(), dchi2_data, (size_t)P * 8);
    for (double v : hd)
        if (std::isnan(v)) return fail(FC_ERR_ARG, "dchi2_data must not be NaN");
    c->stats = fc_stats{};
    c->acc = &c->stats;
    std::vector<int64_t> cnt(P, 0), used(P, 0);
    std::vector<uint8_t> acc(P, 0);
    std::vector<int32_t> open(P);
    for (int32_t i = 0; i < P; ++i) open[i] = i;
    // round r draws U_r new universes per open point with key seed + r: U0, then as many as the point
    // already has (the total doubles), the last round capped at U_max
    for (int round = 0; !open.empty(); ++round) {
        const int64_t have = used[open[0]];  // every open point has had the same rounds
        const int64_t U_r = std::min<int64_t>(round == 0 ? U0 : have, (int64_t)U_max - have);
        const int64_t Pr = (int64_t)open.size();
        if (Pr * U_r > (int64_t)INT32_MAX / 2) return fail(FC_ERR_ARG, "points x universes of a round too large");
        std::vector<int64_t> rps(Pr), rcnt(Pr, 0);
        std::vector<double> rthr(Pr);
        for (int64_t k = 0; k < Pr; ++k) {
            rps[k] = hps[open[k]];
            rthr[k] = hd[open[k]];
        }
        double *dx = nullptr, *dthr = nullptr;
        int64_t* dcnt = nullptr;
        FC_TRY(scratch(c, "ad_x", (size_t)(Pr * U_r), &dx));
        FC_TRY(scratch(c, "ad_thr", (size_t)Pr, &dthr));
        FC_TRY(scratch(c, "ad_cnt", (size_t)Pr, &dcnt));
        FC_TRY(run_sync(c, g, o, rps, (int32_t)U_r, seed + (uint64_t)round, nullptr, dx, nullptr, nullptr, nullptr,
                        nullptr));
        FC_TRY(to_device(c, dthr, rthr.data(), (size_t)Pr * 8));
        FC_CUDA(cudaMemsetAsync(dcnt, 0, (size_t)Pr * 8, c->stream));
        launch_count_below(dx, (int)Pr, (int)U_r, dthr, dcnt, c->stream);
        FC_CUDA(cudaMemcpyAsync(rcnt.data(), dcnt, (size_t)Pr * 8, cudaMemcpyDeviceToHost, c->stream));
        FC_TRY(sync(c));
        c->stats.universes += Pr * U_r;
        std::vector<int32_t> still;
        for (int64_t k = 0; k < Pr; ++k) {
            const int32_t i = open[k];
            cnt[i] += rcnt[k];
            used[i] += U_r;
            const double F = (double)cnt[i] / (double)used[i];
            const double half = z * std::sqrt(cl * (1.0 - cl) / (double)used[i]);
            acc[i] = (F <= cl) ? 1 : 0;
            if (used[i] < U_max && std::fabs(F - cl) <= half) still.push_back(i);
        }
        open.swap(still);
    }
    FC_TRY(put_out(c, accepted, acc.data(), (size_t)P));
    if (U_used) {
        std::vector<int32_t> uu(P);
        for (int32_t i = 0; i < P; ++i) uu[i] = (int32_t)used[i];
        FC_TRY(put_out(c, U_used, uu.data(), (size_t)P * 4));
    }
    if (frac) {
        std::vector<double> f(P);
        for (int32_t i = 0; i < P; ++i) f[i] = (double)cnt[i] / (double)used[i];
        FC_TRY(put_out(c, frac, f.data(), (size_t)P * 8));
    }
    return sync(c);
}

fc_status fc_quantiles(fc_ctx* c, const double* x, int32_t rows, int32_t n, const double* probs, int32_t nq,
                       double* out) {
    if (!c || !x || !probs || !out) return fail(FC_ERR_ARG, "NULL argument");
    if (rows < 0 || n < 1 || n > 16384 || nq < 1 || nq > 1024) return fail(FC_ERR_ARG, "bad sizes (n <= 16384)");
    std::vector<double> hp(nq);
    if (is_device_ptr(probs))
        FC_CUDA(cudaMemcpy(hp.data(), probs, (size_t)nq * 8, cudaMemcpyDeviceToHost));
    else
        memcpy(hp.data(), probs, (size_t)nq * 8);
    for (double p : hp)
        if (!(p >= 0.0 && p <= 1.0)) return fail(FC_ERR_ARG, "probabilities must be in [0, 1]");
    if (rows == 0) return FC_OK;
    std::lock_guard<std::mutex> lk(c->api_mu);
    cudaSetDevice(c->device);
    double *dp = nullptr, *dout = nullptr;
    const double* dx = nullptr;
    FC_TRY(scratch(c, "qp", (size_t)nq, &dp));
    FC_TRY(scratch(c, "qout", (size_t)rows * nq, &dout));
    FC_TRY(quantile_input(c, x, (size_t)rows * n, &dx));
    FC_CUDA(cudaMemcpyAsync(dp, hp.data(), (size_t)nq * 8, cudaMemcpyHostToDevice, c->stream));
    launch_quantiles(dx, rows, n, dp, nq, dout, c->n_sm, c->stream);
    FC_TRY(copy_out(c, out, dout, (size_t)rows * nq * 8));
    return sync(c);
}

fc_status fc_submit(fc_ctx* c, const fc_job* job, uint64_t* ticket) {
    if (!c || !job || !ticket) return fail(FC_ERR_ARG, "NULL argument");
    if (job->P < 0 || job->U < 0 || (job->P > 0 && !job->ps) || (job->P > 0 && job->U > 0 && !job->dchi2))
        return fail(FC_ERR_ARG, "bad job");
    auto jr = std::make_shared<JobRec>();
    jr->job = *job;
    jr->ps.resize(job->P);
    if (job->P > 0) {
        if (is_device_ptr(job->ps)) {
            cudaSetDevice(c->device);
            FC_CUDA(cudaMemcpy(jr->ps.data(), job->ps, (size_t)job->P * 8, cudaMemcpyDeviceToHost));
        } else {
            memcpy(jr->ps.data(), job->ps, (size_t)job->P * 8);
        }
    }
    jr->job.ps = jr->ps.data();
    jr->t_submit = std::chrono::steady_clock::now();
    std::lock_guard<std::mutex> lk(c->q_mu);
    auto it = c->grids.find(job->grid_id);
    if (it == c->grids.end()) return fail(FC_ERR_NOT_FOUND, "unknown grid id");
    const Grid* g = it->second.get();
    if (!g->has_F) return fail(FC_ERR_STATE, "fractional covariance not set (fc_set_frac_cov)");
    FC_TRY(validate_opts(&jr->job.opts, g));
    for (int64_t p : jr->ps)
        if (p < 0 || p >= g->G) return fail(FC_ERR_ARG, "true point index out of range");
    if ((int64_t)job->P * job->U > (int64_t)INT32_MAX / 2) return fail(FC_ERR_ARG, "P * U too large");
    // device memory the job may hold while it runs: per universe its lane state (data, indices,
    // results, work lists) and its share of the scan scratch (A-image row, bounds, candidates,
    // list counts), with the scratch buffers' growth headroom; it must fit the budget
    const size_t n = (size_t)job->P * job->U;
    const size_t need = n * (((size_t)g->nfit * 4 + 64 + (size_t)g->K * 4 + 320 + 17 * 16 + 24) * 5 / 4);
    if (c->budget && need > c->budget) return fail(FC_ERR_BUDGET, "job can never fit the device-memory budget");
    jr->need = need;
    it->second->busy++;
    const uint64_t t = c->next_ticket++;
    c->jobs[t] = jr;
    c->queue.push_back(jr);
    if (!c->worker_started) {
        c->worker = std::thread(worker_main, c);
        c->worker_started = true;
    }
    c->q_cv.notify_one();
    *ticket = t;
    return FC_OK;
}

fc_status fc_poll(fc_ctx* c, uint64_t ticket, double* latency_ms) {
    if (!c) return fail(FC_ERR_ARG, "ctx is NULL");
    std::lock_guard<std::mutex> lk(c->q_mu);
    auto it = c->jobs.find(ticket);
    if (it == c->jobs.end()) return fail(FC_ERR_NOT_FOUND, "unknown ticket");
    const int st = it->second->state.load();
    if (st == FC_PENDING) return FC_PENDING;
    if (latency_ms)
        *latency_ms =
            std::chrono::duration<double, std::milli>(it->second->t_done - it->second->t_submit).count();
    const std::string msg = it->second->error;
    c->jobs.erase(it);
    if (st != FC_OK) return fail((fc_status)st, msg.empty() ? "job failed" : msg);
    return FC_OK;
}

fc_status fc_cancel(fc_ctx* c, uint64_t ticket) {
    if (!c) return fail(FC_ERR_ARG, "ctx is NULL");
    std::lock_guard<std::mutex> lk(c->q_mu);
    auto it = c->jobs.find(ticket);
    if (it == c->jobs.end()) return fail(FC_ERR_NOT_FOUND, "unknown ticket");
    it->second->cancelled.store(true);
    return FC_OK;
}

fc_status fc_set_tuning(fc_ctx* c, int32_t grid_id, const fc_tuning* t) {
    if (!c || !t) return fail(FC_ERR_ARG, "NULL argument");
    std::lock_guard<std::mutex> lk(c->api_mu);
    Grid* g = find_grid(c, grid_id);
    if (!g) return fail(FC_ERR_NOT_FOUND, "unknown grid id");
    if (t->qvec < FC_QVEC_AUTO || t->qvec > FC_QVEC_TC) return fail(FC_ERR_ARG, "bad qvec choice");
    if (t->qvec == FC_QVEC_TC && !qvec_tc_supported(g->K))
        return fail(FC_ERR_ARG, "tensor-core q-vectors need K <= 128");
    if (!screen_config_ok(g->K, t->screen_stages, t->screen_ybuf))
        return fail(FC_ERR_ARG, "screen depth / buffering does not fit this K");
    if (t->cache_slots < 0 || t->cache_slots == 1) return fail(FC_ERR_ARG, "cache_slots must be 0 or >= 2");
    if (t->first_round < FC_ROUND_AUTO || t->first_round > FC_ROUND_LIST) return fail(FC_ERR_ARG, "bad first_round");
    if (t->slot_rows != 0 && t->slot_rows != kQuadRows && t->slot_rows != kBM)
        return fail(FC_ERR_ARG, "slot_rows must be 0, 32 or 128");
    // q-vectors from the other kernel have a different (still certified) bound: recompute them
    if (t->qvec != g->tune.qvec) std::fill(g->q32_ready.begin(), g->q32_ready.end(), 0);
    if (t->cache_slots > 0 && t->cache_slots < g->n_slots) reset_cache(c, g);
    g->tune = *t;
    return sync(c);
}

fc_status fc_get_tuning(fc_ctx* c, int32_t grid_id, fc_tuning* t) {
    if (!c || !t) return fail(FC_ERR_ARG, "NULL argument");
    std::lock_guard<std::mutex> lk(c->api_mu);
    Grid* g = find_grid(c, grid_id);
    if (!g) return fail(FC_ERR_NOT_FOUND, "unknown grid id");
    *t = g->tune;
    return FC_OK;
}

fc_status fc_autotune(fc_ctx* c, int32_t grid_id, const char* cache_path, fc_tuning* out) {
    if (!c) return fail(FC_ERR_ARG, "ctx is NULL");
    std::lock_guard<std::mutex> lk(c->api_mu);
    cudaSetDevice(c->device);
    Grid* g = find_grid(c, grid_id);
    if (!g) return fail(FC_ERR_NOT_FOUND, "unknown grid id");
    if (!g->has_F) return fail(FC_ERR_STATE, "fractional covariance not set (fc_set_frac_cov)");
    char key[512];
    snprintf(key, sizeof key, "fc-tune-v3 dev=%s sms=%d G=%lld nf=%d nfit=%d", c->dev_name.c_str(), c->n_sm,
             (long long)g->G, g->nf, g->nfit);
    auto valid = [&](const fc_tuning& t) {
        return t.qvec >= FC_QVEC_AUTO && t.qvec <= FC_QVEC_TC &&
               (t.qvec != FC_QVEC_TC || qvec_tc_supported(g->K)) &&
               screen_config_ok(g->K, t.screen_stages, t.screen_ybuf) &&
               (t.slot_rows == kQuadRows || t.slot_rows == kBM);
    };
    if (cache_path) {
        if (FILE* f = fopen(cache_path, "r")) {
            char line[768];
            const size_t kl = strlen(key);
            bool hit = false;
            fc_tuning t{};
            while (fgets(line, sizeof line, f)) {
                if (strncmp(line, key, kl) != 0 || line[kl] != ' ') continue;
                fc_tuning r{};
                r.cache_slots = g->tune.cache_slots;
                r.first_round = g->tune.first_round;
                if (sscanf(line + kl, " qvec=%d stages=%d ybuf=%d rows=%d", &r.qvec, &r.screen_stages, &r.screen_ybuf,
                           &r.slot_rows) == 4 &&
                    valid(r)) {
                    t = r;
                    hit = true;
                }
            }
            fclose(f);
            if (hit) {
                if (t.qvec != g->tune.qvec) std::fill(g->q32_ready.begin(), g->q32_ready.end(), 0);
                g->tune = t;
                if (out) *out = t;
                return FC_OK;
            }
        }
    }
    // the timing workload: one scan of 64 evenly spread true points x 256 universes
    const int32_t P = (int32_t)std::min<int64_t>(64, g->G), U = 256;
    std::vector<int64_t> ps(P);
    for (int32_t i = 0; i < P; ++i) ps[i] = (int64_t)i * g->G / P;
    std::vector<double> dchi2((size_t)P * U);
    fc_opts o;
    fc_default_opts(&o);
    o.max_iter = 1;
    const fc_tuning saved = g->tune;
    auto run = [&](const fc_tuning& t, bool cold, fc_stats* st) -> fc_status {
        if (t.qvec != g->tune.qvec || cold) reset_cache(c, g);
        g->tune = t;
        FC_TRY(run_points_impl(c, grid_id, ps.data(), P, 0x5eed, U, &o, dchi2.data(), nullptr, nullptr));
        *st = c->stats;
        return FC_OK;
    };
    fc_tuning best{};
    best.cache_slots = saved.cache_slots;
    best.first_round = saved.first_round;
    best.slot_rows = kQuadRows;
    fc_stats st{};
    fc_status rc = FC_OK;
    // q-vector kernel: covariance stage of a cold cache (P new covariances and q-vectors)
    std::vector<int> qv{FC_QVEC_SIMT};
    if (qvec_tc_supported(g->K)) qv.push_back(FC_QVEC_TC);
    double best_ms = 1e300;
    for (int q : qv) {
        fc_tuning t = best;
        t.qvec = q;
        if ((rc = run(t, true, &st)) != FC_OK) break;  // warm-up: scratch, cache storage
        if ((rc = run(t, true, &st)) != FC_OK) break;
        if (st.ms_cov < best_ms) {
            best_ms = st.ms_cov;
            best.qvec = q;
        }
    }
    // screen depth and A-image buffering, warm cache
    if (rc == FC_OK) {
        best_ms = 1e300;
        const int ks[] = {2, 3, 4, 5, 6, 8};
        for (int stg : ks)
            for (int yb = 1; yb <= 2; ++yb) {
                fc_tuning t = best;
                t.screen_stages = stg;
                t.screen_ybuf = yb;
                if (!screen_config_ok(g->K, stg, yb)) continue;
                if ((rc = run(t, false, &st)) != FC_OK) break;
                if ((rc = run(t, false, &st)) != FC_OK) break;
                if (st.ms_screen < best_ms) {
                    best_ms = st.ms_screen;
                    best.screen_stages = stg;
                    best.screen_ybuf = yb;
                }
            }
    }
    // tile shape: rows per covariance slot, on a short full fit (the 64 points x 256 universes, up to
    // five scans, warm cache), so the refit scans leave covariances as sparse as this grid makes them;
    // prep + screen + rescoring, the best of three runs after a warm-up, and whole tiles must beat the
    // 32-row default by 5 % (a timing job of 1024 one-scan covariances with 8 universes each, dominated
    // by per-tile overheads on small grids, picked whole tiles where a real job runs slower with them)
    if (rc == FC_OK) {
        fc_opts o5 = o;
        o5.max_iter = 5;
        double ms_rows[2] = {1e300, 1e300};
        const int rows_of[2] = {kQuadRows, kBM};
        for (int k = 0; k < 2 && rc == FC_OK; ++k) {
            fc_tuning t = best;
            t.slot_rows = rows_of[k];
            g->tune = t;
            for (int rep = 0; rep < 4 && rc == FC_OK; ++rep) {
                rc = run_points_impl(c, grid_id, ps.data(), P, 0x5eed, U, &o5, dchi2.data(), nullptr, nullptr);
                const double ms = c->stats.ms_prep + c->stats.ms_screen + c->stats.ms_rescore;
                if (rep > 0 && ms < ms_rows[k]) ms_rows[k] = ms;
            }
        }
        best.slot_rows = (ms_rows[1] < 0.95 * ms_rows[0]) ? kBM : kQuadRows;
    }
    reset_cache(c, g);
    if (rc != FC_OK) {
        g->tune = saved;
        return rc;
    }
    g->tune = best;
    if (out) *out = best;
    if (cache_path) {
        if (FILE* f = fopen(cache_path, "a")) {
            fprintf(f, "%s qvec=%d stages=%d ybuf=%d rows=%d\n", key, best.qvec, best.screen_stages, best.screen_ybuf,
                    best.slot_rows);
            fclose(f);
        }
    }
    return sync(c);
}

fc_status fc_get_serve_stats(fc_ctx* c, fc_stats* out) {
    if (!c || !out) return fail(FC_ERR_ARG, "NULL argument");
    std::lock_guard<std::mutex> lk(c->api_mu);
    *out = c->serve_stats;
    out->device_bytes = (int64_t)c->used;
    return FC_OK;
}

fc_status fc_measure_peaks(fc_ctx* c, double* fp64_tflops, double* fp32_tflops) {
    if (!c || !fp64_tflops || !fp32_tflops) return fail(FC_ERR_ARG, "NULL argument");
    std::lock_guard<std::mutex> lk(c->api_mu);
    cudaSetDevice(c->device);
    if (!measure_fma_peaks(c->n_sm, fp64_tflops, fp32_tflops, c->stream))
        return fail(FC_ERR_CUDA, "fma peak probe failed");
    return sync(c);
}

fc_status fc_set_wait_test(fc_ctx* c, uint64_t wait_ns, int64_t screen_stop_after) {
    if (!c) return fail(FC_ERR_ARG, "ctx is NULL");
    if (screen_stop_after < -1) return fail(FC_ERR_ARG, "screen_stop_after must be >= -1");
    if (wait_ns > 2000000000ull) return fail(FC_ERR_ARG, "wait_ns above the built-in limit (2 s)");
    std::lock_guard<std::mutex> lk(c->api_mu);
    c->wait_test = WaitTest{wait_ns, screen_stop_after};
    return FC_OK;
}

fc_status fc_get_decided_by(fc_ctx* c, uint8_t* out, int64_t n) {
    if (!c || (n > 0 && !out)) return fail(FC_ERR_ARG, "NULL argument");
    std::lock_guard<std::mutex> lk(c->api_mu);
    cudaSetDevice(c->device);
    if (c->last_n < 0 || !c->sync_lane.rmask) return fail(FC_ERR_STATE, "no synchronous fit on this context yet");
    if (n != c->last_n)
        return fail(FC_ERR_ARG, "n must be the last fit's universe count (" + std::to_string(c->last_n) + ")");
    if (n == 0) return FC_OK;
    FC_TRY(copy_out(c, out, c->sync_lane.rmask + c->last_base, (size_t)n));
    return sync(c);
}

fc_status fc_get_stats(fc_ctx* c, fc_stats* out) {
    if (!c || !out) return fail(FC_ERR_ARG, "NULL argument");
    *out = c->stats;
    out->device_bytes = (int64_t)c->used;
    return FC_OK;
}

const char* fc_last_error(const fc_ctx*) { return t_last_error.c_str(); }

}  // extern "C"
