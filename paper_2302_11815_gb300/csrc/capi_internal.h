// Internal objects behind the C ABI handles, shared by wost_capi.cpp and
// wost_engine.cpp.
#pragma once

#include <cuda_runtime.h>

#include <chrono>
#include <cstring>
#include <memory>
#include <atomic>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#include "../../include/wost.h"
#include "scene_build.h"
#include "wost_kernels.h"

namespace wost {

// records the thread-local error message and returns s
wost_status fail(wost_status s, const std::string &msg);
wost_status cuda_fail(cudaError_t e, const char *what);
#define CK(expr, what)                                     \
    do {                                                   \
        cudaError_t _e = (expr);                           \
        if (_e != cudaSuccess) return wost::cuda_fail(_e, what); \
    } while (0)

// device allocation owned by a scene or solve, or a part of one (view)
struct DevBuf {
    void *p = nullptr;
    size_t bytes = 0;
    bool owned = true;
    DevBuf() = default;
    DevBuf(const DevBuf &) = delete;
    DevBuf &operator=(const DevBuf &) = delete;
    ~DevBuf() { release(); }
    void release() {
        if (p && owned) cudaFree(p);
        p = nullptr;
        bytes = 0;
        owned = true;
    }
    cudaError_t alloc(size_t n) {
        const cudaError_t e = n ? cudaMalloc(&p, n) : cudaSuccess;
        if (e != cudaSuccess) p = nullptr;
        bytes = p ? n : 0;
        return e;
    }
    // at least n bytes (contents lost when it grows)
    cudaError_t ensure(size_t n) {
        if (bytes >= n) return cudaSuccess;
        release();
        return alloc((n + 65535) & ~(size_t)65535);
    }
    void view(void *base, size_t n) {
        release();
        p = n ? base : nullptr;
        bytes = n;
        owned = false;
    }
    // stream-ordered allocation / release: neither waits for the device,
    // unlike cudaMalloc / cudaFree, which synchronise with all work in flight
    cudaError_t alloc_async(size_t n, cudaStream_t s, cudaMemPool_t pool = nullptr) {
        bytes = n;
        if (!n) return cudaSuccess;
        return pool ? cudaMallocFromPoolAsync(&p, n, pool, s) : cudaMallocAsync(&p, n, s);
    }
    void release_async(cudaStream_t s) {
        if (p) cudaFreeAsync(p, s);
        p = nullptr;
    }
};

// One device allocation for many arrays, filled by one copy: arrays are added
// to a host image, placed (their buffers become views of the allocation) and
// uploaded.
struct DevImage {
    std::vector<unsigned char> host;
    std::vector<std::pair<DevBuf *, std::pair<size_t, size_t>>> parts;
    size_t reserve(size_t n) {
        const size_t at = (host.size() + 255) & ~(size_t)255;
        host.resize(at + n);
        return at;
    }
    template <class T>
    void add(DevBuf &b, const std::vector<T> &v) {
        const size_t n = v.size() * sizeof(T), at = reserve(n);
        if (n) std::memcpy(host.data() + at, v.data(), n);
        parts.push_back({&b, {at, n}});
    }
    cudaError_t place(DevBuf &dev) {
        cudaError_t e = dev.alloc(host.size());
        if (e != cudaSuccess) return e;
        for (auto &q : parts) q.first->view((unsigned char *)dev.p + q.second.first, q.second.second);
        return cudaSuccess;
    }
    cudaError_t upload(const DevBuf &dev) const {
        return cudaMemcpy(dev.p, host.data(), host.size(), cudaMemcpyHostToDevice);
    }
};

// What a solve needs beside its results' memory: streams, events, pinned host
// memory and device buffers.  Setting these up and giving them back took 0.5
// ms per solve, so a scene keeps those of its last finished solves.
struct SolveRes {
    DevBuf main, chain, resume;  // inputs and accumulators; hand-over slots; saved walks
    unsigned char *host = nullptr;  // pinned, mapped: the cancel flag, then kStaging bytes for results
    unsigned char *host_dev = nullptr;
    cudaStream_t stream = nullptr, poll = nullptr;
    cudaEvent_t ev_start = nullptr, ev_done = nullptr, ev_copy = nullptr;
    static constexpr size_t kStagingAt = 256, kStaging = 64u << 10;
    cudaError_t init() {
        cudaError_t e = cudaHostAlloc((void **)&host, kStagingAt + kStaging, cudaHostAllocMapped);
        if (e == cudaSuccess) e = cudaHostGetDevicePointer((void **)&host_dev, host, 0);
        if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&poll, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreate(&ev_start);
        if (e == cudaSuccess) e = cudaEventCreate(&ev_done);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev_copy, cudaEventDisableTiming);
        return e;
    }
    size_t bytes() const { return main.bytes + chain.bytes + resume.bytes; }
    ~SolveRes() {
        for (cudaEvent_t e : {ev_start, ev_done, ev_copy})
            if (e) cudaEventDestroy(e);
        for (cudaStream_t s : {stream, poll})
            if (s) cudaStreamDestroy(s);
        if (host) cudaFreeHost(host);
    }
};

// The resources that a scene's finished solves left for its next ones.  All
// scenes' idle sets are in one list (idle_sets, in the order they were given
// back): a device keeps kAllBytes of them in all, a scene kIdle sets of
// kIdleBytes each at most; the oldest go first, all of a device's when an
// allocation of the library finds no memory there, a scene's with the scene
// (a set given back later is freed then).
struct SolvePool {
    static constexpr size_t kIdle = 4, kIdleBytes = 64u << 20, kAllBytes = 256u << 20;
    int device = 0;
    bool closed = false;  // (guarded by the list's mutex)
    cudaError_t take(std::unique_ptr<SolveRes> &out);
    void give(std::unique_ptr<SolveRes> r);  // (the device is no longer using the set)
    void close();
};
// frees the idle sets of `device`; returns how many
size_t drop_idle(int device);
// alloc(), once more without the device's idle sets if memory is short
template <class F>
inline cudaError_t with_memory(int device, F alloc) {
    const cudaError_t e = alloc();
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();
    return drop_idle(device) ? alloc() : e;
}

// Words (u64) of a batched launch's counters.
constexpr size_t kBatchCounters = 4 + 2 * kMaxStages;
// The chain buffers of dimension di (0: 2D, 1: 3D) of a batched launch, in
// `chain`, for its grid; without memory for them, none (the launch then keeps
// its walks to their ends).
inline cudaError_t batch_chain_buffers(int device, DevBuf &chain, unsigned long long *counters, int di, int block,
                                       int blocks, ChainBuffers *cb) {
    size_t bytes[2];
    for (int i = 0; i < 2; ++i) {
        cb->cap[i] = (unsigned)batch_chain_capacity(block, blocks, i);
        bytes[i] = (size_t)cb->cap[i] * 3 * sizeof(float4);
    }
    const cudaError_t e = with_memory(device, [&] { return chain.ensure(bytes[0] + bytes[1]); });
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        *cb = ChainBuffers{};
        return cudaSuccess;
    }
    if (e != cudaSuccess) return e;
    cb->slots[0] = (float4 *)chain.p;
    cb->slots[1] = (float4 *)((unsigned char *)chain.p + bytes[0]);
    cb->counters = (unsigned int *)(counters + 4 + di * kMaxStages);
    return cudaSuccess;
}

// resources shared by the solves of one batched launch
struct BatchShared {
    // counters: next walk (2D), next walk (3D), guard, -, then each
    // dimension's hand-over counters
    DevBuf jobs[2], counters;
    unsigned long long total[2] = {0, 0};
    cudaEvent_t ev_start = nullptr, ev_done = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;  // the 3D launch's side stream
    cudaStream_t own_stream = nullptr, side = nullptr;
    ~BatchShared() {
        if (ev_done) cudaEventSynchronize(ev_done);
        if (ev_start) cudaEventDestroy(ev_start);
        if (ev_done) cudaEventDestroy(ev_done);
        if (ev_fork) cudaEventDestroy(ev_fork);
        if (ev_join) cudaEventDestroy(ev_join);
        if (side) cudaStreamDestroy(side);
        if (own_stream) cudaStreamDestroy(own_stream);
    }
};

}  // namespace wost

struct wost_engine;

struct wost_scene {
    int device = 0;
    wost::HostScene host;
    wost::SceneView view{};
    wost::DevBuf image;  // every array below, one allocation
    wost::DevBuf bufs[16];
    wost::DevBuf wbufs[6];  // wide layout: nodes and cones of the three trees
    wost::DevBuf xbufs[18];  // per tree: wide top and its cones, parents, leaf parents, treelets, hints
    wost::DevBuf sbufs[4];  // double-sided records (App. B): - side data and flags of D and N
    wost::DevBuf n_rec_of_id;
    unsigned int *guard = nullptr;        // guard word of the query kernels (pinned host memory), its device address
    unsigned int *guard_dev = nullptr;
    std::shared_ptr<wost::SolvePool> pool = std::make_shared<wost::SolvePool>();
    wost::SceneView *view_dev = nullptr;  // device copy of `view` (batched launches)
    wost_scene_info info{};
    int stack_depth = 0;                  // traversal stack entries per walk, one lane per walk
    int stack_depth_team = 0;             // ... per 8-lane team over the 8-wide trees
    int tuned_block = 0;                  // set by wost_scene_autotune (0 = not tuned)
    int tuned_lanes = 1;                  // lanes per walk chosen by wost_scene_autotune
    std::mutex mu;
    ~wost_scene() {
        pool->close();
        if (guard) cudaFreeHost(guard);
    }
};

struct wost_solve_handle {
    wost_scene *scene = nullptr;
    int device = 0;
    int dim = 2;
    int64_t n_points = 0;
    int32_t walks = 0;
    int block = 128;
    int lanes = 1;                        // lanes per walk (persistent / resumable kernels)
    bool warp_ok = false;                 // the scene's own traversal limits: walks may run one per warp
    cudaStream_t stream = nullptr;
    cudaStream_t poll_stream = nullptr;
    bool own_poll_stream = false;  // an engine request whose engine is gone
    cudaEvent_t ev_start = nullptr, ev_done = nullptr;
    std::shared_ptr<wost::BatchShared> batch;  // set for solves started by wost_solve_batch
    unsigned int *batch_guard = nullptr;
    wost_engine *engine = nullptr;             // set for solves submitted to an engine
    std::unique_ptr<wost::SolveRes> res;       // streams, events, memory (not for engine requests)
    std::shared_ptr<wost::SolvePool> res_pool;  // where they go back to
    wost::SolveParams sp{};
    wost::Accumulators acc{};
    wost::DevBuf points, normals, onN;
    wost::DevBuf sum, sumsq, walks_done, steps, globals;  // globals: capped, next_walk, guard, -, hand-over counters
    wost::DevBuf counts;                                   // counting kernel only
    // resumable solves: saved-walk slots of the fixed grid, launch counters
    // (steps_run u64, live u32), launches enqueued so far
    wost::DevBuf slots, rstate;
    int resume_blocks = 0;
    uint64_t launches = 0;
    bool idle = false;  // nothing of it is in flight though no event tells: a resumable solve until its first launch
    std::atomic<bool> handed_out{false};  // the caller has device pointers to the accumulators
    bool resumable() const { return kernel == WOST_KERNEL_RESUMABLE; }
    int kernel = 0;
    int *cancel_host = nullptr;                            // mapped pinned (engine requests: plain host)
    int *cancel_dev = nullptr;
    // engine requests: device buffers come from the stream-ordered allocator
    // and the cancel flag is plain host memory (the engine reads it on the
    // host), so that destroying a request never waits for the device, whose
    // queue the engine keeps full
    bool engine_buffers = false;
    cudaMemPool_t pool = nullptr;  // the engine's memory pool (engine requests)
    // engine requests: set once a round holding some of the request's walks
    // has completed; until then a poll reports no walks without reading
    // the device (its buffers may still be being set up)
    std::atomic<bool> engine_ready{false};
    std::chrono::steady_clock::time_point t_launch;
    double elapsed_done = -1;
    bool done = false;
    wost_status final_status = WOST_OK;                    // engine requests
    std::mutex mu;
    ~wost_solve_handle() {
        // a resumable solve drops the walks it has not drawn
        if (resumable() && !done && cancel_host) *(volatile int *)cancel_host = 1;
        // (a stream of the caller's is used only by a call that failed before
        // its event was recorded: the caller may have destroyed it since)
        if (ev_done && launches) cudaEventSynchronize(ev_done);
        else if (stream && !idle) cudaStreamSynchronize(stream);
        if (res) {
            // reads that the caller enqueued on its own streams, before the
            // memory is another solve's
            if (handed_out) cudaDeviceSynchronize();
            res_pool->give(std::move(res));
            return;
        }
        if (engine_buffers) {
            for (wost::DevBuf *b : {&points, &normals, &onN, &sum, &sumsq, &walks_done, &steps, &globals})
                b->release_async(poll_stream);
            delete cancel_host;
        }
        if (poll_stream && own_poll_stream) cudaStreamDestroy(poll_stream);
    }
};

namespace wost {
// Layout fields of a scene's info for `lanes` lanes per walk.
void set_layout_info(wost_scene *s, int lanes);
// Validates a solve description, allocates and fills the solve's device
// buffers on `stream`, fills h->sp and h->acc.  Does not launch.  With
// fill false the buffers are only allocated: the caller uploads the points,
// normals and flags and clears the accumulators (the serving engine does
// both on streams of its own).
wost_status prepare_solve(wost_scene *scene, const wost_solve_desc *d, cudaStream_t stream, wost_solve_handle *h,
                          bool fill = true);
// u64 words of a solve's globals: 4, then the hand-over counters
constexpr size_t kGlobals = 4 + kMaxStages;
// Zeroes a solve's accumulators and counters on `stream`.
cudaError_t clear_accumulators(wost_solve_handle *h, cudaStream_t stream);
// Blocks until the work queued so far on `stream` (the input copies) is done.
wost_status wait_for_copies(cudaStream_t stream, cudaEvent_t ev);
// Engine side of wost_solve_destroy / wost_cancel for engine requests.
void engine_detach(wost_engine *e, wost_solve_handle *h);
}  // namespace wost
