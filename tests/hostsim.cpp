// A stand-in for the CUDA runtime and the kernel launchers, on which the
// library's host code (wost_capi.cpp) runs without a device: device memory is
// host memory up to a limit, streams and events only record how they are used,
// and a launch is a line of a log.  tests/test_host_cpu.py builds and drives it.
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <new>
#include <string>
#include <vector>

#include "capi_internal.h"

struct CUstream_st {
    bool alive = true;
    bool busy = false;  // launched on, not waited for since
};
struct CUevent_st {
    bool pending = false;
};

// host allocations of the library, refused on demand
static bool refuse_new = false;
void *operator new(size_t n) {
    void *p = refuse_new ? nullptr : std::malloc(n ? n : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, size_t) noexcept { std::free(p); }

namespace {

struct Sim {
    std::map<void *, size_t> mem;
    size_t used = 0, limit = ~(size_t)0;
    int bad = 0;        // uses of a destroyed stream
    bool hold = false;  // launches stay in flight (their events are not ready)
    bool launched = false;
    int fail_record = 0;  // the cudaEventRecord that fails, counted from now on (0: none)
    std::vector<cudaStream_t> streams;
    int to_go = 3;      // launches after which a resumable solve has no walk left to draw; one more ends it
    const int *cancel = nullptr;  // the last launch's cancel flag
    std::string log;
} sim;

cudaError_t use(cudaStream_t s) {
    if (s && !s->alive) ++sim.bad;
    return cudaSuccess;
}
cudaError_t launch(const std::string &what, cudaStream_t s) {
    sim.log += what + "\n";
    sim.launched = true;
    if (s) s->busy = true;
    return use(s);
}
cudaError_t get(void **p, size_t n) {
    *p = nullptr;
    if (n > sim.limit || sim.used > sim.limit - n) return cudaErrorMemoryAllocation;
    *p = std::calloc(n ? n : 1, 1);
    sim.mem[*p] = n;
    sim.used += n;
    return cudaSuccess;
}

}  // namespace

extern "C" {

void sim_reset(size_t limit) {
    sim.limit = limit;
    sim.bad = 0;
    sim.hold = sim.launched = false;
    for (cudaStream_t s : sim.streams) s->busy = false;
    sim.to_go = 3;
    sim.log.clear();
}
void sim_limit(size_t n) { sim.limit = n; }
void sim_to_go(int n) { sim.to_go = n; }
void sim_refuse_new(int on) { refuse_new = on != 0; }
void sim_hold(int on) { sim.hold = on != 0; }
size_t sim_used(void) { return sim.used; }
void sim_fail_record(int n) { sim.fail_record = n; }
int sim_busy(void) {
    int n = 0;
    for (cudaStream_t s : sim.streams) n += s->busy;
    return n;
}
int sim_bad(void) { return sim.bad; }
const char *sim_log(void) { return sim.log.c_str(); }

cudaError_t cudaMalloc(void **p, size_t n) { return get(p, n); }
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) { return get(p, n); }
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t, cudaStream_t) { return get(p, n); }
cudaError_t cudaFree(void *p) {
    if (!p) return cudaSuccess;
    sim.used -= sim.mem.at(p);
    sim.mem.erase(p);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return cudaFree(p); }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return (*p = std::calloc(n, 1)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFreeHost(void *p) {
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaHostGetDevicePointer(void **d, void *h, unsigned) {
    *d = h;
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpy2D(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind) {
    for (size_t i = 0; i < h; ++i) std::memcpy((char *)d + i * dp, (const char *)s + i * sp, w);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t st) {
    std::memcpy(d, s, n);
    return use(st);
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t st) {
    std::memset(d, v, n);
    return use(st);
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    *s = new CUstream_st;
    sim.streams.push_back(*s);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {  // (kept, so that later uses are seen)
    use(s);
    s->alive = false;
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    if (s) s->busy = false;
    return use(s);
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t, unsigned) { return use(s); }
cudaError_t cudaDeviceSynchronize(void) {
    sim.log += "device synchronised\n";
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) {
    *e = new CUevent_st;
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    delete e;
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    if (sim.fail_record > 0 && --sim.fail_record == 0) return cudaErrorUnknown;
    e->pending = sim.launched;
    return use(s);
}
cudaError_t cudaEventQuery(cudaEvent_t e) { return sim.hold && e->pending ? cudaErrorNotReady : cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) {
    if (sim.hold && e->pending) sim.log += sim.cancel && *sim.cancel ? "waiting, cancelled\n" : "waiting\n";
    return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.f;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceCount(int *n) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }

}  // extern "C"

namespace wost {

constexpr int kBlocks = 16;

static uint64_t all_walks(const SolveParams &sp) { return (uint64_t)sp.n_points * (uint64_t)sp.walks_per_point; }

cudaError_t launch_walk_plain(const SceneView &, const SolveParams &sp, const Accumulators &acc, int, cudaStream_t s) {
    *acc.next_walk = all_walks(sp);
    return launch("plain", s);
}
cudaError_t launch_walk_count(const SceneView &, const SolveParams &sp, const Accumulators &acc, unsigned long long *,
                              int, cudaStream_t s) {
    *acc.next_walk = all_walks(sp);
    return launch("counting", s);
}
cudaError_t persistent_grid(int, int, int, int *blocks, int) {
    *blocks = kBlocks;
    return cudaSuccess;
}
cudaError_t batch_grid(int, int, int, int *blocks) {
    *blocks = kBlocks;
    return cudaSuccess;
}
cudaError_t resume_grid(int, int, int, int *blocks, int) {
    *blocks = kBlocks;
    return cudaSuccess;
}
int64_t resume_slots(int block, int blocks, int lanes) { return (int64_t)blocks * (block / lanes); }
uint64_t chain_capacity(uint64_t, int, int, int) { return 1 << 16; }
uint64_t batch_chain_capacity(int, int, int) { return 1 << 16; }
cudaError_t launch_walk_batch(int dim, const BatchHeader *, const BatchJob *, unsigned long long *, unsigned int *, int,
                              const int *, int, int, const ChainBuffers &cb, cudaStream_t s, unsigned long long *,
                              bool) {
    return launch("batch " + std::to_string(dim) + "d" + (cb.slots[0] ? "" : " without slots"), s);
}
cudaError_t launch_walk_persistent(const SceneView &, const SolveParams &sp, const Accumulators &acc, int, int,
                                   cudaStream_t s, int lanes, const SavedWalks &, const HandOver &) {
    *acc.next_walk = all_walks(sp);
    *acc.steps = lanes == 1 ? 1000 : 500;
    return launch(lanes == 1 ? "persistent" : "persistent, 8 lanes", s);
}
cudaError_t launch_walk_warp(const SceneView &, const SolveParams &sp, const Accumulators &acc, const SavedWalks &,
                             uint64_t, cudaStream_t s) {
    *acc.next_walk = all_walks(sp);
    *acc.steps = 1000;
    return launch("one per warp", s);
}
cudaError_t launch_walk_chain(const SceneView &, const SolveParams &sp, const Accumulators &acc, SavedWalks src,
                              uint64_t, const ChainBuffers &, int, int, cudaStream_t s) {
    *acc.next_walk = all_walks(sp);
    *acc.steps = 1000;
    sim.cancel = acc.cancel;
    return launch(src.slots ? "chain from saved walks" : "chain", s);
}
cudaError_t launch_walk_resume(const SceneView &, const SolveParams &sp, const Accumulators &acc, const ResumeState &rs,
                               int iters, int, int, cudaStream_t s, int lanes) {
    const uint64_t total = all_walks(sp);
    sim.cancel = acc.cancel;
    *rs.steps_run += lanes == 1 ? 500 : 1000;  // 8 lanes look faster per launch, a whole solve is not
    --sim.to_go;
    *acc.next_walk = sim.to_go > 0 ? total / 2 : total;
    *rs.live = sim.to_go >= 0 ? 5 : 0;
    return launch("resume " + std::to_string(iters), s);
}
cudaError_t launch_screened_kernels(int, int64_t, const float *, const float *, float, float *, float *,
                                    cudaStream_t s) {
    return launch("screened kernels", s);
}
cudaError_t launch_query_closest(const SceneView &, int64_t, const float *, float *, float *, int32_t *, int,
                                 unsigned int *, cudaStream_t s) {
    return launch("closest", s);
}
cudaError_t launch_query_silhouette(const SceneView &, int64_t, const float *, const float *, float *, int,
                                    unsigned int *, cudaStream_t s) {
    return launch("silhouette", s);
}
cudaError_t launch_query_ray(const SceneView &, int64_t, const float *, const float *, const float *, const int32_t *,
                             const int32_t *, int64_t, int32_t *, float *, int32_t *, int, unsigned int *,
                             cudaStream_t s) {
    return launch("ray", s);
}
cudaError_t launch_query_sample(const SceneView &, int64_t, const float *, const float *, uint32_t, uint32_t, uint32_t,
                                uint32_t, float *, float *, int32_t *, cudaStream_t s) {
    return launch("sample", s);
}
void engine_detach(wost_engine *, wost_solve_handle *) {}

}  // namespace wost
