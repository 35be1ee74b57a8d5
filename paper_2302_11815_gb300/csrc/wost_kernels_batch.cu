// The batched persistent kernel over many solves (wost_solve_batch and the
// serving engine's rounds) in its screened and Poisson-only forms, and their
// launchers (sm_103a).  The Poisson-only form runs when no job of a batch is
// screened: the screened terms enlarge the walk loop's code, and instruction
// supply is what stalls these kernels most.
#include <cuda_runtime.h>

#include <algorithm>

#include "wost_batch.cuh"
#include "wost_screened.cuh"

namespace wost {

namespace {

// the fewest resident blocks per SM of a dimension's forms (their shared
// memory size is set for all of them)
template <int D>
cudaError_t occupancy(int block, size_t sm, int *per_sm) {
    *per_sm = 0;
    for (const void *k : {(const void *)k_walk_batch<D, false, false>, (const void *)k_walk_batch<D, false, true>,
                          (const void *)k_walk_batch<D, true, false>, (const void *)k_walk_batch<D, true, true>}) {
        int n = 0;
        cudaError_t e = smem_limit(k, sm);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, block, sm);
        if (e != cudaSuccess) return e;
        if (!*per_sm || n < *per_sm) *per_sm = n;
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t batch_grid(int dim, int block, int depth, int *blocks_out) {
    int sms = 0, per_sm = 0;
    cudaError_t e = sm_count(&sms);
    const size_t sm = smem_bytes(depth, block);
    if (e == cudaSuccess) e = dim == 2 ? occupancy<2>(block, sm, &per_sm) : occupancy<3>(block, sm, &per_sm);
    // the warp kernels that end a batch are loaded now, not while a graph is captured
    for (int scr = 0; scr < 2 && e == cudaSuccess; ++scr) e = prepare_walk_warp_batch(dim, depth, scr != 0);
    if (e != cudaSuccess) return e;
    *blocks_out = sms * (per_sm > 0 ? per_sm : 1);
    return cudaSuccess;
}

namespace {

template <int D, bool SCR>
cudaError_t launch(const BatchHeader *hdr, const BatchJob *jobs, unsigned long long *counter, unsigned int *guard,
                   int depth, const int *cancel, int block, int blocks, cudaStream_t s, unsigned long long *steps_out,
                   const SavedWalks &src, const HandOver &ho) {
    const auto k = src.slots ? k_walk_batch<D, SCR, true> : k_walk_batch<D, SCR, false>;
    k<<<blocks, block, smem_bytes(depth, block), s>>>(hdr, jobs, counter, guard, depth, cancel, steps_out, src, ho);
    return cudaGetLastError();
}

}  // namespace

uint64_t batch_chain_capacity(int block, int blocks, int which) {
    return std::max<uint64_t>(kTailWalks, ((uint64_t)blocks * (uint64_t)block) >> (which + 1));
}

// As launch_walk_chain, without knowing how many walks the launch will hold
// (a captured graph is replayed over other tables): a launch that begins
// with fewer walks than it would hand over hands them over at once.
cudaError_t launch_walk_batch(int dim, const BatchHeader *hdr, const BatchJob *jobs, unsigned long long *counter,
                              unsigned int *guard, int depth, const int *cancel, int block, int blocks,
                              const ChainBuffers &cb, cudaStream_t s, unsigned long long *steps_out, bool screened) {
    SavedWalks src{};
    const uint64_t resident = (uint64_t)blocks * (uint64_t)block;
    uint64_t walks = ~0ull;
    int sms = 0;
    cudaError_t e = sm_count(&sms);
    if (e != cudaSuccess) return e;
    for (int stage = 0; stage < kMaxStages && walks > kTailWalks; ++stage) {
        const int b = stage & 1;
        const uint64_t held = std::min(walks, resident);
        uint64_t most = held / 2 < kTailWalks * 3 / 2 ? kTailWalks : held / 2;
        most = std::min<uint64_t>(most, cb.cap[b]);
        unsigned int *ctr = cb.slots[b] ? cb.counters + 2 * stage : nullptr;
        const unsigned per_warp = src.per_warp ? src.per_warp : 32u;
        const uint64_t per_block = (uint64_t)(block / 32) * per_warp;
        const int grid =
            walks == ~0ull ? blocks : (int)std::min<uint64_t>((uint64_t)blocks, (walks + per_block - 1) / per_block);
        if (!cb.slots[b]) most = 0;  // (no memory: this launch runs its walks to their ends)
        const HandOver ho{cb.slots[b], ctr, (unsigned)most, (unsigned)grid * (unsigned)per_block};
        e = dim == 2 ? (screened ? launch<2, true>(hdr, jobs, counter, guard, depth, cancel, block, grid, s, steps_out,
                                                   src, ho)
                                 : launch<2, false>(hdr, jobs, counter, guard, depth, cancel, block, grid, s, steps_out,
                                                    src, ho))
                     : (screened ? launch<3, true>(hdr, jobs, counter, guard, depth, cancel, block, grid, s, steps_out,
                                                   src, ho)
                                 : launch<3, false>(hdr, jobs, counter, guard, depth, cancel, block, grid, s, steps_out,
                                                    src, ho));
        if (e != cudaSuccess || !cb.slots[b]) return e;
        src = SavedWalks{cb.slots[b], nullptr, ctr, ctr + 1, nullptr, spread_walks(dim, most, sms)};
        walks = most;
    }
    return launch_walk_warp_batch(dim, hdr, jobs, guard, depth, src, steps_out, screened, s);
}

}  // namespace wost
