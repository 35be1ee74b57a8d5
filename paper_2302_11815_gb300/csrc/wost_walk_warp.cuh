// Walk kernels with one walk per warp (WarpQ, wost_warp.cuh): all of a small
// solve's walks, or the last walks of a large one, which the one-lane kernels
// hand over in saved-walk slots once too few of them are left to fill lanes.
#pragma once

#include "wost_walk.cuh"
#include "wost_warp.cuh"

// Register cap of the one-walk-per-warp kernels.
#ifndef WOST_WARP_REGS
#define WOST_WARP_REGS 96
#endif

namespace wost {

constexpr int kWarpFrontier = 192;  // frontier entries per warp (an overflow falls back to the binary trees)

template <int D, bool WALK = true>
__device__ __forceinline__ WarpQ<D, WALK> make_warp_q(int depth, unsigned int *guard) {
    extern __shared__ int2 smem_stack[];
    WarpQ<D, WALK> q;
    int2 *mine = smem_stack + (threadIdx.x >> 5) * (kWarpFrontier + depth);
    q.fr = mine;
    q.frs = 32;
    q.fcap = kWarpFrontier;
    q.st = Stack{mine + kWarpFrontier, 1, depth, guard, 0u};
    q.lane = threadIdx.x & 31;
    q.new_walk();
    return q;
}

// Walks drawn from the solve's counter, or saved ones (src.slots).  Bound by
// the latency of dependent instructions (2,450 of them per step, 5.8 cycles
// each when a warp runs alone): a step takes 7.1 us alone on the Koch workload
// (one lane 20 us, a full warp of one-lane walks 35 us), and 4,864 walks of 200
// steps run at 1.6e8 steps/s (4.07 ms).  Whole solves, one-lane kernels -> this
// one: 976 Koch walks 1,501 -> 420 ms, 6,144 keyhole walks 173 -> 26 ms, 768
// walks by a crack 6.8 -> 1.1 ms.  Cap of 96 registers: 64 to 128 within 5%.
template <int D, bool SCR>
__global__ void __maxnreg__(WOST_WARP_REGS) k_walk_warp(const __grid_constant__ SceneView sc,
                                                        const __grid_constant__ SolveParams sp,
                                                        const Accumulators acc, const SavedWalks src) {
    WarpQ<D> q = make_warp_q<D>(sp.stack_depth, acc.guard);
    q.scale = sc.scale;
    q.tau = sc.tau;
    q.eps2 = sp.epsilon * sp.epsilon * 1.00001f;
    const uint64_t total = (uint64_t)sp.n_points * (uint64_t)sp.walks_per_point;
    const unsigned n_saved = src.slots ? *src.count : 0u;
    for (;;) {
        unsigned long long my = 0;
        if (q.lane == 0) {
            if (src.slots) my = atomicAdd(src.next, 1u);
            else my = (acc.cancel && *(volatile int *)acc.cancel) ? total : atomicAdd(acc.next_walk, 1ull);
        }
        my = __shfl_sync(0xffffffffu, my, 0);
        Walk w{};
        if (src.slots) {
            if (my >= n_saved) break;
            float4 *slot = src.slots + 3 * (size_t)(src.list ? src.list[my] : (uint32_t)my);
            const bool there = load_walk(slot, w, nullptr, false);
            __syncwarp();
            if (q.lane == 0) slot[2] = make_float4(0.f, 0.f, 0.f, 0.f);  // taken
            if (!there) continue;
        } else {
            if (my >= total) break;
            walk_init<D>(sp, w, (int64_t)(my / (uint64_t)sp.walks_per_point),
                         (uint32_t)(my % (uint64_t)sp.walks_per_point) + sp.first_walk);
        }
        q.new_walk();
        const int began = w.steps;
        while (!walk_step<D, SCR>(sc, sp, w, q, true)) {
        }
        if (q.lane == 0) {
            accumulate(acc, w);
            if (src.steps_run) atomicAdd(src.steps_run, (unsigned long long)(w.steps - began));
        }
        __syncwarp();
    }
}

// The same over a batch's walks: drawn from its counter, or saved ones.
template <int D, bool SCR>
__global__ void __maxnreg__(WOST_WARP_REGS) k_walk_warp_batch(const BatchHeader *__restrict__ hdr,
                                                              const BatchJob *__restrict__ jobs,
                                                              unsigned int *guard, int depth,
                                                              unsigned long long *steps_out, const SavedWalks src) {
    WarpQ<D> q = make_warp_q<D>(depth, guard);
    if (hdr->n_jobs <= 0) return;
    const unsigned n_saved = *src.count;
    unsigned long long ran = 0;
    for (;;) {
        unsigned my = 0;
        if (q.lane == 0) my = atomicAdd(src.next, 1u);
        my = __shfl_sync(0xffffffffu, my, 0);
        if (my >= n_saved) break;
        Walk w{};
        int job = 0;
        load_walk(src.slots + 3 * (size_t)my, w, &job, false);
        const BatchJob &J = jobs[job];
        q.scale = J.scene->scale;
        q.tau = J.scene->tau;
        q.eps2 = J.sp.epsilon * J.sp.epsilon * 1.00001f;
        q.new_walk();
        while (!walk_step<D, SCR>(*J.scene, J.sp, w, q, true)) {
        }
        if (q.lane == 0) {
            accumulate(J.acc, w);
            ran += (unsigned long long)w.steps;
        }
        __syncwarp();
    }
    if (steps_out && q.lane == 0 && ran) atomicAdd(steps_out, ran);
}

template <int D, bool SCR>
static cudaError_t warp_batch_grid(int depth, int block, size_t *sm, int *blocks) {
    *sm = (size_t)(block / 32) * (kWarpFrontier + depth) * sizeof(int2);
    return resident_blocks((const void *)k_walk_warp_batch<D, SCR>, block, *sm, blocks);
}

template <int D, bool SCR>
static cudaError_t warp_batch_launch(const BatchHeader *hdr, const BatchJob *jobs, unsigned int *guard, int depth,
                                     const SavedWalks &src, unsigned long long *steps_out, cudaStream_t s) {
    const int block = 64;
    size_t sm = 0;
    int blocks = 0;
    cudaError_t e = warp_batch_grid<D, SCR>(depth, block, &sm, &blocks);
    if (e != cudaSuccess) return e;
    k_walk_warp_batch<D, SCR><<<blocks, block, sm, s>>>(hdr, jobs, guard, depth, steps_out, src);
    return cudaGetLastError();
}

template <int D, bool SCR>
static cudaError_t walk_warp_launch_d(const SceneView &sc, const SolveParams &sp, const Accumulators &acc,
                                      const SavedWalks &src, uint64_t walks, cudaStream_t s) {
    const int block = 64;
    const size_t sm = (size_t)(block / 32) * (kWarpFrontier + sp.stack_depth) * sizeof(int2);
    const void *k = (const void *)k_walk_warp<D, SCR>;
    int blocks = 0;
    cudaError_t e = resident_blocks(k, block, sm, &blocks);
    if (e != cudaSuccess) return e;
    const uint64_t want = (walks + block / 32 - 1) / (block / 32);
    if (want < (uint64_t)blocks) blocks = (int)want;
    k_walk_warp<D, SCR><<<blocks, block, sm, s>>>(sc, sp, acc, src);
    return cudaGetLastError();
}

template <bool SCR>
static cudaError_t walk_warp_load(int dim) {
    cudaFuncAttributes a;
    return cudaFuncGetAttributes(&a, dim == 2 ? (const void *)k_walk_warp<2, SCR> : (const void *)k_walk_warp<3, SCR>);
}

template <bool SCR>
static cudaError_t walk_warp_launch(const SceneView &sc, const SolveParams &sp, const Accumulators &acc,
                                    const SavedWalks &src, uint64_t walks, cudaStream_t s) {
    return sc.dim == 2 ? walk_warp_launch_d<2, SCR>(sc, sp, acc, src, walks, s)
                       : walk_warp_launch_d<3, SCR>(sc, sp, acc, src, walks, s);
}

}  // namespace wost
