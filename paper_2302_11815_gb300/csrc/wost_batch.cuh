// The batched persistent walk kernel (wost_solve_batch and the serving
// engine's rounds), instantiated in wost_kernels_batch.cu in two forms:
// SCR = true when a job of the batch is screened, SCR = false (the smaller
// Poisson-only code) when none is.
#pragma once

#include "wost_walk.cuh"

namespace wost {

// the job that walk index `my` of a batched launch belongs to
__device__ __forceinline__ int job_of(const BatchJob *jobs, int n_jobs, unsigned long long my) {
    int lo = 0, hi = n_jobs - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (jobs[mid].walk_begin <= my) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}
template <int D>
__device__ __forceinline__ void init_job_walk(const BatchJob &J, unsigned long long my, Walk &w) {
    const SolveParams &sp = J.sp;
    unsigned long long local = my - J.walk_begin;
    int64_t pt = sp.point_begin + (int64_t)(local / (uint64_t)sp.walks_per_point);
    uint32_t j = (uint32_t)(local % (uint64_t)sp.walks_per_point) + sp.first_walk;
    walk_init<D>(sp, w, pt, j);
}

// Batched persistent kernel: many solves (scenes, point sets, walk counts,
// parameters) in one launch.  The walk index space is the concatenation of
// the jobs' walks; a team maps its next index to a job by binary search over
// the jobs' first indices and runs that job's walk on that job's scene.
// steps_out (may be null) receives the walk steps of the finished walks.
// src, ho: walks taken up from (SAVED), and handed over to, another launch (a
// saved walk keeps its job index).  As in k_walk_persistent, the loop is bound
// by its instruction supply, so SAVED is a parameter of the template and the
// stores of a hand-over are behind the loop.  Device time of one scene of 3,800
// points x 480 walks (Koch level 3: x 100; torus of 18,750 candidates: 17,003 x
// 32), ms, without hand-over / all of it in the loop / as it is: disk of 356
// segments 27.9 / 30.0 / 28.5, flower 9.75 / 10.4 / 10.1, annulus 37.2 / 32.0 /
// 30.8, crack 26.8 / 18.1 / 17.4, Koch 356 / 339 / 331, torus 146 / 82 / 80.
// The counter is read on every step: with every fourth to eighth the disk takes
// 28.0, but serving rounds hand over late (six requests 39.8 -> 41 to 42 ms).
template <int D, bool SCR, bool SAVED>
__global__ void WOST_WALK_BOUNDS k_walk_batch(const BatchHeader *__restrict__ hdr,
                                                    const BatchJob *__restrict__ jobs, unsigned long long *counter,
                                                    unsigned int *guard, int stack_depth, const int *cancel,
                                                    unsigned long long *steps_out, const SavedWalks src,
                                                    const HandOver ho) {
    const int n_jobs = hdr->n_jobs;
    const unsigned long long total = SAVED ? (unsigned long long)*src.count : hdr->total;
    if (n_jobs <= 0) return;
    Cnt<false> cnt;
    auto q = make_q<D, false>(stack_depth, guard, cnt, 0u, true);
    const Group g = make_team<1>();
    const int lane = threadIdx.x & 31;
    const unsigned FULL = 0xffffffffu;
    Walk w{};
    int job = -1;
    unsigned int ran = 0;  // steps of this lane's finished walks
    // the launch's counter has run past `total`, or the lane holds no walks
    bool drained = SAVED && src.per_warp && lane >= (int)src.per_warp;
    unsigned first = 0xffffffffu, held;
    // as in k_walk_persistent: the whole warp stays in the loop and
    // reconverges after every step
    for (;;) {
        unsigned need = __ballot_sync(FULL, g.leader() && job < 0 && !drained);
        if (need) {
            int lead = __ffs(need) - 1;
            unsigned long long base = 0;
            if (lane == lead) {
                if constexpr (SAVED) {
                    base = atomicAdd(src.next, (unsigned)__popc(need));
                } else {
                    bool stop = cancel && *(volatile const int *)cancel != 0;
                    base = stop ? total : atomicAdd(counter, (unsigned long long)__popc(need));
                }
            }
            base = __shfl_sync(FULL, base, lead);
            if ((need >> g.base) & 1u) {
                unsigned long long my = base + __popc(need & ((1u << g.base) - 1u));
                if (my >= total) {
                    drained = true;
                } else if constexpr (SAVED) {
                    load_walk(src.slots + 3 * (size_t)my, w, &job);
                } else {
                    const int lo = job_of(jobs, n_jobs, my);
                    // a cancelled solve's remaining walks are skipped: the
                    // team takes another index at the next iteration
                    if (!team_flag(g, jobs[lo].acc.cancel)) {
                        job = lo;
                        init_job_walk<D>(jobs[job], my, w);
                    }
                }
            }
        }
        held = __ballot_sync(FULL, job >= 0);
        if (!held) {
            if (__any_sync(FULL, !drained)) continue;
            break;
        }
        if (ho.slots) {
            if constexpr (SAVED) first = hand_over_at(ho, src.next, total, lane, held);
            else first = hand_over_at(ho, counter, total, lane, held);
            if (first != 0xffffffffu) break;
        }
        // lanes without a job step a dummy reference to job 0 (inactive)
        const BatchJob &J = jobs[job >= 0 ? job : 0];
        if (walk_step<D, SCR>(*J.scene, J.sp, w, q, job >= 0)) {
            if (g.leader()) {
                accumulate(J.acc, w);
                ran += (unsigned int)w.steps;
            }
            job = -1;
        }
        __syncwarp();
    }
    if (first != 0xffffffffu && job >= 0)
        save_walk(ho.slots + 3 * (size_t)(first + __popc(held & ((1u << lane) - 1u))), w, job);
    if (steps_out) {
        unsigned long long r = ran;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(FULL, r, o);
        if (lane == 0 && r) atomicAdd(steps_out, r);
    }
}

}  // namespace wost
