// Host launchers of the walk and query kernels (wost_kernels.cu).
#pragma once

#include <cuda_runtime.h>

#include "wost_internal.h"

namespace wost {

// A solve of at most this many walks runs them one per warp from the start,
// and a larger one hands its last walks over when so many are left.  Measured
// with 4,096 / 8,192 / 16,384 / 32,768 / 65,536: 8,192 keyhole walks 74 / 40 /
// 40 / 39 / 40 ms, 64,000 box-sphere walks 19 / 16 / 13 / 12 / 13 ms, 48,000
// torus walks 80 / 59 / 50 / 44 / 49 ms, 131,072 flower walks (short ones)
// 2.6 / 2.4 / 2.3 / 2.6 / 3.1 ms.
constexpr unsigned kTailWalks = 16384;

// Walks per warp of a one-lane launch over `walks` saved walks on `sms` SMs.
// 2D: full warps (a warp's step takes as long with 8 walks as with 32).  3D:
// spread over 6 warps per SM partition, 24 per SM, as a warp's silhouette
// searches run one after the other (544,096 torus walks 206 -> 185 ms).
inline unsigned spread_walks(int dim, uint64_t walks, int sms) {
    if (dim == 2) return 32u;
    const uint64_t warps = 24u * (uint64_t)(sms > 0 ? sms : 1), w = (walks + warps - 1) / warps;
    return (unsigned)(w < 1 ? 1 : (w > 32 ? 32 : w));
}

cudaError_t launch_walk_plain(const SceneView &sc, const SolveParams &sp, const Accumulators &acc, int block,
                              cudaStream_t s);
cudaError_t launch_walk_count(const SceneView &sc, const SolveParams &sp, const Accumulators &acc,
                              unsigned long long *stats, int block, cudaStream_t s);
cudaError_t persistent_grid(int dim, int block, int depth, int *blocks_out, int lanes = 1);
cudaError_t batch_grid(int dim, int block, int depth, int *blocks_out);
cudaError_t launch_request_stats(const StatJob *jobs, int n_jobs, int64_t max_points, unsigned int *max_var_bits,
                                 unsigned long long *min_walks, unsigned long long *steps_sum,
                                 unsigned long long *walks_sum, cudaStream_t s);
cudaError_t launch_walk_batch(int dim, const BatchHeader *hdr, const BatchJob *jobs, unsigned long long *counter,
                              unsigned int *guard, int depth, const int *cancel, int block, int blocks,
                              const ChainBuffers &cb, cudaStream_t s, unsigned long long *steps_out = nullptr,
                              bool screened = true);
cudaError_t prepare_walk_warp_batch(int dim, int depth, bool screened);
// slots that slot array `which` (0, 1) of a batch's chain has to hold
uint64_t batch_chain_capacity(int block, int blocks, int which);
cudaError_t launch_walk_warp_batch(int dim, const BatchHeader *hdr, const BatchJob *jobs, unsigned int *guard, int depth,
                                   const SavedWalks &src, unsigned long long *steps_out, bool screened,
                                   cudaStream_t s);
// lanes: lanes per walk, 1 (binary trees) or 8 (8-lane teams over the 8-wide
// trees; Poisson solves)
cudaError_t launch_walk_persistent(const SceneView &sc, const SolveParams &sp, const Accumulators &acc, int block,
                                   int blocks, cudaStream_t s, int lanes = 1, const SavedWalks &src = SavedWalks{},
                                   const HandOver &ho = HandOver{});
// one walk per warp: `walks` walks (an upper bound), saved ones or the solve's own
cudaError_t launch_walk_warp(const SceneView &sc, const SolveParams &sp, const Accumulators &acc,
                             const SavedWalks &src, uint64_t walks, cudaStream_t s);
// all of a solve's walks (src.slots null), or `walks` saved ones at most, to
// their ends: launches that hand the remaining walks over to one another
// (block, blocks: the persistent kernel's resident grid)
cudaError_t launch_walk_chain(const SceneView &sc, const SolveParams &sp, const Accumulators &acc, SavedWalks src,
                              uint64_t walks, const ChainBuffers &cb, int block, int blocks, cudaStream_t s);
// Loads every kernel of a chain.  The runtime loads a kernel when it is first
// used, and waits for the device then: the first chain of a process would not
// return before its first launch has ended.
cudaError_t load_chain_kernels(int dim, bool screened);
// slots that the chain's slot array `which` (0, 1) has to hold
uint64_t chain_capacity(uint64_t walks, int block, int blocks, int which);
// resumable solves: grid of the fixed launch, its walk slots, one launch
cudaError_t resume_grid(int dim, int block, int depth, int *blocks_out, int lanes = 1);
int64_t resume_slots(int block, int blocks, int lanes = 1);
cudaError_t launch_walk_resume(const SceneView &sc, const SolveParams &sp, const Accumulators &acc,
                               const ResumeState &rs, int iters, int block, int blocks, cudaStream_t s,
                               int lanes = 1);
cudaError_t launch_screened_kernels(int dim, int64_t n, const float *rho, const float *R, float sigma, float *G,
                                    float *Q, cudaStream_t s);
cudaError_t launch_query_closest(const SceneView &sc, int64_t n, const float *pts, float *dist, float *closest,
                                 int32_t *prim, int depth, unsigned int *guard, cudaStream_t s);
cudaError_t launch_query_silhouette(const SceneView &sc, int64_t n, const float *pts, const float *rmax, float *dist,
                                    int depth, unsigned int *guard, cudaStream_t s);
cudaError_t launch_query_silhouette_lane(const SceneView &sc, int64_t n, const float *pts, const float *rmax,
                                         float *dist, int depth, unsigned int *guard, cudaStream_t s);
cudaError_t launch_query_ray(const SceneView &sc, int64_t n, const float *o, const float *v, const float *tmax,
                             const int32_t *skip, const int32_t *rec_of_id, int64_t n_ids, int32_t *hit, float *t,
                             int32_t *prim, int depth, unsigned int *guard, cudaStream_t s);
cudaError_t launch_query_sample(const SceneView &sc, int64_t n, const float *pts, const float *r, uint32_t k0,
                                uint32_t k1, uint32_t c1, uint32_t c2, float *z, float *pdf, int32_t *prim,
                                cudaStream_t s);
// one query per warp (wost_kernels_query.cu): the lines of the dispatch in
// wost_kernels.cu, which states their measurements
constexpr int64_t kWarpClosest = 2048, kWarpRay2D = 4096, kWarpRay3D = 16384, kWarpSample = 4096;
inline int64_t warp_silhouettes(int dim, int64_t candidates) {
    if (dim == 2) return 16384;
    return candidates <= 256 ? 131072 : candidates <= 384 ? 1 << 20 : INT64_MAX;
}
// A launch of one warp per query takes this many at most (two warps per block:
// its grid stays below 2^31 blocks); a larger array is asked in parts,
// f(first query, how many).
constexpr int64_t kWarpQueries = (int64_t)1 << 31;
template <class F>
inline cudaError_t in_parts(int64_t n, int64_t most, F f) {
    cudaError_t e = cudaSuccess;
    for (int64_t at = 0; at < n && e == cudaSuccess; at += most) e = f(at, n - at < most ? n - at : most);
    return e;
}
cudaError_t launch_query_closest_warp(const SceneView &sc, int64_t n, const float *pts, float *dist, float *closest,
                                      int32_t *prim, int depth, unsigned int *guard, cudaStream_t s);
cudaError_t launch_query_silhouette_warp(const SceneView &sc, int64_t n, const float *pts, const float *rmax,
                                         float *dist, int depth, unsigned int *guard, cudaStream_t s);
cudaError_t launch_query_ray_warp(const SceneView &sc, int64_t n, const float *o, const float *v, const float *tmax,
                                  const int32_t *skip, const int32_t *rec_of_id, int64_t n_ids, int32_t *hit, float *t,
                                  int32_t *prim, int depth, unsigned int *guard, cudaStream_t s);
cudaError_t launch_query_sample_warp(const SceneView &sc, int64_t n, const float *pts, const float *r, uint32_t k0,
                                     uint32_t k1, uint32_t c1, uint32_t c2, float *z, float *pdf, int32_t *prim,
                                     cudaStream_t s);

}  // namespace wost
