// One walk per warp, Poisson instantiations (wost_walk_warp.cuh); a solve
// with sigma > 0 is passed on to the screened ones, wost_kernels_warp_scr.cu.
#include <cuda_runtime.h>

#include "wost_walk_warp.cuh"

namespace wost {

cudaError_t launch_walk_warp(const SceneView &sc, const SolveParams &sp, const Accumulators &acc, const SavedWalks &src,
                             uint64_t walks, cudaStream_t s) {
    if (sp.sigma > 0.f) return launch_walk_warp_scr(sc, sp, acc, src, walks, s);
    return walk_warp_launch<false>(sc, sp, acc, src, walks, s);
}

cudaError_t load_walk_warp(int dim, bool screened) {
    return screened ? load_walk_warp_scr(dim) : walk_warp_load<false>(dim);
}

cudaError_t launch_walk_warp_batch(int dim, const BatchHeader *hdr, const BatchJob *jobs, unsigned int *guard, int depth,
                                   const SavedWalks &src, unsigned long long *steps_out, bool screened,
                                   cudaStream_t s) {
    if (screened) return launch_walk_warp_batch_scr(dim, hdr, jobs, guard, depth, src, steps_out, s);
    return dim == 2 ? warp_batch_launch<2, false>(hdr, jobs, guard, depth, src, steps_out, s)
                    : warp_batch_launch<3, false>(hdr, jobs, guard, depth, src, steps_out, s);
}

cudaError_t prepare_walk_warp_batch(int dim, int depth, bool screened) {
    if (screened) return prepare_walk_warp_batch_scr(dim, depth);
    size_t sm = 0;
    int blocks = 0;
    return dim == 2 ? warp_batch_grid<2, false>(depth, 64, &sm, &blocks) : warp_batch_grid<3, false>(depth, 64, &sm, &blocks);
}

}  // namespace wost
