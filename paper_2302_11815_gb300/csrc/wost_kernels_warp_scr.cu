// One walk per warp, screened instantiations (wost_walk_warp.cuh).
#include <cuda_runtime.h>

#include "wost_screened.cuh"
#include "wost_walk_warp.cuh"

namespace wost {

cudaError_t launch_walk_warp_scr(const SceneView &sc, const SolveParams &sp, const Accumulators &acc,
                                 const SavedWalks &src, uint64_t walks, cudaStream_t s) {
    return walk_warp_launch<true>(sc, sp, acc, src, walks, s);
}

cudaError_t load_walk_warp_scr(int dim) { return walk_warp_load<true>(dim); }

cudaError_t launch_walk_warp_batch_scr(int dim, const BatchHeader *hdr, const BatchJob *jobs, unsigned int *guard,
                                       int depth, const SavedWalks &src, unsigned long long *steps_out,
                                       cudaStream_t s) {
    return dim == 2 ? warp_batch_launch<2, true>(hdr, jobs, guard, depth, src, steps_out, s)
                    : warp_batch_launch<3, true>(hdr, jobs, guard, depth, src, steps_out, s);
}

cudaError_t prepare_walk_warp_batch_scr(int dim, int depth) {
    size_t sm = 0;
    int blocks = 0;
    return dim == 2 ? warp_batch_grid<2, true>(depth, 64, &sm, &blocks) : warp_batch_grid<3, true>(depth, 64, &sm, &blocks);
}

}  // namespace wost
