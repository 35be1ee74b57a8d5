// One walk per warp, Poisson instantiations (wost_walk_warp.cuh); a solve
// with sigma > 0 is passed on to the screened ones, wost_kernels_warp_scr.cu.
#include <cuda_runtime.h>

#include "wost_walk_warp.cuh"

namespace wost {

cudaError_t launch_walk_warp(const SceneView &sc, const SolveParams &sp, const Accumulators &acc, const TailWalks &tw,
                             uint64_t walks, cudaStream_t s) {
    if (sp.sigma > 0.f) return launch_walk_warp_scr(sc, sp, acc, tw, walks, s);
    return walk_warp_launch<false>(sc, sp, acc, tw, walks, s);
}

}  // namespace wost
