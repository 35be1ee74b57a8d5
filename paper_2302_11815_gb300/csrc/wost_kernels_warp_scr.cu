// One walk per warp, screened instantiations (wost_walk_warp.cuh).
#include <cuda_runtime.h>

#include "wost_screened.cuh"
#include "wost_walk_warp.cuh"

namespace wost {

cudaError_t launch_walk_warp_scr(const SceneView &sc, const SolveParams &sp, const Accumulators &acc,
                                 const TailWalks &tw, uint64_t walks, cudaStream_t s) {
    return walk_warp_launch<true>(sc, sp, acc, tw, walks, s);
}

}  // namespace wost
