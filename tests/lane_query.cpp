// Q.2 by one lane per query whatever the array's size, for tests that compare
// it with one warp per query (linked against libwost.so).
#include "capi_internal.h"

extern "C" int lane_query_silhouette(wost_scene *s, int64_t n, const float *pts, const float *rmax, float *dist,
                                     int per_warp) {  // (enqueued on the default stream)
    const auto launch = per_warp ? wost::launch_query_silhouette_warp : wost::launch_query_silhouette_lane;
    cudaError_t e = launch(s->view, n, pts, rmax, dist, s->stack_depth, s->guard_dev, nullptr);
    return (int)e;
}
