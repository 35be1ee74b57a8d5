// Q.1-Q.4 with one query per warp: for arrays of so few queries that one lane
// per query leaves most of the GPU idle and waits for the slowest lane's chain
// of node visits, and for silhouettes in 3D unless the candidates are few
// (warp_silhouettes), as their chains are the longest.  Bound by the latency of
// a warp's rounds (few queries) or by instruction issue (many: 250,000 raster
// points of a plane by the torus take 0.7 to 3 ns each, by plane; on the plane
// of the table in wost_kernels.cu 2.2, one lane each 5.8).  The answers are
// those of the one-lane query kernels (wost_kernels.cu), record for record;
// four queries over 1,000 Koch points 277 -> 128 us.
#include <cuda_runtime.h>

#include "wost_walk_warp.cuh"

namespace wost {

template <int D>
__device__ __forceinline__ WarpQ<D, false> query_warp(const SceneView &sc, int depth, unsigned int *guard) {
    WarpQ<D, false> q = make_warp_q<D, false>(depth, guard);
    q.scale = sc.scale;
    q.tau = sc.tau;
    q.eps2 = INFINITY;
    q.want_rec = true;
    return q;
}

template <int D>
__global__ void k_query_closest_warp(const __grid_constant__ SceneView sc, int64_t n, const float *pts, float *dist,
                                     float *closest, int32_t *prim, int depth, unsigned int *guard) {
    WarpQ<D, false> q = query_warp<D>(sc, depth, guard);
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= n) return;
    const Closest c = q.closest_w(sc.D, load_point<D>(pts, i), INFINITY, true);
    if (q.lane) return;
    dist[i] = sqrtf(c.d2);
    closest[D * i] = c.p.x;
    closest[D * i + 1] = c.p.y;
    if (D == 3) closest[D * i + 2] = c.p.z;
    prim[i] = c.rec >= 0 ? __ldg(sc.D.ids + c.rec) : -1;
}

template <int D>
__global__ void k_query_silhouette_warp(const __grid_constant__ SceneView sc, int64_t n, const float *pts,
                                        const float *rmax, float *dist, int depth, unsigned int *guard) {
    WarpQ<D, false> q = query_warp<D>(sc, depth, guard);
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= n) return;
    const float d = q.silhouette_w(sc.S, load_point<D>(pts, i), rmax[i], true, sc.tau);
    if (q.lane == 0) dist[i] = d;
}

template <int D>
__global__ void k_query_ray_warp(const __grid_constant__ SceneView sc, int64_t n, const float *o, const float *v,
                                 const float *tmax, const int32_t *skip, const int32_t *rec_of_id, int64_t n_ids,
                                 int32_t *hit, float *t, int32_t *prim, int depth, unsigned int *guard) {
    WarpQ<D, false> q = query_warp<D>(sc, depth, guard);
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= n) return;
    int sk = -1;
    if (skip && skip[i] >= 0 && skip[i] < n_ids) sk = rec_of_id[skip[i]];
    const P3 x = load_point<D>(o, i), d = load_point<D>(v, i);
    float tt = tmax[i];
    int r = -1;
    if (sc.N.root != WOST_EMPTY_REF) {
        bool occ, certain;
        r = q.ray2_search(sc.N, x, d, tmax[i], sk, tt, false, d, -1, 0.f, occ, certain);
        if (!certain) {
            Cnt<false> cnt;
            if (q.lane == 0) r = q_ray<D, false>(sc.N, x, d, tmax[i], sk, false, tt, q.st, cnt);
            __syncwarp();
        }
    }
    if (q.lane) return;
    hit[i] = r >= 0;
    t[i] = r >= 0 ? tt : tmax[i];
    prim[i] = r >= 0 ? __ldg(sc.N.ids + r) : -1;
}

template <int D>
__global__ void k_query_sample_warp(const __grid_constant__ SceneView sc, int64_t n, const float *pts, const float *r,
                                    uint32_t k0, uint32_t k1, uint32_t c1, uint32_t c2, float *z, float *pdf,
                                    int32_t *prim) {
    WarpQ<D, false> q = query_warp<D>(sc, 0, nullptr);
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= n) return;
    q.rb = philox10(make_uint4((uint32_t)i, c1, c2, (uint32_t)q.lane), k0, k1);
    const NSample s = q.sample(sc.N, load_point<D>(pts, i), r[i]);
    if (q.lane) return;
    z[D * i] = s.z.x;
    z[D * i + 1] = s.z.y;
    if (D == 3) z[D * i + 2] = s.z.z;
    pdf[i] = s.rec >= 0 ? s.pdf : 0.f;
    prim[i] = s.rec >= 0 ? __ldg(sc.N.ids + s.rec) : -1;
}

namespace {

constexpr int kBlock = 64;
unsigned warps_grid(int64_t n) { return (unsigned)((n + kBlock / 32 - 1) / (kBlock / 32)); }
size_t warps_smem(int depth) { return (size_t)(kBlock / 32) * (kWarpFrontier + depth) * sizeof(int2); }

}  // namespace

cudaError_t launch_query_closest_warp(const SceneView &sc, int64_t n, const float *pts, float *dist, float *closest,
                                      int32_t *prim, int depth, unsigned int *guard, cudaStream_t s) {
    if (sc.dim == 2)
        k_query_closest_warp<2><<<warps_grid(n), kBlock, warps_smem(depth), s>>>(sc, n, pts, dist, closest, prim, depth,
                                                                                 guard);
    else
        k_query_closest_warp<3><<<warps_grid(n), kBlock, warps_smem(depth), s>>>(sc, n, pts, dist, closest, prim, depth,
                                                                                 guard);
    return cudaGetLastError();
}

// (the only one that large arrays take, in 3D)
cudaError_t launch_query_silhouette_warp(const SceneView &sc, int64_t n, const float *pts, const float *rmax,
                                         float *dist, int depth, unsigned int *guard, cudaStream_t s) {
    return in_parts(n, kWarpQueries, [&](int64_t at, int64_t m) {
        const auto k = sc.dim == 2 ? k_query_silhouette_warp<2> : k_query_silhouette_warp<3>;
        k<<<warps_grid(m), kBlock, warps_smem(depth), s>>>(sc, m, pts + at * sc.dim, rmax + at, dist + at, depth, guard);
        return cudaGetLastError();
    });
}

cudaError_t launch_query_ray_warp(const SceneView &sc, int64_t n, const float *o, const float *v, const float *tmax,
                                  const int32_t *skip, const int32_t *rec_of_id, int64_t n_ids, int32_t *hit, float *t,
                                  int32_t *prim, int depth, unsigned int *guard, cudaStream_t s) {
    if (sc.dim == 2)
        k_query_ray_warp<2><<<warps_grid(n), kBlock, warps_smem(depth), s>>>(sc, n, o, v, tmax, skip, rec_of_id, n_ids,
                                                                             hit, t, prim, depth, guard);
    else
        k_query_ray_warp<3><<<warps_grid(n), kBlock, warps_smem(depth), s>>>(sc, n, o, v, tmax, skip, rec_of_id, n_ids,
                                                                             hit, t, prim, depth, guard);
    return cudaGetLastError();
}

cudaError_t launch_query_sample_warp(const SceneView &sc, int64_t n, const float *pts, const float *r, uint32_t k0,
                                     uint32_t k1, uint32_t c1, uint32_t c2, float *z, float *pdf, int32_t *prim,
                                     cudaStream_t s) {
    if (sc.dim == 2)
        k_query_sample_warp<2><<<warps_grid(n), kBlock, warps_smem(0), s>>>(sc, n, pts, r, k0, k1, c1, c2, z, pdf,
                                                                            prim);
    else
        k_query_sample_warp<3><<<warps_grid(n), kBlock, warps_smem(0), s>>>(sc, n, pts, r, k0, k1, c1, c2, z, pdf,
                                                                            prim);
    return cudaGetLastError();
}

}  // namespace wost
