// Warp-cooperative walks: the 32 lanes of a warp carry ONE walk.
//
// A walk is a serial chain of steps, and a step's queries are serial chains
// of node visits.  One lane alone runs ~160 dependent instructions per visit
// (measured: 20 us per step on the Koch workload, 31 us in the keyhole), and
// a full warp of one-lane walks takes 35 us per step, because it runs the
// union of its lanes' paths.  That is the better trade while there are enough
// walks to fill the GPU, and the wrong one for a solve of few walks and for
// the last walks of a long one.  Here the lanes split each query instead: a
// frontier of nodes of the 8-wide trees, four nodes (32 children) per round.
//
// The answers are, bit for bit, those of the one-lane traversals over the
// binary trees, so that a walk does not depend on which kernel runs it.  The
// wide search tests every primitive the binary one can reach and also keeps
// what decides whether the binary one returns the same value: its answer is
// taken when no other candidate lies within rounding of the best one (or
// when it has the same bits) and the best one is not itself on the edge of a
// rounded test; otherwise (a few percent of the queries) lane 0 repeats the
// query over the binary tree.  The reasons are stated at each query.
#pragma once

#include "wost_device.cuh"
#include "wost_group.cuh"

namespace wost {

// Nearest-candidate search state of one lane: the smallest value seen, and
// the smallest one with different bits.
struct LaneBest {
    float d2, alt;
    int rec;
    bool dup;  // another candidate has the same bits as d2
    __device__ __forceinline__ void clear() {
        d2 = alt = INFINITY;
        rec = -1;
        dup = false;
    }
    // true if v is the new best (strictly smaller)
    __device__ __forceinline__ bool add(float v, int r) {
        if (v < d2) {
            alt = d2;
            d2 = v;
            rec = r;
            dup = false;
            return true;
        }
        if (v == d2) dup = true;
        else if (v < alt) alt = v;
        return false;
    }
};

__device__ __forceinline__ float warp_min(float v) {  // non-negative floats (and +inf) order like their bits
    return __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(v)));
}

// Uniforms of slots 1, 2, ... computed one slot per lane; every lane of the
// warp draws the same sequence.
struct WarpStream {
    uint4 mine;  // lane j holds slot j
    int i;
    __device__ __forceinline__ float next() {
        const int src = 1 + (i >> 2), c = i & 3;
        const uint32_t w = c == 0 ? mine.x : (c == 1 ? mine.y : (c == 2 ? mine.z : mine.w));
        ++i;
        return u01(__shfl_sync(0xffffffffu, w, src));
    }
};
// draws of one sample: at most one per level, one per leaf primitive, two for the point
static_assert(4 * 31 >= WOST_MAX_DEPTH + 2 + WOST_MAX_LEAF + 2, "slots 1..31 hold every draw of a Neumann sample");

// Is the accepted hit of ray o + t v on primitive p clear of every rounded
// decision: inside the primitive by more than the rounding of its
// coordinates there (then the ray also meets, in single precision, the boxes
// that hold the primitive), and inside (0, tmax) by more than rounding?
// The error terms: u is a quotient of cross products over the determinant,
// so its rounding grows with 1 / |determinant| (grazing rays); margin kEdgeTol
// of the hit test doubled.  te: the rounding of t.
template <int D>
__device__ __forceinline__ bool hit_clear(const Prim<D> &p, P3 o, P3 v, float t, float tmax, float scale, float &te) {
    const float vl = rsqrtf(dotp<D>(v, v));
    if constexpr (D == 2) {
        const P3 e = p.b - p.a, ao = p.a - o;
        const float inv = __fdividef(1.f, v.x * e.y - v.y * e.x);
        const float u = (ao.x * v.y - ao.y * v.x) * inv;
        const float ai = (fabsf(ao.x) + fabsf(ao.y)) * fabsf(inv) * 1e-6f;
        const float ue = ai * (fabsf(v.x) + fabsf(v.y)) + 2.f * kEdgeTol +
                         4e-6f * scale * rsqrtf(fmaxf(dotp<D>(e, e), 1e-30f));
        te = ai * (fabsf(e.x) + fabsf(e.y)) + 4e-6f * scale * vl;
        return u > ue && u < 1.f - ue && t > te && t < tmax - te;
    } else {
        const P3 e1 = p.b - p.a, e2 = p.c - p.a, pv = crossp(v, e2), tv = o - p.a;
        const float inv = __fdividef(1.f, dotp<D>(e1, pv));
        const float u = dotp<D>(tv, pv) * inv;
        const P3 qv = crossp(tv, e1);
        const float w = dotp<D>(v, qv) * inv;
        const float l1 = maxabs3(e1) + maxabs3(e2), lt = maxabs3(tv), lv = maxabs3(v);
        const float ai = lt * l1 * fabsf(inv) * 4e-6f;
        // shortest altitude ~ |normal| / longest edge
        const P3 nn = crossp(e1, e2);
        const float ue = ai * lv + 2.f * kEdgeTol + 4e-6f * scale * 2.f * l1 * rsqrtf(fmaxf(dotp<D>(nn, nn), 1e-30f));
        te = ai * l1 + 4e-6f * scale * vl;
        return u > ue && w > ue && u + w < 1.f - ue && t > te && t < tmax - te;
    }
}

// The binary-tree queries, out of line: lane 0's second opinion.  All lanes
// call them (the 2D ones are warp-wide) and get lane 0's answer.
template <int D>
__device__ __noinline__ Closest closest_binary(const TreeView &T, P3 x, Stack st, float bound2) {
    Cnt<false> cnt;
    const bool first = (threadIdx.x & 31) == 0;
    Closest c;
    c.d2 = bound2;
    c.rec = -1;
    c.s0 = c.s1 = 0.f;
    c.p = x;
    if constexpr (WOST_POSTPONE_LEAVES && D == 2) {
        c = q_closest_w<D, false>(T, x, st, cnt, bound2, first);
    } else {
        if (first) c = q_closest<D, false>(T, x, st, cnt, bound2);
    }
    __syncwarp();
    const unsigned F = 0xffffffffu;
    c.d2 = __shfl_sync(F, c.d2, 0);
    c.rec = __shfl_sync(F, c.rec, 0);
    c.s0 = __shfl_sync(F, c.s0, 0);
    c.s1 = __shfl_sync(F, c.s1, 0);
    c.p = mk(__shfl_sync(F, c.p.x, 0), __shfl_sync(F, c.p.y, 0), __shfl_sync(F, c.p.z, 0));
    return c;
}
template <int D>
__device__ __noinline__ float silhouette_binary(const TreeView &T, P3 x, float rmax, Stack st) {
    Cnt<false> cnt;
    const bool first = (threadIdx.x & 31) == 0;
    float r = rmax;
    if constexpr (WOST_POSTPONE_LEAVES && D == 2) {
        r = q_silhouette_w<D, false>(T, x, rmax, st, cnt, first);
    } else {
        if (first) r = q_silhouette<D, false>(T, x, rmax, st, cnt);
    }
    __syncwarp();
    return __shfl_sync(0xffffffffu, r, 0);
}
struct RayAnswer {
    int hit;
    float t;
    bool occ;
};
template <int D>
__device__ __noinline__ RayAnswer ray2_binary(const TreeView &T, P3 o, P3 va, float tmaxA, bool wantB, P3 vb, int skipB,
                                              float tmaxB, Stack st) {
    Cnt<false> cnt;
    const bool first = (threadIdx.x & 31) == 0;
    RayAnswer a{-1, tmaxA, false};
    if constexpr (WOST_POSTPONE_LEAVES && D == 2) {
        a.hit = q_ray2_w<D, false>(T, o, va, tmaxA, a.t, wantB, vb, skipB, tmaxB, a.occ, st, cnt, first);
    } else {
        if (first) a.hit = q_ray2<D, false>(T, o, va, tmaxA, a.t, wantB, vb, skipB, tmaxB, a.occ, st, cnt);
    }
    __syncwarp();
    a.hit = __shfl_sync(0xffffffffu, a.hit, 0);
    a.t = __shfl_sync(0xffffffffu, a.t, 0);
    a.occ = __shfl_sync(0xffffffffu, (int)a.occ, 0) != 0;
    return a;
}

// Query policy: the whole warp answers the queries of its one walk.
template <int D>
struct WarpQ {
    static constexpr bool kWarp = true;
    static constexpr unsigned FULL = 0xffffffffu;
    // A list of at most this many records is tested outright, 32 at a time: a
    // round of tests costs less than a round of nodes, and four rounds of
    // them less than the tree's two levels of nodes and one of leaves.
    static constexpr int kBrute = 128;
    int2 *fr;      // frontier (shared memory): (node reference, key)
    int fcap;
    Stack st;      // lane 0's stack for the binary trees
    float scale;   // largest coordinate of the scene
    float eps;
    int lane;
    // per step
    bool want_rec;  // the closest record itself will be used, not only the distance
    uint4 rb;       // slot `lane` of the step's random numbers
    // the previous step's answers: their distance from the new position
    // bounds the new answer (it is found again if it is still the best)
    int last_d, last_s;

    __device__ __forceinline__ void new_walk() { last_d = last_s = -1; }
    __device__ __forceinline__ void begin_step(const SolveParams &sp, const Walk &w, bool lost) {
        want_rec = lost || w.steps + 1 >= sp.max_steps;
        rb = philox10(make_uint4(w.index, w.point, (uint32_t)w.steps, (uint32_t)lane), sp.key0, sp.key1);
    }
    __device__ __forceinline__ uint4 slot0() const {
        return make_uint4(__shfl_sync(FULL, rb.x, 0), __shfl_sync(FULL, rb.y, 0), __shfl_sync(FULL, rb.z, 0),
                          __shfl_sync(FULL, rb.w, 0));
    }

    // Rounding of a distance.  A computed closest point lies within ~3 ulp of
    // the largest coordinate of its primitive's box, so a box's computed
    // distance exceeds that of a primitive in it by at most tau1, and the
    // one-lane traversal can miss a primitive only in favour of one less than
    // tau1 farther.  near2(d2): the square of (distance + 4 tau1).
    __device__ __forceinline__ float near2(float d2) const {
        const float tau = 6e-7f * scale;
        const float s = sqrtf(d2) * 1.000001f + tau;
        return s * s;
    }

    // One frontier search.  box(child, node ref, c, key) decides whether a
    // child is kept (key orders the visits), prim(k) tests record k, bound()
    // is the current pruning key (entries beyond it are dropped), after()
    // runs, for the whole warp, after a round that tested records.  Returns
    // false when the frontier overflows.
    template <class BOX, class PRIM, class BOUND, class AFTER>
    __device__ __forceinline__ bool search(const float4 *wnodes, uint32_t root, BOX box, PRIM prim, BOUND bound,
                                           AFTER after) {
        const int g = lane >> 3, c = lane & 7;
        int sp = 1;
        if (lane == 0) fr[0] = make_int2((int)root, 0);
        __syncwarp();
#pragma unroll 1
        while (sp > 0) {
            int n = min(sp, 4);
            if (sp - n + 8 * n > fcap) n = 1;
            if (sp - 1 + 8 > fcap) return false;
            bool on = g < n, leaf = false, hit = false;
            uint32_t ref = 0, cref = 0;
            float key = 0.f;
            if (on) {
                const int2 e = fr[sp - 1 - g];
                ref = (uint32_t)e.x;
                on = __int_as_float(e.y) <= bound();
            }
            sp -= n;
            if (on) {
                leaf = is_leaf(ref);
                if (leaf) {
                    const uint32_t f = leaf_first(ref), cnt = leaf_count(ref);
#pragma unroll 1
                    for (uint32_t j = c; j < cnt; j += 8) prim(f + j);
                } else {
                    const WChild ch = load_wchild(wnodes, ref, c);
                    cref = ch.ref;
                    hit = !ref_empty(ch.ref) && box(ch, ref, c, key);
                }
            }
            if (__any_sync(FULL, leaf)) after();  // (a barrier too: the popped entries are read)
            const unsigned hits = __ballot_sync(FULL, hit);
            if (hits) {
                // the nearest child on top, the others below it in any order
                const unsigned kb = hit ? __float_as_uint(key) : 0xffffffffu;
                const unsigned near = __reduce_min_sync(FULL, kb);
                const int top = __ffs(__ballot_sync(FULL, hit && kb == near)) - 1;
                const int cnt = __popc(hits);
                if (hit) {
                    int pos = __popc(hits & ((1u << lane) - 1u)) - (lane > top ? 1 : 0);
                    if (lane == top) pos = cnt - 1;
                    fr[sp + pos] = make_int2((int)cref, __float_as_int(key));
                }
                sp += cnt;
            }
            __syncwarp();
        }
        return true;
    }

    // Q.1.  Certain when every record within near2 of the best has the
    // best's bits (the one-lane search then returns those bits, whatever
    // order it meets the records in), and, if the record itself is used, when
    // there is only one.
    __device__ __forceinline__ Closest closest_w(const TreeView &T, P3 x, float bound2, bool act) {
        Closest best;
        best.d2 = bound2;
        best.rec = -1;
        best.s0 = best.s1 = 0.f;
        best.p = x;
        if (!act) return best;
        LaneBest lb;
        lb.clear();
        float s0 = 0.f, s1 = 0.f, B = bound2;
        P3 q = x;
        auto test = [&](uint32_t k) {
            const Prim<D> p = load_prim<D>(T.prims, k);
            float t0, t1;
            const P3 qq = prim_closest<D>(p, x, t0, t1);
            const P3 dq = qq - x;
            if (lb.add(dotp<D>(dq, dq), (int)k)) {
                s0 = t0;
                s1 = t1;
                q = qq;
            }
        };
        bool ok = T.root != WOST_EMPTY_REF;
        if (T.n_prims <= kBrute) {
#pragma unroll 1
            for (uint32_t k = lane; k < (uint32_t)T.n_prims; k += 32) test(k);
        } else {
            if (last_d >= 0) {
                const Prim<D> p = load_prim<D>(T.prims, (uint32_t)last_d);
                float t0, t1;
                const P3 dq = prim_closest<D>(p, x, t0, t1) - x;
                B = fminf(B, near2(near2(dotp<D>(dq, dq))));
            }
            ok = search(
                T.wnodes, T.wroot,
                [&](const WChild &ch, uint32_t, int, float &key) {
                    key = box_dist2<D>(ch.lo, ch.hi, x);
                    return key < B;
                },
                test, [&] { return B; }, [&] { B = fminf(B, near2(near2(warp_min(lb.d2)))); });
        }
        const float m = warp_min(lb.d2);
        const float lim = near2(m);
        const unsigned at = __ballot_sync(FULL, lb.d2 == m);
        bool amb = (lb.d2 != m && lb.d2 <= lim) || lb.alt <= lim;
        const bool rec_used = want_rec || !(sqrtf(m) >= eps);
        if (rec_used) amb = amb || (lb.d2 == m && lb.dup) || __popc(at) != 1;
        // (a bound that comes near the answer, no answer, NaN: not certain)
        if (!ok || __any_sync(FULL, amb) || !(near2(lim) < bound2)) {
            best = closest_binary<D>(T, x, st, D == 3 && m < INFINITY ? fminf(bound2, near2(lim)) : bound2);
        } else {
            const int src = __ffs(at) - 1;
            best.d2 = m;
            best.rec = __shfl_sync(FULL, lb.rec, src);
            best.s0 = __shfl_sync(FULL, s0, src);
            best.s1 = __shfl_sync(FULL, s1, src);
            best.p.x = __shfl_sync(FULL, q.x, src);
            best.p.y = __shfl_sync(FULL, q.y, src);
            if constexpr (D == 3) best.p.z = __shfl_sync(FULL, q.z, src);
        }
        last_d = best.rec;
        return best;
    }

    // Q.2.  Certain, beside the near ties of Q.1, when the best candidate is
    // not grazing: the normals on both sides of the view direction by more
    // than the cone test's padding can lose in single precision (a cone's
    // half angle of 3.4e-4 or less rounds to 0), so that no cone that holds
    // them is culled.  A boundary candidate (n1 = 0) is never culled.
    __device__ __forceinline__ float silhouette_w(const TreeView &T, P3 x, float rmax, bool act) {
        if (!act || T.root == WOST_EMPTY_REF) return rmax;
        const float r2 = rmax * rmax;
        LaneBest lb;
        lb.clear();
        float B = r2;
        auto test = [&](uint32_t k) { lb.add(sil_test<D>(T.prims, k, x, r2), (int)k); };
        bool ok = true;
        if (T.n_prims <= 3 * kBrute) {
#pragma unroll 2
            for (uint32_t k = lane; k < (uint32_t)T.n_prims; k += 32) test(k);
        } else {
            if (last_s >= 0) {
                const float d2 = sil_test<D>(T.prims, (uint32_t)last_s, x, r2);
                if (d2 < r2) B = fminf(B, near2(near2(d2)));
            }
            ok = search(
                T.wnodes, T.wroot,
                [&](const WChild &ch, uint32_t ref, int c, float &key) {
                    key = box_dist2<D>(ch.lo, ch.hi, x);
                    bool keep = key < B;
                    if (keep && key > 0.f)
                        keep = has_silhouette<D>(ch.lo, ch.hi, __ldg(T.wcones + (size_t)ref * WOST_WIDE + c), x);
                    return keep;
                },
                test, [&] { return B; }, [&] { B = fminf(B, near2(near2(warp_min(lb.d2)))); });
        }
        const float m = warp_min(lb.d2);
        if (ok && m == INFINITY) return rmax;
        const float lim = near2(m);
        const unsigned at = __ballot_sync(FULL, lb.d2 == m);
        bool amb = (lb.d2 != m && lb.d2 <= lim) || lb.alt <= lim;
        const int k = __shfl_sync(FULL, lb.rec, at ? __ffs(at) - 1 : 0);
        bool certain = ok && !__any_sync(FULL, amb) && near2(lim) < r2;
        if (certain) certain = sil_clear<D>(T.prims, (uint32_t)k, x);
        last_s = k;
        return certain ? sqrtf(m) : silhouette_binary<D>(T, x, rmax, st);
    }

    template <int DD>
    __device__ __forceinline__ static bool sil_clear(const float4 *prims, uint32_t k, P3 x) {
        P3 pe, n0, n1;
        if constexpr (DD == 2) {
            const float4 q0 = __ldg(prims + 2 * (size_t)k), q1 = __ldg(prims + 2 * (size_t)k + 1);
            pe = mk(q0.x, q0.y, 0.f);
            n0 = mk(q1.x, q1.y, 0.f);
            n1 = mk(q1.z, q1.w, 0.f);
        } else {
            const float4 q0 = __ldg(prims + 3 * (size_t)k), q1 = __ldg(prims + 3 * (size_t)k + 1),
                         q2 = __ldg(prims + 3 * (size_t)k + 2);
            const P3 a = mk(q0.x, q0.y, q0.z), b = mk(q1.x, q1.y, q1.z);
            n0 = mk(q0.w, q1.w, q2.x);
            n1 = mk(q2.y, q2.z, q2.w);
            pe = a + (b - a) * seg_param(a, b, x, 1);
        }
        const P3 v = pe - x;
        if (n1.x == 0.f && n1.y == 0.f && n1.z == 0.f) return true;
        const float lim = 4e-4f * sqrtf(dotp<DD>(v, v));
        return fabsf(dotp<DD>(v, n0)) > lim && fabsf(dotp<DD>(v, n1)) > lim;
    }

    // Q.4 over the binary tree, every lane alike; the uniforms come from the
    // lanes' slots.
    __device__ __forceinline__ NSample sample(const TreeView &T, P3 x, float r) {
        WarpStream rng{rb, 0};
        Cnt<false> cnt;
        return q_sample<D, false>(T, x, r, rng, cnt);
    }

    // Q.3 and the visibility ray.  Every primitive of every wide leaf that
    // either ray's [0, tmax] meets is tested against both (the binary search
    // tests a subset: its boxes are smaller, and ray A's end shrinks).
    // Certain: no hit at all; or the nearest hit clear of rounding (hit_clear)
    // and the next one farther by more than its rounding.  An occluder that is
    // clear of rounding occludes; none accepted, no occlusion.
    __device__ __forceinline__ int ray2_w(const TreeView &T, P3 o, P3 va, float tmaxA, float &t_out, bool wantB, P3 vb,
                                          int skipB, float tmaxB, bool &occB, bool act) {
        t_out = tmaxA;
        occB = false;
        if (!act || T.root == WOST_EMPTY_REF) return -1;
        const P3 ia = mk(1.f / va.x, 1.f / va.y, D == 3 ? 1.f / va.z : 0.f);
        P3 ib = mk(0.f, 0.f, 0.f);
        if (wantB) ib = mk(1.f / vb.x, 1.f / vb.y, D == 3 ? 1.f / vb.z : 0.f);
        // a zero component makes the slab test drop boxes that touch the ray
        // (0 x inf): such a ray is lane 0's
        const bool axis = va.x == 0.f || va.y == 0.f || (D == 3 && va.z == 0.f) ||
                          (wantB && (vb.x == 0.f || vb.y == 0.f || (D == 3 && vb.z == 0.f)));
        LaneBest lb;
        lb.clear();
        bool clearA = false, occ = false, occ_maybe = false;
        float teA = 0.f;
        auto test = [&](uint32_t k) {
            const Prim<D> p = load_prim<D>(T.prims, k);
            float t, te;
            if (prim_ray<D>(p, o, va, tmaxA, t, kEdgeTol) && lb.add(t, (int)k)) {
                clearA = hit_clear<D>(p, o, va, t, tmaxA, scale, te);
                teA = te;
            }
            if (wantB && (int)k != skipB && prim_ray<D>(p, o, vb, tmaxB, t, 0.f)) {
                if (hit_clear<D>(p, o, vb, t, tmaxB, scale, te)) occ = true;
                else occ_maybe = true;
            }
        };
        bool ok = !axis;
        if (!ok) {
        } else if (T.n_prims <= kBrute) {
#pragma unroll 1
            for (uint32_t k = lane; k < (uint32_t)T.n_prims; k += 32) test(k);
        } else {
            ok = search(
                T.wnodes, T.wroot,
                [&](const WChild &ch, uint32_t, int, float &key) {
                    key = 0.f;
                    return box_ray<D>(ch.lo, ch.hi, o, ia, tmaxA) != INFINITY ||
                           (wantB && box_ray<D>(ch.lo, ch.hi, o, ib, tmaxB) != INFINITY);
                },
                test, [&] { return 0.f; }, [&] {});
        }
        const float m = warp_min(lb.d2);
        bool certain = ok;
        int hit = -1;
        if (m < INFINITY) {
            const unsigned at = __ballot_sync(FULL, lb.d2 == m);
            const int src = __ffs(at) - 1;
            const float lim = m + __shfl_sync(FULL, teA, src);
            const bool bad = lane == src ? (!clearA || lb.dup || lb.alt <= lim) : lb.d2 <= lim;
            certain = certain && !__any_sync(FULL, bad);
            hit = __shfl_sync(FULL, lb.rec, src);
            t_out = m;
        }
        if (wantB) {
            occB = __any_sync(FULL, occ);
            certain = certain && (occB || !__any_sync(FULL, occ_maybe));
        }
        if (!certain) {
            const RayAnswer a = ray2_binary<D>(T, o, va, tmaxA, wantB, vb, skipB, tmaxB, st);
            t_out = a.t;
            occB = a.occ;
            hit = a.hit;
        }
        return hit;
    }
};

}  // namespace wost
