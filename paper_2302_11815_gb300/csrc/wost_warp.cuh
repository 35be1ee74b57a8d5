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
// wide search tests every primitive the binary one can reach, so its best
// value is at most the binary one's; it is the binary one's unless rounding
// keeps that search from the record that has it, which is checked (the
// reasons are stated at each query).  Where the check fails, lane 0 repeats
// the query over the binary tree (at most 1.7% of the searches on seven scenes).
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
// warp draws the same sequence.  `mine` of lane j: slot j; `u`: draw j of the
// first 32.
struct WarpStream {
    uint4 mine;
    float u;
    int i, lane;
    __device__ __forceinline__ float at(int n, int src) const {
        const uint32_t x = __shfl_sync(0xffffffffu, mine.x, src), y = __shfl_sync(0xffffffffu, mine.y, src),
                       z = __shfl_sync(0xffffffffu, mine.z, src), w = __shfl_sync(0xffffffffu, mine.w, src);
        return u01(n & 2 ? (n & 1 ? w : z) : (n & 1 ? y : x));
    }
    __device__ __forceinline__ WarpStream(uint4 m, int l) : mine(m), u(0.f), i(0), lane(l) { u = at(l, 1 + (l >> 2)); }
    __device__ __forceinline__ float next() {
        const int n = i++;
        return n < 32 ? __shfl_sync(0xffffffffu, u, n) : at(n, 1 + (n >> 2));
    }
};
// draws of one sample: at most one per level, one per leaf primitive, two for the point
static_assert(4 * 31 >= WOST_MAX_DEPTH + 2 + WOST_MAX_LEAF + 2, "slots 1..31 hold every draw of a Neumann sample");

__device__ __forceinline__ float sqrt_fast(float a) {
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}

// has_silhouette (the cone test of the one-lane search) with fast square
// roots and the slack that covers them: true wherever that one is.  (An ulp
// of sv moves cv, at least 0.014 here, by 1.3e-5.)
template <int D>
__device__ __forceinline__ bool may_have_silhouette(const float lo[3], const float hi[3], float4 cone, P3 x) {
    const float ct = cone.w;
    const P3 c = mk(0.5f * (lo[0] + hi[0]), 0.5f * (lo[1] + hi[1]), 0.5f * (lo[2] + hi[2]));
    const P3 av = c - x;
    const float l2 = dotp<D>(av, av);
    const P3 ext = mk(hi[0] - lo[0], hi[1] - lo[1], hi[2] - lo[2]);
    const float rb2 = 0.25f * dotp<D>(ext, ext);
    const float il = rsqrtf(l2);
    const float sv = sqrt_fast(rb2) * il, cv = sqrt_fast(fmaxf(0.f, 1.f - sv * sv));
    const float st = sqrt_fast(fmaxf(0.f, 1.f - ct * ct));
    const float cphi = (cone.x * av.x + cone.y * av.y + (D == 3 ? cone.z * av.z : 0.f)) * il;
    return ct <= 0.f || l2 <= rb2 * 1.0002f || ct * cv - st * sv <= 3e-5f ||
           fabsf(cphi) <= st * cv + ct * sv + 3e-5f;
}

// Is the accepted hit of ray o + t v on primitive p clear of every rounded
// decision: inside the primitive by more than the rounding of its
// coordinates there (then the ray also meets, in single precision, the boxes
// that hold the primitive), and inside (0, tmax) by more than rounding?
// The error terms: u is a quotient of cross products over the determinant,
// so its rounding grows with 1 / |determinant| (grazing rays); margin kEdgeTol
// of the hit test doubled.  te: the rounding of t.
// scale: the largest coordinate of the boundary and of o.
// Returns te, negative if the hit is not clear (out of line: two call sites).
template <int D>
__device__ __noinline__ float hit_clear(const float4 *prims, uint32_t k, P3 o, P3 v, float t, float tmax, float scale) {
    const Prim<D> p = load_prim<D>(prims, k);
    float te;
    const float vl = rsqrtf(dotp<D>(v, v));
    if constexpr (D == 2) {
        const P3 e = p.b - p.a, ao = p.a - o;
        const float inv = __fdividef(1.f, v.x * e.y - v.y * e.x);
        const float u = (ao.x * v.y - ao.y * v.x) * inv;
        const float ai = (fabsf(ao.x) + fabsf(ao.y)) * fabsf(inv) * 1e-6f;
        const float ue = ai * (fabsf(v.x) + fabsf(v.y)) + 2.f * kEdgeTol +
                         4e-6f * scale * rsqrtf(fmaxf(dotp<D>(e, e), 1e-30f));
        te = ai * (fabsf(e.x) + fabsf(e.y)) + 4e-6f * scale * vl;
        return u > ue && u < 1.f - ue && t > te && t < tmax - te ? te : -1.f;
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
        return u > ue && w > ue && u + w < 1.f - ue && t > te && t < tmax - te ? te : -1.f;
    }
}

// The binary-tree queries, out of line: lane 0's second opinion.  All lanes
// call them (the 2D ones are warp-wide) and get lane 0's answer.
// WALK: as the walk kernels search (2D: postponed leaves), or as the query
// kernels do; their order differs, and with it the answer among ties.
template <int D, bool WALK>
__device__ __noinline__ Closest closest_binary(const TreeView &T, P3 x, Stack st, float bound2) {
    Cnt<false> cnt;
    const bool first = (threadIdx.x & 31) == 0;
    Closest c;
    c.d2 = bound2;
    c.rec = -1;
    c.s0 = c.s1 = 0.f;
    c.p = x;
    if constexpr (WOST_POSTPONE_LEAVES && D == 2 && WALK) {
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

// lim, lim2: the squares of distance + tau and + 2 tau (tau: see beyond)
struct Near {
    float lim, lim2;
    __device__ __forceinline__ Near(float d2, float tau) {
        const float s = sqrt_fast(d2) * 1.000002f + tau;
        lim = s * s;
        lim2 = (s + tau) * (s + tau);
    }
};

// the box of the child at `at` (parent node * 2 + side)
template <int D>
__device__ __forceinline__ float box_dist2_at(const TreeView &T, uint32_t at, P3 x) {
    if (at == WOST_EMPTY_REF) return box_dist2<D>(T.root_lo, T.root_hi, x);
    const Node<D> n = load_node<D>(T.nodes, at >> 1);
    return at & 1u ? box_dist2<D>(n.lo1, n.hi1, x) : box_dist2<D>(n.lo0, n.hi0, x);
}

template <int D>
__device__ __noinline__ float coop_distance(const TreeView &T, P3 x, float tau, int2 *fr, int frs, int fcap);

// Query policy: the whole warp answers the queries of its one walk (WALK), or
// one query of an array of queries.
template <int D, bool WALK = true>
struct WarpQ {
    static constexpr bool kWarp = true;
    static constexpr unsigned FULL = 0xffffffffu;
    // A list of at most this many records is tested outright, 32 at a time: a
    // round of tests costs less than a round of nodes, and four rounds of
    // them less than the tree's two levels of nodes and one of leaves.
    static constexpr int kBrute = 128;
    // frontier (shared memory): entry j, (node reference, key), at
    // fr[(j / 32) * frs + j % 32]
    int2 *fr;
    int frs, fcap;
    Stack st;      // lane 0's stack for the binary trees
    float scale, tau;  // of the scene
    float eps2;    // square of epsilon, rounded up
    int lane;
    // per step
    bool want_rec;  // the closest record itself will be used, not only the distance
    uint4 rb;       // slot `lane` of the step's random numbers
    // the previous step's answers: their distance from the new position
    // bounds the new answer (it is found again if it is still the best)
    int last_d, last_s;
    int hit_s;  // a candidate on the Neumann primitive hit last
    // The walk's distance to the Dirichlet boundary is at least dlow (less
    // than 0: not known) and at most its dbound; they are of the previous
    // step's position px plus or minus the length of its move, `moved`, except
    // after steps that skipped Q.1 (skipped), when they have grown apart.
    // hug: the previous step's silhouette was near against dlow.
    float dlow, moved;
    P3 px;
    bool skipped, hug;

    __device__ __forceinline__ void new_walk() {
        last_d = last_s = hit_s = -1;
        dlow = -1.f;
        skipped = hug = false;
    }
    // After a step from x: Q.1's answer dD there (or, skipped, an upper bound),
    // the length of the move, the silhouette distance.
    __device__ __forceinline__ void moved_on(P3 x, float dD, float len, float dsil, bool skip) {
        dlow = (skip ? dlow : dD) * 0.999999f - len - tau;
        px = x;
        moved = len;
        skipped = skip;
        hug = dsil < 0.5f * dlow;
    }
    // Q.2 ahead of Q.1: true if a silhouette lies nearer than the Dirichlet
    // boundary can (then d is Q.2's answer whatever Q.1's is, and the step is
    // no epsilon-shell hit), and Q.1's record is not needed.
    __device__ __forceinline__ bool near_silhouette(const TreeView &S, P3 xq, float epsilon, float &d) {
        if (!hug || want_rec || !(dlow > 1.001f * epsilon + tau) || S.root == WOST_EMPTY_REF) return false;
        const float lim = dlow * 0.9999f - tau;
        if (!(lim > 0.f)) return false;
        const SilAnswer a = coop_silhouette<D>(S, xq, lim, hint_bound(S, xq, lim * lim), tau, fr, frs, fcap);
        if (a.rec >= 0) last_s = a.rec;
        d = a.d;
        return a.certain && a.rec >= 0;
    }

    __device__ __forceinline__ void hit(const TreeView &N, int rec) { hit_s = (int)__ldg(N.hints + rec); }
    __device__ __forceinline__ void begin_step(const SolveParams &sp, const Walk &w, bool lost) {
        want_rec = lost || w.steps + 1 >= sp.max_steps;
        rb = philox10(make_uint4(w.index, w.point, (uint32_t)w.steps, (uint32_t)lane), sp.key0, sp.key1);
    }
    __device__ __forceinline__ uint4 slot0() const {
        return make_uint4(__shfl_sync(FULL, rb.x, 0), __shfl_sync(FULL, rb.y, 0), __shfl_sync(FULL, rb.z, 0),
                          __shfl_sync(FULL, rb.w, 0));
    }

    __device__ __forceinline__ int2 &entry(int j) const { return fr[(j >> 5) * frs + (j & 31)]; }

    // One frontier search over tree T.  box(child, cone, key) decides whether
    // a child is kept (cone: its record; key orders the visits), prim(k)
    // tests record k, bound() is the current pruning key (entries beyond it
    // are dropped), after() runs, for the whole warp, after a round that
    // tested records.  A list of at most `brute` records is tested outright.
    // Else the first round tests the tree's top, one subtree per lane; a
    // later one takes the up to four nearest entries still within the bound
    // (of the top 32, looked at together, so that a bound that tightens late
    // costs no rounds of its own).  Returns false when the frontier overflows.
    // (One call site each for box and prim: the code is walked through once
    // per query, so its size is latency.)
    template <class BOX, class PRIM, class BOUND, class AFTER>
    __device__ __forceinline__ bool search(const TreeView &T, int brute, BOX box, PRIM prim, BOUND bound, AFTER after) {
        const int g = lane >> 3, c = lane & 7;
        int sp = 0;
        // this round's work of the lane: a child record, or records j0, j0 + js, ... < j1
        const float4 *child = T.wtop + 2 * lane, *cone = T.wtopcones + lane;
        uint32_t j0 = 0, j1 = 0, js = 8;
        if (T.n_prims <= brute) {
            child = nullptr;
            j0 = (uint32_t)lane;
            j1 = (uint32_t)T.n_prims;
            js = 32;
        }
#pragma unroll 1
        for (;;) {
            uint32_t cref = 0;
            float key = 0.f;
            bool hit = false;
            if (child) {
                const WChild ch = load_wchild(child, 0, 0);
                cref = ch.ref;
                hit = !ref_empty(cref) && box(ch, cone, key);
            }
            const bool tests = __any_sync(FULL, j0 < j1);
            if (tests) {
#pragma unroll 1
                for (uint32_t j = j0; j < j1; j += js) prim(j);
                __syncwarp();
                after();
            }
            const unsigned hits = __ballot_sync(FULL, hit);
            unsigned m = hits, m1, m2, m3;
            uint32_t from = cref;  // this lane's entry of the candidates in m
            if (sp == 0 && __popc(hits) <= 4) {
                // few enough: visited at once, without the frontier
                if (!hits) return true;
                m1 = m & (m - 1u);
                m2 = m1 & (m1 - 1u);
                m3 = m2 & (m2 - 1u);
            } else {
                if (hit) entry(sp + __popc(hits & ((1u << lane) - 1u))) = make_int2((int)cref, __float_as_int(key));
                sp += __popc(hits);
                __syncwarp();
                // entries to visit: the four nearest within the bound
                float ekey = 0.f;
                m = 0;
                while (sp > 0) {
                    const int n = min(sp, 32);
                    bool alive = false;
                    if (lane < n) {
                        const int2 e = entry(sp - 1 - lane);
                        from = (uint32_t)e.x;
                        ekey = __int_as_float(e.y);
                        alive = ekey <= bound();
                    }
                    m = __ballot_sync(FULL, alive);
                    if (m) break;
                    sp -= n;
                }
                if (!m) return true;
                const int n = min(sp, 32);
                unsigned rest = 0u;
                if (__popc(m) > 4) {
                    // the four nearest of them; the others stay
                    unsigned kb = (m >> lane) & 1u ? __float_as_uint(ekey) : 0xffffffffu, sel = 0u;
#pragma unroll 1
                    for (int i = 0; i < 4; ++i) {
                        const unsigned at = __ballot_sync(FULL, kb == __reduce_min_sync(FULL, kb));
                        const unsigned one = at & (0u - at);
                        sel |= one;
                        if ((one >> lane) & 1u) kb = 0xffffffffu;
                    }
                    rest = m & ~sel;
                    m = sel;
                }
                m1 = m & (m - 1u);
                m2 = m1 & (m1 - 1u);
                m3 = m2 & (m2 - 1u);
                const int kept = __popc(rest);
                if (sp - n + kept + 32 > fcap) {  // one at a time while space is short
                    rest |= m1;
                    m &= ~m1;
                    m1 = m2 = m3 = 0u;
                    if (sp - n + __popc(rest) + 8 > fcap) return false;
                }
                __syncwarp();
                if ((rest >> lane) & 1u)
                    entry(sp - n + __popc(rest >> lane >> 1)) = make_int2((int)from, __float_as_int(ekey));
                sp += __popc(rest) - n;
            }
            const unsigned mine = g == 0 ? m : (g == 1 ? m1 : (g == 2 ? m2 : m3));
            const uint32_t ref = __shfl_sync(FULL, from, mine ? __ffs(mine) - 1 : 0);
            child = nullptr;
            j0 = j1 = 0;
            js = 8;
            if (mine && is_leaf(ref)) {
                j0 = leaf_first(ref) + c;
                j1 = leaf_first(ref) + leaf_count(ref);
            } else if (mine) {
                child = T.wnodes + (size_t)ref * (2 * WOST_WIDE) + 2 * c;
                cone = T.wcones + (size_t)ref * WOST_WIDE + c;
            }
        }
    }

    // Q.1.  The one-lane search prunes a box whose computed distance is not
    // below the best value so far.  It reaches the record with the smallest
    // value m, in whatever order it goes, if the box of that record's leaf is
    // computed no farther than m (those above it are no farther either:
    // rounding is monotonic): m is then its answer.  Where rounding puts the
    // box beyond m (a vertex computed just outside it), m is still the answer
    // if no record with other bits lies within rounding.  Which of several
    // records with the bits of m it returns depends on its order.
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
        // the records around the last answer (neighbours in leaf order are
        // neighbours in space) bound the new one
        if (last_d >= 0 && T.n_prims > kBrute) {
            const int k = min(max(last_d - 16 + lane, 0), T.n_prims - 1);
            B = fminf(B, beyond(warp_min(prim_dist2<D>(T.prims, (uint32_t)k, x)), tau));
        }
        if (ok)
            ok = search(
                T, kBrute,
                [&](const WChild &ch, const float4 *, float &key) {
                    key = box_dist2<D>(ch.lo, ch.hi, x);
                    return key < B;
                },
                test, [&] { return B; }, [&] { B = fminf(B, beyond(warp_min(lb.d2), tau)); });
        const float m = warp_min(lb.d2);
        const Near nr(m, tau);
        const unsigned at = __ballot_sync(FULL, lb.d2 == m);
        const bool tie = __any_sync(FULL, (lb.d2 != m && lb.d2 <= nr.lim) || lb.alt <= nr.lim);
        const int src = at ? __ffs(at) - 1 : 0, k = __shfl_sync(FULL, lb.rec, src);
        bool certain = ok && m < bound2;  // (no answer, NaN: not certain)
        if (want_rec || !(m >= eps2))  // the record is used
            certain = certain && __popc(at) == 1 && !__any_sync(FULL, lb.d2 == m && lb.dup);
        if (certain && (tie || !(nr.lim2 < bound2))) certain = box_dist2_at<D>(T, __ldg(T.leaf_parents + k), x) <= m;
        if (!certain) {
            if (WALK && skipped && bound2 < INFINITY) {
                // the bound the one-lane walk has here: Q.1's answer at the
                // previous position, which was skipped
                const float b = (coop_distance<D>(T, px, tau, fr, frs, fcap) + moved) * 1.0001f + 1e-6f;
                bound2 = b * b;
            }
            best = closest_binary<D, WALK>(T, x, st, D == 3 && m < INFINITY ? fminf(bound2, nr.lim2) : bound2);
        } else {
            best.d2 = m;
            best.rec = k;
            best.s0 = __shfl_sync(FULL, s0, src);
            best.s1 = __shfl_sync(FULL, s1, src);
            best.p.x = __shfl_sync(FULL, q.x, src);
            best.p.y = __shfl_sync(FULL, q.y, src);
            if constexpr (D == 3) best.p.z = __shfl_sync(FULL, q.z, src);
        }
        last_d = best.rec;
        return best;
    }

    // Q.2.  As Q.1 (only the distance is used), and the best candidate must
    // not be culled: one that is not grazing (sil_certain) never is.  Of a
    // grazing one (common on flat walls, where rounding decides the signs)
    // the cone tests above it decide: a candidate whose leaf is culled is
    // none, and the best one's whole path is tested.
    // B: a bound on the squared distance (beyond that of a certain candidate,
    // or rmax^2).
    __device__ __forceinline__ SilAnswer silhouette_search(const TreeView &T, P3 x, float rmax, float B) {
        const float r2 = rmax * rmax;
        LaneBest lb;
        lb.clear();
        bool clear = false;
        auto test = [&](uint32_t k) {
            const float d2 = sil_test<D>(T.prims, k, x, r2);
            if (d2 < INFINITY && d2 <= B) {
                const bool cl = sil_certain<D>(T.prims, k, x) < INFINITY;
                if (!cl && !reached(T, T.leaf_parents[k], x)) return;
                if (lb.add(d2, (int)k)) clear = cl;
            }
        };
        const bool ok = search(
            T, 3 * kBrute,
            [&](const WChild &ch, const float4 *cone, float &key) {
                const float4 cn = __ldg(cone);
                key = box_dist2<D>(ch.lo, ch.hi, x);
                bool keep = key < B;
                if (keep && key > 0.f) keep = may_have_silhouette<D>(ch.lo, ch.hi, cn, x);
                return keep;
            },
            test, [&] { return B; }, [&] { B = fminf(B, beyond(warp_min(lb.d2), tau)); });
        const float m = warp_min(lb.d2);
        const Near nr(m, tau);
        bool certain = ok;
        if (m == INFINITY) return SilAnswer{rmax, -1, ok};
        const unsigned at = __ballot_sync(FULL, lb.d2 == m);
        const bool tie = __any_sync(FULL, (lb.d2 != m && lb.d2 <= nr.lim) || lb.alt <= nr.lim);
        const int src = __ffs(at) - 1;
        const int k = __shfl_sync(FULL, lb.rec, src);
        if (certain && (tie || !(nr.lim2 < r2))) certain = box_dist2_at<D>(T, __ldg(T.leaf_parents + k), x) <= m;
        if (certain && !__shfl_sync(FULL, (int)clear, src)) certain = path_reached(T, (uint32_t)k, x);
        return SilAnswer{sqrtf(m), k, certain};
    }

    // the candidates around the last answer and around the last hit bound the
    // new one
    __device__ __forceinline__ float hint_bound(const TreeView &T, P3 x, float B) const {
        if ((last_s < 0 && hit_s < 0) || T.n_prims <= 3 * kBrute) return B;
        const int mid = (lane < 16 && last_s >= 0) || hit_s < 0 ? last_s : hit_s;
        const int k = min(max(mid - 8 + (lane & 15), 0), T.n_prims - 1);
        return fminf(B, beyond(warp_min(sil_certain<D>(T.prims, (uint32_t)k, x)), tau));
    }

    __device__ __forceinline__ float silhouette_w(const TreeView &T, P3 x, float rmax, bool act, float) {
        if (!act || T.root == WOST_EMPTY_REF) return rmax;
        const SilAnswer a = coop_silhouette<D>(T, x, rmax, hint_bound(T, x, rmax * rmax), tau, fr, frs, fcap);
        if (a.rec >= 0) last_s = a.rec;
        if (a.certain) return a.d;
        // the one-lane search among the candidates near the best one, if
        // it finds one there (culled candidates can leave none)
        const Near nr(a.d * a.d, tau);
        const float rn = sqrtf(nr.lim2) * 1.000001f;
        if (rn < rmax) {
            const float t = silhouette_binary<D>(T, x, rn, st);
            if (t * t <= nr.lim) return t;
        }
        return silhouette_binary<D>(T, x, rmax, st);
    }

    // does the binary search enter the child at `at` (parent * 2 + side)?
    __device__ __noinline__ static bool reached(const TreeView &T, uint32_t at, P3 x) {
        if (at == WOST_EMPTY_REF)
            return !(box_dist2<D>(T.root_lo, T.root_hi, x) > 0.f) ||
                   has_silhouette<D>(T.root_lo, T.root_hi, T.root_cone, x);
        const Node<D> n = load_node<D>(T.nodes, at >> 1);
        float lo[3], hi[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            lo[a] = at & 1u ? n.lo1[a] : n.lo0[a];
            hi[a] = at & 1u ? n.hi1[a] : n.hi0[a];
        }
        return !(box_dist2<D>(lo, hi, x) > 0.f) ||
               has_silhouette<D>(lo, hi, load_cone<D>(T.cones, at >> 1, (int)(at & 1u)), x);
    }
    // ... and every one above record k?  (lane i tests the i-th from below)
    __device__ __forceinline__ bool path_reached(const TreeView &T, uint32_t k, P3 x) const {
        uint32_t at = __ldg(T.leaf_parents + k), mine = WOST_EMPTY_REF;
        for (int i = 0; at != WOST_EMPTY_REF; ++i) {
            if (i == 31) return false;  // deeper than the warp is wide: undecided
            if (lane == i) mine = at;
            at = __ldg(T.parents + (at >> 1));
        }
        return __all_sync(FULL, reached(T, mine, x));  // (a lane without an entry tests the root)
    }

    // Q.4 over the binary tree; the uniforms come from the lanes' slots.  The
    // descent is a chain of one decision per level, each on the two children's
    // weights: the lanes compute the decisions of a five-level treelet at
    // once, so a level costs a shuffle and a comparison instead of a node
    // fetch and two weights (480 cycles).
    __device__ __forceinline__ NSample sample(const TreeView &T, P3 x, float r) {
        Cnt<false> cnt;
        NSample out;
        out.rec = -1;
        out.pdf = 0.f;
        out.z = x;
        out.s0 = out.s1 = 0.f;
        const float r2 = r * r;
        if (T.root == WOST_EMPTY_REF || box_dist2<D>(T.root_lo, T.root_hi, x) > r2) return out;
        WarpStream rng(rb, lane);
        uint32_t ref = T.root, t = 0;
        float pdf = 1.f;
        const int depth = 31 - __clz(lane + 1);  // of heap position `lane` in a treelet
#pragma unroll 1
        for (int level = 0; !is_leaf(ref); level += 5) {
            if (level > WOST_MAX_DEPTH) return out;
            const uint32_t *tl = T.treelets + 64 * (size_t)t;
            const uint32_t node = lane < 31 ? __ldg(tl + lane) : WOST_EMPTY_REF, exit = __ldg(tl + 32 + lane);
            uint32_t next = WOST_EMPTY_REF;
            bool live = false, first = false;
            float f = 0.f;
            // the draw that a walk arriving at this position takes
            const int n = rng.i + depth;
            const float u = __shfl_sync(FULL, rng.u, n & 31);
            const float ub = rng.i + 4 >= 32 ? rng.at(n, min(1 + (n >> 2), 31)) : u;
            if (node != WOST_EMPTY_REF) {
                const Node<D> nd = load_node<D>(T.nodes, node);
                const float w0 = child_weight<D>(nd.lo0, nd.hi0, x, r2), w1 = child_weight<D>(nd.lo1, nd.hi1, x, r2);
                const float tot = w0 + w1, p0 = __fdividef(w0, tot);
                live = tot > 0.f;
                first = (n < 32 ? u : ub) < p0;  // the decision and the pdf use this same p0
                f = first ? p0 : 1.f - p0;
                next = first ? nd.r0 : nd.r1;
            }
            const unsigned lives = __ballot_sync(FULL, live), firsts = __ballot_sync(FULL, first),
                           ends = __ballot_sync(FULL, is_leaf(next));
            int pos = 0, last;
            do {
                if (!((lives >> pos) & 1u)) return out;
                pdf *= __shfl_sync(FULL, f, pos);
                last = pos;
                pos = 2 * pos + 2 - (int)((firsts >> pos) & 1u);
                ++rng.i;
            } while (pos < 31 && !((ends >> last) & 1u));
            ref = __shfl_sync(FULL, next, last);
            if (!is_leaf(ref)) t = __shfl_sync(FULL, exit, pos - 31);
        }
        sample_leaf<D, false>(T, x, r2, ref, pdf, rng, cnt, out);
        return out;
    }

    // Q.3 and the visibility ray.  Every primitive of every wide leaf that
    // either ray's [0, tmax] meets is tested against both (the binary search
    // tests a subset: its boxes are smaller, and ray A's end shrinks).
    // Certain: no hit at all; or the nearest hit clear of rounding (hit_clear)
    // and the next one farther by more than its rounding.  An occluder that is
    // clear of rounding occludes; none accepted, no occlusion.
    // skipA: a record ray A does not meet (-1: none).
    __device__ __forceinline__ int ray2_search(const TreeView &T, P3 o, P3 va, float tmaxA, int skipA, float &t_out,
                                               bool wantB, P3 vb, int skipB, float tmaxB, bool &occB, bool &certain) {
        t_out = tmaxA;
        occB = false;
        // fast reciprocals: the boxes are widened by more than they, and the
        // rounding of the one-lane slab test, can move its planes: that grows
        // with |plane - o|.  A walk's origin is within 3 scale of zero (it ends
        // outside the grown bounding box), a query's is anywhere.
        const float reach = WALK ? scale : fmaxf(scale, maxabs3(o));
        const P3 ia = mk(__fdividef(1.f, va.x), __fdividef(1.f, va.y), D == 3 ? __fdividef(1.f, va.z) : 0.f);
        P3 ib = mk(0.f, 0.f, 0.f);
        if (wantB) ib = mk(__fdividef(1.f, vb.x), __fdividef(1.f, vb.y), D == 3 ? __fdividef(1.f, vb.z) : 0.f);
        const float pad = 8e-6f * reach;
        // a zero component makes the slab test drop boxes that touch the ray
        // (0 x inf): such a ray is lane 0's
        auto flat = [](P3 v) {
            return fminf(fminf(fabsf(v.x), fabsf(v.y)), D == 3 ? fabsf(v.z) : INFINITY) < 1e-30f;
        };
        const bool axis = flat(va) || (wantB && flat(vb));
        LaneBest lb;
        lb.clear();
        bool occ = false, occ_maybe = false;
        float teA = -1.f;
        auto test = [&](uint32_t k) {
            const Prim<D> p = load_prim<D>(T.prims, k);
            float t;
            if ((int)k != skipA && prim_ray<D>(p, o, va, tmaxA, t, kEdgeTol) && lb.add(t, (int)k))
                teA = hit_clear<D>(T.prims, k, o, va, t, tmaxA, reach);
            if (wantB && (int)k != skipB && prim_ray<D>(p, o, vb, tmaxB, t, 0.f)) {
                if (hit_clear<D>(T.prims, k, o, vb, t, tmaxB, reach) >= 0.f) occ = true;
                else occ_maybe = true;
            }
        };
        bool ok = !axis && (WALK || reach < INFINITY);
        if (ok)
            ok = search(
                T, kBrute,
                [&](const WChild &ch, const float4 *, float &key) {
                    key = 0.f;
                    const float lo[3] = {ch.lo[0] - pad, ch.lo[1] - pad, ch.lo[2] - pad};
                    const float hi[3] = {ch.hi[0] + pad, ch.hi[1] + pad, ch.hi[2] + pad};
                    return box_ray<D>(lo, hi, o, ia, tmaxA) != INFINITY ||
                           (wantB && box_ray<D>(lo, hi, o, ib, tmaxB) != INFINITY);
                },
                test, [&] { return 0.f; }, [&] {});
        const float m = warp_min(lb.d2);
        certain = ok;
        int hit = -1;
        if (m < INFINITY) {
            const unsigned at = __ballot_sync(FULL, lb.d2 == m);
            const int src = __ffs(at) - 1;
            const float lim = m + __shfl_sync(FULL, teA, src);
            const bool bad = lane == src ? (!(teA >= 0.f) || lb.dup || lb.alt <= lim) : lb.d2 <= lim;
            certain = certain && !__any_sync(FULL, bad);
            hit = __shfl_sync(FULL, lb.rec, src);
            t_out = m;
        }
        if (wantB) {
            occB = __any_sync(FULL, occ);
            certain = certain && (occB || !__any_sync(FULL, occ_maybe));
        }
        return hit;
    }

    __device__ __forceinline__ int ray2_w(const TreeView &T, P3 o, P3 va, float tmaxA, float &t_out, bool wantB, P3 vb,
                                          int skipB, float tmaxB, bool &occB, bool act) {
        t_out = tmaxA;
        occB = false;
        if (!act || T.root == WOST_EMPTY_REF) return -1;
        bool certain;
        int hit = ray2_search(T, o, va, tmaxA, -1, t_out, wantB, vb, skipB, tmaxB, occB, certain);
        if (!certain) {
            const RayAnswer a = ray2_binary<D>(T, o, va, tmaxA, wantB, vb, skipB, tmaxB, st);
            t_out = a.t;
            occB = a.occ;
            hit = a.hit;
        }
        return hit;
    }
};

// the distance alone (to within the ties that only a one-lane search decides)
template <int D>
__device__ __noinline__ float coop_distance(const TreeView &T, P3 x, float tau, int2 *fr, int frs, int fcap) {
    WarpQ<D> q;
    q.fr = fr;
    q.frs = frs;
    q.fcap = fcap;
    q.lane = threadIdx.x & 31;
    q.tau = tau;
    float B = INFINITY, best = INFINITY;
    q.search(
        T, WarpQ<D>::kBrute,
        [&](const WChild &ch, const float4 *, float &key) {
            key = box_dist2<D>(ch.lo, ch.hi, x);
            return key < B;
        },
        [&](uint32_t k) { best = fminf(best, prim_dist2<D>(T.prims, k, x)); }, [&] { return B; },
        [&] { B = fminf(B, beyond(warp_min(best), tau)); });
    return sqrtf(warp_min(best));
}

// One copy of the silhouette search for every caller, and for the one-lane
// kernels, whose warps would otherwise wait for the lane with the longest
// search (every lane calls it with the same arguments).
template <int D>
__device__ __noinline__ SilAnswer coop_silhouette(const TreeView &T, P3 x, float rmax, float bound2, float tau,
                                                  int2 *fr, int frs, int fcap) {
    WarpQ<D> q;
    q.fr = fr;
    q.frs = frs;
    q.fcap = fcap;
    q.lane = threadIdx.x & 31;
    q.tau = tau;
    return q.silhouette_search(T, x, rmax, fminf(rmax * rmax, bound2));
}

}  // namespace wost
