// Boundary queries of 3D walks by groups of lanes: closest Dirichlet point,
// closest silhouette, first Neumann hit, crossing count (the per-lane
// traversals of geom.cuh serve 2D).
//
// A warp keeps one walk per lane, but its queries are answered by groups of
// lanes: a group takes one pending query of the warp at a time, tests the
// children of a node (or as many primitives of a leaf) in one go, one per
// lane, and takes the next pending query when it is done.  A node visit is
// one coalesced load, and the traversal stack is the group's, in shared
// memory.
//
// Why: with one query per lane a 3D walk ran 3-4 active lanes of 32 (every
// lane at another node, the warp waiting for its longest query), one L2
// round trip per primitive of a leaf, and a launch lasted as long as its
// slowest walk, 0.5-2 ms a step.  With groups all lanes of a visit do work,
// a leaf is one or a few round trips, and so is a node.  What bounds it now: L2
// round trips and instruction fetch (35% of issue slots, 20 active lanes of 32 on
// the icosphere); figures at plain_walk_kernel.
//
// Closest points: groups of eight lanes over eight-wide nodes of oriented
// caps and boxes (geom.cuh), nearest node first.  The bounds carry a margin above the
// rounding of the distances, so the search returns the minimum over all
// primitives (ties to the smaller id) in whatever order it visits them.  The
// query is defined by the box tree, though (coop_closest).
// Silhouettes, rays, Neumann samples: groups of four or eight lanes over
// four-wide nodes of boxes, depth first, children nearest first.  An edge's or a hit's FP32 value can
// lie below its box's by rounding (a ray hit by its edge slack, ray_prim), so
// the result can depend on which box was opened first, and the summed weight of
// the Neumann sample on the order of its terms: the order of visits is part of
// these queries.
// All lanes of the warp run every call together.
#pragma once
#include "geom.cuh"

namespace wost {

constexpr int kGrpStack = 64;     // stack entries per query (checked when the scene is built)

struct alignas(16) CoopWarp {     // shared memory of one warp
    uint2 stack[8][kGrpStack + 1];         // (key, node or leaf); +1: groups start in different banks
    float best[32];               // results by lane
    int slot[32];
    int pad[4];
};

// shared memory of the calling warp in a kernel of NW warps (3D kernels)
template <int D, int NW>
__device__ __forceinline__ CoopWarp *coop_shared() {
    if constexpr (D == 3) {
        __shared__ CoopWarp s[NW];
        return &s[threadIdx.x >> 5];
    } else {
        return nullptr;
    }
}
__host__ __device__ constexpr int coop_bytes(int D, int warps) { return D == 3 ? warps * (int)sizeof(CoopWarp) : 0; }

enum : int { kCoopPoint = 0, kCoopPointBox = 1, kCoopSil = 2, kCoopExit = 3, kCoopAny = 4, kCoopCount = 5, kCoopPick = 6 };

// What the lanes of a calling warp hold: walks of one scene, walks whose scenes
// may differ (a pointer per lane), or few walks of one scene (the wavefront)
enum : int { kModeSolo = 0, kModeMulti = 1, kModeFew = 2 };

// Lanes per group.  Closest points: one per child and leaf primitive.
// Silhouettes and rays: one per child, four rounds for a leaf of 16; with few
// walks per warp the longer chain costs more than the shared visits save
// (silhouettes, eight lanes: guided icosphere 63.2 -> 59.2 ms, plain icosphere
// 80 -> 82).  The Neumann sample's leaves are long (a philox draw and a log
// per primitive): flux slab 19.6 -> 18.8 ms with eight.
__host__ __device__ constexpr int group_lanes(int kind, int mode) {
    return kind == kCoopPoint || kind == kCoopPick || (kind == kCoopSil && mode == kModeFew) ? 8 : 4;
}

// monotonic map of a float (not NaN) to an int
__device__ __forceinline__ int order_key(float f) {
    const int i = __float_as_int(f);
    return i ^ ((i >> 31) & 0x7fffffff);
}
template <int G>
__device__ __forceinline__ int group_min(int v) {
#pragma unroll
    for (int o = G / 2; o; o >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
template <int G>
__device__ __forceinline__ float group_min(float v) {
#pragma unroll
    for (int o = G / 2; o; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

template <int kKind>
__device__ __forceinline__ const DevBVH &coop_bvh(const DevScene &sc, bool dirichlet = false) {
    if (kKind == kCoopPoint || kKind == kCoopPointBox) return sc.dir;
    if (kKind == kCoopSil) return sc.sil;
    if (kKind == kCoopPick) return sc.neu;
    if (kKind == kCoopCount) return dirichlet ? sc.dir : sc.neu;
    return sc.neu;
}

// One query per lane that wants one; all lanes of the warp call.
//   kCoopPoint  best_io: in the bound (squared), out the squared distance
//               (kCoopPointBox: the same over the box tree)
//   kCoopSil    best_io: in the bound (squared), out the squared distance
//   kCoopExit   first exit through the Neumann boundary along v within
//               best_io, from t > -(rounding band of a position)
//               (ray_prim, kExit), aux: slot skipped
//   kCoopAny    first hit of either orientation, aux: slot skipped
//   kCoopCount  crossings along v (returned), aux != 0: of the Dirichlet BVH
//   kCoopPick   neumann_pick: best_io: in r^2, out W; v: the bits of point, walk
//               and step, aux and key1: the key
// Returns the leaf slot (-1: none within the bound).
// Out of line: the walk's state is saved once around the call instead of
// competing with the traversal for registers (the kernels run at 64 to 96 per
// thread).
struct CoopResult {
    int slot;
    float best;
    uint32_t nodes, prims;   // visits of the queries this lane's group answered (its first lane counts)
};
template <int kKind, int kMode>
__device__ __noinline__ CoopResult coop_query(uint32_t sh_addr, const DevScene *scene_p, bool want, float x0, float x1,
                                              float x2, float v0, float v1, float v2, float best_io, int aux, uint32_t key1,
                                              int *err) {
    CoopWarp &sh = *reinterpret_cast<CoopWarp *>(__cvta_shared_to_generic(sh_addr));
    const DevScene &scene = *scene_p;
    const float x[3] = {x0, x1, x2}, v[3] = {v0, v1, v2};
    CoopResult res{kKind == kCoopCount ? 0 : -1, best_io, 0u, 0u};
    constexpr unsigned kFull = 0xffffffffu;
    constexpr bool kRay = kKind >= kCoopExit && kKind <= kCoopCount;
    constexpr bool kMulti = kMode == kModeMulti;
    constexpr int G = group_lanes(kKind, kMode), NG = 32 / G;   // lanes per group, groups
    constexpr int NW = kKind == kCoopPoint ? 8 : 4;   // children per node
    const int lane = threadIdx.x & 31, sub = lane & (G - 1), g = lane / G, base = g * G;
    uint2 *stack = sh.stack[g];
    want = want && coop_bvh<kKind>(scene, aux != 0).nprims > 0;
    unsigned todo = __ballot_sync(kFull, want);
    if (todo == 0) return res;
    __syncwarp();   // the results of the warp's previous query have been read
    float inv[3] = {0.f, 0.f, 0.f};
    if (kRay) {
#pragma unroll
        for (int k = 0; k < 3; ++k) inv[k] = 1.f / v[k];   // +-inf for a zero component is fine in the slab test
    }
    // the group's query
    bool busy = false;
    int cur = 0, ref = 0, sp = 0, gaux = -1;
    uint32_t gkey1 = 0;        // kCoopPick
    float best = 0.f, gx[3] = {0.f, 0.f, 0.f}, gv[3] = {0.f, 0.f, 0.f}, ginv[3] = {0.f, 0.f, 0.f};
    const DevScene *gs = &scene;
    // this lane's candidate of the group's query
    float lb = 0.f;
    int ls = -1, lid = INT_MAX;
    float W = 0.f;             // kCoopPick: summed weight of the group's query
    for (;;) {
        const unsigned idle = __ballot_sync(kFull, !busy);
        if (todo && idle) {
            // the idle groups take the next pending lanes in order
            const int rank = __popc(idle & ((1u << base) - 1u)) / G, n = __popc(idle) / G;
            unsigned mine = todo;
#pragma unroll 1
            for (int i = 0; i < rank; ++i) mine &= mine - 1u;
#pragma unroll 1
            for (int i = 0; i < n; ++i) todo &= todo - 1u;
            const bool take = !busy && mine != 0;
            const int from = take ? __ffs(mine) - 1 : lane;
            const float b0 = __shfl_sync(kFull, best_io, from);
            const int a0 = __shfl_sync(kFull, aux, from);
            const uint32_t nk1 = kKind == kCoopPick ? __shfl_sync(kFull, key1, from) : 0u;
            float nx[3], nv[3], ni[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                nx[k] = __shfl_sync(kFull, x[k], from);
                if (kRay || kKind == kCoopPick) nv[k] = __shfl_sync(kFull, v[k], from);
                if (kRay) ni[k] = __shfl_sync(kFull, inv[k], from);
            }
            const DevScene *ns = gs;
            if (kMulti)
                ns = reinterpret_cast<const DevScene *>(
                    __shfl_sync(kFull, reinterpret_cast<unsigned long long>(&scene), from));
            if (take) {
                busy = true;
                cur = from;
                ref = 0;
                sp = 0;
                best = b0;
                gaux = a0;
                gkey1 = nk1;
                W = 0.f;
                gs = ns;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    gx[k] = nx[k];
                    if (kRay || kKind == kCoopPick) gv[k] = nv[k];
                    if (kRay) ginv[k] = ni[k];
                }
                lb = __int_as_float(0x7f800000);
                ls = -1;
                lid = kKind == kCoopCount ? 0 : INT_MAX;
            }
        }
        if (!__any_sync(kFull, busy)) break;
        const DevScene &sc = kMulti ? *gs : scene;
        const DevBVH &bv = coop_bvh<kKind>(sc, gaux != 0);
        const float tneg = kKind == kCoopExit ? kRoundBand * sc.scale : 0.f;

        bool fin = false;
        // the next entry of the stack
        auto pop = [&](bool need) {
            while (__any_sync(kFull, need)) {
                const int i = sp - 1 - sub;
                if constexpr (kKind == kCoopPoint) {
                    // the nearest of the top eight that is still within the
                    // bound; eight that are not go together.  An entry below
                    // the top is taken only while a whole depth-first
                    // traversal fits above the stack; taking the top one then
                    // never needs more space than the entries there already do.
                    const int window = sp - 1 + bv.need <= kGrpStack ? G : 1;
                    const bool in = need && i >= 0 && sub < window;
                    uint2 e = make_uint2(0u, 0u);
                    if (in) e = stack[i];
                    const bool ok = in && __uint_as_float(e.x) <= best;
                    const int m = group_min<G>(ok ? (order_key(__uint_as_float(e.x)) & ~(G - 1)) | sub : INT_MAX);
                    const int win = m & (G - 1);
                    const int rwin = __shfl_sync(kFull, (int)e.y, base + win);
                    const unsigned kt = __shfl_sync(kFull, e.x, base), rt = __shfl_sync(kFull, e.y, base);
                    if (need) {
                        if (m == INT_MAX) {
                            sp = max(sp - window, 0);
                            if (sp == 0) { need = false; fin = true; }
                        } else {
                            ref = rwin;
                            if (sub == win && win != 0) stack[i] = make_uint2(kt, rt);
                            --sp;
                            need = false;
                        }
                    }
                } else {
                    // the top one that is still within the bound
                    const bool in = need && i >= 0;
                    uint2 e = make_uint2(0u, 0u);
                    if (in) e = stack[i];
                    const unsigned okm = __ballot_sync(kFull, in && __uint_as_float(e.x) <= best) >> base & ((1u << G) - 1u);
                    const int win = okm ? __ffs(okm) - 1 : 0;
                    const int rwin = __shfl_sync(kFull, (int)e.y, base + win);
                    if (need) {
                        if (okm) {
                            ref = rwin;
                            sp -= win + 1;
                            need = false;
                        } else {
                            sp = max(sp - G, 0);
                            if (sp == 0) { need = false; fin = true; }
                        }
                    }
                }
                __syncwarp();
            }
        };

        // ---- nodes, until every group that searches holds a leaf ----
        while (__any_sync(kFull, busy && !fin && ref >= 0)) {
            const bool at = busy && !fin && ref >= 0;
            float key = 0.f;
            int cref = kEmptyRef;
            bool ok = false;
            if (at && (G == NW || sub < NW)) {
                if constexpr (kKind == kCoopPoint) {
                    const float4 *p = sc.dir_caps + (size_t)cap_f4(3) * ref;
                    const float4 bl = ldn(p + 2 * G + sub), bh = ldn(p + 3 * G + sub);   // lo.xyz, hi.x | hi.yz
                    const float ex = fmaxf(fmaxf(bl.x - gx[0], gx[0] - bl.w), 0.f);
                    const float ey = fmaxf(fmaxf(bl.y - gx[1], gx[1] - bh.x), 0.f);
                    const float ez = fmaxf(fmaxf(bl.z - gx[2], gx[2] - bh.y), 0.f);
                    key = fmaxf(cap_d2_3(ldn(p + sub), ldn(p + G + sub), gx), ex * ex + ey * ey + ez * ez);
                    cref = __float_as_int(bh.z);
                    ok = cref != kEmptyRef && key <= best;
                } else {
                    const float4 *p = bv.nodes + (size_t)node_f4<3>() * ref + sub;
                    const float4 a = ldn(p), b = ldn(p + NW);   // lo.xyz, hi.x | hi.yz, child, -
                    cref = __float_as_int(b.z);
                    const float lo[3] = {a.x, a.y, a.z}, hi[3] = {a.w, b.x, b.y};
                    if constexpr (kRay) {
                        float e = -tneg, xm = best;
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            const float t0 = (lo[k] - tneg - gx[k]) * ginv[k], t1 = (hi[k] + tneg - gx[k]) * ginv[k];
                            e = fmaxf(e, fminf(t0, t1));
                            xm = fminf(xm, fmaxf(t0, t1));
                        }
                        key = e;
                        ok = cref != kEmptyRef && e <= xm;
                    } else {
                        float far2 = 0.f, u[3], dd[3];
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            u[k] = lo[k] - gx[k];
                            const float w = gx[k] - hi[k];
                            const float df = fmaxf(fabsf(u[k]), fabsf(w));
                            dd[k] = fmaxf(fmaxf(u[k], w), 0.f);
                            far2 += df * df;
                        }
                        key = box_d2(dd[0], dd[1], dd[2]);
                        ok = cref != kEmptyRef && (kKind == kCoopPick ? key < best : key <= best);
                        if constexpr (kKind == kCoopSil) {
                            const float4 *fp = sc.sil_facing + (size_t)facing_f4(3) * ref;
                            const float4 f = ldn(fp + sub);   // axis, d0
                            const float2 h = reinterpret_cast<const float2 *>(fp + NW)[sub];   // d1, s^2
                            const float q = -(f.x * u[0] + f.y * u[1] + f.z * u[2]);
                            ok = ok && !facing_prunes(q, f.w, h.x, h.y, far2, sc.tau);
                        }
                    }
                }
                res.nodes += sub == 0;
            }
            const unsigned m = __ballot_sync(kFull, ok) >> base & ((1u << G) - 1u);
            const int n = __popc(m);
            int pos;   // >= 0: push this lane's child there
            int nref;
            if constexpr (kKind == kCoopPoint) {
                const int near = group_min<G>(ok ? (order_key(key) & ~(G - 1)) | sub : INT_MAX) & (G - 1);
                nref = __shfl_sync(kFull, cref, base + near);
                pos = ok && sub != near ? sp + __popc(m & ~(1u << near) & ((1u << sub) - 1u)) : -1;
            } else {
                // sort the children by key (a network of four: strict
                // comparisons, children not taken last)
                float kk = ok ? key : __int_as_float(0x7f800000);
                auto swap = [&](int other) {
                    const float ko = __shfl_sync(kFull, kk, base + other);
                    const int ro = __shfl_sync(kFull, cref, base + other);
                    if (sub < other ? ko < kk : (sub > other && kk < ko)) { kk = ko; cref = ro; }
                };
                swap(G == NW || sub < NW ? sub ^ 1 : sub);
                swap(G == NW || sub < NW ? sub ^ 2 : sub);
                swap(sub == 1 || sub == 2 ? 3 - sub : sub);
                key = kk;
                nref = __shfl_sync(kFull, cref, base);
                pos = at && sub >= 1 && sub < n ? sp + n - 1 - sub : -1;
            }
            if (at && m) {
                if (pos >= 0) {
                    if (pos < kGrpStack) stack[pos] = make_uint2(__float_as_uint(key), (unsigned)cref);
                    else atomicOr(err, 1);
                }
                sp = min(sp + n - 1, kGrpStack);
                ref = nref;
            }
            __syncwarp();
            pop(at && !m);
        }

        // ---- leaves ----
        const bool at = busy && !fin;
        const int s0 = leaf_start(ref), cnt = at ? leaf_count(ref) : 0;
        for (int b = 0; __any_sync(kFull, b < cnt); b += G) {
            const int s = s0 + b + sub;
            float wt = 0.f;
            if (b + sub < cnt) {
                float t;
                bool cand;
                if (kKind == kCoopPoint || kKind == kCoopPointBox) {
                    float a[3], bb[3], c[3];
                    load_tri(bv.prims, s, a, bb, c);
                    t = tri_d2_fast(a, bb, c, gx);
                    cand = t <= best;
                } else if (kKind == kCoopSil) {
                    cand = sil_elem<3>(bv.prims, s, gx, sc.tau, best, t);
                } else if (kKind == kCoopExit) {
                    cand = s != gaux && ray_prim<3, true>(bv.prims, s, gx, gv, t, tneg) && t <= best;
                } else if (kKind == kCoopAny) {
                    cand = s != gaux && ray_prim<3>(bv.prims, s, gx, gv, t) && t <= best;
                } else if (kKind == kCoopPick) {
                    wt = neumann_weight<3>(bv, s, gx, best);
                    cand = wt > 0.f;
                    if (cand)
                        t = neumann_key(__ldg(bv.ids + s), wt, __float_as_uint(gv[0]), __float_as_uint(gv[1]),
                                        __float_as_uint(gv[2]), (uint32_t)gaux, gkey1);
                } else {
                    lid += ray_prim<3>(bv.prims, s, gx, gv, t) ? 1 : 0;
                    cand = false;
                }
                if (cand && t <= lb) {
                    const int id = __ldg(bv.ids + s);
                    if (t < lb || id < lid) { lb = t; ls = s; lid = id; }
                }
            }
            if constexpr (kKind == kCoopPick) {   // in the order of the primitives
#pragma unroll
                for (int j = 0; j < G; ++j) W += __shfl_sync(kFull, wt, base + j);
            }
        }
        if (sub == 0) res.prims += cnt;
        if (kKind != kCoopCount && kKind != kCoopPick) best = fminf(best, group_min<G>(at ? lb : __int_as_float(0x7f800000)));
        pop(at);

        // ---- results ----
        if (__any_sync(kFull, fin)) {
            if (kKind == kCoopCount) {
                int n = lid;
#pragma unroll
                for (int o = G / 2; o; o >>= 1) n += __shfl_xor_sync(kFull, n, o);
                if (fin && sub == 0) sh.slot[cur] = n;
            } else {
                const float top = kKind == kCoopPick ? group_min<G>(lb) : best;
                const int id = ls >= 0 && lb == top ? lid : INT_MAX;
                const int mid = group_min<G>(id);
                if (kKind == kCoopPick && fin) best = W;   // (returned in place of the bound)
                if (fin) {
                    if (mid == INT_MAX) {
                        if (sub == 0) { sh.best[cur] = best; sh.slot[cur] = -1; }
                    } else if (id == mid) {
                        sh.best[cur] = best;
                        sh.slot[cur] = ls;
                    }
                }
            }
            if (fin) busy = false;
        }
    }
    __syncwarp();
    if (want) {
        if (kKind != kCoopCount) res.best = sh.best[lane];
        res.slot = sh.slot[lane];
    }
    return res;
}

// the call, with the visits added to the lane's counters
template <int kKind, int kMode>
__device__ __forceinline__ int coop_run(CoopWarp &sh, const DevScene &sc, bool want, const float *x, const float *v,
                                        float &best, int aux, int *err, volatile Visits *vis, uint32_t key1 = 0) {
    const CoopResult r = coop_query<kKind, kMode>((uint32_t)__cvta_generic_to_shared(&sh), &sc, want, x[0], x[1], x[2],
                                                   v[0], v[1], v[2], best, aux, key1, err);
    best = r.best;
    if (kKind == kCoopPoint) add_visits(vis, &Visits::dnodes, r.nodes, &Visits::dprims, r.prims);
    else if (kKind == kCoopPointBox) add_visits(vis, &Visits::nodes, r.nodes, &Visits::dprims, r.prims);
    else if (kKind == kCoopSil) add_visits(vis, &Visits::snodes, r.nodes, &Visits::sprims, r.prims);
    else add_visits(vis, &Visits::nodes, r.nodes, &Visits::nprims, r.prims);
    return r.slot;
}

// Closest Dirichlet primitive: leaf slot, squared distance in d2.  A search of
// the boxes opens every box at or below the smallest FP32 distance, so it finds
// the minimum over all primitives unless that one's FP32 distance lies below
// the distance of its own box (both are rounded; an edge shared by triangles
// of several leaves), where the order of visits decides.  The answer of the
// caps is therefore the boxes' answer whenever the primitive's distance is not
// below that of its own bounding box, which its leaf's box contains; the few
// others are searched again in the boxes.
template <int kMode>
__device__ __forceinline__ int coop_closest(CoopWarp &sh, const DevScene &sc, bool want, const float *x, float &d2,
                                            int *err, volatile Visits *vis) {
    d2 = __int_as_float(0x7f800000);
    int slot = coop_run<kCoopPoint, kMode>(sh, sc, want, x, x, d2, -1, err, vis);
    bool again = false;
    if (slot >= 0) {
        float a[3], b[3], c[3], dd[3];
        load_tri(sc.dir.prims, slot, a, b, c);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const float lo = fminf(fminf(a[i], b[i]), c[i]), hi = fmaxf(fmaxf(a[i], b[i]), c[i]);
            dd[i] = fmaxf(fmaxf(lo - x[i], x[i] - hi), 0.f);
        }
        again = d2 < box_d2(dd[0], dd[1], dd[2]);
    }
    if (__any_sync(0xffffffffu, again)) {
        float e2 = __int_as_float(0x7f800000);
        const int e = coop_run<kCoopPointBox, kMode>(sh, sc, again, x, x, e2, -1, err, vis);
        if (again) { slot = e; d2 = e2; }
    }
    return slot;
}

}  // namespace wost
