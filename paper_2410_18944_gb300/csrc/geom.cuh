// Boundary queries of one walk step (Sec. 3.2, Sec. 5.3): closest Dirichlet
// point (epsilon-shell test, R_D), closest Neumann silhouette (R_S), first
// Neumann hit along a ray (next point on the star boundary).  Stack-based
// traversal of a binary BVH with child boxes in the parent; node and
// primitive loads are 16-byte vector loads through the read-only path.
// Ties between equal distances go to the smaller original primitive id.
#pragma once
#include <climits>

#include "common.cuh"

namespace wost {

constexpr int kStack = 64;

// width of the band (relative to the scene scale) inside which an FP32
// distance or hit parameter may be on the wrong side of its threshold:
// 16 units of 2^-24
constexpr float kRoundBand = 16.f * 5.9604645e-8f;

// The 2D closest-point, closest-silhouette and ray queries compiled out of line
// (a call per query; the caller's live registers no longer add to the
// traversal's), or inlined into the walk step.  One GB300, star of 4096
// segments: out of line plain walks take 24.2 against 20.4 ms, the walks of a
// training batch 38.4 against 38.7; inlined is the default.
#ifndef WOST_QUERY_NOINLINE
#define WOST_QUERY_NOINLINE 0
#endif
#if WOST_QUERY_NOINLINE
#define WOST_QUERY_FN __noinline__
#else
#define WOST_QUERY_FN
#endif

// BVH nodes.  2D: binary, child boxes in the parent (3 float4), one query per
// lane (this file).  3D: four children per node, 4 x (lo.xyz, hi.x), then
// 4 x (hi.yz, child, -), one query per group of lanes (coop.cuh).
constexpr int kEmptyRef = INT_MIN;   // child slot without a child (wide nodes)

// float4 per node
template <int D>
__host__ __device__ constexpr int node_f4() {
    return D == 2 ? 3 : 8;
}

// Per-thread visit counts of the traversals (algorithmic-traffic accounting):
// nodes of caps (closest point), of boxes with facing bounds (silhouettes) and
// of boxes alone, primitives.  A query counts in registers of its own and adds
// to these at its end.  They are volatile, kept in memory: totals that stayed in
// registers cost the traversals more than the adds per query (training batch of
// the star, counted per visit in registers 51.9 ms, so 50.9).
struct Visits {
    uint32_t dnodes = 0, snodes = 0, nodes = 0, dprims = 0, sprims = 0, nprims = 0;
};
__device__ __forceinline__ void add_visits(volatile Visits *vis, uint32_t Visits::*nodes, uint32_t nv, uint32_t Visits::*prims,
                                           uint32_t pv) {
    if (!vis) return;
    vis->*nodes = vis->*nodes + nv;
    vis->*prims = vis->*prims + pv;
}

// squared distance from the distances along the axes, with its rounding
// spelled out: whether a box is opened is decided on this value
__device__ __forceinline__ float box_d2(float dx, float dy, float dz) {
    return __fmaf_rn(dz, dz, __fmaf_rn(dx, dx, __fmul_rn(dy, dy)));
}

// keys of the children of a binary 2D node: squared distance from x to the box
__device__ __forceinline__ void node_keys_d2(const float4 *nodes, int node, const float *x, float *k, int *r) {
    const float4 a = ldn(nodes + 3 * node), b = ldn(nodes + 3 * node + 1), q = ldn(nodes + 3 * node + 2);
    float ax = fmaxf(fmaxf(a.x - x[0], x[0] - a.z), 0.f), ay = fmaxf(fmaxf(a.y - x[1], x[1] - a.w), 0.f);
    float bx = fmaxf(fmaxf(b.x - x[0], x[0] - b.z), 0.f), by = fmaxf(fmaxf(b.y - x[1], x[1] - b.w), 0.f);
    k[0] = ax * ax + ay * ay;
    k[1] = bx * bx + by * by;
    r[0] = __float_as_int(q.x);
    r[1] = __float_as_int(q.y);
}

// keys of the children of a binary 2D node: entry parameter of the ray
// o + t v (inv = 1/v) into the child box grown by pad, from t > -pad, +inf if
// it misses within tmax (exit casts grow the boxes, so that crossings within
// the rounding band of a primitive are not pruned)
__device__ __forceinline__ void node_keys_ray(const float4 *nodes, int node, const float *o, const float *inv,
                                              float tmax, float *kk, int *r, float pad) {
    const float4 a = ldn(nodes + 3 * node), b = ldn(nodes + 3 * node + 1), q = ldn(nodes + 3 * node + 2);
    const float lo0[2] = {a.x, a.y}, hi0[2] = {a.z, a.w}, lo1[2] = {b.x, b.y}, hi1[2] = {b.z, b.w};
    r[0] = __float_as_int(q.x);
    r[1] = __float_as_int(q.y);
    float e0 = -pad, x0 = tmax, e1 = -pad, x1 = tmax;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        float a0 = (lo0[k] - pad - o[k]) * inv[k], b0 = (hi0[k] + pad - o[k]) * inv[k];
        float a1 = (lo1[k] - pad - o[k]) * inv[k], b1 = (hi1[k] + pad - o[k]) * inv[k];
        e0 = fmaxf(e0, fminf(a0, b0));
        x0 = fminf(x0, fmaxf(a0, b0));
        e1 = fmaxf(e1, fminf(a1, b1));
        x1 = fminf(x1, fmaxf(a1, b1));
    }
    kk[0] = e0 <= x0 ? e0 : __int_as_float(0x7f800000);
    kk[1] = e1 <= x1 ? e1 : __int_as_float(0x7f800000);
}

// Traversal stack of a lane (2D): key and node or leaf in one 8-byte entry
struct LaneStack {
    uint2 e[kStack];
    int sp = 0;
    __device__ __forceinline__ void push(float key, int ref, int *err) {
        if (sp < kStack) e[sp++] = make_uint2(__float_as_uint(key), (unsigned)ref);
        else atomicOr(err, 1);
    }
    // the top entry whose key is within best; false if there is none
    __device__ __forceinline__ bool pop(float best, int &ref) {
        while (sp > 0) {
            const uint2 t = e[--sp];
            if (__uint_as_float(t.x) <= best) { ref = (int)t.y; return true; }
        }
        return false;
    }
};

// Continue at the nearer of the two children with h[c] (ties: the first) and
// push the other.  Returns false if no child is taken.
__device__ __forceinline__ bool take_children(const float *k, const int *r, const bool *h, int &ref, LaneStack &st,
                                              int *err) {
    if (h[0] && h[1]) {
        const bool second = k[1] < k[0];
        st.push(second ? k[0] : k[1], second ? r[0] : r[1], err);
        ref = second ? r[1] : r[0];
        return true;
    }
    if (h[0] || h[1]) ref = h[0] ? r[0] : r[1];
    return h[0] || h[1];
}

// ---- oriented caps ------------------------------------------------------------
// Bound of the closest-point search: a cap around the primitives of a child,
// centre c, axis a (their mean normal), half thickness h along a and radius r
// across it (3D: a flat cylinder; 2D: an oriented box).  A boundary patch is
// thin along its normal, so seen from the front, as walks see the boundary,
// the cap's distance is that of the patch within curvature x r^2; the distance
// to its axis-aligned box falls short by about r, and a search from afar has
// to open every patch whose box is nearer than the closest point: patches
// within about sqrt(r R) of it (R: the walk's distance) instead of a few r.
// h and r carry a margin of 1e-6 x the scene's extent and its distance from the
// origin, and the axis is 1e-6 short of unit length, so that the distance is
// too, for points far outside the scene (rounding grows with their distance):
// together more than the rounding of this distance and of a primitive's own.
// Every primitive at or below the bound is tested, whatever the order of visits
// (3D, outside the scene by more than a few extents: but for the last units of
// a box's own distance).
// Per node: 2D (2 children) (c.xy, a.xy) of each, (h0, r0, h1, r1), (ref0,
// ref1, -, -); 3D (8 children) 8 x (c.xyz, h), 8 x (a.xyz, r), and the children's
// boxes grown by the margin with the references, 8 x (lo.xyz, hi.x), 8 x (hi.yz,
// ref, -): a large curved patch has a thick cap, and the greater of the two
// distances bounds (genus-3: 51 -> 43 nodes and 51 -> 38 triangles per step).
__host__ __device__ constexpr int cap_f4(int d) { return d == 2 ? 4 : 32; }

// squared distance from x to the cap (c, a as loaded; 2D: c = (c.xy, a.xy))
__host__ __device__ __forceinline__ float cap_d2_2(float4 c, float h, float r, const float *x) {
    const float ux = x[0] - c.x, uy = x[1] - c.y;
    const float s = fmaxf(fabsf(c.z * ux + c.w * uy) - h, 0.f), l = fmaxf(fabsf(c.z * uy - c.w * ux) - r, 0.f);
    return s * s + l * l;
}
__host__ __device__ __forceinline__ float cap_d2_3(float4 c, float4 a, const float *x) {
    const float u[3] = {x[0] - c.x, x[1] - c.y, x[2] - c.z};
    const float q = a.x * u[0] + a.y * u[1] + a.z * u[2];
    const float n = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    // squared distance to the axis, less the axis' 2e-6 of q^2 and the rounding
    // of n and q^2
    const float w = fmaxf(n * (1.f - 4e-6f) - q * q, 1e-30f);
    const float s = fmaxf(fabsf(q) - c.w, 0.f), l = fmaxf(w * rsqrtf(w) - a.w, 0.f);
    return s * s + l * l;
}

// ---- primitive distances ----------------------------------------------------
template <typename R>
__device__ __forceinline__ R seg_d2(R ax, R ay, R bx, R by, R px, R py, R &qx, R &qy) {
    R ex = bx - ax, ey = by - ay;
    R ee = ex * ex + ey * ey;
    R t = ee > R(0) ? ((px - ax) * ex + (py - ay) * ey) / ee : R(0);
    t = t < R(0) ? R(0) : (t > R(1) ? R(1) : t);
    qx = ax + t * ex;
    qy = ay + t * ey;
    R dx = px - qx, dy = py - qy;
    return dx * dx + dy * dy;
}

// the FP32 distance of seg_d2, bit for bit, dividing only where the foot lies
// inside the segment (few of a leaf's segments; star of 4096: 21.7 -> 21.1 ms)
__device__ __forceinline__ float seg_d2_fast(float4 s, const float *x) {
    const float ex = s.z - s.x, ey = s.w - s.y;
    const float ee = ex * ex + ey * ey, dot = (x[0] - s.x) * ex + (x[1] - s.y) * ey;
    float t = dot > 0.f ? 1.f : 0.f;
    if (dot > 0.f && dot < ee) t = dot / ee;
    const float dx = x[0] - __fmaf_rn(t, ex, s.x), dy = x[1] - __fmaf_rn(t, ey, s.y);
    return dx * dx + dy * dy;
}

template <typename R>
__device__ __forceinline__ R seg3_d2(const R *a, const R *b, const R *p) {
    R e[3], ap[3], ee = 0, t = 0;
    for (int i = 0; i < 3; ++i) { e[i] = b[i] - a[i]; ap[i] = p[i] - a[i]; ee += e[i] * e[i]; t += ap[i] * e[i]; }
    t = ee > R(0) ? t / ee : R(0);
    t = t < R(0) ? R(0) : (t > R(1) ? R(1) : t);
    R s = 0;
    for (int i = 0; i < 3; ++i) { R d = ap[i] - t * e[i]; s += d * d; }
    return s;
}

// closest point on a triangle by Voronoi regions (Ericson 2004, Sec. 5.1.5)
template <typename R>
__device__ __forceinline__ R tri_d2(const R *a, const R *b, const R *c, const R *p, R *q) {
    R ab[3], ac[3], ap[3], bp[3], cp[3];
    for (int i = 0; i < 3; ++i) { ab[i] = b[i] - a[i]; ac[i] = c[i] - a[i]; ap[i] = p[i] - a[i]; bp[i] = p[i] - b[i]; cp[i] = p[i] - c[i]; }
    auto dot = [](const R *u, const R *v) { return u[0] * v[0] + u[1] * v[1] + u[2] * v[2]; };
    R d1 = dot(ab, ap), d2 = dot(ac, ap);
    R d3 = dot(ab, bp), d4 = dot(ac, bp);
    R d5 = dot(ab, cp), d6 = dot(ac, cp);
    R vc = d1 * d4 - d3 * d2, vb = d5 * d2 - d1 * d6, va = d3 * d6 - d5 * d4;
    if (d1 <= R(0) && d2 <= R(0)) {
        for (int i = 0; i < 3; ++i) q[i] = a[i];
    } else if (d3 >= R(0) && d4 <= d3) {
        for (int i = 0; i < 3; ++i) q[i] = b[i];
    } else if (vc <= R(0) && d1 >= R(0) && d3 <= R(0)) {
        R v = d1 / (d1 - d3);
        for (int i = 0; i < 3; ++i) q[i] = a[i] + v * ab[i];
    } else if (d6 >= R(0) && d5 <= d6) {
        for (int i = 0; i < 3; ++i) q[i] = c[i];
    } else if (vb <= R(0) && d2 >= R(0) && d6 <= R(0)) {
        R w = d2 / (d2 - d6);
        for (int i = 0; i < 3; ++i) q[i] = a[i] + w * ac[i];
    } else if (va <= R(0) && (d4 - d3) >= R(0) && (d5 - d6) >= R(0)) {
        R w = (d4 - d3) / ((d4 - d3) + (d5 - d6));
        for (int i = 0; i < 3; ++i) q[i] = b[i] + w * (c[i] - b[i]);
    } else {
        R den = R(1) / (va + vb + vc);
        R v = vb * den, w = vc * den;
        for (int i = 0; i < 3; ++i) q[i] = a[i] + v * ab[i] + w * ac[i];
    }
    R s = 0;
    for (int i = 0; i < 3; ++i) { R d = p[i] - q[i]; s += d * d; }
    return s;
}

// The FP32 distance of tri_d2, bit for bit, without its branches: the region
// selects base point, edge and quotient, and one division serves all regions
// (the lanes of a group test different triangles and fall into different
// regions, so every branch of tri_d2 would run, most with a division).  A zero
// weight leaves a coordinate as it is: fma(0, e, a) = a.
__device__ __forceinline__ float tri_d2_fast(const float *a, const float *b, const float *c, const float *p) {
    float ab[3], ac[3], ap[3], bp[3], cp[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) { ab[i] = b[i] - a[i]; ac[i] = c[i] - a[i]; ap[i] = p[i] - a[i]; bp[i] = p[i] - b[i]; cp[i] = p[i] - c[i]; }
    auto dot = [](const float *u, const float *v) { return u[0] * v[0] + u[1] * v[1] + u[2] * v[2]; };
    const float d1 = dot(ab, ap), d2 = dot(ac, ap);
    const float d3 = dot(ab, bp), d4 = dot(ac, bp);
    const float d5 = dot(ab, cp), d6 = dot(ac, cp);
    const float vc = d1 * d4 - d3 * d2, vb = d5 * d2 - d1 * d6, va = d3 * d6 - d5 * d4;
    const float e43 = d4 - d3, e56 = d5 - d6;
    // the first of tri_d2's regions that holds: A, B, AB, C, AC, BC, face
    const bool rA = d1 <= 0.f && d2 <= 0.f;
    const bool rB = !rA && d3 >= 0.f && d4 <= d3;
    const bool rAB = !rA && !rB && vc <= 0.f && d1 >= 0.f && d3 <= 0.f;
    const bool n3 = rA || rB || rAB;
    const bool rC = !n3 && d6 >= 0.f && d5 <= d6;
    const bool rAC = !n3 && !rC && vb <= 0.f && d2 >= 0.f && d6 <= 0.f;
    const bool n5 = n3 || rC || rAC;
    const bool rBC = !n5 && va <= 0.f && e43 >= 0.f && e56 >= 0.f;
    const bool face = !n5 && !rBC;
    float num = 0.f, den = 1.f;
    if (rAB) { num = d1; den = d1 - d3; }
    if (rAC) { num = d2; den = d2 - d6; }
    if (rBC) { num = e43; den = e43 + e56; }
    if (face) { num = 1.f; den = va + vb + vc; }
    const float t = num / den;
    const float v = face ? vb * t : (rAC ? 0.f : t), w = face ? vc * t : (rAC ? t : 0.f);
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float base = rB || rBC ? b[i] : (rC ? c[i] : a[i]);
        const float dir = rBC ? c[i] - b[i] : ab[i];
        const float q = __fmaf_rn(w, ac[i], __fmaf_rn(v, dir, base));
        const float d = p[i] - q;
        s += d * d;
    }
    return s;
}

__device__ __forceinline__ void load_tri(const float4 *__restrict__ P, int s, float *a, float *b, float *c) {
    float4 u = ldn(P + 3 * s), v = ldn(P + 3 * s + 1), w = ldn(P + 3 * s + 2);
    a[0] = u.x; a[1] = u.y; a[2] = u.z; b[0] = u.w; b[1] = v.x; b[2] = v.y; c[0] = v.z; c[1] = v.w; c[2] = w.x;
}

// ---- warp-synchronous traversal ------------------------------------------------
// Every traversal below runs as a loop whose iterations are taken together by
// all lanes of the warp that entered it (a warp vote at the loop head): in one
// iteration each unfinished lane processes one inner node or one leaf, then
// pops its stack if needed.  Lanes that diverge inside an iteration
// re-converge at its end, instead of drifting apart for the rest of the
// traversal.
// ---- closest Dirichlet primitive (2D) ---------------------------------------
// returns the leaf slot of the closest primitive (-1 if none); best = squared distance
__device__ inline WOST_QUERY_FN int closest_dirichlet(const DevBVH &bv, const float4 *caps, const float *x, float &best,
                                                         int *err, volatile Visits *vis = nullptr) {
    constexpr int kBW = 2;
    best = __int_as_float(0x7f800000);
    if (bv.nprims == 0) return -1;
    const unsigned mask = __activemask();
    int best_slot = -1, best_id = 0x7fffffff;
    LaneStack st;
    int ref = 0;
    bool done = false;
    uint32_t nv = 0, pv = 0;
    // while-while: descend inner nodes together until every lane holds a
    // leaf (or is done), then test the leaves together
    while (__any_sync(mask, !done)) {
        while (__any_sync(mask, !done && ref >= 0)) {
            if (done || ref < 0) continue;
            float k[kBW];
            int r[kBW];
            bool h[kBW];
            const float4 *p = caps + cap_f4(2) * ref;
            const float4 hr = ldn(p + 2), q = ldn(p + 3);
            k[0] = cap_d2_2(ldn(p), hr.x, hr.y, x);
            k[1] = cap_d2_2(ldn(p + 1), hr.z, hr.w, x);
            r[0] = __float_as_int(q.x);
            r[1] = __float_as_int(q.y);
            ++nv;
#pragma unroll
            for (int c = 0; c < kBW; ++c) h[c] = k[c] <= best;
            if (!take_children(k, r, h, ref, st, err)) done = !st.pop(best, ref);
        }
        if (!done && ref < 0) {
            int s0 = leaf_start(ref), cnt = leaf_count(ref);
            pv += cnt;
            for (int s = s0; s < s0 + cnt; ++s) {
                float4 p = ldn(bv.prims + s);
                const float d2 = seg_d2_fast(p, x);
                if (d2 <= best) {
                    int id = __ldg(bv.ids + s);
                    if (d2 < best || id < best_id) { best = d2; best_slot = s; best_id = id; }
                }
            }
            done = !st.pop(best, ref);
        }
    }
    add_visits(vis, &Visits::dnodes, nv, &Visits::dprims, pv);
    return best_slot;
}

// FP64 distance (and closest point) from x to Dirichlet leaf slot s
template <int D>
__device__ __forceinline__ double dirichlet_dist64(const DevBVH &bv, int s, const float *x, double *q) {
    double p[3] = {x[0], x[1], D == 3 ? x[2] : 0.0};
    if (D == 2) {
        const double *v = bv.prims64 + 4 * (size_t)s;
        double d2 = seg_d2<double>(v[0], v[1], v[2], v[3], p[0], p[1], q[0], q[1]);
        return sqrt(d2);
    } else {
        const double *v = bv.prims64 + 9 * (size_t)s;
        return sqrt(tri_d2<double>(v, v + 3, v + 6, p, q));
    }
}

// ---- closest silhouette ------------------------------------------------------
// Silhouette rule: o = signed distance of x to the plane of an adjacent
// Neumann primitive (positive on the domain side); front o > tau, back
// o < -tau, edge-on otherwise; a silhouette has one neighbour seen from the
// back and the other from the front or edge-on.  Elements flagged "always"
// border the Neumann set.  Search radius starts at sqrt(best) (cap).
__device__ __forceinline__ bool sil_rule(float o0, float o1, float tau) {
    int c0 = o0 > tau ? 1 : (o0 < -tau ? -1 : 0);
    int c1 = o1 > tau ? 1 : (o1 < -tau ? -1 : 0);
    return (c0 == -1 && c1 >= 0) || (c1 == -1 && c0 >= 0);
}

// Facing bound of a silhouette-BVH child: no element below it can be a
// silhouette from x when all of its planes are seen from the front (no
// o < -tau) or all from the back (every o < -tau).  Per child the host stores
// a unit axis a, s = sin t of the largest angle t between a and the normals
// below it, and the range [d0, d1] of a . (v - lo) over the planes' points v
// (lo: the child box's lower corner).  With A = a . (x - lo) - d1 > 0 every v
// has a . (x - v) >= A, so x sees v under an angle from a whose cosine is at
// least A / L, L the distance from x to the far corner of the box, and a
// normal within t of a faces x when A >= L s (from the back: d0 - a . (x - lo)
// in place of A).  The slab [d0, d1] is what makes the bound sharp for the
// flat patches of a mesh: x may stand closer to a patch than the patch is
// wide.  A bound from the patch's bounding sphere and normal cone alone
// leaves every patch within about sqrt(2 rho / curvature) of a point on the
// boundary unpruned (rho the patch radius), this one those within a few rho.
// Rounding: o in a leaf, A and L err by less than 6e-7 L together, which the
// stored s carries (scene.cu, facing_bound); planes seen from the front may lie up to tau
// behind x, of which half is used (tau / 2, cos t >= 0.6), and from the back
// every o has to be below -tau.
// Per node: 2D (2 children) a.x, a.y, d0, d1 of each child, then both s^2;
// 3D (4 children) 4 x (a.xyz, d0), then 4 x (d1, s^2).
__host__ __device__ constexpr int facing_f4(int d) { return d == 2 ? 3 : 6; }

// q = a . (x - lo), far2 = squared distance to the far corner of the box
__device__ __forceinline__ bool facing_prunes(float q, float d0, float d1, float s2, float far2, float tau) {
    const float m = fmaxf(q - d1 + 0.5f * tau, d0 - q - 1.01f * tau);
    return m > 0.f && m * m >= s2 * far2;
}

// One inner node of the 2D silhouette search: keys of the children (squared
// distance to the box) and which of them can hold a silhouette within best.
__device__ __forceinline__ void node_keys_sil(const float4 *nodes, const float4 *facing, int node, const float *x,
                                              float best, float tau, float *k, int *r, bool *h) {
    const float4 bx[2] = {ldn(nodes + 3 * node), ldn(nodes + 3 * node + 1)}, q = ldn(nodes + 3 * node + 2);
    const float4 f[2] = {ldn(facing + 3 * node), ldn(facing + 3 * node + 1)}, s = ldn(facing + 3 * node + 2);
    r[0] = __float_as_int(q.x);
    r[1] = __float_as_int(q.y);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const float ux = bx[c].x - x[0], vx = x[0] - bx[c].z, uy = bx[c].y - x[1], vy = x[1] - bx[c].w;
        const float dx = fmaxf(fmaxf(ux, vx), 0.f), dy = fmaxf(fmaxf(uy, vy), 0.f);
        const float fx = fmaxf(fabsf(ux), fabsf(vx)), fy = fmaxf(fabsf(uy), fabsf(vy));
        k[c] = dx * dx + dy * dy;
        h[c] = k[c] <= best && !facing_prunes(-(f[c].x * ux + f[c].y * uy), f[c].z, f[c].w, c == 0 ? s.x : s.y,
                                              fx * fx + fy * fy, tau);
    }
}

// Silhouette element s: whether it is a silhouette from x within best, and
// its squared distance.  The facing tests come first: most elements of a
// smooth boundary fail them, and skip the edge distance and its division.
// An element without two neighbours ("always") carries zero normals.
template <int D>
__device__ __forceinline__ bool sil_elem(const float4 *prims, int s, const float *x, float tau, float best, float &d2) {
    if (D == 2) {
        float4 e0 = ldn(prims + 2 * s), e1 = ldn(prims + 2 * s + 1);
        float rx = x[0] - e0.x, ry = x[1] - e0.y;
        d2 = rx * rx + ry * ry;
        const float o0 = e0.z * rx + e0.w * ry;
        const float o1 = e1.x * rx + e1.y * ry;
        return d2 <= best && (e1.z != 0.f || sil_rule(o0, o1, tau));
    }
    const float4 e0 = ldn(prims + 3 * s), e1 = ldn(prims + 3 * s + 1), e2 = ldn(prims + 3 * s + 2);
    const float a[3] = {e0.x, e0.y, e0.z}, b[3] = {e0.w, e1.x, e1.y};
    const float r[3] = {x[0] - a[0], x[1] - a[1], x[2] - a[2]};
    const float o0 = e1.z * r[0] + e1.w * r[1] + e2.x * r[2];
    const float o1 = e2.y * r[0] + e2.z * r[1] + e2.w * r[2];
    const bool always = e1.z == 0.f && e1.w == 0.f && e2.x == 0.f;
    if (!(always || sil_rule(o0, o1, tau))) return false;
    d2 = seg3_d2<float>(a, b, x);
    return d2 <= best;
}

__device__ inline WOST_QUERY_FN int closest_silhouette(const DevBVH &bv, const float *x, float tau, float &best, int *err,
                                   const float4 *facing, volatile Visits *vis = nullptr) {
    constexpr int kBW = 2;
    if (bv.nprims == 0) return -1;
    const unsigned mask = __activemask();
    int best_slot = -1, best_id = 0x7fffffff;
    LaneStack st;
    int ref = 0;
    bool done = false;
    uint32_t nv = 0, pv = 0;
    // while-while: descend inner nodes together until every lane holds a
    // leaf (or is done), then test the leaves together
    while (__any_sync(mask, !done)) {
        while (__any_sync(mask, !done && ref >= 0)) {
            if (done || ref < 0) continue;
            float k[kBW];
            int r[kBW];
            bool h[kBW];
            node_keys_sil(bv.nodes, facing, ref, x, best, tau, k, r, h);
            ++nv;
            if (!take_children(k, r, h, ref, st, err)) done = !st.pop(best, ref);
        }
        if (!done && ref < 0) {
            int s0 = leaf_start(ref), cnt = leaf_count(ref);
            pv += cnt;
            for (int s = s0; s < s0 + cnt; ++s) {
                float d2;
                if (sil_elem<2>(bv.prims, s, x, tau, best, d2)) {
                    int id = __ldg(bv.ids + s);
                    if (d2 < best || id < best_id) { best = d2; best_slot = s; best_id = id; }
                }
            }
            done = !st.pop(best, ref);
        }
    }
    add_visits(vis, &Visits::snodes, nv, &Visits::sprims, pv);
    return best_slot;
}

// ---- ray cast against Neumann primitives --------------------------------------
// kExit: count only primitives the ray leaves the domain through.  The
// boundary is closed and oriented (2D: domain left of a -> b; 3D: triangles
// counter-clockwise seen from outside), so from inside the domain the first
// crossing is always such an exit; an entry hit can only come from a start
// point that rounding put a hair outside the boundary, and taking it would
// put the walker on the wrong side.  2D: exit iff cross(v, b - a) > 0;
// 3D: exit iff v . ((b - a) x (c - a)) > 0, i.e. the Moller-Trumbore
// determinant (b - a) . (v x (c - a)) is negative.  Exit hits count from
// t > -tneg and within about tneg of the primitive (segment parameter /
// barycentric slack tneg over the length / smallest height): a walker that
// stands on a Neumann primitive within rounding of its end vertex and heads
// out through the next primitive crosses it at t ~ 0, and rounding can put
// that crossing slightly behind the start or past the primitive's end; a
// start point inside the domain has no exit crossing behind it.
template <int D, bool kExit = false>
__device__ __forceinline__ bool ray_prim(const float4 *__restrict__ P, int s, const float *o, const float *v, float &t,
                                         float tneg = 0.f) {
    if (D == 2) {
        float4 p = ldn(P + s);
        float ex = p.z - p.x, ey = p.w - p.y;
        float ax = p.x - o[0], ay = p.y - o[1];
        float den = v[0] * ey - v[1] * ex;
        if (kExit ? !(den > 0.f) : den == 0.f) return false;
        float tt = (ax * ey - ay * ex) / den;
        float ss = (ax * v[1] - ay * v[0]) / den;
        const float eta = kExit ? tneg * rsqrtf(ex * ex + ey * ey) : 0.f;
        if (ss < -eta || ss > 1.f + eta || !(tt > (kExit ? -tneg : 0.f))) return false;
        t = tt;
        return true;
    } else {
        float a[3], b[3], c[3];
        load_tri(P, s, a, b, c);
        float e1[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]}, e2[3] = {c[0] - a[0], c[1] - a[1], c[2] - a[2]};
        float pv[3] = {v[1] * e2[2] - v[2] * e2[1], v[2] * e2[0] - v[0] * e2[2], v[0] * e2[1] - v[1] * e2[0]};
        float det = e1[0] * pv[0] + e1[1] * pv[1] + e1[2] * pv[2];
        if (kExit ? !(det < 0.f) : det == 0.f) return false;
        float eta = 0.f;
        if (kExit) {
            float n0 = e1[1] * e2[2] - e1[2] * e2[1], n1 = e1[2] * e2[0] - e1[0] * e2[2], n2 = e1[0] * e2[1] - e1[1] * e2[0];
            float e3[3] = {e2[0] - e1[0], e2[1] - e1[1], e2[2] - e1[2]};
            float l2 = fmaxf(fmaxf(e1[0] * e1[0] + e1[1] * e1[1] + e1[2] * e1[2], e2[0] * e2[0] + e2[1] * e2[1] + e2[2] * e2[2]),
                             e3[0] * e3[0] + e3[1] * e3[1] + e3[2] * e3[2]);
            eta = tneg * sqrtf(l2) * rsqrtf(n0 * n0 + n1 * n1 + n2 * n2);
        }
        float inv = 1.f / det;
        float tv[3] = {o[0] - a[0], o[1] - a[1], o[2] - a[2]};
        float u = (tv[0] * pv[0] + tv[1] * pv[1] + tv[2] * pv[2]) * inv;
        if (u < -eta || u > 1.f + eta) return false;
        float qv[3] = {tv[1] * e1[2] - tv[2] * e1[1], tv[2] * e1[0] - tv[0] * e1[2], tv[0] * e1[1] - tv[1] * e1[0]};
        float w = (v[0] * qv[0] + v[1] * qv[1] + v[2] * qv[2]) * inv;
        if (w < -eta || u + w > 1.f + eta) return false;
        float tt = (e2[0] * qv[0] + e2[1] * qv[1] + e2[2] * qv[2]) * inv;
        if (!(tt > (kExit ? -tneg : 0.f))) return false;
        t = tt;
        return true;
    }
}

// FP64 re-test of a hit: the same intersection in double precision
template <int D, bool kExit = false>
__device__ __forceinline__ bool ray_prim64(const DevBVH &bv, int s, const float *of, const float *vf, double &t,
                                           double tneg = 0.0) {
    double o[3] = {of[0], of[1], D == 3 ? of[2] : 0.0}, v[3] = {vf[0], vf[1], D == 3 ? vf[2] : 0.0};
    if (D == 2) {
        const double *p = bv.prims64 + 4 * (size_t)s;
        double ex = p[2] - p[0], ey = p[3] - p[1], ax = p[0] - o[0], ay = p[1] - o[1];
        double den = v[0] * ey - v[1] * ex;
        if (kExit ? !(den > 0.0) : den == 0.0) return false;
        double tt = (ax * ey - ay * ex) / den, ss = (ax * v[1] - ay * v[0]) / den;
        const double eta = kExit ? tneg / sqrt(ex * ex + ey * ey) : 0.0;
        if (ss < -eta || ss > 1.0 + eta || !(tt > (kExit ? -tneg : 0.0))) return false;
        t = tt;
        return true;
    } else {
        const double *a = bv.prims64 + 9 * (size_t)s, *b = a + 3, *c = a + 6;
        double e1[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]}, e2[3] = {c[0] - a[0], c[1] - a[1], c[2] - a[2]};
        double pv[3] = {v[1] * e2[2] - v[2] * e2[1], v[2] * e2[0] - v[0] * e2[2], v[0] * e2[1] - v[1] * e2[0]};
        double det = e1[0] * pv[0] + e1[1] * pv[1] + e1[2] * pv[2];
        if (kExit ? !(det < 0.0) : det == 0.0) return false;
        double eta = 0.0;
        if (kExit) {
            double n0 = e1[1] * e2[2] - e1[2] * e2[1], n1 = e1[2] * e2[0] - e1[0] * e2[2], n2 = e1[0] * e2[1] - e1[1] * e2[0];
            double e3[3] = {e2[0] - e1[0], e2[1] - e1[1], e2[2] - e1[2]};
            double l2 = fmax(fmax(e1[0] * e1[0] + e1[1] * e1[1] + e1[2] * e1[2], e2[0] * e2[0] + e2[1] * e2[1] + e2[2] * e2[2]),
                             e3[0] * e3[0] + e3[1] * e3[1] + e3[2] * e3[2]);
            eta = tneg * sqrt(l2 / (n0 * n0 + n1 * n1 + n2 * n2));
        }
        double inv = 1.0 / det;
        double tv[3] = {o[0] - a[0], o[1] - a[1], o[2] - a[2]};
        double u = (tv[0] * pv[0] + tv[1] * pv[1] + tv[2] * pv[2]) * inv;
        if (u < -eta || u > 1.0 + eta) return false;
        double qv[3] = {tv[1] * e1[2] - tv[2] * e1[1], tv[2] * e1[0] - tv[0] * e1[2], tv[0] * e1[1] - tv[1] * e1[0]};
        double w = (v[0] * qv[0] + v[1] * qv[1] + v[2] * qv[2]) * inv;
        if (w < -eta || u + w > 1.0 + eta) return false;
        double tt = (e2[0] * qv[0] + e2[1] * qv[1] + e2[2] * qv[2]) * inv;
        if (!(tt > (kExit ? -tneg : 0.0))) return false;
        t = tt;
        return true;
    }
}

// first Neumann hit with 0 < t <= tmax, skipping leaf slot `skip`; returns
// slot or -1 (kExit: exit hits only, from t > -tneg, see ray_prim)
template <bool kExit = false>
__device__ WOST_QUERY_FN int ray_neumann(const DevBVH &bv, const float *o, const float *v, float tmax, int skip, float &thit,
                           int *err, volatile Visits *vis = nullptr, float tneg = 0.f) {
    constexpr int kBW = 2;
    thit = tmax;
    if (bv.nprims == 0) return -1;
    const unsigned mask = __activemask();
    float inv[3];
#pragma unroll
    for (int k = 0; k < 2; ++k) inv[k] = 1.f / v[k];   // +-inf for a zero component is fine in the slab test
    float best = tmax;
    int best_slot = -1, best_id = 0x7fffffff;
    LaneStack st;
    int ref = 0;
    bool done = false;
    uint32_t nv = 0, pv = 0;
    // while-while: descend inner nodes together until every lane holds a
    // leaf (or is done), then test the leaves together
    while (__any_sync(mask, !done)) {
        while (__any_sync(mask, !done && ref >= 0)) {
            if (done || ref < 0) continue;
            float k[kBW];
            int r[kBW];
            bool h[kBW];
            node_keys_ray(bv.nodes, ref, o, inv, best, k, r, kExit ? tneg : 0.f);
            ++nv;
#pragma unroll
            for (int c = 0; c < kBW; ++c) h[c] = k[c] <= best;
            if (!take_children(k, r, h, ref, st, err)) done = !st.pop(best, ref);
        }
        if (!done && ref < 0) {
            int s0 = leaf_start(ref), cnt = leaf_count(ref);
            pv += cnt;
            for (int s = s0; s < s0 + cnt; ++s) {
                float t;
                if (s != skip && ray_prim<2, kExit>(bv.prims, s, o, v, t, tneg) && t <= best) {
                    int id = __ldg(bv.ids + s);
                    if (t < best || id < best_id) { best = t; best_slot = s; best_id = id; }
                }
            }
            done = !st.pop(best, ref);
        }
    }
    thit = best;
    add_visits(vis, &Visits::nodes, nv, &Visits::nprims, pv);
    return best_slot;
}

// ---- Neumann boundary sample of <N> (Sec. 3.2, Eq. wost_estm) ---------------
// Every Neumann primitive closer to x than r is a candidate with weight w its
// length (2D) or area (3D).  The candidate with the smallest key -log(u)/w,
// u in (0, 1] from the Philox counter (pid, wid, step, P_NKEY | id), is
// chosen: probability w / W (W = the summed weight) whatever order the
// traversal visits the candidates in (weighted sampling with keys,
// Efraimidis & Spirakis 2006); ties go to the smaller id.  Returns the leaf
// slot of the choice (-1 if there is no candidate) and W.
//
// weight of leaf slot s, 0 if it is not within the ball (r2 = r^2)
template <int D>
__device__ __forceinline__ float neumann_weight(const DevBVH &bv, int s, const float *x, float r2) {
    float d2, w;
    if (D == 2) {
        float4 p = ldn(bv.prims + s);
        float qx, qy;
        d2 = seg_d2<float>(p.x, p.y, p.z, p.w, x[0], x[1], qx, qy);
        w = sqrtf((p.z - p.x) * (p.z - p.x) + (p.w - p.y) * (p.w - p.y));
    } else {
        float a[3], b[3], c[3];
        load_tri(bv.prims, s, a, b, c);
        d2 = tri_d2_fast(a, b, c, x);
        float e1[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]}, e2[3] = {c[0] - a[0], c[1] - a[1], c[2] - a[2]};
        float n0 = e1[1] * e2[2] - e1[2] * e2[1], n1 = e1[2] * e2[0] - e1[0] * e2[2], n2 = e1[0] * e2[1] - e1[1] * e2[0];
        w = 0.5f * sqrtf(n0 * n0 + n1 * n1 + n2 * n2);
    }
    return d2 < r2 && w > 0.f ? w : 0.f;
}
__device__ __forceinline__ float neumann_key(int id, float w, uint32_t pid, uint32_t wid, uint32_t step, uint32_t k0,
                                             uint32_t k1) {
    U4 u = philox(pid, wid, step, P_NKEY | (uint32_t)id, k0, k1);
    const float uu = ((float)(u.x >> 8) + 1.f) * (1.0f / 16777216.0f);   // (0, 1]
    return -logf(uu) / w;
}

// 2D (one query per lane; 3D: kCoopPick, coop.cuh)
__device__ inline int neumann_pick(const DevBVH &bv, const float *x, float r, uint32_t pid, uint32_t wid, uint32_t step,
                                   uint32_t k0, uint32_t k1, float &W, int *err, volatile Visits *vis = nullptr) {
    constexpr int kBW = 2;
    W = 0.f;
    if (bv.nprims == 0) return -1;
    const float r2 = r * r;
    const unsigned mask = __activemask();
    int best_slot = -1, best_id = 0x7fffffff;
    float best_key = __int_as_float(0x7f800000);
    LaneStack st;
    int ref = 0;
    bool done = false;
    uint32_t nv = 0, pv = 0;
    const float lim = r2;   // the search radius never shrinks
    while (__any_sync(mask, !done)) {
        while (__any_sync(mask, !done && ref >= 0)) {
            if (done || ref < 0) continue;
            float k[kBW];
            int rr[kBW];
            bool h[kBW];
            node_keys_d2(bv.nodes, ref, x, k, rr);
            ++nv;
#pragma unroll
            for (int c = 0; c < kBW; ++c) h[c] = k[c] < r2;
            if (!take_children(k, rr, h, ref, st, err)) done = !st.pop(lim, ref);
        }
        if (!done && ref < 0) {
            int s0 = leaf_start(ref), cnt = leaf_count(ref);
            pv += cnt;
            for (int s = s0; s < s0 + cnt; ++s) {
                const float w = neumann_weight<2>(bv, s, x, r2);
                if (!(w > 0.f)) continue;
                const int id = __ldg(bv.ids + s);
                const float key = neumann_key(id, w, pid, wid, step, k0, k1);
                W += w;
                if (key < best_key || (key == best_key && id < best_id)) { best_key = key; best_slot = s; best_id = id; }
            }
            done = !st.pop(lim, ref);
        }
    }
    add_visits(vis, &Visits::nodes, nv, &Visits::nprims, pv);
    return best_slot;
}

// number of crossings of the ray o + t v (t > 0) with all primitives of a 2D BVH
__device__ inline int ray_count(const DevBVH &bv, const float *o, const float *v, int *err) {
    constexpr int kBW = 2;
    if (bv.nprims == 0) return 0;
    const unsigned mask = __activemask();
    float inv[3];
#pragma unroll
    for (int k = 0; k < 2; ++k) inv[k] = 1.f / v[k];
    const float big = 3.0e38f;
    int cnt = 0, ref = 0;
    LaneStack st;
    bool done = false;
    while (__any_sync(mask, !done)) {
        if (done) continue;
        bool pop = false;
        if (ref >= 0) {
            float k[kBW];
            int r[kBW];
            bool h[kBW];
            node_keys_ray(bv.nodes, ref, o, inv, big, k, r, 0.f);
#pragma unroll
            for (int c = 0; c < kBW; ++c) h[c] = k[c] <= big;
            if (!take_children(k, r, h, ref, st, err)) pop = true;
        } else {
            int s0 = leaf_start(ref), c = leaf_count(ref);
            for (int s = s0; s < s0 + c; ++s) {
                float t;
                cnt += ray_prim<2>(bv.prims, s, o, v, t) ? 1 : 0;
            }
            pop = true;
        }
        if (pop) done = !st.pop(big, ref);
    }
    return cnt;
}

}  // namespace wost
