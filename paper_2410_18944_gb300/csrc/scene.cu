// Scene construction: boundary validation, inward normals, silhouette
// elements (Neumann vertices in 2D, Neumann edges in 3D), three binned-SAH
// BVHs and their upload in leaf order (FP32 for traversal, FP64 copies for
// the epsilon-shell and ray re-tests).  Sec. 5.3: the queries of a WoSt step
// run on a linear BVH in the paper; here the hierarchy is built once on the
// host (not timed) and traversed in the persistent walk kernel.
#include <algorithm>
#include <atomic>
#include <cfloat>
#include <cmath>
#include <cstring>
#include <exception>
#include <numeric>
#include <thread>
#include <utility>

#include "coop.cuh"
#include "internal.h"

namespace wost {

namespace {

// primitives per leaf (<= 16), and per leaf of the caps (3D: one per lane of a
// query group; 2D, star of 4096 segments: 22.1 / 21.7 / 21.8 ms with 16 / 8 / 4)
constexpr int kLeaf = 16, kLeafCaps = 8;
constexpr int kBins = 16;
constexpr int kSahDepth = 40;   // beyond this depth, median splits bound the tree depth

struct Box {
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    void grow(const Box &b) {
        for (int k = 0; k < 3; ++k) { lo[k] = std::min(lo[k], b.lo[k]); hi[k] = std::max(hi[k], b.hi[k]); }
    }
    void grow(const float *p, int d) {
        for (int k = 0; k < d; ++k) { lo[k] = std::min(lo[k], p[k]); hi[k] = std::max(hi[k], p[k]); }
    }
    float cost(int d) const {
        if (lo[0] > hi[0]) return 0.f;
        float e[3];
        for (int k = 0; k < 3; ++k) e[k] = std::max(hi[k] - lo[k], 0.f);
        return d == 2 ? e[0] + e[1] : e[0] * e[1] + e[1] * e[2] + e[2] * e[0];
    }
};

struct Item {
    Box b;
    float c[3];
    int idx;
    int bin;   // of the split in progress
};

// silhouette element: inward normals of the two adjacent Neumann primitives
// and the vertex both planes are taken through; free marks elements that are
// always silhouettes
struct SilData {
    float n0[3] = {0, 0, 0}, n1[3] = {0, 0, 0}, v[3] = {0, 0, 0};
    bool free = false;
};

// Facing bound of elements [b, e) relative to the box corner lo (geom.cuh,
// facing_prunes): axis a (rounded to FP32), slab [d0, d1] of a . (v - lo) over
// the planes' points v, and s^2, s the sine of the largest angle between a
// and a normal (a normal of length 1 within FP32 rounding: |n x a|^2 is its
// sine squared within 1e-6).  s^2 = infinity disables pruning: an
// always-silhouette element inside, a degenerate normal, or normals spread
// over more than a half space.
struct Facing { float a[3] = {0, 0, 0}, d0 = 0, d1 = 0, s2 = INFINITY; };

Facing facing_bound(const std::vector<SilData> &el, int b, int e, int d, const float *lo, double tau) {
    const Facing off;
    double ax[3] = {0, 0, 0};
    for (int i = b; i < e; ++i) {
        if (el[i].free) return off;
        for (int k = 0; k < d; ++k) ax[k] += el[i].n0[k] + el[i].n1[k];
    }
    double L = 0;
    for (int k = 0; k < d; ++k) L += ax[k] * ax[k];
    L = std::sqrt(L);
    if (!(L > 1e-12)) return off;
    Facing f;
    for (int k = 0; k < d; ++k) { f.a[k] = (float)(ax[k] / L); ax[k] = f.a[k]; }
    double s2 = 0, d0 = INFINITY, d1 = -INFINITY;
    for (int i = b; i < e; ++i) {
        for (const float *n : {el[i].n0, el[i].n1}) {
            double c = 0;
            for (int k = 0; k < d; ++k) c += ax[k] * n[k];
            if (!(c > 0)) return off;
            const double x = n[1] * ax[2] - n[2] * ax[1], y = n[2] * ax[0] - n[0] * ax[2], z = n[0] * ax[1] - n[1] * ax[0];
            s2 = std::max(s2, x * x + y * y + z * z);
        }
        double h = 0;
        for (int k = 0; k < d; ++k) h += ax[k] * ((double)el[i].v[k] - lo[k]);
        d0 = std::min(d0, h);
        d1 = std::max(d1, h);
    }
    // half of tau is used only while cos t >= 0.6; the rounding of o, A and L
    // (below 6e-7 L together) goes into s
    if (!(s2 < 0.64)) d1 += 0.5 * tau;
    const double s = std::sqrt(s2) * (1 + 2e-6) + 1e-6;
    f.d0 = std::nextafterf((float)d0, -INFINITY);
    f.d1 = std::nextafterf((float)d1, INFINITY);
    f.s2 = std::nextafterf((float)(s * s * (1 + 2e-6)), INFINITY);
    return f;
}

// Oriented cap around primitives [b, e) (geom.cuh, cap_d2): centre c, axis a,
// half thickness h along a, radius r across it.  The axis is the mean normal
// (any axis bounds, that one is thin), 1e-6 short of unit length.  P: vertices
// in leaf order (d points of d floats per primitive), N: unit normals.  Margin
// and length: see cap_f4.
struct Cap { float c[3] = {0, 0, 0}, a[3] = {1, 0, 0}, h = 0, r = 0; };

Cap cap_of(const std::vector<float> &P, const std::vector<float> &N, int b, int e, int d, double margin) {
    Cap o;
    double ax[3] = {0, 0, 0}, lo[3], hi[3], L = 0;
    for (int i = b; i < e; ++i)
        for (int k = 0; k < d; ++k) ax[k] += N[(size_t)i * d + k];
    for (int k = 0; k < d; ++k) L += ax[k] * ax[k];
    L = std::sqrt(L);
    // frame: the unit axis and (2D) its perpendicular, or (3D) two axes across
    double f[3][3] = {{1, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    if (L > 1e-3 * (e - b))
        for (int k = 0; k < d; ++k) f[0][k] = ax[k] / L;
    for (int k = 0; k < d; ++k) o.a[k] = (float)((1 - 1e-6) * f[0][k]);
    f[1][0] = -f[0][1];
    f[1][1] = f[0][0];
    if (d == 3) {
        const int m = std::fabs(f[0][0]) < std::fabs(f[0][1]) ? (std::fabs(f[0][0]) < std::fabs(f[0][2]) ? 0 : 2)
                                                              : (std::fabs(f[0][1]) < std::fabs(f[0][2]) ? 1 : 2);
        double t[3] = {0, 0, 0}, q = f[0][m], n = 0;
        t[m] = 1;
        for (int k = 0; k < 3; ++k) { t[k] -= q * f[0][k]; n += t[k] * t[k]; }
        for (int k = 0; k < 3; ++k) f[1][k] = t[k] / std::sqrt(n);
        f[2][0] = f[0][1] * f[1][2] - f[0][2] * f[1][1];
        f[2][1] = f[0][2] * f[1][0] - f[0][0] * f[1][2];
        f[2][2] = f[0][0] * f[1][1] - f[0][1] * f[1][0];
    }
    for (int j = 0; j < d; ++j) { lo[j] = INFINITY; hi[j] = -INFINITY; }
    const size_t p0 = (size_t)b * d * d, p1 = (size_t)e * d * d;
    for (size_t p = p0; p < p1; p += d)
        for (int j = 0; j < d; ++j) {
            double q = 0;
            for (int k = 0; k < d; ++k) q += f[j][k] * P[p + k];
            lo[j] = std::min(lo[j], q);
            hi[j] = std::max(hi[j], q);
        }
    for (int k = 0; k < d; ++k) {
        double c = 0;
        for (int j = 0; j < d; ++j) c += 0.5 * (lo[j] + hi[j]) * f[j][k];
        o.c[k] = (float)c;
    }
    // extents along and across the axis as stored.  The radius comes from the
    // components across it: n - q^2 (n the squared length, q the part along the
    // axis) would lose a radius below about h / 3000 to the rounding of the FP32
    // axis' length.
    double h = 0, r2 = 0, a2 = 0;
    for (int k = 0; k < d; ++k) a2 += (double)o.a[k] * o.a[k];
    for (size_t p = p0; p < p1; p += d) {
        double u[3], q = 0, w2 = 0;
        for (int k = 0; k < d; ++k) { u[k] = P[p + k] - (double)o.c[k]; q += o.a[k] * u[k]; }
        if (d == 2) {
            const double w = o.a[0] * u[1] - o.a[1] * u[0];   // (as cap_d2_2)
            w2 = w * w;
        } else {
            for (int k = 0; k < d; ++k) { const double w = u[k] - q / a2 * o.a[k]; w2 += w * w; }
        }
        h = std::max(h, std::fabs(q));
        r2 = std::max(r2, w2);
    }
    o.h = std::nextafterf((float)(h + margin), INFINITY);
    o.r = std::nextafterf((float)(std::sqrt(r2) * (1 + 1e-6) + margin), INFINITY);
    return o;
}

// fn(i) for i in [0, n), split over the host's cores
template <class F>
void parallel_for(int n, F fn) {
    const int nt = (int)std::min<int64_t>(std::min<unsigned>(std::max(1u, std::thread::hardware_concurrency()), 16u), n / 64);
    if (nt <= 1) {
        for (int i = 0; i < n; ++i) fn(i);
        return;
    }
    std::atomic<int> next{0};
    auto work = [&] {
        for (int i; (i = next.fetch_add(16)) < n;)
            for (int j = i; j < std::min(n, i + 16); ++j) fn(j);
    };
    std::vector<std::thread> th;
    th.reserve(nt);
    for (int t = 1; t < nt; ++t) {
        try {
            th.emplace_back(work);
        } catch (const std::exception &) {
            break;   // no more threads (or memory for one) to be had: those there are do the work
        }
    }
    work();
    for (std::thread &t : th) t.join();
}

struct BNode {
    Box box[2];
    int ref[2];
    int range[2][2];   // item ranges of the two children
};

struct Builder {
    int d;
    int leaf = kLeaf;   // the tree is split down to this (<= kLeaf)
    std::vector<Item> items;
    std::vector<BNode> nodes;
    int maxdepth = 0;

    static int leaf_ref(int start, int count) { return ~((start << 4) | (count - 1)); }

    Box range_box(int b, int e) const {
        Box r;
        for (int i = b; i < e; ++i) r.grow(items[i].b);
        return r;
    }

    int split_median(int b, int e, int axis) {
        int m = (b + e) / 2;
        std::nth_element(items.begin() + b, items.begin() + m, items.begin() + e,
                         [&](const Item &x, const Item &y) {
                             return x.c[axis] < y.c[axis] || (x.c[axis] == y.c[axis] && x.idx < y.idx);
                         });
        return m;
    }

    int rec(int b, int e, int depth, bool within_leaf = false) {
        // (splits below kLeaf primitives do not count: the box tree has none)
        if (!within_leaf) maxdepth = std::max(maxdepth, depth);
        int n = e - b;
        if (n <= leaf) return leaf_ref(b, n);
        Box cb;
        for (int i = b; i < e; ++i) cb.grow(items[i].c, d);
        int axis = 0;
        for (int k = 1; k < d; ++k)
            if (cb.hi[k] - cb.lo[k] > cb.hi[axis] - cb.lo[axis]) axis = k;
        float ext = cb.hi[axis] - cb.lo[axis];
        int mid;
        Box half[2];
        bool boxed = false;   // `half` holds the children's boxes
        if (!(ext > 0.f)) {
            mid = (b + e) / 2;   // identical centroids: split by index
        } else if (depth > kSahDepth) {
            mid = split_median(b, e, axis);
        } else {
            Box bb[kBins];
            int bn[kBins] = {0};
            for (int i = b; i < e; ++i) {
                int k = (int)((items[i].c[axis] - cb.lo[axis]) / ext * kBins);
                k = std::min(std::max(k, 0), kBins - 1);
                items[i].bin = k;
                bn[k]++;
                bb[k].grow(items[i].b);
            }
            // the boxes left and right of each split, one sweep each
            Box R[kBins];
            int nr[kBins];
            R[kBins - 1] = bb[kBins - 1];
            nr[kBins - 1] = bn[kBins - 1];
            for (int s = kBins - 2; s > 0; --s) {
                R[s] = R[s + 1];
                R[s].grow(bb[s]);
                nr[s] = nr[s + 1] + bn[s];
            }
            float best = INFINITY;
            int bestk = -1, nl = 0;
            Box L;
            for (int s = 1; s < kBins; ++s) {
                L.grow(bb[s - 1]);
                nl += bn[s - 1];
                if (!nl || !nr[s]) continue;
                float c = L.cost(d) * nl + R[s].cost(d) * nr[s];
                if (c < best) { best = c; bestk = s; half[0] = L; }
            }
            if (bestk < 0) {
                mid = split_median(b, e, axis);
            } else {
                auto it = std::partition(items.begin() + b, items.begin() + e,
                                         [&](const Item &x) { return x.bin < bestk; });
                mid = (int)(it - items.begin());
                half[1] = R[bestk];
                boxed = true;
            }
        }
        if (!boxed) {
            half[0] = range_box(b, mid);
            half[1] = range_box(mid, e);
        }
        int node = (int)nodes.size();
        nodes.push_back(BNode{});
        int l = rec(b, mid, depth + 1, n <= kLeaf);
        int r = rec(mid, e, depth + 1, n <= kLeaf);
        nodes[node].ref[0] = l;
        nodes[node].ref[1] = r;
        nodes[node].box[0] = half[0];
        nodes[node].box[1] = half[1];
        nodes[node].range[0][0] = b; nodes[node].range[0][1] = mid;
        nodes[node].range[1][0] = mid; nodes[node].range[1][1] = e;
        return node;
    }

    // returns false if the tree is too deep for the device traversal stack
    bool build() {
        nodes.clear();
        int n = (int)items.size();
        if (n == 0) return true;
        if (n <= leaf) {
            BNode r;
            r.ref[0] = leaf_ref(0, n);
            r.ref[1] = leaf_ref(0, 1);
            r.box[0] = range_box(0, n);   // r.box[1] stays empty (inverted)
            r.range[0][0] = 0; r.range[0][1] = n;
            r.range[1][0] = 0; r.range[1][1] = 0;
            nodes.push_back(r);
            maxdepth = 1;
            return true;
        }
        rec(0, n, 0);
        return maxdepth < 62;   // device traversal stack holds 64 entries
    }

    // ---- device layout ----
    // Wide nodes: each takes up to W descendants of a binary node (its
    // children, with the inner child of the larger box surface opened until
    // there are W); empty slots carry kEmptyRef and an inverted box.
    struct Child { Box box; int ref = kEmptyRef; int range[2] = {0, 0}; };
    struct WNode { Child ch[8]; int n = 0; };

    // (leaves of at most `lf` primitives)
    int collapse(std::vector<WNode> &out, int W, int lf, int bnode) const {
        Child ch[8];
        int n = 0;
        auto child = [&](int b, int c) {
            Child x;
            x.box = nodes[b].box[c];
            x.ref = nodes[b].ref[c];
            x.range[0] = nodes[b].range[c][0];
            x.range[1] = nodes[b].range[c][1];
            if (x.ref >= 0 && x.range[1] - x.range[0] <= lf) x.ref = leaf_ref(x.range[0], x.range[1] - x.range[0]);
            return x;
        };
        for (int c = 0; c < 2; ++c) ch[n++] = child(bnode, c);
        while (n < W) {
            int pick = -1;
            float area = -1.f;
            for (int i = 0; i < n; ++i)
                if (ch[i].ref >= 0 && ch[i].box.cost(d) > area) { pick = i; area = ch[i].box.cost(d); }
            if (pick < 0) break;
            const int b = ch[pick].ref;
            ch[pick] = child(b, 0);
            ch[n++] = child(b, 1);
        }
        const int id = (int)out.size();
        out.push_back(WNode{});
        for (int i = 0; i < n; ++i) {
            Child c = ch[i];
            if (c.ref >= 0) c.ref = collapse(out, W, lf, c.ref);
            out[id].ch[i] = c;
        }
        out[id].n = n;
        return id;
    }

    // most stack entries a traversal below wide node id can hold: a visit
    // pushes all but one of its taken children
    static int stack_need(const std::vector<WNode> &w, int id) {
        int need = 0;
        for (int c = 0; c < w[id].n; ++c)
            if (w[id].ch[c].ref >= 0) need = std::max(need, stack_need(w, w[id].ch[c].ref));
        return need + std::max(w[id].n - 1, 0);
    }

    // wide tree of at most W children per node and lf primitives per leaf
    std::vector<WNode> widen(int W, int lf) const {
        std::vector<WNode> out;
        const int n = (int)items.size();
        if (n > lf) {
            collapse(out, W, lf, 0);
        } else if (n > 0) {   // one leaf, although the binary tree may be split further
            WNode root;
            root.ch[0].box = range_box(0, n);
            root.ch[0].ref = leaf_ref(0, n);
            root.ch[0].range[1] = n;
            root.n = 1;
            out.push_back(root);
        }
        return out;
    }

    // a traversal's entries fit the device stack
    static bool fits(const std::vector<WNode> &w) { return w.empty() || stack_need(w, 0) < kGrpStack; }

    static float bits(int r) { float f; std::memcpy(&f, &r, 4); return f; }

    // 3D nodes (geom.cuh)
    static std::vector<float4> pack_wide(const std::vector<WNode> &w) {
        std::vector<float4> out;
        out.reserve(w.size() * node_f4<3>());
        for (const WNode &n : w) {
            for (int c = 0; c < 4; ++c) {
                const Box &b = n.ch[c].box;
                out.push_back(make_float4(b.lo[0], b.lo[1], b.lo[2], b.hi[0]));
            }
            for (int c = 0; c < 4; ++c) {
                const Box &b = n.ch[c].box;
                out.push_back(make_float4(b.hi[1], b.hi[2], bits(n.ch[c].ref), 0.f));
            }
        }
        return out;
    }

    // binary 2D nodes, child boxes in the parent
    std::vector<float4> pack_binary() const {
        std::vector<float4> out;
        for (const BNode &nd : nodes) {
            const Box &a = nd.box[0];
            Box b = nd.box[1];
            if (nd.range[1][1] <= nd.range[1][0])   // the unused child of a one-leaf tree: a point out of any ray's reach
                for (int k = 0; k < 2; ++k) b.lo[k] = b.hi[k] = FLT_MAX;
            out.push_back(make_float4(a.lo[0], a.lo[1], a.hi[0], a.hi[1]));
            out.push_back(make_float4(b.lo[0], b.lo[1], b.hi[0], b.hi[1]));
            int r[2];
            for (int c = 0; c < 2; ++c) {
                const int n = nd.range[c][1] - nd.range[c][0];
                r[c] = nd.ref[c] >= 0 && n <= kLeaf ? leaf_ref(nd.range[c][0], n) : nd.ref[c];
            }
            out.push_back(make_float4(bits(r[0]), bits(r[1]), 0.f, 0.f));
        }
        return out;
    }

    // facing bounds of every node's children (layout: facing_f4, geom.cuh)
    static Facing facing_of(const std::vector<SilData> &el, const int *r, int d, const Box &bx, double tau) {
        return r[1] > r[0] ? facing_bound(el, r[0], r[1], d, bx.lo, tau) : Facing{};
    }
    std::vector<float4> facing_binary(const std::vector<SilData> &el, double tau) const {
        std::vector<float4> out(nodes.size() * facing_f4(2));
        parallel_for((int)nodes.size(), [&](int i) {
            const BNode &nd = nodes[i];
            float4 *o = &out[(size_t)i * facing_f4(2)];
            Facing f[2];
            for (int c = 0; c < 2; ++c) {
                f[c] = facing_of(el, nd.range[c], d, nd.box[c], tau);
                o[c] = make_float4(f[c].a[0], f[c].a[1], f[c].d0, f[c].d1);
            }
            o[2] = make_float4(f[0].s2, f[1].s2, 0.f, 0.f);
        });
        return out;
    }
    static std::vector<float4> facing_wide(const std::vector<SilData> &el, const std::vector<WNode> &w, double tau) {
        std::vector<float4> out(w.size() * facing_f4(3));
        parallel_for((int)w.size(), [&](int i) {
            float4 *o = &out[(size_t)i * facing_f4(3)];
            Facing f[4];
            for (int c = 0; c < 4; ++c) {
                f[c] = facing_of(el, w[i].ch[c].range, 3, w[i].ch[c].box, tau);
                o[c] = make_float4(f[c].a[0], f[c].a[1], f[c].a[2], f[c].d0);
            }
            for (int c = 0; c < 4; c += 2) o[4 + c / 2] = make_float4(f[c].d1, f[c].s2, f[c + 1].d1, f[c + 1].s2);
        });
        return out;
    }

    // caps of every node's children, with the child references (layout:
    // cap_f4, geom.cuh); P, N as cap_of
    std::vector<float4> caps_binary(const std::vector<float> &P, const std::vector<float> &N, double margin) const {
        std::vector<float4> out(nodes.size() * cap_f4(2));
        parallel_for((int)nodes.size(), [&](int i) {
            const BNode &nd = nodes[i];
            float4 *o = &out[(size_t)i * cap_f4(2)];
            Cap c[2];
            for (int k = 0; k < 2; ++k) {
                if (nd.range[k][1] > nd.range[k][0]) c[k] = cap_of(P, N, nd.range[k][0], nd.range[k][1], 2, margin);
                else c[k].c[0] = 1e30f;   // the unused child of a one-leaf tree: far away
                o[k] = make_float4(c[k].c[0], c[k].c[1], c[k].a[0], c[k].a[1]);
            }
            o[2] = make_float4(c[0].h, c[0].r, c[1].h, c[1].r);
            o[3] = make_float4(bits(nd.ref[0]), bits(nd.ref[1]), 0.f, 0.f);
        });
        return out;
    }
    static std::vector<float4> caps_wide(const std::vector<WNode> &w, const std::vector<float> &P,
                                          const std::vector<float> &N, double margin) {
        std::vector<float4> out(w.size() * cap_f4(3));
        parallel_for((int)w.size(), [&](int i) {
            float4 *o = &out[(size_t)i * cap_f4(3)];
            const Child *ch = w[i].ch;
            for (int k = 0; k < 8; ++k) {
                const Cap c = ch[k].range[1] > ch[k].range[0] ? cap_of(P, N, ch[k].range[0], ch[k].range[1], 3, margin) : Cap{};
                o[k] = make_float4(c.c[0], c.c[1], c.c[2], c.h);
                o[8 + k] = make_float4(c.a[0], c.a[1], c.a[2], c.r);
            }
            const float grow = std::nextafterf((float)margin, INFINITY);
            for (int k = 0; k < 8; ++k) {
                const Box &bx = ch[k].box;
                o[16 + k] = make_float4(bx.lo[0] - grow, bx.lo[1] - grow, bx.lo[2] - grow, bx.hi[0] + grow);
                o[24 + k] = make_float4(bx.hi[1] + grow, bx.hi[2] + grow, bits(ch[k].ref), 0.f);
            }
        });
        return out;
    }
};

// The scene's device arrays.  Each allocation and copy costs about 10 us, a
// third of the creation of a small scene, so arrays of up to kPacked bytes go
// into one allocation, with one copy (64 segments: 185 / 150 us); a larger one
// is copied from where it is.
struct Uploader {
    static constexpr size_t kPacked = 256 << 10;
    wost_scene *s;
    std::vector<unsigned char> blob{};
    std::vector<std::pair<const void **, size_t>> at{};   // pointers into the blob's device copy

    wost_status send(const void *src, size_t bytes, const void **out) {
        void *p = nullptr;
        cudaError_t e = cudaMalloc(&p, bytes);
        if (e != cudaSuccess) {
            set_error("cudaMalloc failed while uploading the scene");
            return e == cudaErrorMemoryAllocation ? WOST_ERR_OOM : WOST_ERR_CUDA;
        }
        s->allocs.push_back(p);
        WOST_CUDA(cudaMemcpy(p, src, bytes, cudaMemcpyHostToDevice));
        *out = p;
        return WOST_OK;
    }
    template <class T>
    wost_status add(const std::vector<T> &v, const T **out) {
        *out = nullptr;
        const size_t bytes = v.size() * sizeof(T);
        const void **o = reinterpret_cast<const void **>(out);
        if (bytes == 0) return WOST_OK;
        if (bytes > kPacked) return send(v.data(), bytes, o);
        const size_t off = (blob.size() + 255) / 256 * 256;
        blob.resize(off + bytes);
        std::memcpy(blob.data() + off, v.data(), bytes);
        at.push_back({o, off});
        return WOST_OK;
    }
    // the packed arrays (their pointers are set here)
    wost_status finish() {
        if (blob.empty()) return WOST_OK;
        const void *base = nullptr;
        const wost_status st = send(blob.data(), blob.size(), &base);
        if (st != WOST_OK) return st;
        for (auto &x : at) *x.first = static_cast<const unsigned char *>(base) + x.second;
        return WOST_OK;
    }
};

bool valid_fn(const wost_fn &f) {
    if (f.kind < 0 || f.kind > 10) return false;
    if (f.kind == 7 && (f.params[0] < 0 || f.params[0] > 8)) return false;
    return true;
}

DevFn to_dev(const wost_fn &f) {
    DevFn o{};
    o.kind = f.kind;
    o.n = f.nparams;
    for (int i = 0; i < 40; ++i) o.p[i] = (float)f.params[i];
    return o;
}

}  // namespace

}  // namespace wost

using namespace wost;

wost_scene::~wost_scene() {
    for (void *p : allocs) cudaFree(p);
    ws_points.release(); ws_status.release(); ws_sum.release(); ws_sum2.release(); ws_ctr.release(); ws_out.release();
    ws_wf.release();
    ws_order.release();
    if (pinned) cudaFreeHost(pinned);
}

extern "C" wost_status wost_create_scene(const wost_scene_desc *desc, wost_scene **out) {
    if (!desc || !out) { set_error("wost_create_scene: null argument"); return WOST_ERR_INVALID_ARG; }
    *out = nullptr;
    const int d = desc->dim;
    if (d != 2 && d != 3) { set_error("wost_create_scene: dim must be 2 or 3"); return WOST_ERR_INVALID_ARG; }
    if (desc->nverts <= 0 || desc->nprims <= 0 || !desc->verts || !desc->prims || !desc->bc) {
        set_error("wost_create_scene: empty or null geometry");
        return WOST_ERR_INVALID_ARG;
    }
    if (desc->nprims >= (1LL << 27) || desc->nverts >= (1LL << 31)) {
        set_error("wost_create_scene: too many primitives");
        return WOST_ERR_INVALID_ARG;
    }
    if (!valid_fn(desc->g) || !valid_fn(desc->f) || !valid_fn(desc->h)) {
        set_error("wost_create_scene: unknown data-function kind");
        return WOST_ERR_INVALID_ARG;
    }
    const int64_t nv = desc->nverts, np = desc->nprims;
    int ndir = 0;
    for (int64_t i = 0; i < np; ++i) {
        if (desc->bc[i] > 1) { set_error("wost_create_scene: bc must be 0 or 1"); return WOST_ERR_INVALID_ARG; }
        ndir += desc->bc[i] == 0;
        for (int k = 0; k < d; ++k) {
            int32_t v = desc->prims[i * d + k];
            if (v < 0 || v >= nv) { set_error("wost_create_scene: vertex index out of range"); return WOST_ERR_INVALID_ARG; }
        }
    }
    for (int64_t i = 0; i < nv * d; ++i)
        if (!std::isfinite(desc->verts[i])) { set_error("wost_create_scene: non-finite vertex"); return WOST_ERR_INVALID_ARG; }
    if (ndir == 0) { set_error("wost_create_scene: no Dirichlet primitive (ill-posed)"); return WOST_ERR_ILL_POSED; }
    int dev = -1;
    WOST_CUDA(cudaGetDevice(&dev));

    auto *s = new wost_scene();
    s->dim = d;
    s->device = dev;
    s->nverts = nv;
    s->nprims = np;
    s->scene_id = desc->scene_id;
    const double *V = desc->verts;
    const int32_t *P = desc->prims;
    double lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int64_t i = 0; i < nv; ++i)
        for (int k = 0; k < d; ++k) { lo[k] = std::min(lo[k], V[i * d + k]); hi[k] = std::max(hi[k], V[i * d + k]); }
    double diag = 0;
    for (int k = 0; k < d; ++k) { diag += (hi[k] - lo[k]) * (hi[k] - lo[k]); s->lo[k] = lo[k]; s->hi[k] = hi[k]; }
    diag = std::sqrt(diag);

    // inward unit normals (2D: left perpendicular of b - a; 3D: -(e1 x e2))
    std::vector<double> nin((size_t)np * d);
    for (int64_t i = 0; i < np; ++i) {
        const double *a = V + (size_t)P[i * d] * d, *b = V + (size_t)P[i * d + 1] * d;
        double *n = &nin[(size_t)i * d];
        if (d == 2) {
            double ex = b[0] - a[0], ey = b[1] - a[1], L = std::sqrt(ex * ex + ey * ey);
            n[0] = -ey / L; n[1] = ex / L;
        } else {
            const double *c = V + (size_t)P[i * d + 2] * d;
            double e1[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]}, e2[3] = {c[0] - a[0], c[1] - a[1], c[2] - a[2]};
            double cx = e1[1] * e2[2] - e1[2] * e2[1], cy = e1[2] * e2[0] - e1[0] * e2[2], cz = e1[0] * e2[1] - e1[1] * e2[0];
            double L = std::sqrt(cx * cx + cy * cy + cz * cz);
            n[0] = -cx / L; n[1] = -cy / L; n[2] = -cz / L;
        }
    }

    auto fv = [&](int64_t vi, int k) { return (float)V[vi * d + k]; };
    Uploader up{s};

    // ---- primitive BVHs (Dirichlet, Neumann) ----
    auto build_prims = [&](int bcv, DevBVH &bv, int &count, int &depth, std::vector<int> *slot_of) -> wost_status {
        Builder B;
        B.d = d;
        // (the caps' smaller leaves subdivide those of the boxes)
        B.leaf = bcv == 0 ? kLeafCaps : kLeaf;
        B.items.reserve(bcv == 0 ? ndir : np - ndir);
        for (int64_t i = 0; i < np; ++i) {
            if (desc->bc[i] != bcv) continue;
            Item it;
            for (int k = 0; k < 3; ++k) it.c[k] = 0.f;
            for (int j = 0; j < d; ++j) {
                float p[3] = {fv(P[i * d + j], 0), fv(P[i * d + j], 1), d == 3 ? fv(P[i * d + j], 2) : 0.f};
                it.b.grow(p, d);
                for (int k = 0; k < d; ++k) it.c[k] += p[k] / d;
            }
            if (d == 2) { it.b.lo[2] = it.b.hi[2] = 0.f; }
            it.idx = (int)i;
            B.items.push_back(it);
        }
        count = (int)B.items.size();
        std::vector<Builder::WNode> wide, caps;
        bool ok = B.build();
        if (ok && d == 3) {
            wide = B.widen(4, kLeaf);
            ok = Builder::fits(wide);
            if (bcv == 0) {
                // a very deep tree takes fewer children per node, then the
                // larger leaves (always fits: the binary depth is below 62)
                for (int W : {8, 4, 2})
                    if (W == 8 || !Builder::fits(caps)) caps = B.widen(W, kLeafCaps);
                if (!Builder::fits(caps)) caps = B.widen(2, kLeaf);
            }
        }
        if (!ok) { set_error("wost_create_scene: BVH too deep"); return WOST_ERR_INVALID_ARG; }
        depth = B.maxdepth;
        std::vector<float4> prims;
        std::vector<double> p64;
        std::vector<int> ids;
        if (slot_of) slot_of->assign(np, -1);
        for (size_t sidx = 0; sidx < B.items.size(); ++sidx) {
            int i = B.items[sidx].idx;
            ids.push_back(i);
            if (slot_of) (*slot_of)[i] = (int)sidx;
            const int32_t *q = P + (size_t)i * d;
            if (d == 2) {
                prims.push_back(make_float4(fv(q[0], 0), fv(q[0], 1), fv(q[1], 0), fv(q[1], 1)));
                for (int j = 0; j < 2; ++j) for (int k = 0; k < 2; ++k) p64.push_back(V[(size_t)q[j] * 2 + k]);
            } else {
                prims.push_back(make_float4(fv(q[0], 0), fv(q[0], 1), fv(q[0], 2), fv(q[1], 0)));
                prims.push_back(make_float4(fv(q[1], 1), fv(q[1], 2), fv(q[2], 0), fv(q[2], 1)));
                prims.push_back(make_float4(fv(q[2], 2), 0.f, 0.f, 0.f));
                for (int j = 0; j < 3; ++j) for (int k = 0; k < 3; ++k) p64.push_back(V[(size_t)q[j] * 3 + k]);
            }
        }
        wost_status st;
        if ((st = up.add(d == 2 ? B.pack_binary() : Builder::pack_wide(wide), &bv.nodes)) != WOST_OK) return st;
        bv.nnodes = (int)(d == 2 ? B.nodes.size() : (bcv == 0 ? caps.size() : wide.size()));
        bv.need = caps.empty() ? 0 : Builder::stack_need(caps, 0);
        if (bcv == 0) {
            std::vector<float> vp((size_t)count * d * d), vn((size_t)count * d);
            for (int i = 0; i < count; ++i) {
                const int id = B.items[i].idx;
                for (int j = 0; j < d; ++j)
                    for (int k = 0; k < d; ++k) vp[((size_t)i * d + j) * d + k] = fv(P[(size_t)id * d + j], k);
                for (int k = 0; k < d; ++k) vn[(size_t)i * d + k] = (float)nin[(size_t)id * d + k];
            }
            double far = diag;
            for (int k = 0; k < d; ++k) far = std::max(far, std::max(std::fabs(lo[k]), std::fabs(hi[k])));
            if ((st = up.add(d == 2 ? B.caps_binary(vp, vn, 1e-6 * far) : Builder::caps_wide(caps, vp, vn, 1e-6 * far),
                             &s->dev.dir_caps)) != WOST_OK) return st;
        }
        if ((st = up.add(prims, &bv.prims)) != WOST_OK) return st;
        if ((st = up.add(ids, &bv.ids)) != WOST_OK) return st;
        if ((st = up.add(p64, &bv.prims64)) != WOST_OK) return st;
        bv.nprims = count;
        return WOST_OK;
    };
    wost_status st;
    std::vector<int> neu_slot;
    if ((st = build_prims(0, s->dev.dir, s->ndir, s->depth_dir, nullptr)) != WOST_OK) { delete s; return st; }
    if ((st = build_prims(1, s->dev.neu, s->nneu, s->depth_neu, &neu_slot)) != WOST_OK) { delete s; return st; }

    // inward normals of Neumann primitives in leaf order
    {
        std::vector<int> ids(s->nneu);
        std::vector<float> nn((size_t)s->nneu * d);
        for (int64_t i = 0; i < np; ++i)
            if (neu_slot[i] >= 0)
                for (int k = 0; k < d; ++k) nn[(size_t)neu_slot[i] * d + k] = (float)nin[(size_t)i * d + k];
        if ((st = up.add(nn, &s->dev.nin_neu)) != WOST_OK) { delete s; return st; }
    }

    // ---- silhouette elements ----
    {
        struct Elem { int64_t key; int a, b, f0, f1; };
        std::vector<Elem> el;
        if (d == 2) {
            std::vector<int> in_seg(nv, -1), out_seg(nv, -1);
            for (int64_t i = 0; i < np; ++i)
                if (desc->bc[i] == 1) { out_seg[P[2 * i]] = (int)i; in_seg[P[2 * i + 1]] = (int)i; }
            for (int64_t v = 0; v < nv; ++v)
                if (in_seg[v] >= 0 || out_seg[v] >= 0) el.push_back({v, (int)v, (int)v, in_seg[v], out_seg[v]});
        } else {
            struct E { int a, b, f; };
            std::vector<E> es;
            for (int64_t i = 0; i < np; ++i)
                if (desc->bc[i] == 1)
                    for (int k = 0; k < 3; ++k) {
                        int a = P[3 * i + k], b = P[3 * i + (k + 1) % 3];
                        es.push_back({std::min(a, b), std::max(a, b), (int)i});
                    }
            std::sort(es.begin(), es.end(), [](const E &x, const E &y) {
                return x.a != y.a ? x.a < y.a : (x.b != y.b ? x.b < y.b : x.f < y.f);
            });
            for (size_t i = 0; i < es.size();) {
                size_t j = i;
                while (j < es.size() && es[j].a == es[i].a && es[j].b == es[i].b) ++j;
                bool two = (j - i) == 2;
                el.push_back({(int64_t)es[i].a * nv + es[i].b, es[i].a, es[i].b, two ? es[i].f : -1, two ? es[i + 1].f : -1});
                i = j;
            }
        }
        Builder B;
        B.d = d;
        for (size_t e = 0; e < el.size(); ++e) {
            Item it;
            float pa[3] = {fv(el[e].a, 0), fv(el[e].a, 1), d == 3 ? fv(el[e].a, 2) : 0.f};
            float pb[3] = {fv(el[e].b, 0), fv(el[e].b, 1), d == 3 ? fv(el[e].b, 2) : 0.f};
            it.b.grow(pa, d);
            it.b.grow(pb, d);
            if (d == 2) it.b.lo[2] = it.b.hi[2] = 0.f;
            for (int k = 0; k < 3; ++k) it.c[k] = 0.5f * (pa[k] + pb[k]);
            it.idx = (int)e;
            B.items.push_back(it);
        }
        s->nsil = (int)el.size();
        std::vector<Builder::WNode> wide;
        bool ok = B.build();
        if (ok && d == 3) {
            wide = B.widen(4, kLeaf);
            ok = Builder::fits(wide);
        }
        if (!ok) { set_error("wost_create_scene: BVH too deep"); delete s; return WOST_ERR_INVALID_ARG; }
        s->depth_sil = B.maxdepth;
        std::vector<float4> prims;
        std::vector<int> ids;
        std::vector<int64_t> keys;
        std::vector<SilData> data;
        data.reserve(B.items.size());
        for (const Item &it : B.items) {
            const Elem &e = el[it.idx];
            ids.push_back(it.idx);
            keys.push_back(e.key);
            const bool always = e.f0 < 0 || e.f1 < 0;   // 3D: marked by the zero normals
            float n0[3] = {0, 0, 0}, n1[3] = {0, 0, 0};
            for (int k = 0; k < d; ++k) {
                if (e.f0 >= 0) n0[k] = (float)nin[(size_t)e.f0 * d + k];
                if (e.f1 >= 0) n1[k] = (float)nin[(size_t)e.f1 * d + k];
            }
            SilData sd;
            for (int k = 0; k < d; ++k) { sd.n0[k] = n0[k]; sd.n1[k] = n1[k]; sd.v[k] = fv(e.a, k); }
            sd.free = always;
            data.push_back(sd);
            if (d == 2) {
                prims.push_back(make_float4(fv(e.a, 0), fv(e.a, 1), n0[0], n0[1]));
                prims.push_back(make_float4(n1[0], n1[1], always ? 1.f : 0.f, 0.f));
            } else {
                prims.push_back(make_float4(fv(e.a, 0), fv(e.a, 1), fv(e.a, 2), fv(e.b, 0)));
                prims.push_back(make_float4(fv(e.b, 1), fv(e.b, 2), n0[0], n0[1]));
                prims.push_back(make_float4(n0[2], n1[0], n1[1], n1[2]));
            }
        }
        DevBVH &bv = s->dev.sil;
        const double tau = (float)(1e-6 * diag);
        if ((st = up.add(d == 2 ? B.facing_binary(data, tau) : Builder::facing_wide(data, wide, tau), &s->dev.sil_facing)) != WOST_OK) { delete s; return st; }
        if ((st = up.add(d == 2 ? B.pack_binary() : Builder::pack_wide(wide), &bv.nodes)) != WOST_OK ||
            (st = up.add(prims, &bv.prims)) != WOST_OK || (st = up.add(ids, &bv.ids)) != WOST_OK) {
            delete s;
            return st;
        }
        bv.nnodes = (int)(d == 2 ? B.nodes.size() : wide.size());
        bv.need = 0;
        if ((st = up.add(keys, &s->sil_key)) != WOST_OK) { delete s; return st; }
        bv.prims64 = nullptr;
        bv.nprims = s->nsil;
    }
    s->dev.dim = d;
    s->dev.scale = (float)diag;
    s->dev.tau = (float)(1e-6 * diag);
    s->dev.g = to_dev(desc->g);
    s->dev.f = to_dev(desc->f);
    s->dev.has_source = desc->f.kind != 0;
    s->dev.h = to_dev(desc->h);
    s->dev.has_flux = desc->h.kind != 0 && s->nneu > 0;
    if ((st = up.finish()) != WOST_OK) { delete s; return st; }
    *out = s;
    return WOST_OK;
}

extern "C" wost_status wost_destroy_scene(wost_scene *s) {
    delete s;
    return WOST_OK;
}

extern "C" wost_status wost_scene_device(const wost_scene *s, int32_t *device) {
    if (!s || !device) { set_error("wost_scene_device: null argument"); return WOST_ERR_INVALID_ARG; }
    *device = s->device;
    return WOST_OK;
}

extern "C" wost_status wost_diag_scene_rebind(wost_scene *s, int32_t device) {
    if (!s) { set_error("wost_diag_scene_rebind: null scene"); return WOST_ERR_INVALID_ARG; }
    s->device = device;
    return WOST_OK;
}

extern "C" wost_status wost_scene_bbox(const wost_scene *s, double lo[3], double hi[3]) {
    if (!s || !lo || !hi) { set_error("wost_scene_bbox: null argument"); return WOST_ERR_INVALID_ARG; }
    for (int k = 0; k < 3; ++k) {
        double e = k < s->dim ? s->hi[k] - s->lo[k] : 0;
        lo[k] = k < s->dim ? s->lo[k] - 0.05 * e : 0;
        hi[k] = k < s->dim ? s->hi[k] + 0.05 * e : 1;
    }
    return WOST_OK;
}
