// One walk-on-stars step, shared by the plain and the guided persistent
// kernels (Sec. 3.2 Eq. wost_estm, reparameterised as in Sec. 4.1):
//   1. closest Dirichlet point; stop inside the epsilon-shell (FP64 re-test)
//      or at the step cap, adding T g(xbar) to the point's FP64 sums;
//   2. star radius r = max(min(R_D, R_S), eps) from the closest silhouette;
//   0. Russian roulette from step rr_depth on (after the epsilon-shell test):
//      go on with probability q (throughput / q), else end with value 0;
//   3. source term -(r^2 / 2d) f(y), y ~ Green-function density, if visible,
//      and the Neumann term -<N> when the flux is nonzero;
//   4. (caller) direction nu and step weight;
//   5. first Neumann hit within r (FP64 re-test of the winner) or x + r nu.
// Random numbers: Philox4x32-10, counter (point, walk, step, purpose).
#pragma once
#include "coop.cuh"

namespace wost {

struct WalkArgs {
    DevScene sc;
    const double *points;      // npoints * D
    const uint8_t *status;     // 0 walk, 1 shell, 2 outside
    int64_t npoints;
    int walk_begin;
    unsigned long long total;  // work items = npoints * walks in this launch
    unsigned long long *work_ctr;
    double *sum, *sum2;
    float eps;
    double eps64;
    int maxsteps;
    uint32_t key0, key1;
    unsigned long long *stat;  // [0] walk-steps, [1] truncated, [2] walks, [3..6] node/Dirichlet/silhouette/Neumann visits
    int *err;
    int rr_depth;              // Russian roulette from this step on (0 = off)
    float rr_q;                // survival probability of a roulette step
    // single-scene guided launches only (nullptr elsewhere): the order in
    // which a launch hands out the points of each walk index (a
    // permutation of [0, npoints)), and per point the walk-steps its walks
    // take in this launch
    const uint32_t *order;
    unsigned *plen;
    int lanes;                 // plain walks: plain_lanes
};

// what one step needs besides the walk state: the walk's scene and the
// solve's scalars (scene and keys differ per job in a multi-scene batch)
struct StepEnv {
    const DevScene &sc;
    float eps;
    double eps64;
    int maxsteps;
    uint32_t key0, key1;
    int *err;
    int rr_depth;
    float rr_q;
};

__device__ __forceinline__ StepEnv env_of(const WalkArgs &a) {
    return StepEnv{a.sc, a.eps, a.eps64, a.maxsteps, a.key0, a.key1, a.err, a.rr_depth, a.rr_q};
}

// Russian roulette (Sec. 6.1 enables it beyond 128 steps; the survival rule
// is a reading: a fixed probability q).  A step k >= rr_depth that survives
// divides the throughput by q, and for the suffix pass its weight and
// non-recursive terms carry the same 1 / q: roulette_scale(k).
__device__ __forceinline__ bool roulette_on(const StepEnv &a, int k) { return a.rr_depth > 0 && k >= a.rr_depth; }
__device__ __forceinline__ float roulette_scale(const StepEnv &a, int k) {
    return roulette_on(a, k) ? 1.f / a.rr_q : 1.f;
}
// the step's roulette draw (counter purpose P_RR): true if the walk goes on
__device__ __forceinline__ bool roulette_survives(const StepEnv &a, uint32_t pid, uint32_t wid, int k) {
    U4 u = philox(pid, wid, (uint32_t)k, P_RR, a.key0, a.key1);
    return u01(u.x) < a.rr_q;
}

template <int D>
struct Walk {
    float x[D], n[D];
    float T, acc;
    uint32_t pid, wid;
    int k, prim;     // prim: Neumann leaf slot the walker stands on, -1 if interior
    int job;         // job of a multi-scene batch (unused by single solves)
};

template <int D>
__device__ __forceinline__ void uniform_dir(float u0, float u1, float *v) {
    if (D == 2) {
        float s, c;
        sincospif(2.f * u0, &s, &c);
        v[0] = c;
        v[1] = s;
    } else {
        float z = 1.f - 2.f * u0, s, c;
        float st = sqrtf(fmaxf(0.f, 1.f - z * z));
        sincospif(2.f * u1, &s, &c);
        v[0] = st * c;
        v[1] = st * s;
        v[2] = z;
    }
}

template <int D>
__device__ __forceinline__ float dotv(const float *a, const float *b) {
    float s = a[0] * b[0] + a[1] * b[1];
    if (D == 3) s += a[2] * b[2];
    return s;
}

template <int D>
__device__ __forceinline__ void reflect(float *v, const float *n) {
    float t = 2.f * dotv<D>(v, n);
#pragma unroll
    for (int i = 0; i < D; ++i) v[i] -= t * n[i];
}

// Beta(2,2) by inversion of F(s) = 3 s^2 - 2 s^3 (trigonometric root)
__device__ __forceinline__ float beta22_inv(float u) {
    return 0.5f + cosf((acosf(1.f - 2.f * u) + 4.f * WOST_PI) / 3.f);
}

template <int D>
__device__ __forceinline__ void start_walk(Walk<D> &w, const WalkArgs &a, unsigned long long item) {
    w.pid = (uint32_t)(item % (unsigned long long)a.npoints);
    w.wid = (uint32_t)(a.walk_begin + item / (unsigned long long)a.npoints);
#pragma unroll
    for (int i = 0; i < D; ++i) { w.x[i] = (float)a.points[(size_t)w.pid * D + i]; w.n[i] = 0.f; }
    w.T = 1.f;
    w.acc = 0.f;
    w.k = 0;
    w.prim = -1;
}

__device__ __forceinline__ void finish_walk(const WalkArgs &a, uint32_t pid, float value) {
    atomicAdd(a.sum + pid, (double)value);
    atomicAdd(a.sum2 + pid, (double)value * (double)value);
}

// Neumann contribution <N> of a step (Sec. 3.2, Eq. wost_estm), entering the
// estimate with a minus sign: z on the Neumann boundary inside B(x, r) with
// density 1 / W (neumann_pick, then uniform on the chosen primitive), counted
// when it faces x (inside B there is no silhouette, so every Neumann point
// there that faces x is on the star's boundary).
//   <N> = G(x, z) h(z) W / alpha,  G = ln(r / |z - x|) / 2 pi  (2D),
//                                      (1 / |z - x| - 1 / r) / 4 pi  (3D),
// h the flux along the normal into the domain, alpha = 1/2 on a Neumann point.
// Lanes with `act` (3D: the whole warp calls).
template <int D, int kMode>
__device__ __forceinline__ float neumann_term(CoopWarp *sh, const Walk<D> &w, const DevScene &sc, bool act, float r,
                                              uint32_t k0, uint32_t k1, int *err, volatile Visits *vis) {
    float W;
    int js;
    if constexpr (D == 2) {
        js = neumann_pick(sc.neu, w.x, r, w.pid, w.wid, (uint32_t)w.k, k0, k1, W, err, vis);
    } else {
        const float ctr[3] = {__uint_as_float(w.pid), __uint_as_float(w.wid), __int_as_float(w.k)};
        W = r * r;
        js = coop_run<kCoopPick, kMode>(*sh, sc, act, w.x, ctr, W, (int)k0, err, vis, k1);
    }
    if (js < 0) return 0.f;
    U4 u = philox(w.pid, w.wid, (uint32_t)w.k, P_NEU, k0, k1);
    const float u0 = u01(u.x), u1 = u01(u.y);
    float z[3];
    if (D == 2) {
        const float4 p = ldn(sc.neu.prims + js);
        z[0] = (1.f - u0) * p.x + u0 * p.z;
        z[1] = (1.f - u0) * p.y + u0 * p.w;
    } else {
        float a[3], b[3], c[3];
        load_tri(sc.neu.prims, js, a, b, c);
        const float su = sqrtf(u0);
#pragma unroll
        for (int i = 0; i < 3; ++i) z[i] = (1.f - su) * a[i] + su * (1.f - u1) * b[i] + su * u1 * c[i];
    }
    float dz[D], dd2 = 0.f, facing = 0.f;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        dz[i] = z[i] - w.x[i];
        dd2 += dz[i] * dz[i];
        facing += dz[i] * __ldg(sc.nin_neu + (size_t)js * D + i);   // normals by leaf slot
    }
    const float dd = sqrtf(dd2);
    if (!(dd > 0.f) || !(dd < r) || !(facing < 0.f)) return 0.f;
    const float G = D == 2 ? logf(r / dd) * (0.5f / WOST_PI) : (1.f / dd - 1.f / r) * (0.25f / WOST_PI);
    return G * eval_fn<D>(sc.h, z) * W * (w.prim >= 0 ? 2.f : 1.f);
}

// The queries of a step: per lane in 2D (called by the lanes that want one),
// by groups of lanes in 3D (called by the whole warp).  kMode: coop.cuh.
template <int D, int kMode>
__device__ __forceinline__ int query_dirichlet(CoopWarp *sh, const DevScene &sc, bool want, const float *x, float &d2,
                                               int *err, volatile Visits *vis) {
    if constexpr (D == 2) {
        return closest_dirichlet(sc.dir, sc.dir_caps, x, d2, err, vis);
    } else {
        return coop_closest<kMode>(*sh, sc, want, x, d2, err, vis);
    }
}

template <int D, int kMode>
__device__ __forceinline__ int query_silhouette(CoopWarp *sh, const DevScene &sc, bool want, const float *x, float &d2,
                                                 int *err, volatile Visits *vis) {
    if constexpr (D == 2) return closest_silhouette(sc.sil, x, sc.tau, d2, err, sc.sil_facing, vis);
    else return coop_run<kCoopSil, kMode>(*sh, sc, want, x, x, d2, -1, err, vis);
}

// first exit through the Neumann boundary within tmax, re-tested in FP64 when
// the FP32 hit lies within its rounding band below tmax
template <int D, int kMode>
__device__ __forceinline__ int query_exit(CoopWarp *sh, const DevScene &sc, bool want, const float *x, const float *v,
                                          float tmax, int skip, float &th, int *err, volatile Visits *vis) {
    const float tneg = kRoundBand * sc.scale;
    int hit;
    if constexpr (D == 2) {
        hit = ray_neumann<true>(sc.neu, x, v, tmax, skip, th, err, vis, tneg);
    } else {
        th = tmax;
        hit = coop_run<kCoopExit, kMode>(*sh, sc, want, x, v, th, skip, err, vis);
    }
    if (hit >= 0 && tmax - th <= kRoundBand * (sc.scale + tmax)) {
        double t64;
        if (!ray_prim64<D, true>(sc.neu, hit, x, v, t64, tneg) || t64 > (double)tmax) hit = -1;
    }
    return hit;
}

// Steps 1-3 of the lanes with `act` (3D: the whole warp calls).  Returns true
// if the walk ended (its value already added; term_value 0 after a lost
// roulette draw).  On return false: r (star radius) and S (this step's source
// and Neumann terms, times the step's roulette scale, as the suffix pass of a
// recorded walk takes them).
template <int D, int kMode>
__device__ __forceinline__ bool step_geometry(CoopWarp *sh, Walk<D> &w, const StepEnv &a, bool act, float &r, float &S,
                                              float &term_value, bool &truncated, volatile Visits *vis) {
    if (D == 2 && !act) return false;
    const DevScene &sc = a.sc;
    float bd2;
    const int slot = query_dirichlet<D, kMode>(sh, sc, act, w.x, bd2, a.err, vis);
    const float RD = sqrtf(bd2);
    bool ended = false;
    if (act) {
        // eps-shell decision: in FP64 when the FP32 distance lies within its
        // rounding band around eps (elsewhere both precisions agree)
        double q64[3];
        bool have64 = false, shell;
        if (fabsf(RD - a.eps) <= kRoundBand * (sc.scale + RD)) {
            shell = dirichlet_dist64<D>(sc.dir, slot, w.x, q64) <= a.eps64;
            have64 = true;
        } else {
            shell = RD <= a.eps;
        }
        if (shell || w.k >= a.maxsteps) {
            if (!have64) dirichlet_dist64<D>(sc.dir, slot, w.x, q64);
            float xb[3] = {(float)q64[0], (float)q64[1], D == 3 ? (float)q64[2] : 0.f};
            term_value = eval_fn<D>(sc.g, xb);
            w.acc += w.T * term_value;
            truncated = !shell;
            ended = true;
        } else if (roulette_on(a, w.k)) {
            if (!roulette_survives(a, w.pid, w.wid, w.k)) {
                term_value = 0.f;
                truncated = false;
                ended = true;
            } else {
                w.T *= 1.f / a.rr_q;
            }
        }
    }
    if (D == 2 && ended) return true;
    const bool go = act && !ended;
    float bs = RD * RD;
    query_silhouette<D, kMode>(sh, sc, go, w.x, bs, a.err, vis);
    if (go) {
        float R = fminf(sqrtf(bs), RD);
        r = fmaxf(R, a.eps);
        S = 0.f;
    }
    const bool source = go && sc.has_source;
    if (D == 2 ? source : __any_sync(0xffffffffu, source)) {
        float vs[D] = {}, rho = 0.f;
        if (source) {
            U4 u = philox(w.pid, w.wid, (uint32_t)w.k, P_SRC, a.key0, a.key1);
            uniform_dir<D>(u01(u.x), u01(u.y), vs);
            if (w.prim >= 0 && dotv<D>(vs, w.n) < 0.f) reflect<D>(vs, w.n);
            rho = D == 2 ? r * sqrtf(u01(u.z) * u01(u.w)) : r * beta22_inv(u01(u.z));
        }
        float th;
        const int hs = query_exit<D, kMode>(sh, sc, source, w.x, vs, rho, w.prim, th, a.err, vis);
        if (source) {
            if (hs < 0) {
                float y[3];
#pragma unroll
                for (int i = 0; i < D; ++i) y[i] = w.x[i] + rho * vs[i];
                S = -(r * r / (2.f * D)) * eval_fn<D>(sc.f, y);
            }
            if (!sc.has_flux) w.acc += w.T * S;
        }
    }
    const bool flux = go && sc.has_flux;
    if (D == 2 ? flux : __any_sync(0xffffffffu, flux)) {
        const float N = neumann_term<D, kMode>(sh, w, sc, flux, r, a.key0, a.key1, a.err, vis);
        if (flux) {
            S -= N;
            w.acc += w.T * S;
        }
    }
    if (go) S *= roulette_scale(a, w.k);
    return ended;
}

// Step 5 of the lanes with `act` (3D: the whole warp calls): ray cast within
// r and move.
template <int D, int kMode>
__device__ __forceinline__ void step_move(CoopWarp *sh, Walk<D> &w, const StepEnv &a, bool act, const float *nu, float r,
                                          volatile Visits *vis) {
    if (D == 2 && !act) return;
    const DevScene &sc = a.sc;
    float th;
    const int hit = query_exit<D, kMode>(sh, sc, act, w.x, nu, r, w.prim, th, a.err, vis);
    if (!act) return;
    if (hit >= 0) {
        // an exit hit arrives from the inside, the side the walk is on, so
        // the walker's normal is the primitive's inward normal (Sec. 4.1,
        // normal convention at Eq. angular_req).  The walker stands at the
        // hit point moved tneg along that normal: a rounded hit point may lie
        // on either side of the boundary, and every later query (silhouettes,
        // exit casts near a vertex) needs a start point inside the domain.
        const float tneg = kRoundBand * sc.scale;
        th = fmaxf(th, 0.f);
#pragma unroll
        for (int i = 0; i < D; ++i) {
            w.n[i] = __ldg(sc.nin_neu + (size_t)hit * D + i);
            w.x[i] += th * nu[i] + tneg * w.n[i];
        }
        w.prim = hit;
    } else {
#pragma unroll
        for (int i = 0; i < D; ++i) w.x[i] += r * nu[i];
        w.prim = -1;
    }
    w.k++;
}

// crossings of the ray x + t v (t > 0) with the whole boundary
template <int D, int kMode>
__device__ __forceinline__ int count_crossings(CoopWarp *sh, const DevScene &sc, bool want, const float *x,
                                               const float *v, int *err) {
    if constexpr (D == 2) {
        return ray_count(sc.dir, x, v, err) + ray_count(sc.neu, x, v, err);
    } else {
        float far = 3.0e38f;
        const int n = coop_run<kCoopCount, kMode>(*sh, sc, want, x, v, far, 1, err, nullptr);
        return n + coop_run<kCoopCount, kMode>(*sh, sc, want, x, v, far, 0, err, nullptr);
    }
}

// Status of a query point: 2 outside (odd/even crossing count of a fixed
// ray against all primitives), 1 inside the epsilon-shell (val = g at the
// closest Dirichlet point, FP64 distance test), 0 to be walked.
// (3D: the whole warp calls, `act`: the lanes with a point)
template <int D, int kMode>
__device__ __forceinline__ uint8_t classify_point(CoopWarp *sh, const DevScene &sc, double eps64, const double *p,
                                                  bool act, int *err, double &val) {
    float x[D] = {};
    if (act)
        for (int k = 0; k < D; ++k) x[k] = (float)p[k];
    const float dir[3] = {0.5377844f, 0.7924136f, 0.2876523f};
    float v[D], nn = 0.f;
    for (int k = 0; k < D; ++k) { v[k] = dir[k]; nn += v[k] * v[k]; }
    for (int k = 0; k < D; ++k) v[k] *= rsqrtf(nn);
    if (D == 2 && !act) return 0;
    const int c = count_crossings<D, kMode>(sh, sc, act, x, v, err);
    val = 0.0;
    const bool inside = act && (c & 1) != 0;
    if (D == 2 && !inside) {
        val = __longlong_as_double(0x7ff8000000000000LL);
        return 2;
    }
    float bd2;
    const int slot = query_dirichlet<D, kMode>(sh, sc, inside, x, bd2, err, nullptr);
    if (!inside) {
        val = __longlong_as_double(0x7ff8000000000000LL);
        return 2;
    }
    double q[3];
    if (dirichlet_dist64<D>(sc.dir, slot, x, q) <= eps64) {
        float xb[3] = {(float)q[0], (float)q[1], D == 3 ? (float)q[2] : 0.f};
        val = eval_fn<D>(sc.g, xb);
        return 1;
    }
    return 0;
}

// mean and variance of the mean of one point from its FP64 sums (Sec. 3.2);
// shell / outside points take their classification value
__device__ __forceinline__ void finalize_point(uint8_t status, double shell, double sum, double sum2, int nw,
                                               double *mean, double *var) {
    if (status != 0) {
        *mean = shell;
        if (var) *var = status == 1 ? 0.0 : shell;
        return;
    }
    double m = sum / nw;
    *mean = m;
    if (var) {
        double v = nw > 1 ? (sum2 - nw * m * m) / ((double)nw * (nw - 1)) : 0.0;
        *var = v > 0 ? v : 0.0;
    }
}

// Block-level sum of the per-thread counters into the launch statistics
// stat[0..7]: walk-steps, truncated, walks, node / Dirichlet / silhouette /
// Neumann visits, float4 words of the visited nodes.  Summed over each warp
// first (a 64-bit shared atomic per thread and counter ran one lane at a time,
// at the end of every iteration of the wavefront: guided star, 4 walks per
// point, 33.4 / 29.2 ms); out of line, so that it takes no part in the walk
// loops' register allocation.
__device__ __noinline__ inline void flush_counts(unsigned long long *stat, unsigned long long steps, unsigned long long trunc,
                                                 unsigned long long walks, unsigned long long nodes, uint32_t dprims,
                                                 uint32_t sprims, uint32_t nprims, unsigned long long words) {
    __shared__ unsigned long long red[8];
    if (threadIdx.x < 8) red[threadIdx.x] = 0;
    __syncthreads();
    unsigned long long c[8] = {steps, trunc, walks, nodes, dprims, sprims, nprims, words};
#pragma unroll
    for (int i = 0; i < 8; ++i) {
#pragma unroll
        for (int o = 16; o; o >>= 1) c[i] += __shfl_xor_sync(0xffffffffu, c[i], o);
        if ((threadIdx.x & 31) == 0 && c[i]) atomicAdd(&red[i], c[i]);
    }
    __syncthreads();
    if (threadIdx.x < 8 && red[threadIdx.x]) atomicAdd(stat + threadIdx.x, red[threadIdx.x]);
}
template <int D>
__device__ __forceinline__ void flush_stats(unsigned long long *stat, unsigned long long steps,
                                            unsigned long long trunc, unsigned long long walks, const volatile Visits &v) {
    const unsigned long long nd = v.dnodes, ns = v.snodes, nb = v.nodes;
    flush_counts(stat, steps, trunc, walks, nd + ns + nb, v.dprims, v.sprims, v.nprims,
                 nd * cap_f4(D) + ns * (node_f4<D>() + facing_f4(D)) + nb * node_f4<D>());
}

}  // namespace wost
