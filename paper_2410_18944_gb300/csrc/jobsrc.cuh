// Where a walk's work comes from.  The persistent walk loops (plain here,
// guided in guided_ws.cuh) are written once against a "job source":
//   SoloSrc  - one scene, one point set, one field: everything lives in the
//              kernel's argument block (wost_solve);
//   BatchSrc - many scenes of uneven size, each with its own points, walk
//              count, eps, step cap, seed and field, in a device job table
//              (wost_solve_batch).  Work items are laid out job-major, so the
//              walks in flight at any moment belong to few jobs.
// A source hands out work items, starts a walk from an item, gives the
// step its scene and scalars (StepEnv), and owns the per-point sums and the
// training-record buffer the walk writes to.  Either way every walk draws
// from the same Philox streams, counter (point, walk, step, purpose) and key
// (seed_lo, seed_hi + scene_id), so a job of a batch walks exactly as the
// same problem solved alone.
#pragma once
#include "field.cuh"
#include "walkstep.cuh"

namespace wost {

constexpr int kRecFloats = 12;   // training record: x[3] nu[3] n[3] on_neumann q target

// destination of finished training records (Sec. 5.2): buffer, counters
// ([0] appended, [1] dropped), capacity
struct RecDest {
    float *out;
    unsigned long long *ctr;
    long long cap;
};

// ---------------------------------------------------------------------------
// one scene
// ---------------------------------------------------------------------------
template <int D>
struct SoloSrc {
    const WalkArgs &a;
    const DevField *f;   // guided only
    RecDest rd;
    const DevScene *sc;  // the scene view the steps use (a.sc, or a copy on staged nodes)

    __device__ __forceinline__ unsigned long long *work_ctr() const { return a.work_ctr; }
    __device__ __forceinline__ unsigned long long total() const { return a.total; }
    __device__ __forceinline__ unsigned lanes() const { return a.lanes; }
    __device__ __forceinline__ bool start(Walk<D> &w, unsigned long long item) const {
        if (a.order) {   // the same walk index, another point
            const unsigned long long p = item % (unsigned long long)a.npoints;
            item = item - p + a.order[p];
        }
        start_walk<D>(w, a, item);
        return a.status[w.pid] == 0;
    }
    __device__ __forceinline__ StepEnv env(const Walk<D> &) const {
        return StepEnv{*sc, a.eps, a.eps64, a.maxsteps, a.key0, a.key1, a.err, a.rr_depth, a.rr_q};
    }
    __device__ __forceinline__ void finish(const Walk<D> &w) const {
        finish_walk(a, w.pid, w.acc);
        if (a.plen) atomicAdd(a.plen + w.pid, (unsigned)w.k + 1u);
    }
    __device__ __forceinline__ const DevField &field(const Walk<D> &) const { return *f; }
    __device__ __forceinline__ RecDest rec(const Walk<D> &) const { return rd; }
    __device__ __forceinline__ int job(const Walk<D> &) const { return 0; }
    __device__ __forceinline__ const uint4 *wimg(int) const { return f->wimg; }
    __device__ __forceinline__ const float *b3(int) const { return f->b3; }
};

// Staging of a scene's traversal data in shared memory.  A walk step is a
// chain of dependent loads of BVH nodes and leaf primitives, so their
// latency is the step's latency; a kernel with shared memory to spare keeps
// as much of the data there as fits.  Regions, in the order they are taken:
// the three BVHs' nodes (of the Dirichlet BVH its caps), the silhouette facing
// bounds, then the Dirichlet,
// Neumann and silhouette primitives.
constexpr int kStageRegions = 7;

__host__ __device__ __forceinline__ void stage_regions(const DevScene &s, const float4 **src, int *cnt) {
    const int nb = s.dim == 2 ? node_f4<2>() : node_f4<3>();   // float4 per node
    const int pd = s.dim == 2 ? 1 : 3;       // per Dirichlet / Neumann primitive
    const int ps = s.dim == 2 ? 2 : 3;       // per silhouette element
    src[0] = s.dir_caps; cnt[0] = s.dir.nnodes * cap_f4(s.dim);
    src[1] = s.neu.nodes; cnt[1] = s.neu.nnodes * nb;
    src[2] = s.sil.nodes; cnt[2] = s.sil.nnodes * nb;
    src[3] = s.sil_facing; cnt[3] = s.sil_facing ? facing_f4(s.dim) * s.sil.nnodes : 0;
    src[4] = s.dir.prims; cnt[4] = s.dir.nprims * pd;
    src[5] = s.neu.prims; cnt[5] = s.neu.nprims * pd;
    src[6] = s.sil.prims; cnt[6] = s.sil.nprims * ps;
}

// Which regions fit in budget_f4 float4 (bit r = region r), greedily in
// order: all node regions or none, then whole primitive arrays.
__host__ __forceinline__ int stage_plan(const DevScene &s, int budget_f4, int *total_f4) {
    const float4 *src[kStageRegions];
    int cnt[kStageRegions];
    stage_regions(s, src, cnt);
    int mask = 0, used = 0;
    const int nodes = cnt[0] + cnt[1] + cnt[2] + cnt[3];
    if (nodes <= budget_f4) {
        mask = 0xF;
        used = nodes;
        for (int r = 4; r < kStageRegions; ++r)
            if (cnt[r] > 0 && used + cnt[r] <= budget_f4) { mask |= 1 << r; used += cnt[r]; }
    }
    *total_f4 = used;
    return mask;
}

// Copies the regions in `mask` into shared memory `dst` (all threads of the
// block take part) and makes `out` (shared) a copy of the scene view whose
// pointers name the staged copies.
__device__ __forceinline__ void stage_scene(const DevScene &in, DevScene &out, float4 *dst, int mask) {
    const float4 *src[kStageRegions];
    int cnt[kStageRegions];
    stage_regions(in, src, cnt);
    float4 *start[kStageRegions];
    float4 *d = dst;
    for (int r = 0; r < kStageRegions; ++r) {
        start[r] = d;
        if (!(mask >> r & 1) || cnt[r] == 0) continue;
        for (int i = threadIdx.x; i < cnt[r]; i += blockDim.x) d[i] = __ldg(src[r] + i);
        d += cnt[r];
    }
    if (threadIdx.x == 0) {
        out = in;
        auto take = [&](int r) { return (mask >> r & 1) && cnt[r] > 0; };
        if (take(0)) out.dir_caps = start[0];
        if (take(1)) out.neu.nodes = start[1];
        if (take(2)) out.sil.nodes = start[2];
        if (take(3)) out.sil_facing = start[3];
        if (take(4)) out.dir.prims = start[4];
        if (take(5)) out.neu.prims = start[5];
        if (take(6)) out.sil.prims = start[6];
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------
// many scenes
// ---------------------------------------------------------------------------
struct DevJob {
    DevScene sc;
    DevField f;                  // the job's field (guided batches)
    const double *points;        // npoints * D (device)
    int64_t npoints;
    int64_t point_off;           // first row of the job in the batch's per-point arrays
    int nwalks;
    int maxsteps;
    float eps;
    double eps64;
    uint32_t key0, key1;
    int rr_depth;                // Russian roulette from this step on (0 = off)
    float rr_q;                  // its survival probability
    RecDest rd;                  // the field's record buffer
    double *out_mean, *out_var;  // npoints each (device; out_var nullable)
};

// a contiguous run of work items of one launch: walks [walk_begin,
// walk_begin + n) of every point of one job, items ordered walk-major
// within the run (item = walk * npoints + point)
struct DevSeg {
    unsigned long long item_begin;
    int job;
    int walk_begin;
};

struct BatchArgs {
    const DevJob *jobs;
    const DevSeg *segs;
    int nseg;
    unsigned long long total;        // items in this launch
    unsigned long long *work_ctr;
    const uint8_t *status;           // per point of the batch: 0 walk, 1 shell, 2 outside
    double *sum, *sum2;              // per point of the batch (FP64)
    unsigned long long *stat;        // launch statistics (as WalkArgs::stat)
    int *err;
};

// index of the last segment whose item_begin <= item (segments sorted)
__device__ __forceinline__ int find_seg(const DevSeg *segs, int nseg, unsigned long long item) {
    int lo = 0, hi = nseg - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (__ldg(&segs[mid].item_begin) <= item) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

template <int D>
struct BatchSrc {
    const BatchArgs &b;

    __device__ __forceinline__ unsigned long long *work_ctr() const { return b.work_ctr; }
    __device__ __forceinline__ unsigned long long total() const { return b.total; }
    __device__ __forceinline__ unsigned lanes() const { return D == 2 ? 0 : 32; }
    __device__ __forceinline__ bool start(Walk<D> &w, unsigned long long item) const {
        const int s = find_seg(b.segs, b.nseg, item);
        const DevSeg sg = b.segs[s];
        const DevJob &J = b.jobs[sg.job];
        const unsigned long long local = item - sg.item_begin, np = (unsigned long long)J.npoints;
        w.job = sg.job;
        w.pid = (uint32_t)(local % np);
        w.wid = (uint32_t)(sg.walk_begin + local / np);
#pragma unroll
        for (int i = 0; i < D; ++i) { w.x[i] = (float)J.points[(size_t)w.pid * D + i]; w.n[i] = 0.f; }
        w.T = 1.f;
        w.acc = 0.f;
        w.k = 0;
        w.prim = -1;
        return b.status[J.point_off + w.pid] == 0;
    }
    __device__ __forceinline__ StepEnv env(const Walk<D> &w) const {
        const DevJob &J = b.jobs[w.job];
        return StepEnv{J.sc, J.eps, J.eps64, J.maxsteps, J.key0, J.key1, b.err, J.rr_depth, J.rr_q};
    }
    __device__ __forceinline__ void finish(const Walk<D> &w) const {
        const size_t i = (size_t)b.jobs[w.job].point_off + w.pid;
        atomicAdd(b.sum + i, (double)w.acc);
        atomicAdd(b.sum2 + i, (double)w.acc * (double)w.acc);
    }
    __device__ __forceinline__ const DevField &field(const Walk<D> &w) const { return b.jobs[w.job].f; }
    __device__ __forceinline__ RecDest rec(const Walk<D> &w) const { return b.jobs[w.job].rd; }
    __device__ __forceinline__ int job(const Walk<D> &w) const { return w.job; }
    __device__ __forceinline__ const uint4 *wimg(int j) const { return b.jobs[j].f.wimg; }
    __device__ __forceinline__ const float *b3(int j) const { return b.jobs[j].f.b3; }
};

// How a plain launch of `total` walks on `warps` warps hands out its items
// (WorkCursor).  2D: 0, from the counter, so that a warp starts on consecutive
// points and shares the nodes of their first step; a launch of less than one
// walk per lane goes round the warps instead (32), which leaves each warp fewer
// lanes to wait for (64-segment problem, 52k walks: see plain_walk_kernel).
// 3D: round the warps, the lanes of a warp that hold walks: a warp has four to
// eight queries in flight at a time, so more walks than that only amortise the
// step logic, but a warp that is left with many long walks holds up the end of
// the launch; half the lanes where there are fewer than two walks per lane,
// all of them where every step has a Neumann sample too.  Measured on one GB300,
// 16 / 32 lanes at 0.84, 1, 1.5, 1.9, 2.4 and 4 walks per lane: genus-3 60 / 67,
// 70 / 80, 85 / 90, 101 / 105, 118 / 126, 180 / 182 ms; icosphere 42.8 / 42.0,
// 46 / 50, 58.8 / 58.1, 70 / 67, 83 / 78, 128 / 110 ms; flux slab at 0.84 walks
// 16.1 / 15.0 ms.
inline int plain_lanes(const DevScene &s, unsigned long long total, long long warps) {
    const unsigned long long lanes = 32ull * (unsigned long long)warps;
    if (s.dim == 2) return total <= lanes ? 32 : 0;
    return s.has_flux || total >= 2 * lanes ? 32 : 16;
}

// A lane's next work item: from the launch's counter, warp-aggregated, after
// (lanes > 0) the first items have gone round the warps (warp w's lane l takes
// item l * warps + w; the counter then counts the items after those).  Long
// walks come in runs of neighbouring points, or first where the launch is
// ordered, and in 3D a warp that held a run of them would outlast all others.
// The first items belong to their warps: a CTA that does not fit the GPU beside
// the others holds its items until one of them leaves (correct, but a launch of
// few walks then takes two waves; wost_solve_plain_static in 3D, whose kernel
// fits four of its eight CTAs per SM: flux slab, 131k walks, 18.8 ms against the
// 15.4 of wost_solve).
struct WorkCursor {
    bool first = true;
    __device__ __forceinline__ unsigned long long next(unsigned long long *ctr, unsigned warp, unsigned warps,
                                                       unsigned lanes) {
        if (first && lanes > 0) {
            first = false;
            return (unsigned long long)(threadIdx.x & 31) * warps + warp;
        }
        return (unsigned long long)lanes * warps + warp_fetch_add(ctr, true);
    }
};

// ---------------------------------------------------------------------------
// The plain persistent walk loop (uniform directions, Sec. 3.2).
// Every lane of a warp stays in the loop until the whole warp is out of
// work, and one loop iteration is one step of every active lane: lanes
// cannot drift into different phases of the step, so the warp re-converges
// after each query (2D: a lane without a walk is predicated off; 3D: it takes
// part in the queries of the others, coop.cuh).
// ---------------------------------------------------------------------------
template <int D, int kMode, class Src>
__device__ __forceinline__ void plain_loop(CoopWarp *sh, const Src &src, unsigned long long *stat) {
    Walk<D> w;
    volatile Visits vis;
    bool active = false, exhausted = false;
    unsigned long long nsteps = 0, ntrunc = 0, nwalks = 0;
    if (D == 3) {   // lanes without a walk take part in the groups' queries
        w.job = 0;
        w.prim = -1;
        w.k = 0;
        for (int i = 0; i < D; ++i) w.x[i] = 0.f;
        exhausted = (threadIdx.x & 31) >= src.lanes();
    }
    WorkCursor cursor;
    const unsigned warps = gridDim.x * (blockDim.x / 32), warp = (threadIdx.x / 32) * gridDim.x + blockIdx.x;
    for (;;) {
        if (!active && !exhausted) {
            unsigned long long item = cursor.next(src.work_ctr(), warp, warps, src.lanes());
            if (item >= src.total()) exhausted = true;
            else if (src.start(w, item)) { active = true; nwalks++; }
        }
        if (!__any_sync(0xffffffffu, active || !exhausted)) break;
        __syncwarp();
        if (D == 2 ? !active : !__any_sync(0xffffffffu, active)) continue;
        nsteps += active;
        const StepEnv env = src.env(w);
        float r = 0.f, S, gv;
        bool trunc = false;
        bool ended = step_geometry<D, kMode>(sh, w, env, active, r, S, gv, trunc, &vis);
        float nu[D] = {};
        if (active && !ended) {
            U4 u = philox(w.pid, w.wid, (uint32_t)w.k, P_DIR, env.key0, env.key1);
            uniform_dir<D>(u01(u.x), u01(u.y), nu);
            if (w.prim >= 0) {
                float dn = dotv<D>(nu, w.n);
                if (dn < 0.f) reflect<D>(nu, w.n);
                ended = dn == 0.f;   // zero density at the tangent plane (Eq. angular_req)
            }
        }
        if (active && ended) {
            src.finish(w);
            ntrunc += trunc;
            active = false;
        }
        step_move<D, kMode>(sh, w, env, active, nu, r, &vis);
    }
    flush_stats<D>(stat, nsteps, ntrunc, nwalks, vis);
}

}  // namespace wost
