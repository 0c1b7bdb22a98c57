// Team synchronisation primitives and the lazy edge checks shared by the
// wavefront kernels (plan.cu: one query per team; plan_multi.cu: all queries
// of a batch advancing together).
#pragma once

#include <climits>

#include "common.cuh"
#include "internal.h"

namespace gmtk {

constexpr int kDefaultSpinLimit = 1 << 22;

__host__ __device__ constexpr size_t smem_round16(size_t b) { return (b + 15) / 16 * 16; }

__device__ __forceinline__ int ldcg_i(const int* p) { return __ldcg(p); }
__device__ __forceinline__ unsigned ldcg_u(const unsigned* p) { return __ldcg(p); }
__device__ __forceinline__ float ldcg_f(const float* p) { return __ldcg(p); }

// Every team also names its CTAs (cta() in [0, ctas())), so that work can be
// dealt to CTAs round-robin.
struct BlockTeam {
    static constexpr bool kSingle = true;
    static constexpr bool kSharedCtl = true;  // the team's counters can live in shared memory
    __device__ __forceinline__ int id() const { return blockIdx.x; }
    __device__ __forceinline__ int cta() const { return 0; }
    __device__ __forceinline__ int ctas() const { return 1; }
    __device__ __forceinline__ int rank() const { return threadIdx.x; }
    __device__ __forceinline__ int size() const { return blockDim.x; }
    __device__ __forceinline__ bool sync(PlanCtl*) const {
        __syncthreads();
        return true;
    }
};

// Sense-reversing barrier over all CTAs of a cooperative grid.  Every poll is
// counted; after spin_limit polls (or once another CTA has reported an error)
// the wait gives up, records GMT_ERR_TIMEOUT and returns false, so the kernel
// ends with an error status instead of hanging.
struct GridTeam {
    static constexpr bool kSharedCtl = false;
    unsigned expected;
    int spin_limit;
    __device__ __forceinline__ int id() const { return 0; }
    __device__ __forceinline__ int cta() const { return blockIdx.x; }
    __device__ __forceinline__ int ctas() const { return gridDim.x; }
    __device__ __forceinline__ int rank() const { return blockIdx.x * blockDim.x + threadIdx.x; }
    __device__ __forceinline__ int size() const { return gridDim.x * blockDim.x; }
    __device__ bool sync(PlanCtl* ctl) const {
        __syncthreads();
        if (threadIdx.x == 0) {
            const unsigned gen = ld_acquire(&ctl->bar_gen);
            const unsigned arrived = atom_add_acq_rel(&ctl->bar_count, 1u);
            if (arrived == expected - 1) {
                ctl->bar_count = 0;
                st_release(&ctl->bar_gen, gen + 1);
            } else {
                int spins = 0;
                while (ld_acquire(&ctl->bar_gen) == gen) {
                    if (ld_volatile(&ctl->error) != 0) break;
                    if (++spins > spin_limit) {
                        atomicCAS(&ctl->error, 0, (int)GMT_ERR_TIMEOUT);
                        break;
                    }
                    __nanosleep(64);
                }
            }
            __threadfence();
        }
        __syncthreads();
        return ld_volatile(&ctl->error) == 0;
    }
};

// All CTAs of one thread-block cluster (up to 16 SMs of a GPC).  The barrier
// is the hardware cluster barrier (arrive.release / wait.acquire at cluster
// scope); it cannot wait forever because every thread of the cluster reaches
// every barrier (all exits from the iteration loop are uniform).
struct ClusterTeam {
    static constexpr bool kSingle = false;
    static constexpr bool kSharedCtl = true;
    __device__ __forceinline__ static unsigned cta_rank() {
        unsigned r;
        asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
        return r;
    }
    __device__ __forceinline__ static unsigned cluster_ctas() {
        unsigned n;
        asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(n));
        return n;
    }
    __device__ __forceinline__ int id() const { return (int)(blockIdx.x / cluster_ctas()); }
    __device__ __forceinline__ int cta() const { return (int)cta_rank(); }
    __device__ __forceinline__ int ctas() const { return (int)cluster_ctas(); }
    __device__ __forceinline__ int rank() const { return (int)(cta_rank() * blockDim.x + threadIdx.x); }
    __device__ __forceinline__ int size() const { return (int)(cluster_ctas() * blockDim.x); }
    __device__ __forceinline__ bool sync(PlanCtl*) const {
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        return true;
    }
};

// ------------------------------------------------------------- lane groups
// A group of W lanes (W = 32: the warp; W = 16: half a warp) working on one
// edge: its lane index, its lanes' mask, and votes whose bit i is lane i of
// the group.  Two groups of one warp may call these at the same time with
// their own masks.
template <int W>
struct LaneGroup {
    static_assert(W == 32 || W == 16 || W == 8, "lane groups of 8, 16 or 32 lanes");
    __device__ __forceinline__ static int base() { return (int)(threadIdx.x & 31) & ~(W - 1); }
    __device__ __forceinline__ static int lane() { return (int)threadIdx.x & (W - 1); }
    __device__ __forceinline__ static unsigned mask() {
        return W == 32 ? 0xffffffffu : ((1u << (W & 31)) - 1u) << base();
    }
    __device__ __forceinline__ static unsigned ballot(bool p) {
        const unsigned b = __ballot_sync(mask(), p);
        return W == 32 ? b : (b >> base()) & ((1u << (W & 31)) - 1u);
    }
    __device__ __forceinline__ static bool any(bool p) { return __any_sync(mask(), p); }
};

// ------------------------------------------------------------ team counters
// The wavefront's team-wide counters (PlanCtl's group, queue and commit
// words): in the control block in global memory (SH = false), or in a copy in
// the shared memory of the team's first CTA (SH = true: a CTA or a cluster),
// reached through the cluster's shared window, where a dependent atomic takes
// about a third of a global one's latency (measured on GB300: 261 against 707
// cycles; a load 219 against 307).  Field addresses are those of the control
// block; `base` maps them into the copy.  The ordering of the memory model
// holds in both: barrier.cluster (or __syncthreads) orders the copy's
// accesses across the team, and the fences of the global path also order the
// queue's global entries against these counters (acquire/release at cluster
// scope covers both state spaces).
template <bool SH>
struct TeamCtl {
    PlanCtl* g;
    unsigned base;  // SH: shared::cluster address of the copy in CTA 0
    template <class T>
    __device__ __forceinline__ unsigned at(const T* f) const {
        return base + (unsigned)((const char*)f - (const char*)g);
    }
    __device__ __forceinline__ int add(int* f, int v) const {
        if (!SH) return atomicAdd(f, v);
        int r;
        asm volatile("atom.shared::cluster.add.u32 %0, [%1], %2;" : "=r"(r) : "r"(at(f)), "r"(v) : "memory");
        return r;
    }
    __device__ __forceinline__ unsigned add(unsigned* f, unsigned v) const {
        if (!SH) return atomicAdd(f, v);
        unsigned r;
        asm volatile("atom.shared::cluster.add.u32 %0, [%1], %2;" : "=r"(r) : "r"(at(f)), "r"(v) : "memory");
        return r;
    }
    __device__ __forceinline__ unsigned long long add(unsigned long long* f, unsigned long long v) const {
        if (!SH) return atomicAdd(f, v);
        unsigned long long r;
        asm volatile("atom.shared::cluster.add.u64 %0, [%1], %2;" : "=l"(r) : "r"(at(f)), "l"(v) : "memory");
        return r;
    }
    __device__ __forceinline__ void min(unsigned* f, unsigned v) const {
        if (!SH) { atomicMin(f, v); return; }
        unsigned r;
        asm volatile("atom.shared::cluster.min.u32 %0, [%1], %2;" : "=r"(r) : "r"(at(f)), "r"(v) : "memory");
    }
    // 64-bit minimum: a compare-and-swap loop in the copy (on GB300 the
    // native 64-bit atomic minimum through the cluster's shared window lost
    // updates under contention in a test of 16 CTAs, while 64-bit add and CAS
    // were exact); every failed CAS returns a smaller value, so the loop ends.
    __device__ __forceinline__ void min(unsigned long long* f, unsigned long long v) const {
        if (!SH) { atomicMin(f, v); return; }
        const unsigned a = at(f);
        unsigned long long cur;
        asm volatile("ld.relaxed.cluster.shared::cluster.u64 %0, [%1];" : "=l"(cur) : "r"(a) : "memory");
        while (v < cur) {
            unsigned long long prev;
            asm volatile("atom.shared::cluster.cas.b64 %0, [%1], %2, %3;" : "=l"(prev) : "r"(a), "l"(cur), "l"(v) : "memory");
            if (prev == cur) break;
            cur = prev;
        }
    }
    __device__ __forceinline__ void cas(int* f, int cmp, int v) const {
        if (!SH) { atomicCAS(f, cmp, v); return; }
        int r;
        asm volatile("atom.shared::cluster.cas.b32 %0, [%1], %2, %3;" : "=r"(r) : "r"(at(f)), "r"(cmp), "r"(v) : "memory");
    }
    // relaxed (volatile) load; acquire load at cluster scope
    __device__ __forceinline__ int ld(const int* f) const {
        if (!SH) return ld_volatile(f);
        int r;
        asm volatile("ld.relaxed.cluster.shared::cluster.u32 %0, [%1];" : "=r"(r) : "r"(at(f)) : "memory");
        return r;
    }
    __device__ __forceinline__ unsigned ld(const unsigned* f) const {
        if (!SH) return __ldcg(f);
        unsigned r;
        asm volatile("ld.relaxed.cluster.shared::cluster.u32 %0, [%1];" : "=r"(r) : "r"(at(f)) : "memory");
        return r;
    }
    __device__ __forceinline__ unsigned long long ld(const unsigned long long* f) const {
        if (!SH) return __ldcg(f);
        unsigned long long r;
        asm volatile("ld.relaxed.cluster.shared::cluster.u64 %0, [%1];" : "=l"(r) : "r"(at(f)) : "memory");
        return r;
    }
    __device__ __forceinline__ unsigned ld_acq(const unsigned* f) const {
        if (!SH) return ld_acquire(f);
        unsigned r;
        asm volatile("ld.acquire.cluster.shared::cluster.u32 %0, [%1];" : "=r"(r) : "r"(at(f)) : "memory");
        return r;
    }
    // plain stores (the writer then passes a team barrier before any reader)
    __device__ __forceinline__ void st(int* f, int v) const {
        if (!SH) { *f = v; return; }
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(at(f)), "r"(v) : "memory");
    }
    __device__ __forceinline__ void st(unsigned* f, unsigned v) const {
        if (!SH) { *f = v; return; }
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(at(f)), "r"(v) : "memory");
    }
    __device__ __forceinline__ void st(unsigned long long* f, unsigned long long v) const {
        if (!SH) { *f = v; return; }
        asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(at(f)), "l"(v) : "memory");
    }
};

// The shared::cluster address of `p` (this CTA's shared memory) in CTA `rank`
// of the cluster (a launch without clusters is a cluster of one CTA).
__device__ __forceinline__ unsigned cluster_map(const void* p, unsigned rank) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

// ---------------------------------------------------------------- edge check
// Both checks first keep only the boxes that meet an axis-aligned bound of
// every point the check will evaluate (one box per lane, a lane group's width
// at a time), then test the points against those boxes alone.  The bound is inflated by far
// more than the rounding of the point formulas, so a box that holds one of
// the computed points is never dropped: the verdict equals testing every
// point against every box.

// Geometric edge y -> x of length L: m = max(2, ceil(L/spacing) + 1) points
// p_k = y + t_k (x - y), t_k = k/(m-1); collision if one lies in a closed box.
// Without the grid, boxes that do not meet the segment's bounding box (every
// computed p_k lies within a few ulps of it) are set aside W at a time first.
template <int DP, int W = 32>
__device__ __forceinline__ bool segment_free_warp(const float* y, const float* x, float L, float spacing,
                                                  const BoxSet<DP>& B, const BoxGridArgs& grid) {
    using LG = LaneGroup<W>;
    const int lane = LG::lane();
    int m = (int)ceilf(L / spacing) + 1;
    if (m < 2) m = 2;
    const float denom = (float)(m - 1);
    if (grid.use) {
        for (int k0 = 0; k0 < m; k0 += W) {
            const int k = k0 + lane;
            bool hit = false;
            if (k < m) {
                const float t = (float)k / denom;
                float p[DP];
#pragma unroll
                for (int a = 0; a < DP; ++a) p[a] = y[a] + t * (x[a] - y[a]);
                hit = in_any_box_grid<DP>(p, B.lo, B.hi, grid);
            }
            if (LG::any(hit)) return false;
        }
        return true;
    }
    float lo[DP], hi[DP];
#pragma unroll
    for (int a = 0; a < DP; ++a) {
        const float e = 1e-5f * (fabsf(x[a]) + fabsf(y[a])) + 1e-30f;
        lo[a] = fminf(x[a], y[a]) - e;
        hi[a] = fmaxf(x[a], y[a]) + e;
    }
    for (int b0 = 0; b0 < B.count; b0 += W) {
        const int b = b0 + lane;
        const unsigned near = LG::ballot(b < B.count && B.meets(b, lo, hi));
        if (!near) continue;
        for (int k0 = 0; k0 < m; k0 += W) {
            const int k = k0 + lane;
            bool hit = false;
            if (k < m) {
                const float t = (float)k / denom;
                float p[DP];
#pragma unroll
                for (int a = 0; a < DP; ++a) p[a] = y[a] + t * (x[a] - y[a]);
                for (unsigned w = near; w; w &= w - 1) hit = hit | B.holds(b0 + __ffs(w) - 1, p);
            }
            if (LG::any(hit)) return false;
        }
    }
    return true;
}

// Least and greatest value over a lane group, one instruction each (a NaN is
// passed over).
__device__ __forceinline__ float group_min(unsigned mask, float v) {
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, %2;" : "=f"(r) : "f"(v), "r"(mask));
    return r;
}
__device__ __forceinline__ float group_max(unsigned mask, float v) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, %2;" : "=f"(r) : "f"(v), "r"(mask));
    return r;
}

// Does one of the lane group's points (has: the lane holds one) lie in a box?
// Only the boxes that meet the bounding box of the group's computed points can
// hold one (no rounding is in between, so nothing is inflated); one box per
// lane, W at a time.
template <int W>
__device__ __forceinline__ bool points_hit(const float* p, bool has, const BoxSet<3>& B) {
    using LG = LaneGroup<W>;
    float lo[3], hi[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        lo[a] = group_min(LG::mask(), has ? p[a] : f_inf());
        hi[a] = group_max(LG::mask(), has ? p[a] : -f_inf());
    }
    bool hit = false;
    for (int b0 = 0; b0 < B.count; b0 += W) {
        const int b = b0 + LG::lane();
        const unsigned near = LG::ballot(b < B.count && B.meets(b, lo, hi));
        if (near && has && !hit) hit = in_near_boxes<3>(p, B, b0, near);
    }
    return hit;
}

// Double-integrator edge: `points` samples of the Hermite trajectory at
// s_k = k/(points-1); collision if one lies in a box or outside the position
// bounds.  basis: the points' Hermite basis (points entries), or NULL to
// compute it.  (The boxes used to be filtered against the hull of the cubic's
// Bezier control points, which a chunk's own points fill only in part.)
template <int W = 32>
__device__ __forceinline__ bool trajectory_free_warp(const float* y, const float* x, float tau, int points,
                                                     const float* plo, const float* phi, const BoxSet<3>& B,
                                                     const BoxGridArgs& grid, const float4* basis = nullptr) {
    using LG = LaneGroup<W>;
    const int lane = LG::lane();
    const float denom = (float)(points - 1);
    for (int k0 = 0; k0 < points; k0 += W) {
        const int k = k0 + lane;
        bool hit = false;
        float p[3] = {0.0f, 0.0f, 0.0f};
        if (k < points) {
            hermite_point(y, x, tau, basis ? basis[k] : hermite_basis((float)k / denom), p);
#pragma unroll
            for (int a = 0; a < 3; ++a) hit = hit | (p[a] < plo[a]) | (p[a] > phi[a]);
            if (grid.use && !hit) hit = in_any_box_grid<3>(p, B.lo, B.hi, grid);
        }
        if (LG::any(hit)) return false;
        if (!grid.use && B.count > 0 && LG::any(points_hit<W>(p, k < points, B))) return false;
    }
    return true;
}

// Dubins airplane edge y -> x of cost c along its shortest word P:
// m = max(2, ceil(c / spacing) + 1) trajectory points at fractions k / (m - 1);
// a point in a box or outside the position bounds collides.  Every lane walks
// the segment start poses once, then its own points.
template <int W = 32>
__device__ __forceinline__ bool dubins_free_warp(const float* y, const float* x, const DubPath& P, float c,
                                                 float spacing, float rho, const float* plo, const float* phi,
                                                 const BoxSet<3>& B, const BoxGridArgs& grid) {
    using LG = LaneGroup<W>;
    const int lane = LG::lane();
    if (P.word >= kDubNone) return false;  // no word: never an edge (its cost would be +inf)
    const DubSegs G = dubins_segments(y, P, rho);
    int m = (int)ceilf(c / spacing) + 1;
    if (m < 2) m = 2;
    const float denom = (float)(m - 1);
    for (int k0 = 0; k0 < m; k0 += W) {
        const int k = k0 + lane;
        bool hit = false;
        float p[3] = {0.0f, 0.0f, 0.0f};
        if (k < m) {
            dubins_point(y, x, G, (float)k / denom, p);
#pragma unroll
            for (int a = 0; a < 3; ++a) hit = hit | (p[a] < plo[a]) | (p[a] > phi[a]);
            if (grid.use && !hit) hit = in_any_box_grid<3>(p, B.lo, B.hi, grid);
        }
        if (LG::any(hit)) return false;
        if (!grid.use && B.count > 0 && LG::any(points_hit<W>(p, k < m, B))) return false;
    }
    return true;
}

// The lazy collision check (Alg. 1) of in-edge be of the node with state sx,
// whose chosen parent is node by: the cached verdict if there is one, else
// the check of that edge, kept in the cache.  Run by a group of W lanes.
template <int KIND, int DP, int W>
__device__ __forceinline__ bool lazy_check(const PlanArgs& A, int by, int be, const float* sx, const BoxSet<DP>& B,
                                           const float4* basis, bool& computed) {
    constexpr int D = KIND == GMT_COST_DI ? 6 : (KIND == GMT_COST_DUBINS ? 4 : DP);
    float sy[D];
#pragma unroll
    for (int a = 0; a < D; ++a) sy[a] = __ldg(&A.X[(size_t)a * A.pitch + by]);
    const int cached = A.verdict ? (int)__ldcg(&A.verdict[be]) : 0;
    computed = cached == 0;
    if (cached != 0) return cached == 1;
    bool free_edge;
    if constexpr (KIND == GMT_COST_EUCLID) {
        free_edge = segment_free_warp<DP, W>(sy, sx, __ldg(&A.in_cost[be]), A.seg_spacing, B, A.grid);
    } else if constexpr (KIND == GMT_COST_DUBINS) {
        // the edge's shortest word: stored by the graph build, or recomputed
        DubPath P;
        if (A.in_path) {
            const float4 w = __ldg(reinterpret_cast<const float4*>(A.in_path) + be);
            P = DubPath{__float_as_int(w.w), w.x, w.y, w.z, ((w.x + w.y) + w.z) * A.rho};
        } else {
            P = dubins_path(sy, sx, A.rho);
        }
        free_edge = dubins_free_warp<W>(sy, sx, P, __ldg(&A.in_cost[be]), A.seg_spacing, A.rho, A.pos_lo, A.pos_hi,
                                        B, A.grid);
    } else {
        // arrival time of the edge: stored by the graph build, or recomputed
        const float tau = A.in_tau ? __ldg(&A.in_tau[be]) : di_tau(di_coef(sy, sx), A.r);
        free_edge = trajectory_free_warp<W>(sy, sx, tau, A.traj_points, A.pos_lo, A.pos_hi, B, A.grid, basis);
    }
    if (A.verdict && LaneGroup<W>::lane() == 0) A.verdict[be] = free_edge ? 1 : 2;
    return free_edge;
}

// Lazy parent (Alg. 1, Sec. III-A), one lane's share of a group of W lanes:
// over the in-row entries r0 + lane, r0 + lane + W, ... the minimum (cost, index) of
// fl(ocost[y] + in_cost[e]) among open y (ocost < +inf); *be = its edge, -1
// if none.  (cost, index) is a total order, so the order of the entries does
// not matter: four chunks of W are taken at a time, their column and cost
// loads issued together, then their snapshot gathers.
template <int W = 32>
__device__ __forceinline__ void lane_parent_min(const int* __restrict__ in_col, const float* __restrict__ in_cost,
                                                const float* ocost, int r0, int r1, int lane, float* bc_out,
                                                int* by_out, int* be_out) {
    const float INF = f_inf();
    float bc = INF;
    int by = INT_MAX, be = -1;
    for (int eb = r0; eb < r1; eb += 4 * W) {
        int ys[4];
        float ic[4], oc[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int e = eb + W * u + lane;
            ys[u] = e < r1 ? __ldg(&in_col[e]) : -1;
            ic[u] = e < r1 ? __ldg(&in_cost[e]) : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) oc[u] = ys[u] >= 0 ? ldcg_f(&ocost[ys[u]]) : INF;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (oc[u] < INF) {
                const float c = oc[u] + ic[u];
                if (c < bc || (c == bc && ys[u] < by)) { bc = c; by = ys[u]; be = eb + W * u + lane; }
            }
        }
    }
    *bc_out = bc;
    *by_out = by;
    *be_out = be;
}


}  // namespace gmtk
