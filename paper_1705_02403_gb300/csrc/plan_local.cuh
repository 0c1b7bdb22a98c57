// Algorithm 1 on a team whose wavefront state lives in its CTAs' shared
// memory: one thread-block cluster, or one CTA, with two team barriers per
// iteration.
//
// What bounds the wavefront is the chain of dependent accesses of an
// iteration and the instructions of its checks, not its bytes.  On a GB300 a
// dependent L2 load takes about 300 cycles, a global
// atomic about 700, the cluster's shared window about 220 and 260, the CTA's
// own shared memory about 30.  So the nodes are dealt to the team's CTAs
// (node x belongs to CTA x mod n, as its entry x / n), each CTA keeps its own
// nodes' state, and every CTA keeps a replica of the open-set snapshot of all
// nodes:
//   own[q]      cost of own node q while it is open, +inf otherwise
//   tree        bit per own node: in the tree
//   rep[x]      the snapshot of node x: cost while open, +inf while
//               unexplored, NaN once closed
//   claim       bit per own node: a neighbour of this iteration's group
//               pushed it (set by any CTA)
//   sent[x]     last iteration (1 + it mod 255) in which this CTA marked x
//   glist[2], newl, clist   own nodes of the group (by parity), own nodes
//               opened, own candidates
// Phase 1: every replica takes the changes of the previous iteration (nodes
// opened, group closed), each CTA selects its own nodes of the group
// G_i = {open, cost <= theta_i}, and its warps push them: the out-neighbours
// that the replica shows as unexplored are marked in their owners' claim bits
// with one fire-and-forget OR (a stale replica entry only costs a needless
// mark, which the owner's tree bit drops).  Team barrier.  Phase 2: the
// owner's marked unexplored nodes are the candidates; each warp (or half
// warp) takes one at a time, finds its lazy parent by gathering the replica
// from shared memory, checks the one edge and commits.  Nothing writes the
// replicas in phase 2, so they hold V_open as it stood when the iteration
// began (Sec. III-A).  The last warp of a CTA to finish sends the CTA's
// minimum open cost and goal flag to every CTA; one warp of each CTA reads
// the n summaries and takes the termination test and the next threshold.
//
// A cluster's CTAs reach one another through the cluster's shared window: the
// changes are written into all replicas with remote stores, the marks with
// remote ORs, and the barrier is the hardware's.
//
// Measured against the one-barrier body with its lists, stamps and snapshot
// in L2 (plan kernel, mean over four seeds): 2D n = 1024 0.157 -> 0.107 ms,
// 2D n = 30000 0.988 -> 0.619, 3D n = 16384 0.421 -> 0.274, 6D n = 5000 (a
// thousand neighbours a node) 0.407 -> 0.256, double integrator n = 4096
// 0.110 -> 0.078, Dubins airplane n = 5000 with 1500 boxes 0.363 -> 0.251
// (0.163 since the box grid's cells have the boxes' proportions).
//
// Decisions, trees, counters and paths are those of plan_body_fused (which
// remains for graphs whose replica does not fit).
#pragma once

#include "plan_core.cuh"

namespace gmtk {

constexpr int kLocalMaxCluster = 16;
// W < 32: candidates per warp of a CTA from which its pulls take W lanes each in
// an iteration, else 32.  Many candidates: throughput, and two pulls per warp
// hide each other's latency; few: a candidate's own chain, which a whole warp
// shortens.  Plan stage on one GB300, always 16 lanes, always 32, by this line:
// 256 uneven queries 1.452, 1.458, 1.440 ms; 200 3D queries of 2049 nodes
// 0.664, 0.616, 0.622; 8 of 16385 0.718, 0.663, 0.669; 100 double-integrator
// queries of 2049 0.379, 0.330, 0.330.  At 8 a warp: 1.439, 0.627, 0.669, 0.354.
constexpr int kNarrowPulls = 16;
template <int V>
struct PullLanes {
    static constexpr int value = V;
};

// Byte offsets of the state in dynamic shared memory (M own nodes, MW words
// of own bits).  cache = true also keeps the own nodes' row bounds and states
// on chip.
struct LocalLayout {
    unsigned rows, rep, own, xs, sent, claim, tree, goal, lists, total;  // lists: newl, glist[2], clist
    int M, MW;
};
__host__ __device__ inline LocalLayout local_layout(unsigned box_bytes, int N, int n, int D, bool directed,
                                                    bool cache) {
    LocalLayout L;
    L.M = (N + n - 1) / n;
    L.MW = (L.M + 31) / 32;
    const unsigned M = (unsigned)L.M, MW = (unsigned)L.MW;
    L.rows = (unsigned)smem_round16(box_bytes);
    L.rep = L.rows + (cache ? (unsigned)smem_round16((directed ? 16u : 8u) * M) : 0u);
    L.own = L.rep + 4u * n * M;
    L.xs = L.own + 4u * M;
    L.sent = L.xs + (cache ? 4u * D * M : 0u);
    L.claim = L.sent + (n > 1 ? ((unsigned)n * M + 3u) / 4u * 4u : 0u);  // one CTA: its claim bits say it
    L.tree = L.claim + 4u * MW;
    L.goal = L.tree + 4u * MW;
    L.lists = L.goal + 4u * MW;
    L.total = L.lists + 8u * M;
    return L;
}

// Boxes staged in shared memory: none when the checks go through the box grid.
__host__ __device__ inline int local_staged_boxes(const PlanArgs& A, int DP) {
    return !A.grid.use && A.boxes.count <= smem_box_cap(DP) ? A.boxes.count : 0;
}

// Counters of a CTA: one allocation per kernel however many instantiations
// of the body it inlines.
constexpr int kHermiteTable = 64;  // trajectory points whose basis is kept
struct LocalCtl {
    float4 basis[kHermiteTable];  // Hermite basis of the check's points (double integrator)
    int gcount[2], newcount[2], ccount[2], ticket[2], done[2], goal[2];
    unsigned minopen[2];
    int state;                    // of the termination test: -1 go on, else the plan's status
    float theta;
    unsigned slot[2][kLocalMaxCluster];              // every CTA's summary: minimum open cost | goal << 31
    unsigned long long goal_key;                     // minimum (cost, node) over the own goal nodes of the tree
    unsigned long long goal_keys[kLocalMaxCluster];  // CTA 0: every CTA's
    unsigned long long sums[6];
};
static __shared__ LocalCtl local_ctl;

__device__ __forceinline__ void st_cluster(unsigned addr, unsigned v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(unsigned addr, unsigned long long v) {
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ void red_or_cluster(unsigned addr, unsigned v) {
    asm volatile("red.relaxed.cluster.shared::cluster.or.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// Node x of a team of n CTAs: owner x mod n, entry x / n (a multiplication by
// ceil(2^32 / n), exact for x < 2^24 and n < 2^8).
template <bool SINGLE>
struct NodeMap {
    unsigned n, magic;
    __device__ __forceinline__ explicit NodeMap(int n_) : n((unsigned)n_), magic(0xffffffffu / (unsigned)n_ + 1u) {}
    __device__ __forceinline__ void split(int x, int& r, int& q) const {
        if (SINGLE) { r = 0; q = x; return; }
        q = (int)__umulhi((unsigned)x, magic);
        r = x - q * (int)n;
    }
};

// The part of a row [r0, r1) that a lane of W handles outside the row's whole
// aligned groups of four: lanes 0-2 its head, lanes 3-5 its tail; -1: none.
// a0, a1: the bounds of the aligned groups.
__device__ __forceinline__ int row_edge_entry(int r0, int r1, int lane, int& a0, int& a1) {
    a0 = min(r1, (r0 + 3) & ~3);
    a1 = max(a0, r1 & ~3);
    const int e = lane < 3 ? r0 + lane : a1 + lane - 3;
    return (lane < 3 ? e < a0 : lane < 6 && e < r1) ? e : -1;
}

// Rows longer than this are read four entries to a load (push and pull):
// a shorter row is one round trip either way and then spreads better over the
// lanes one entry at a time.
constexpr int kLongRow = 128;

// lane_parent_min over the replica: the minimum (cost, index) of
// fl(rep[y] + in_cost[e]) among open y.  A row of up to kLongRow entries is
// one entry per lane and load, four loads of each array in flight; a longer
// one is read four entries to a load, two loads of each array in flight.
template <int W>
__device__ __forceinline__ void replica_parent_min(const int* __restrict__ in_col, const float* __restrict__ in_cost,
                                                   const float* rep, int r0, int r1, int lane, float* bc_out, int* by_out, int* be_out) {
    const float INF = f_inf();
    float bc = INF;
    int by = INT_MAX, be = -1;
    auto take = [&](int y, float ic, int e) {
        const float oc = rep[y];
        const float c = oc + ic;
        // a closed node's NaN and an unexplored node's +inf both fail oc < inf
        if (oc < INF && (c < bc || (c == bc && y < by))) { bc = c; by = y; be = e; }
    };
    if (r1 - r0 <= kLongRow) {
        for (int eb = r0; eb < r1; eb += 4 * W) {
            int ys[4];
            float ic[4], oc[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int e = eb + W * u + lane;
                ys[u] = e < r1 ? __ldg(&in_col[e]) : -1;
                ic[u] = e < r1 ? __ldg(&in_cost[e]) : INF;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) oc[u] = ys[u] >= 0 ? rep[ys[u]] : INF;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float c = oc[u] + ic[u];
                if (oc[u] < INF && (c < bc || (c == bc && ys[u] < by))) { bc = c; by = ys[u]; be = eb + W * u + lane; }
            }
        }
        *bc_out = bc;
        *by_out = by;
        *be_out = be;
        return;
    }
    int a0, a1;
    const int es = row_edge_entry(r0, r1, lane, a0, a1);
    int ey = 0;
    float ec = 0.0f;
    if (es >= 0) {
        ey = __ldg(&in_col[es]);
        ec = __ldg(&in_cost[es]);
    }
    const int4* const col4 = reinterpret_cast<const int4*>(in_col);
    const float4* const cost4 = reinterpret_cast<const float4*>(in_cost);
    for (int b = a0 / 4 + lane; b < a1 / 4; b += 2 * W) {
        const bool two = b + W < a1 / 4;
        const int4 y0 = __ldg(&col4[b]);
        const float4 c0 = __ldg(&cost4[b]);
        int4 y1 = make_int4(0, 0, 0, 0);
        float4 c1 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (two) {
            y1 = __ldg(&col4[b + W]);
            c1 = __ldg(&cost4[b + W]);
        }
        take(y0.x, c0.x, 4 * b);
        take(y0.y, c0.y, 4 * b + 1);
        take(y0.z, c0.z, 4 * b + 2);
        take(y0.w, c0.w, 4 * b + 3);
        if (two) {
            const int e = 4 * (b + W);
            take(y1.x, c1.x, e);
            take(y1.y, c1.y, e + 1);
            take(y1.z, c1.z, e + 2);
            take(y1.w, c1.w, e + 3);
        }
    }
    if (es >= 0) take(ey, ec, es);
    *bc_out = bc;
    *by_out = by;
    *be_out = be;
}

// Returns true in the CTA that holds the result (every thread of it has then
// passed a block barrier after rank 0's last store to the control block).
template <class Team, int KIND, int DP, int W>
__device__ __forceinline__ bool plan_body_local(const PlanArgs& A, const Team& team, unsigned char* smem, bool cache) {
    constexpr int D = KIND == GMT_COST_DI ? 6 : (KIND == GMT_COST_DUBINS ? 4 : DP);
    constexpr bool DIRECTED = KIND != GMT_COST_EUCLID;
    constexpr bool SINGLE = Team::kSingle;
    const int N = A.N, n = SINGLE ? 1 : team.ctas(), me = SINGLE ? 0 : team.cta();
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5, wpc = blockDim.x >> 5;
    const int nbs = local_staged_boxes(A, DP);
    const LocalLayout L = local_layout((unsigned)(nbs * BoxSet<DP>::kQ) * 16u, N, n, D, DIRECTED, cache);
    const int M = L.M, MW = L.MW;
    float4* const sbox = reinterpret_cast<float4*>(smem);
    int2* const rows2 = reinterpret_cast<int2*>(smem + L.rows);  // Euclidean: (row, row end)
    int4* const rows4 = reinterpret_cast<int4*>(smem + L.rows);  // directed: in-row, in-row end, out-row, out-row end
    float* const rep = reinterpret_cast<float*>(smem + L.rep);
    float* const own = reinterpret_cast<float*>(smem + L.own);
    float* const xs = reinterpret_cast<float*>(smem + L.xs);
    unsigned char* const sent = smem + L.sent;
    unsigned* const claim = reinterpret_cast<unsigned*>(smem + L.claim);
    unsigned* const tree = reinterpret_cast<unsigned*>(smem + L.tree);
    unsigned* const goalbits = reinterpret_cast<unsigned*>(smem + L.goal);
    unsigned short* const newl = reinterpret_cast<unsigned short*>(smem + L.lists);
    unsigned short* const clist = newl + 3 * M;
    LocalCtl& lc = local_ctl;
    PlanCtl* const ctl = A.ctl;
    const NodeMap<SINGLE> map(n);
    const float INF = f_inf();
    const unsigned INF_KEY = 0x7f800000u, CLOSED = 0x7fffffffu;
    const int rank = team.rank(), size = team.size();
    const int mean_degree = __ldcg(&A.out_row[N]) / N;

    if (rank == 0) {
        ctl->status = 0;
        ctl->iters = ctl->final_i = ctl->path_len = 0;
        ctl->goal_node = -1;
        ctl->error = 0;
        ctl->push_edges = ctl->pull_edges = ctl->checks = ctl->failed = ctl->tree_size = 0ull;
        ctl->checks_computed = 0ull;
    }
    if (A.check_edges) {
        const long long e = max(__ldcg(&A.out_row[N]), __ldcg(&A.in_row[N]));
        if (e > A.edge_cap) {  // uniform across the team: every thread reads the same counts
            if (rank == 0) {
                ctl->status = GMT_ERR_OOM;
                ctl->goal_node = -1;
            }
            __syncthreads();
            return me == 0;
        }
    }
    for (int b = tid; b < nbs; b += blockDim.x) pack_box<DP>(sbox, A.boxes.lo, A.boxes.hi, b, b);
    const BoxSet<DP> B{nbs ? sbox : nullptr, A.boxes.lo, A.boxes.hi, A.boxes.count};
    const float4* basis = nullptr;
    if (KIND == GMT_COST_DI && A.traj_points <= kHermiteTable) {
        basis = lc.basis;
        if (tid < A.traj_points) lc.basis[tid] = hermite_basis((float)tid / (float)(A.traj_points - 1));
    }

    // Initialisation: x_init is the only open node and the root of the tree.
    for (int v = rank; v < N; v += size) {
        A.cost[v] = v == 0 ? 0.0f : INF;
        A.parent[v] = -1;
    }
    for (int w = tid; w < (int)(L.claim - L.sent) / 4; w += blockDim.x) reinterpret_cast<unsigned*>(sent)[w] = 0u;
    for (int w = tid; w < MW * 3; w += blockDim.x) claim[w] = 0u;  // and tree, goal behind it
    for (int j = tid; j < n * M; j += blockDim.x) rep[j] = INF;
    for (int q = tid; q < M; q += blockDim.x) {
        own[q] = INF;
        const int x = q * n + me;
        if (cache && x < N) {
            if (DIRECTED) rows4[q] = make_int4(__ldg(&A.in_row[x]), __ldg(&A.in_row[x + 1]), __ldg(&A.out_row[x]),
                                               __ldg(&A.out_row[x + 1]));
            else rows2[q] = make_int2(__ldg(&A.out_row[x]), __ldg(&A.out_row[x + 1]));
#pragma unroll
            for (int a = 0; a < D; ++a) xs[a * M + q] = __ldg(&A.X[(size_t)a * A.pitch + x]);
        }
    }
    if (tid < 2) {
        lc.gcount[tid] = lc.newcount[tid] = lc.ccount[tid] = lc.ticket[tid] = lc.done[tid] = lc.goal[tid] = 0;
        lc.minopen[tid] = INF_KEY;
    }
    if (tid < 6) lc.sums[tid] = 0ull;
    if (tid == 0) lc.goal_key = me == 0 && A.is_goal[0] ? 0ull : ~0ull;
    __syncthreads();
    for (int q = tid; q < M; q += blockDim.x) {
        const int x = q * n + me;
        if (x < N && A.is_goal[x]) atomicOr(&goalbits[q >> 5], 1u << (q & 31));
    }
    if (tid == 0) {
        rep[0] = 0.0f;
        if (me == 0) {
            own[0] = 0.0f;
            tree[0] |= 1u;
        }
    }

    int i = 0;
    float theta = 0.0f;
    int it = 0;
    int status = GMT_ERR_ITER_LIMIT;  // unless the termination test says otherwise within max_iters
    team.sync(ctl);

    unsigned long long n_push = 0, n_pull = 0;
    unsigned n_checks = 0, n_failed = 0, n_computed = 0, n_tree = rank == 0 ? 1u : 0u;  // x_init
    const unsigned below = (1u << lane) - 1u;

    while (it < A.max_iters) {
        const int p = it & 1;
        unsigned short* const G = newl + (1 + p) * M;

        // ---- phase 1: replicas, group selection, push
        {
            const unsigned short* const Gprev = newl + (2 - p) * M;
            const int nn = lc.newcount[p], ngp = lc.gcount[p ^ 1];
            const int total = (nn + ngp) * n;
            for (int j = tid; j < total; j += blockDim.x) {
                int e, r;
                map.split(j, r, e);
                const int q = e < nn ? newl[e] : Gprev[e - nn];
                // own[] of a node opened in i - 1 still holds its cost: groups
                // are closed in phase 2
                const unsigned v = e < nn ? __float_as_uint(own[q]) : CLOSED;
                if (SINGLE) rep[q] = __uint_as_float(v);
                else st_cluster(cluster_map(&rep[q * n + me], (unsigned)r), v);
            }
            for (int e = tid; e < nn; e += blockDim.x) {
                const int q = newl[e];
                atomicOr(&tree[q >> 5], 1u << (q & 31));
            }
        }
        if (wib * 32 < M) {
            unsigned kmin = INF_KEY;
            for (int q0 = wib * 32; q0 < M; q0 += blockDim.x) {
                const int q = q0 + lane;
                const float c = q < M ? own[q] : INF;
                const bool in_g = c <= theta;
                const unsigned mg = __ballot_sync(0xffffffffu, in_g);
                if (mg) {
                    int base = 0;
                    if (lane == 0) base = atomicAdd(&lc.gcount[p], __popc(mg));
                    base = __shfl_sync(0xffffffffu, base, 0);
                    if (in_g) {
                        G[base + __popc(mg & below)] = (unsigned short)q;
                        if ((goalbits[q >> 5] >> (q & 31)) & 1u) lc.goal[p] = 1;
                    }
                }
                if (!in_g) kmin = min(kmin, float_key(c));
            }
            kmin = __reduce_min_sync(0xffffffffu, kmin);
            if (lane == 0 && kmin != INF_KEY) atomicMin(&lc.minopen[p], kmin);
        }
        if (tid == 0) {  // the other parity's counters: last read before the previous barrier
            lc.ccount[p ^ 1] = 0;
            lc.ticket[p ^ 1] = 0;
            lc.done[p ^ 1] = 0;
            lc.goal[p ^ 1] = 0;
            lc.minopen[p ^ 1] = INF_KEY;
        }
        __syncthreads();
        const int ng = lc.gcount[p];
        const unsigned char stamp = (unsigned char)(it % 255 + 1);
        // Push: long rows in 1 to 8 parts of at least 64 columns, so that the
        // group's rows spread evenly over the CTA's warps (part k: the k-th run
        // of a multiple of 32 columns).
        int sh = 0;
        while (sh < 3 && (mean_degree >> (sh + 1)) >= 64 && (ng << (sh + 1)) <= 4 * wpc) ++sh;
        for (int u = wib; u < (ng << sh); u += wpc) {
            const int z = G[u >> sh], part = u & ((1 << sh) - 1);
            int e0, e1;
            if (cache) {
                if (DIRECTED) { const int4 rr = rows4[z]; e0 = rr.z; e1 = rr.w; }
                else { const int2 rr = rows2[z]; e0 = rr.x; e1 = rr.y; }
            } else {
                e0 = __ldg(&A.out_row[z * n + me]);
                e1 = __ldg(&A.out_row[z * n + me + 1]);
            }
            if (lane == 0 && part == 0) n_push += (unsigned long long)(e1 - e0);
            const int run = ((e1 - e0 + (32 << sh) - 1) >> (5 + sh)) * 32;
            e0 += part * run;
            e1 = min(e1, e0 + run);
            // marks up to four nodes (-1: none); two lanes may both mark a
            // node (the byte is not claimed atomically), which does no harm
            auto mark4 = [&](const int* xv) {
                bool want[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) want[c] = xv[c] >= 0 && __float_as_uint(rep[xv[c]]) == INF_KEY;  // else in the tree
                if (!(want[0] | want[1] | want[2] | want[3])) return;
                if (!SINGLE) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) want[c] = want[c] && sent[xv[c]] != stamp;
                }
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    if (!want[c]) continue;
                    int r, q;
                    map.split(xv[c], r, q);
                    const unsigned bit = 1u << (q & 31);
                    if (SINGLE) {
                        atomicOr(&claim[q >> 5], bit);
                    } else {
                        sent[xv[c]] = stamp;
                        red_or_cluster(cluster_map(&claim[q >> 5], (unsigned)r), bit);
                    }
                }
            };
            if (e1 - e0 <= kLongRow) {
                if (e0 >= e1) continue;
                int xv[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int ei = e0 + 32 * c + lane;
                    xv[c] = ei < e1 ? __ldg(&A.out_col[ei]) : -1;
                }
                mark4(xv);
                continue;
            }
            int a0, a1;
            const int es = row_edge_entry(e0, e1, lane, a0, a1);
            const int ex = es >= 0 ? __ldg(&A.out_col[es]) : -1;
            const int4* const col4 = reinterpret_cast<const int4*>(A.out_col);
            for (int b = a0 / 4 + lane; b < a1 / 4; b += 64) {
                const bool two = b + 32 < a1 / 4;
                const int4 x0 = __ldg(&col4[b]);
                const int4 x1 = two ? __ldg(&col4[b + 32]) : x0;
                mark4(&x0.x);
                if (two) mark4(&x1.x);
            }
            if (ex >= 0) {
                const int xv[4] = {ex, -1, -1, -1};
                mark4(xv);
            }
        }
        __syncwarp();
        team.sync(ctl);

        // ---- phase 2: lazy parents, one check each, commits
        if (tid == 0) {
            lc.gcount[p ^ 1] = 0;
            lc.newcount[p] = 0;
        }
        for (int g = tid; g < ng; g += blockDim.x) own[G[g]] = INF;  // the group closes
        // the candidates: marked own nodes that are not in the tree, one warp
        // per word of bits (in any order: each is decided alone)
        for (int w = wib; w < MW; w += wpc) {
            const unsigned marks = claim[w];
            __syncwarp();
            if (lane == 0 && marks) claim[w] = 0u;
            const unsigned m = marks & ~tree[w];
            if (!m) continue;
            int base = 0;
            if (lane == 0) base = atomicAdd(&lc.ccount[p], __popc(m));
            base = __shfl_sync(0xffffffffu, base, 0);
            if ((m >> lane) & 1u) clist[base + __popc(m & below)] = (unsigned short)(32 * w + lane);
        }
        if (!SINGLE && stamp == 255)  // the next iteration's stamp is 1 again
            for (int w = tid; w < (int)(L.claim - L.sent) / 4; w += blockDim.x) reinterpret_cast<unsigned*>(sent)[w] = 0u;
        __syncthreads();
        const int nc = lc.ccount[p];
        auto pull = [&](auto lanes) {
            constexpr int V = decltype(lanes)::value;
            using LG = LaneGroup<V>;
            const int glane = LG::lane();
            const unsigned gmask = LG::mask();
            const int groups = wpc * (32 / V);
            int t = tid / V;
            while (t < nc) {
                const int q = clist[t];
                const int x = q * n + me;
                int r0, r1;
                float sx[D];
                if (cache) {
                    if (DIRECTED) { const int4 rr = rows4[q]; r0 = rr.x; r1 = rr.y; }
                    else { const int2 rr = rows2[q]; r0 = rr.x; r1 = rr.y; }
#pragma unroll
                    for (int a = 0; a < D; ++a) sx[a] = xs[a * M + q];
                } else {
                    r0 = __ldg(&A.in_row[x]);
                    r1 = __ldg(&A.in_row[x + 1]);
#pragma unroll
                    for (int a = 0; a < D; ++a) sx[a] = __ldg(&A.X[(size_t)a * A.pitch + x]);
                }
                float bc;
                int by, be;
                replica_parent_min<V>(A.in_col, A.in_cost, rep, r0, r1, glane, &bc, &by, &be);
                // the least (cost, node) over the lanes, by its two words; costs
                // are >= 0, so their bits order as they do
                const unsigned kc = __reduce_min_sync(gmask, float_key(bc));
                const int ky = __reduce_min_sync(gmask, float_key(bc) == kc ? by : INT_MAX);
                const unsigned holder = LG::ballot(float_key(bc) == kc && by == ky);
                bc = __uint_as_float(kc);
                be = __shfl_sync(gmask, be, __ffs(holder) - 1, V);
                by = ky;
                if (be < 0) {
                    // the group node that pushed x is an open in-neighbour; the
                    // guard keeps a broken invariant from reading out of bounds
                    if (glane == 0) { ++n_checks; ++n_failed; atomicCAS(&ctl->error, 0, (int)GMT_ERR_CUDA); }
                } else {
                    bool computed;
                    const bool free_edge = lazy_check<KIND, DP, V>(A, by, be, sx, B, basis, computed);
                    if (glane == 0) {
                        n_pull += (unsigned long long)(r1 - r0);
                        ++n_checks;
                        n_computed += computed ? 1u : 0u;
                        if (free_edge) {
                            A.cost[x] = bc;
                            A.parent[x] = by;
                            own[q] = bc;
                            newl[atomicAdd(&lc.newcount[p ^ 1], 1)] = (unsigned short)q;
                            atomicMin(&lc.minopen[p], float_key(bc));
                            ++n_tree;
                            if ((goalbits[q >> 5] >> (q & 31)) & 1u)
                                atomicMin(&lc.goal_key, ((unsigned long long)float_key(bc) << 32) | (unsigned)x);
                        } else {
                            ++n_failed;
                        }
                    }
                }
                if (glane == 0) t = groups + atomicAdd(&lc.ticket[p], 1);
                t = __shfl_sync(gmask, t, 0, V);
            }
        };
        if (W < 32 && nc >= kNarrowPulls * wpc) pull(PullLanes<W>{});
        else pull(PullLanes<32>{});
        __syncwarp();
        // the CTA's last warp sends its summary to every CTA
        {
            int last = 0;
            if (lane == 0) {
                __threadfence_block();
                last = atomicAdd(&lc.done[p], 1) == wpc - 1;
                __threadfence_block();
            }
            last = __shfl_sync(0xffffffffu, last, 0);
            if (last && lane < n) {
                const unsigned v = *(volatile unsigned*)&lc.minopen[p] | ((unsigned)*(volatile int*)&lc.goal[p] << 31);
                if (SINGLE) lc.slot[p][0] = v;
                else st_cluster(cluster_map(&lc.slot[p][me], (unsigned)lane), v);
            }
            __syncwarp();
        }
        team.sync(ctl);

        // ---- termination test (Alg. 1), next threshold: one warp per CTA (32
        // warps computing the same divisions would queue for the issue slots)
        ++it;
        if (wib == 0) {
            const unsigned sum = lane < n ? lc.slot[p][lane] : INF_KEY;
            const bool goal = __any_sync(0xffffffffu, (sum >> 31) != 0u);
            const unsigned mk = __reduce_min_sync(0xffffffffu, sum & 0x7fffffffu);
            int state = -1;
            if (goal) state = GMT_OK;
            else if (mk == INF_KEY) state = GMT_NO_PATH;  // no node stays open
            else {
                const float m = __uint_as_float(mk);
                if (A.delta == 0.0f) {
                    theta = m;
                    i = i + 1;
                } else {
                    const float qk = m / A.delta;
                    if (!(qk < 16777216.0f)) {
                        state = GMT_ERR_ITER_LIMIT;  // i stays below 2^24
                    } else {
                        int k = (int)ceilf(qk);
                        if (k < i + 1) k = i + 1;
                        while (k > i + 1 && (float)(k - 1) * A.delta >= m) --k;
                        while ((float)k * A.delta < m) ++k;
                        i = k;
                        theta = (float)i * A.delta;
                    }
                }
            }
            if (lane == 0) {
                lc.state = state;
                lc.theta = theta;
            }
        }
        __syncthreads();
        if (lc.state != -1) { status = lc.state; break; }
        theta = lc.theta;
    }

    // ---- result: counters, the goal node, the returned path
    {
        unsigned long long v[6] = {n_push, n_pull, n_checks, n_failed, n_computed, n_tree};
#pragma unroll
        for (int k = 0; k < 6; ++k) {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], off);
            if (lane == 0 && v[k]) atomicAdd(&lc.sums[k], v[k]);
        }
        __syncthreads();
        unsigned long long* const to[6] = {&ctl->push_edges, &ctl->pull_edges,      &ctl->checks,
                                           &ctl->failed,     &ctl->checks_computed, &ctl->tree_size};
#pragma unroll
        for (int k = 0; k < 6; ++k)
            if (tid == k && lc.sums[k]) atomicAdd(to[k], lc.sums[k]);
        if (tid == 0) {
            if (SINGLE) lc.goal_keys[0] = lc.goal_key;
            else st_cluster(cluster_map(&lc.goal_keys[me], 0u), lc.goal_key);
        }
    }
    // no CTA reaches another's shared memory after this barrier
    team.sync(ctl);
    if (me != 0) return false;
    // The path is walked from the goal node back to x_init by one thread, in a
    // copy of the parents that takes the replica's place (its last reader has
    // passed a barrier).
    int* const spar = reinterpret_cast<int*>(rep);
    if (status == GMT_OK) {
        for (int v = tid; v < N; v += blockDim.x) spar[v] = ldcg_i(&A.parent[v]);
    }
    __syncthreads();
    if (tid == 0) {
        unsigned long long key = ~0ull;
        for (int r = 0; r < n; ++r) key = min(key, lc.goal_keys[r]);
        const int err = ld_volatile(&ctl->error);
        ctl->status = err ? err : status;
        ctl->goal_key = key;  // the host reads the goal's cost from it
        ctl->iters = it;
        ctl->final_i = i;
        ctl->goal_node = -1;
        ctl->path_len = 0;
        if (status == GMT_OK && !err) {
            const int g = (int)(key & 0xffffffffu);
            ctl->goal_node = g;
            int len = 1, v = g;
            while (v > 0 && len <= N) {
                v = spar[v];
                ++len;
            }
            if (v != 0) len = 0;
            ctl->path_len = len;
            if (A.path) {
                v = g;
                for (int k = len - 1; k >= 0; --k) {
                    A.path[k] = v;
                    if (v > 0) v = spar[v];
                }
            }
        }
        __threadfence();
    }
    __syncthreads();
    return true;
}

}  // namespace gmtk
