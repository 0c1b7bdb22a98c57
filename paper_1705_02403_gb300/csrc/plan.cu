// Algorithm 1 (Group Marching Tree) as one persistent CUDA kernel.
//
// A "team" of threads runs every wavefront iteration of one plan without
// returning to the host: one CTA (block barriers), one thread-block cluster
// (hardware cluster barriers) or a cooperative grid (bounded global barriers,
// co-residency guaranteed by the cooperative launch).
//
// A CTA or a cluster keeps the wavefront's state in its shared memory
// (plan_body_local, plan_local.cuh) when it fits and the rows start on 16-byte
// boundaries; other graphs and cooperative grids keep it in global memory
// (plan_body_fused, plan_fused.cuh).  Both take the same decisions.
#include <algorithm>
#include <mutex>

#include "plan_core.cuh"
#include "plan_fused.cuh"
#include "plan_local.cuh"

namespace gmtk {

// The first warp copies the final control block to the caller's mapped host
// copy (src: a block whose writers have all passed a barrier since), then sets
// the caller's word.
__device__ __forceinline__ void publish_ctl(const PlanArgs& A, int rank) {
    constexpr int n = (int)(sizeof(PlanCtl) / sizeof(int));
    for (int t = rank; t < n; t += 32)
        reinterpret_cast<int*>(A.host_ctl)[t] = __ldcg(reinterpret_cast<const int*>(A.ctl) + t);
    if (!A.host_done) return;
    __threadfence_system();
    __syncwarp();
    if (rank == 0) *(volatile int*)A.host_done = 1;
}

// Lanes per candidate pull.  A single plan's team has hundreds of warps for a
// frontier of a few hundred candidates, and narrower pulls only lengthen each
// candidate's chain (32, 16, 8 lanes, plan kernel on one GB300: 2D n = 1024
// 105, 119, 140 us; 3D n = 16384 271, 290, 329; 6D n = 5000 266, 304, 382;
// double integrator n = 4096 85, 114, 161; Dubins n = 5000 177, 178, 201).  A
// batch's small teams may see many candidates per warp: half a warp each then
// (kNarrowPulls), and always in the scratch kernel (256 queries 2.41 -> 2.26 ms).
constexpr int kPlanPullLanes = 32;
constexpr int kBatchPullLanes = 16;

// One plan on a team that spans several SMs (or one CTA whose state does not
// fit its shared memory): the one-barrier wavefront (A.ocost holds 2 N floats).
template <class Team, int KIND, int DP>
__global__ void __launch_bounds__(1024, 1) plan_kernel(PlanArgs A, Team team) {
    extern __shared__ float sbox[];
    unsigned dyn_smem;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn_smem));
    plan_body_fused<Team, KIND, DP, kPlanPullLanes>(A, team, sbox, dyn_smem);
    if (A.host_ctl) {
        team.sync(A.ctl);  // every warp's counters and rank 0's result are in
        if (team.rank() < 32) publish_ctl(A, team.rank());
    }
}

// One plan on a team that keeps the wavefront's state in its shared memory.
template <class Team, int KIND, int DP>
__global__ void __launch_bounds__(1024, 1) plan_local_kernel(PlanArgs A, Team team, bool cache) {
    extern __shared__ __align__(16) unsigned char plan_smem[];
    if (plan_body_local<Team, KIND, DP, kPlanPullLanes>(A, team, plan_smem, cache) && A.host_ctl && threadIdx.x < 32)
        publish_ctl(A, threadIdx.x);
}

// Persistent batched wavefront: every team (a CTA, or a cluster) takes the next
// query from a device queue (every query of the batch, of any kind, ordered by
// decreasing size), runs the one-barrier wavefront on it with its own scratch
// slice, and repeats until the queue is empty.  Queries never wait for each
// other, so teams need no co-scheduling beyond their own CTAs.  ALL_KINDS =
// false: a lean instantiation for batches of geometric queries only.
template <class Team, bool ALL_KINDS>
__global__ void __launch_bounds__(1024, 1) plan_batch_kernel(const PlanArgs* __restrict__ queries,
                                                          const int* __restrict__ order, int nq,
                                                          int* __restrict__ next, int* __restrict__ slot,
                                                          BatchScratch scratch, Team team) {
    extern __shared__ float sbox[];
    const int team_id = team.id();
    for (;;) {
        if (team.rank() == 0) slot[team_id] = atomicAdd(next, 1);
        team.sync(nullptr);
        const int k = __ldcg(&slot[team_id]);
        if (k >= nq) break;
        PlanArgs A = queries[order[k]];
        const size_t nm = (size_t)scratch.max_nodes;
        A.ocost = scratch.ocost + team_id * 2 * nm;
        A.stamp = scratch.stamp + team_id * nm;
        assign_plan_lists(A, scratch.lists + team_id * plan_list_stride(nm), nm);
        unsigned dyn_smem;
        asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn_smem));
        // counters in the control block: in this kernel (four bodies inlined)
        // the shared copy cost registers and measured no faster
        constexpr int W = kBatchPullLanes;
        constexpr bool SH = false;
        if (ALL_KINDS && A.kind == GMT_COST_DI) plan_body_fused<Team, GMT_COST_DI, 3, W, SH>(A, team, sbox, dyn_smem);
        else if (ALL_KINDS && A.kind == GMT_COST_DUBINS)
            plan_body_fused<Team, GMT_COST_DUBINS, 3, W, SH>(A, team, sbox, dyn_smem);
        else if (A.dp == 2) plan_body_fused<Team, GMT_COST_EUCLID, 2, W, SH>(A, team, sbox, dyn_smem);
        else plan_body_fused<Team, GMT_COST_EUCLID, 3, W, SH>(A, team, sbox, dyn_smem);
        team.sync(nullptr);
    }
}

// The same with the wavefront's state in the team's shared memory
// (plan_local.cuh), when the batch's largest query fits; a query that leaves
// room also keeps its rows and states there.
template <class Team, bool ALL_KINDS>
__global__ void __launch_bounds__(1024, 1) plan_batch_local_kernel(const PlanArgs* __restrict__ queries,
                                                                const int* __restrict__ order, int nq,
                                                                int* __restrict__ next, int* __restrict__ slot,
                                                                Team team) {
    extern __shared__ __align__(16) unsigned char plan_smem[];
    __shared__ PlanArgs args;
    unsigned dyn_smem;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn_smem));
    const int team_id = team.id();
    for (;;) {
        if (team.rank() == 0) slot[team_id] = atomicAdd(next, 1);
        team.sync(nullptr);
        const int k = __ldcg(&slot[team_id]);
        if (k >= nq) break;
        {
            const int* src = reinterpret_cast<const int*>(&queries[order[k]]);
            for (int t = threadIdx.x; t < (int)(sizeof(PlanArgs) / sizeof(int)); t += blockDim.x)
                reinterpret_cast<int*>(&args)[t] = __ldg(src + t);
        }
        __syncthreads();
        const PlanArgs& A = args;
        const unsigned box_bytes =
            (unsigned)(A.dp == 2 ? local_staged_boxes(A, 2) * BoxSet<2>::kQ : local_staged_boxes(A, 3) * BoxSet<3>::kQ) * 16u;
        const bool cache =
            local_layout(box_bytes, A.N, team.ctas(), A.d, A.kind != GMT_COST_EUCLID, true).total <= dyn_smem;
        constexpr int W = kBatchPullLanes;
        if (ALL_KINDS && A.kind == GMT_COST_DI) plan_body_local<Team, GMT_COST_DI, 3, W>(A, team, plan_smem, cache);
        else if (ALL_KINDS && A.kind == GMT_COST_DUBINS)
            plan_body_local<Team, GMT_COST_DUBINS, 3, W>(A, team, plan_smem, cache);
        else if (A.dp == 2) plan_body_local<Team, GMT_COST_EUCLID, 2, W>(A, team, plan_smem, cache);
        else plan_body_local<Team, GMT_COST_EUCLID, 3, W>(A, team, plan_smem, cache);
        team.sync(nullptr);  // the next query reuses the shared memory and the slot
    }
}

// ----------------------------------------------------------------- launcher
cudaError_t allow_full_smem(const void* kernel) {
    static std::mutex mu;
    static struct { int dev; const void* kernel; } done[256];
    static int n = 0;
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);  // held until it is set: nobody launches before
    for (int k = 0; k < n; ++k)
        if (done[k].dev == dev && done[k].kernel == kernel) return cudaSuccess;
    cudaFuncAttributes a;
    e = cudaFuncGetAttributes(&a, kernel);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)a.sharedSizeBytes);
    if (e == cudaSuccess && n < 256) {  // past the table: set again at each call, to the same value
        done[n].dev = dev;
        done[n++].kernel = kernel;
    }
    return e;
}

namespace {
// Dynamic shared memory a CTA of the local kernels can have.
size_t plan_local_room() {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return (size_t)optin - kPlanStaticSmem - sizeof(LocalCtl);
}

// Does the wavefront's state of an N-node plan fit the shared memory of n
// CTAs, and with the own nodes' rows and states beside it?  CTAs of at most
// 512 threads are kept small enough for two of them to share an SM where the
// row cache is what would prevent it.
bool plan_local_fits(int N, int n, int D, bool directed, size_t box_bytes, int threads, size_t* bytes, bool* cache) {
    if (N < 1 || N > (1 << 20) || (N + n - 1) / n > 65535) return false;
    const size_t room = plan_local_room();
    const size_t with = local_layout((unsigned)box_bytes, N, n, D, directed, true).total;
    const size_t without = local_layout((unsigned)box_bytes, N, n, D, directed, false).total;
    *cache = with <= (threads <= 512 ? std::min(room, (size_t)110 * 1024) : room);
    *bytes = *cache ? with : without;
    return *bytes <= room;
}

template <class Kern, class Team>
cudaError_t launch_local(Kern kern, const PlanArgs& a, const Team& team, bool cache, int n, int threads, size_t smem,
                         cudaStream_t st) {
    cudaError_t e = allow_full_smem((const void*)kern);
    if (e == cudaSuccess && n > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = n;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, a, team, cache);
}

template <int KIND, int DP>
cudaError_t plan_t(const PlanArgs& a, int blocks, int threads, int cluster, cudaStream_t st) {
    const int nbs = a.boxes.count <= smem_box_cap(DP) ? a.boxes.count : 0;
    const size_t smem = plan_smem_bytes(nbs, DP, a.N);
    // one cluster or one CTA: the wavefront's state in its shared memory, when
    // it fits (and the rows can be read four entries at a time)
    const bool aligned = (((uintptr_t)a.out_col | (uintptr_t)a.in_col | (uintptr_t)a.in_cost) & 15) == 0;
    const int n = cluster > 1 ? cluster : 1;
    size_t local = 0;
    bool cache = false;
    if ((cluster > 1 || blocks <= 1) && aligned &&
        plan_local_fits(a.N, n, a.d, KIND != GMT_COST_EUCLID,
                        (size_t)local_staged_boxes(a, DP) * BoxSet<DP>::kQ * 16, threads, &local, &cache))
        return n == 1 ? launch_local(plan_local_kernel<BlockTeam, KIND, DP>, a, BlockTeam{}, cache, 1, threads, local, st)
                      : launch_local(plan_local_kernel<ClusterTeam, KIND, DP>, a, ClusterTeam{}, cache, n, threads,
                                     local, st);
    if (cluster > 1) {
        auto kern = plan_kernel<ClusterTeam, KIND, DP>;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(cluster);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = cluster;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kern, a, ClusterTeam{});
    }
    if (blocks <= 1) {
        plan_kernel<BlockTeam, KIND, DP><<<1, threads, smem, st>>>(a, BlockTeam{});
        return cudaGetLastError();
    }
    GridTeam team;
    team.expected = (unsigned)blocks + ((a.debug_flags & GMT_DEBUG_UNREACHABLE_BARRIER) ? 1u : 0u);
    team.spin_limit = a.spin_limit > 0 ? a.spin_limit : kDefaultSpinLimit;
    PlanArgs args = a;
    void* params[] = {&args, &team};
    return cudaLaunchCooperativeKernel((const void*)plan_kernel<GridTeam, KIND, DP>, dim3(blocks), dim3(threads),
                                       params, smem, st);
}

template <int KIND, int DP>
int occupancy_t(int threads) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const size_t smem = plan_smem_bytes(smem_box_cap(DP), DP, 12 * 1024);  // the most a launch asks for
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, plan_kernel<GridTeam, KIND, DP>, threads, smem);
    return per_sm * sms;
}
}  // namespace

cudaError_t launch_plan(const PlanArgs& a, int blocks, int threads, cudaStream_t st, int cluster) {
    if (a.kind == GMT_COST_DI) return plan_t<GMT_COST_DI, 3>(a, blocks, threads, cluster, st);
    if (a.kind == GMT_COST_DUBINS) return plan_t<GMT_COST_DUBINS, 3>(a, blocks, threads, cluster, st);
    switch (a.dp) {
        case 2: return plan_t<GMT_COST_EUCLID, 2>(a, blocks, threads, cluster, st);
        case 3: return plan_t<GMT_COST_EUCLID, 3>(a, blocks, threads, cluster, st);
        case 4: return plan_t<GMT_COST_EUCLID, 4>(a, blocks, threads, cluster, st);
        case 5: return plan_t<GMT_COST_EUCLID, 5>(a, blocks, threads, cluster, st);
        case 6: return plan_t<GMT_COST_EUCLID, 6>(a, blocks, threads, cluster, st);
        case 7: return plan_t<GMT_COST_EUCLID, 7>(a, blocks, threads, cluster, st);
        case 8: return plan_t<GMT_COST_EUCLID, 8>(a, blocks, threads, cluster, st);
        case 9: return plan_t<GMT_COST_EUCLID, 9>(a, blocks, threads, cluster, st);
        case 10: return plan_t<GMT_COST_EUCLID, 10>(a, blocks, threads, cluster, st);
        default: return cudaErrorInvalidValue;
    }
}

namespace {
template <int KIND, int DP>
cudaError_t load_plan_t(int cluster) {
    cudaFuncAttributes a;
    cudaError_t e = cluster > 1 ? cudaFuncGetAttributes(&a, plan_local_kernel<ClusterTeam, KIND, DP>)
                                : cudaFuncGetAttributes(&a, plan_local_kernel<BlockTeam, KIND, DP>);
    if (e == cudaSuccess)
        e = cluster > 1 ? cudaFuncGetAttributes(&a, plan_kernel<ClusterTeam, KIND, DP>)
                        : cudaFuncGetAttributes(&a, plan_kernel<BlockTeam, KIND, DP>);
    return e;
}
}  // namespace

cudaError_t load_plan_kernel(int kind, int dp, int cluster) {
    if (kind == GMT_COST_DI) return load_plan_t<GMT_COST_DI, 3>(cluster);
    if (kind == GMT_COST_DUBINS) return load_plan_t<GMT_COST_DUBINS, 3>(cluster);
    return dp == 2 ? load_plan_t<GMT_COST_EUCLID, 2>(cluster) : load_plan_t<GMT_COST_EUCLID, 3>(cluster);
}

// Largest cluster size (16, 8, 4, 2) for which one cluster of `threads`-thread
// CTAs can be resident with all the shared memory a plan may ask for; 0 if
// none.  (The kernel that keeps its state in global memory needs less.)
int plan_max_cluster(int kind, int dp, int threads) {
    auto kern = kind == GMT_COST_DI       ? plan_local_kernel<ClusterTeam, GMT_COST_DI, 3>
                : kind == GMT_COST_DUBINS ? plan_local_kernel<ClusterTeam, GMT_COST_DUBINS, 3>
                : dp == 2                 ? plan_local_kernel<ClusterTeam, GMT_COST_EUCLID, 2>
                                          : plan_local_kernel<ClusterTeam, GMT_COST_EUCLID, 3>;
    if (allow_full_smem((const void*)kern) != cudaSuccess ||
        cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
        return 0;
    for (int c = 16; c >= 2; c /= 2) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(c);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = plan_local_room();
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = c;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n > 0) return c;
    }
    cudaGetLastError();
    return 0;
}

namespace {
// Launch configuration of a batched kernel: `teams` clusters of `cluster` CTAs.
struct BatchLaunch {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    BatchLaunch(int teams, int cluster, int threads, size_t smem, cudaStream_t st) {
        cfg.gridDim = dim3(teams * cluster);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = cluster;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
};
template <class Kern>
cudaError_t batch_attributes(Kern kern, int cluster) {
    cudaError_t e = allow_full_smem((const void*)kern);
    if (e == cudaSuccess && cluster > 8)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

// Calls f(kernel, team) with the batched kernel of a shape (scratch kernels
// take the scratch before the team).
template <bool ALL_KINDS, class FL, class FS>
auto with_batch_kernel(int cluster, bool local, const FL& fl, const FS& fs) {
    if (local)
        return cluster <= 1 ? fl(plan_batch_local_kernel<BlockTeam, ALL_KINDS>, BlockTeam{})
                            : fl(plan_batch_local_kernel<ClusterTeam, ALL_KINDS>, ClusterTeam{});
    return cluster <= 1 ? fs(plan_batch_kernel<BlockTeam, ALL_KINDS>, BlockTeam{})
                        : fs(plan_batch_kernel<ClusterTeam, ALL_KINDS>, ClusterTeam{});
}

template <bool ALL_KINDS>
cudaError_t plan_batch_t(const PlanArgs* queries, const int* order, int nq, int* next, int* slot,
                         const BatchScratch& scratch, int teams, int threads, int cluster, size_t smem, bool local,
                         cudaStream_t st) {
    cluster = cluster < 1 ? 1 : cluster;
    BatchLaunch L(teams, cluster, threads, smem, st);
    return with_batch_kernel<ALL_KINDS>(
        cluster, local,
        [&](auto kern, auto team) {
            cudaError_t e = batch_attributes(kern, cluster);
            return e != cudaSuccess ? e : cudaLaunchKernelEx(&L.cfg, kern, queries, order, nq, next, slot, team);
        },
        [&](auto kern, auto team) {
            cudaError_t e = batch_attributes(kern, cluster);
            return e != cudaSuccess ? e
                                    : cudaLaunchKernelEx(&L.cfg, kern, queries, order, nq, next, slot, scratch, team);
        });
}

template <bool ALL_KINDS>
int batch_teams_t(int threads, int cluster, size_t smem, bool local) {
    cluster = cluster < 1 ? 1 : cluster;
    BatchLaunch L(1, cluster, threads, smem, nullptr);
    auto count = [&](auto kern, auto) {
        int n = 0;
        if (batch_attributes(kern, cluster) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, kern, &L.cfg) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        return n;
    };
    return with_batch_kernel<ALL_KINDS>(cluster, local, count, count);
}
}  // namespace

cudaError_t launch_plan_batch(const PlanArgs* queries, const int* order, int nq, int* next, int* slot,
                              const BatchScratch& scratch, int teams, int threads, int cluster, size_t smem,
                              bool local, bool all_kinds, cudaStream_t st) {
    return all_kinds
               ? plan_batch_t<true>(queries, order, nq, next, slot, scratch, teams, threads, cluster, smem, local, st)
               : plan_batch_t<false>(queries, order, nq, next, slot, scratch, teams, threads, cluster, smem, local, st);
}

int plan_batch_max_teams(int threads, int cluster, size_t smem, bool local, bool all_kinds) {
    return all_kinds ? batch_teams_t<true>(threads, cluster, smem, local) : batch_teams_t<false>(threads, cluster, smem, local);
}

size_t plan_local_bytes(int kind, int d, int dp, int N, int boxes, int n) {
    if (N < 1 || N > (1 << 20) || (N + n - 1) / n > 65535) return SIZE_MAX;
    const int staged = boxes <= smem_box_cap(dp) ? boxes : 0;
    const size_t bytes = local_layout((unsigned)(staged * (dp == 2 ? BoxSet<2>::kQ : BoxSet<3>::kQ)) * 16u, N, n, d,
                                      kind != GMT_COST_EUCLID, false)
                             .total;
    return bytes <= plan_local_room() ? bytes : SIZE_MAX;
}

int plan_max_coresident_blocks(int kind, int dp, int threads) {
    if (kind == GMT_COST_DI) return occupancy_t<GMT_COST_DI, 3>(threads);
    if (kind == GMT_COST_DUBINS) return occupancy_t<GMT_COST_DUBINS, 3>(threads);
    switch (dp) {
        case 2: return occupancy_t<GMT_COST_EUCLID, 2>(threads);
        case 3: return occupancy_t<GMT_COST_EUCLID, 3>(threads);
        case 4: return occupancy_t<GMT_COST_EUCLID, 4>(threads);
        case 5: return occupancy_t<GMT_COST_EUCLID, 5>(threads);
        case 6: return occupancy_t<GMT_COST_EUCLID, 6>(threads);
        case 7: return occupancy_t<GMT_COST_EUCLID, 7>(threads);
        case 8: return occupancy_t<GMT_COST_EUCLID, 8>(threads);
        case 9: return occupancy_t<GMT_COST_EUCLID, 9>(threads);
        case 10: return occupancy_t<GMT_COST_EUCLID, 10>(threads);
        default: return 0;
    }
}

}  // namespace gmtk
