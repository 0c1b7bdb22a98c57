// Cell-list neighbour build for one graph (kernels in cells_body.cuh).
#include <cmath>

#include "cells_body.cuh"

namespace gmtk {

template <int D>
__global__ void __launch_bounds__(256) cells_count_kernel(SpaceArgs s, const float* __restrict__ X, CellGrid cg,
                                                          int* __restrict__ cell_of, int* __restrict__ cnt) {
    cell_count_node<D>(s, X, cg, cell_of, cnt, blockIdx.x * blockDim.x + threadIdx.x);
}

__global__ void __launch_bounds__(256) cells_scatter_kernel(int N, const int* __restrict__ cell_of,
                                                            const int* __restrict__ start, int* __restrict__ cnt,
                                                            int* __restrict__ sorted) {
    cell_scatter_node(N, cell_of, start, cnt, sorted, blockIdx.x * blockDim.x + threadIdx.x);
}

template <int D, bool FILL>
__global__ void __launch_bounds__(kCellWarps * 32) cells_tile_kernel(SpaceArgs s, const float* __restrict__ X,
                                                                     CellGrid cg, const int* __restrict__ start,
                                                                     const int* __restrict__ sorted,
                                                                     int* __restrict__ out_count,
                                                                     int* __restrict__ max_deg,
                                                                     const int* __restrict__ row,
                                                                     int* __restrict__ col, float* __restrict__ cost,
                                                                     int* __restrict__ overflow, int words, int rank_words,
                                                                     long long cap) {
    extern __shared__ __align__(16) int cell_buf[];
    if (FILL && cap > 0 && (long long)__ldg(&row[s.N]) > cap) return;  // the caller rebuilds
    cell_tile<D, FILL>(s, X, cg, start, sorted, out_count, max_deg, row, col, cost, overflow, cell_buf, words,
                       rank_words, blockIdx.x);
}

// ---- box grid (checks against many boxes)
// The cell range [c0, c1] of box b on the grid's axes (empty when lo > hi).
__device__ __forceinline__ void box_grid_range(const BoxGridArgs& grid, const int* g, const float* inv_h,
                                               const float* lo, const float* hi, int* c0, int* c1) {
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        c0[a] = box_grid_cell(grid, lo[a], a, g[a], inv_h[a]);
        c1[a] = box_grid_cell(grid, hi[a], a, g[a], inv_h[a]);
    }
}

// One thread per box: counts it in each cell it overlaps, or lists it as big.
__global__ void __launch_bounds__(256) box_grid_count_kernel(BoxArgs boxes, int dp, BoxGridArgs grid,
                                                             int* __restrict__ cnt, int* __restrict__ big,
                                                             int* __restrict__ nbig) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= boxes.count) return;
    const int g[2] = {grid.g, grid.g};
    int c0[2], c1[2];
    box_grid_range(grid, g, grid.inv_h, boxes.lo + (size_t)b * dp, boxes.hi + (size_t)b * dp, c0, c1);
    if (c0[0] > c1[0] || c0[1] > c1[1]) return;  // lo > hi: the box holds no point
    if ((c1[0] - c0[0] + 1) * (c1[1] - c0[1] + 1) > kBoxGridMaxCells) {
        big[atomicAdd(nbig, 1)] = b;
        return;
    }
    for (int cy = c0[1]; cy <= c1[1]; ++cy)
        for (int cx = c0[0]; cx <= c1[0]; ++cx) atomicAdd(&cnt[cy * grid.g + cx], 1);
}

// Entry t of the grid's list is box b (and its packed copy, in 2D and 3D).
__device__ __forceinline__ void box_grid_put(const BoxArgs& boxes, int dp, int b, int t, int* list, float4* packed) {
    list[t] = b;
    if (!packed) return;
    if (dp == 2) pack_box<2>(packed, boxes.lo, boxes.hi, b, t);
    else pack_box<3>(packed, boxes.lo, boxes.hi, b, t);
}

// One warp per box, a lane per cell of its range: writes it into its cells'
// lists (cnt counts back down to 0).
__global__ void __launch_bounds__(256) box_grid_scatter_kernel(BoxArgs boxes, int dp, BoxGridArgs grid,
                                                               const int* __restrict__ start, int* __restrict__ cnt,
                                                               int* __restrict__ list, float4* __restrict__ packed) {
    const int b = (int)((blockIdx.x * (unsigned)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (b >= boxes.count) return;
    int g[2] = {grid.g, grid.g};
    float inv[2] = {grid.inv_h[0], grid.inv_h[1]};
    if (grid.shape) {
        const float4 s = __ldg(grid.shape);
        g[0] = __float_as_int(s.x);
        g[1] = __float_as_int(s.y);
        inv[0] = s.z;
        inv[1] = s.w;
    }
    int c0[2], c1[2];
    box_grid_range(grid, g, inv, boxes.lo + (size_t)b * dp, boxes.hi + (size_t)b * dp, c0, c1);
    if (c0[0] > c1[0] || c0[1] > c1[1]) return;
    const int nx = c1[0] - c0[0] + 1, n = nx * (c1[1] - c0[1] + 1);
    if (n > kBoxGridMaxCells || lane >= n) return;
    const int c = (c0[1] + lane / nx) * g[0] + c0[0] + lane % nx;
    box_grid_put(boxes, dp, b, start[c] + atomicSub(&cnt[c], 1) - 1, list, packed);
}

// Shapes a grid of uneven boxes is chosen among: 2^x by 2^y cells.
constexpr int kShapeFine = 11;  // cells per axis are at most 2^kShapeFine
__constant__ uchar2 kBoxGridShapes[32] = {
    {10, 4}, {9, 5}, {8, 6}, {7, 7}, {6, 8}, {5, 9}, {4, 10}, {3, 11}, {9, 3}, {8, 4}, {7, 5},
    {6, 6},  {5, 7}, {4, 8}, {3, 9}, {8, 2}, {7, 3}, {6, 4},  {5, 5},  {4, 6}, {3, 7}, {2, 8},
    {6, 2},  {5, 3}, {4, 4}, {3, 5}, {2, 6}, {4, 2}, {3, 3},  {2, 4},  {3, 1}, {2, 2}};

// The shape with the fewest boxes to test at a point: the mean list over the
// cells, and every box over more than kBoxGridMaxCells cells; an entry to write
// weighs as 0.15 tests.  From at most 1024 boxes, one of every `step` by a hash
// (obstacles may alternate).  One block of 1024 threads; cost[32] and g[2] in
// shared memory, g the exponents of the result once the block has passed its
// next barrier.
__device__ __forceinline__ void box_grid_choose(const BoxArgs& boxes, int dp, const BoxGridArgs& grid,
                                                unsigned* cost, int* g) {
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid < 32) cost[tid] = 0u;
    const int step = (boxes.count + 1023) / 1024, of = (boxes.count + step - 1) / step;
    const int s = tid * step + (int)(((unsigned)tid * 2654435761u >> 16) % (unsigned)step);
    int c0[2] = {1, 1}, c1[2] = {0, 0};
    if (s < boxes.count) {
        const int fine[2] = {1 << kShapeFine, 1 << kShapeFine};
        const float inv[2] = {(float)fine[0] / grid.span[0], (float)fine[1] / grid.span[1]};
        box_grid_range(grid, fine, inv, boxes.lo + (size_t)s * dp, boxes.hi + (size_t)s * dp, c0, c1);
    }
    const bool ok = c0[0] <= c1[0] && c0[1] <= c1[1];  // else it holds no point
    __syncthreads();
    for (int k = 0; k < 32; ++k) {
        const int sx = kShapeFine - kBoxGridShapes[k].x, sy = kShapeFine - kBoxGridShapes[k].y;
        const int n = ((c1[0] >> sx) - (c0[0] >> sx) + 1) * ((c1[1] >> sy) - (c0[1] >> sy) + 1);
        // entries in the low half (at most 1024 x 32), big boxes in the high
        const unsigned v = __reduce_add_sync(0xffffffffu, !ok ? 0u : n > kBoxGridMaxCells ? 1u << 16 : (unsigned)n);
        if (lane == 0 && v) atomicAdd(&cost[k], v);
    }
    __syncthreads();
    if (tid < 32) {
        const float n = (float)(cost[lane] & 0xffffu), scale = (float)boxes.count / (float)of;
        const float cells = (float)(1 << (kBoxGridShapes[lane].x + kBoxGridShapes[lane].y));
        const float tests = scale * (n / cells + (float)(cost[lane] >> 16)) + 0.15f * n / (float)of;
        const unsigned best = __reduce_min_sync(0xffffffffu, (__float_as_uint(tests) & ~31u) | (unsigned)lane);
        if (lane == (int)(best & 31u)) {
            g[0] = 1 << kBoxGridShapes[lane].x;
            g[1] = 1 << kBoxGridShapes[lane].y;
        }
    }
}

// The counts, the shape and the prefix by one block, its cell counts in shared
// memory: a plan with many boxes builds the grid before the wavefront (and a
// build before sampling), so dependent launches and a memset cost more than the
// work.  With few boxes it writes the lists too, else it leaves the counts to
// box_grid_scatter_kernel.  The block also chooses the grid's
// shape: cells of the mean box's proportions, down to about a quarter of its
// area (a box then lies in about nine).  Obstacles cut into thin slices get thin
// cells: 1500 strips a hundred times wider than high list 2.9 boxes an occupied
// cell (9 at most) on 16 x 1024 cells, 25 (59 at most) on 64 x 64; the Dubins plan
// kernel at n = 5000 went from 0.251 to 0.163 ms, its Halton sampler from 43 to 21
// us.  The area is the boxes' mean, not the product of their mean extents, which
// slices along both axes make far larger.  Where the shape leaves more than
// kBoxGridFewBig boxes over too many cells to be listed, every point would test
// them all, and box_grid_choose picks another: 1500 squares, a tenth of them four
// times wider, 2D n = 1000, a build and plan 1351 -> 258 us (400 on square cells).
constexpr int kBoxGridFewBig = 4;
static_assert(kBoxGridMaxCells <= 32, "the scatter takes a box's cells in one warp");
__global__ void __launch_bounds__(1024) box_grid_block_kernel(BoxArgs boxes, int dp, BoxGridArgs grid,
                                                              int* __restrict__ start, int* __restrict__ list,
                                                              float4* __restrict__ packed, int* __restrict__ big,
                                                              int* __restrict__ nbig, float4* __restrict__ shape,
                                                              int* __restrict__ counts) {
    extern __shared__ int cnt[];  // kBoxGridCells
    __shared__ int warp_sum[32];
    __shared__ float ext[4][32];
    __shared__ unsigned cost[32];
    __shared__ int s_big, s_g[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // mean extents and area of the boxes that hold points
    float w[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (int b = tid; b < boxes.count; b += 1024) {
        const float dx = boxes.hi[(size_t)b * dp] - boxes.lo[(size_t)b * dp];
        const float dy = boxes.hi[(size_t)b * dp + 1] - boxes.lo[(size_t)b * dp + 1];
        if (!(dx >= 0.0f) || !(dy >= 0.0f)) continue;
        const float mx = fminf(dx, grid.span[0]), my = fminf(dy, grid.span[1]);
        w[0] += mx;
        w[1] += my;
        w[2] += 1.0f;
        w[3] += mx * my;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) w[k] += __shfl_xor_sync(0xffffffffu, w[k], o);
        if (lane == 0) ext[k][warp] = w[k];
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            w[k] = ext[k][lane];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) w[k] += __shfl_xor_sync(0xffffffffu, w[k], o);
        }
        if (lane == 0) {
            const float n = fmaxf(w[2], 1.0f);
            const float fx = fmaxf(w[0] / (n * grid.span[0]), 1e-4f), fy = fmaxf(w[1] / (n * grid.span[1]), 1e-4f);
            const float area = fmaxf(w[3] / (n * grid.span[0] * grid.span[1]), 1e-8f);
            int P = 1;
            while (P < kBoxGridCells && 2.0f * (float)P * area <= 4.0f) P *= 2;
            int gy = 1;
            while (gy < P && fx * (float)(P / gy) > 2.0f * fy * (float)gy) gy *= 2;
            s_g[0] = P / gy;
            s_g[1] = gy;
            s_big = 0;
        }
    }
    int g[2], cells;
    float inv[2];
    for (int attempt = 0;; ++attempt) {
        for (int c = tid; c < kBoxGridCells; c += 1024) cnt[c] = 0;
        __syncthreads();
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            g[a] = s_g[a];
            inv[a] = (float)g[a] / grid.span[a];
        }
        cells = g[0] * g[1];
        for (int b = tid; b < boxes.count; b += 1024) {
            int c0[2], c1[2];
            box_grid_range(grid, g, inv, boxes.lo + (size_t)b * dp, boxes.hi + (size_t)b * dp, c0, c1);
            if (c0[0] > c1[0] || c0[1] > c1[1]) continue;  // lo > hi: the box holds no point
            if ((c1[0] - c0[0] + 1) * (c1[1] - c0[1] + 1) > kBoxGridMaxCells) {
                big[atomicAdd(&s_big, 1)] = b;
                continue;
            }
            for (int cy = c0[1]; cy <= c1[1]; ++cy)
                for (int cx = c0[0]; cx <= c1[0]; ++cx) atomicAdd(&cnt[cy * g[0] + cx], 1);
        }
        __syncthreads();
        if (attempt || s_big <= kBoxGridFewBig) break;  // uniform: nothing writes s_big before the next barrier
        box_grid_choose(boxes, dp, grid, cost, s_g);
        if (tid == 0) s_big = 0;  // read by all before the barriers of the choice
    }
    if (tid == 0) *shape = make_float4(__int_as_float(g[0]), __int_as_float(g[1]), inv[0], inv[1]);
    // exclusive prefix of the counts: a warp's run of cells, 32 at a time (a
    // run per thread would meet 16-way bank conflicts)
    constexpr int kPer = kBoxGridCells / 1024;
    const int c0w = warp * 32 * kPer + lane;
    int v[kPer], x[kPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        v[k] = cnt[c0w + 32 * k];
        x[k] = v[k];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x[k], o);
            if (lane >= o) x[k] += y;
        }
        const int total = __shfl_sync(0xffffffffu, x[k], 31);
        x[k] += sum - v[k];
        sum += total;
    }
    if (lane == 31) warp_sum[warp] = sum;
    __syncthreads();
    if (warp == 0) {
        int t = warp_sum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        warp_sum[lane] = t;
    }
    __syncthreads();
    const int before = warp > 0 ? warp_sum[warp - 1] : 0, at = warp_sum[31];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int c = c0w + 32 * k;
        cnt[c] = before + x[k];  // from here on the cell's next free entry
        if (c < cells) start[c] = before + x[k];
        if (counts && c < cells) counts[c] = v[k];
    }
    if (tid == 1023) {
        start[cells] = at;  // the cells past the grid's are empty
        *nbig = s_big;
    }
    if (counts) return;  // the whole chip writes the lists
    __syncthreads();
    for (int b = tid; b < boxes.count; b += 1024) {
        int c0[2], c1[2];
        box_grid_range(grid, g, inv, boxes.lo + (size_t)b * dp, boxes.hi + (size_t)b * dp, c0, c1);
        if (c0[0] > c1[0] || c0[1] > c1[1]) continue;
        if ((c1[0] - c0[0] + 1) * (c1[1] - c0[1] + 1) > kBoxGridMaxCells) continue;
        for (int cy = c0[1]; cy <= c1[1]; ++cy)
            for (int cx = c0[0]; cx <= c1[0]; ++cx)
                box_grid_put(boxes, dp, b, atomicAdd(&cnt[cy * g[0] + cx], 1), list, packed);
    }
}

cudaError_t launch_box_grid(int dp, BoxArgs boxes, const BoxGridArgs& grid, int* cnt, int* start, int* list,
                            float4* packed, int* big, int* nbig, float4* shape, cudaStream_t st) {
    if (dp < 2 || boxes.count < 1 || grid.g > 64) return cudaErrorInvalidValue;
    if (boxes.count <= kBoxGridBlockMax) {
        constexpr int smem = kBoxGridCells * (int)sizeof(int);
        cudaError_t e = cudaFuncSetAttribute(box_grid_block_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        const bool spread = boxes.count > kBoxGridFuseMax;
        box_grid_block_kernel<<<1, 1024, smem, st>>>(boxes, dp, grid, start, list, packed, big, nbig, shape,
                                                     spread ? cnt : nullptr);
        e = cudaGetLastError();
        if (e != cudaSuccess || !spread) return e;
    } else {
        cudaError_t e = cudaMemsetAsync(cnt, 0, (size_t)grid.g * grid.g * sizeof(int), st);
        if (e == cudaSuccess) e = cudaMemsetAsync(nbig, 0, sizeof(int), st);
        if (e != cudaSuccess) return e;
        box_grid_count_kernel<<<(unsigned)((boxes.count + 255) / 256), 256, 0, st>>>(boxes, dp, grid, cnt, big, nbig);
        e = launch_scan(cnt, start, grid.g * grid.g, st);
        if (e != cudaSuccess) return e;
    }
    box_grid_scatter_kernel<<<(unsigned)((boxes.count + 7) / 8), 256, 0, st>>>(boxes, dp, grid, start, cnt, list, packed);
    return cudaGetLastError();
}

bool make_cell_grid(int kind, int d, const float* lo, const float* hi, float r, int N, bool batched, CellGrid* cg,
                    bool* pays) {
    if (kind != GMT_COST_EUCLID || (d != 2 && d != 3) || !(r > 0.0f)) return false;
    // cell side: at least 1.01 r, and coarse enough for at most 2^16 cells
    double h = (double)r * 1.01;
    for (;;) {
        double cells = 1.0;
        for (int a = 0; a < d; ++a) cells *= std::floor(((double)hi[a] - (double)lo[a]) / h) + 1.0;
        if (cells <= 65536.0) break;
        h *= 1.25;
    }
    double frac = 1.0;
    long long ncells = 1;
    for (int a = 0; a < 3; ++a) {
        cg->g[a] = 1;
        cg->lo[a] = 0.0f;
        if (a >= d) continue;
        const double L = (double)hi[a] - (double)lo[a];
        cg->g[a] = (int)std::floor(L / h) + 1;
        cg->lo[a] = lo[a];
        frac *= std::min(1.0, 3.0 * h / L);
        ncells *= cg->g[a];
    }
    // keep h >= 1.01 r for the rounded reciprocal too
    cg->inv_h = (float)(1.0 / h);
    while ((double)r * 1.01 * (double)cg->inv_h > 1.0) cg->inv_h = std::nextafter(cg->inv_h, 0.0f);
    cg->ncells = (int)ncells;
    cg->list_only = 0;
    // measured on one GB300 (Theorem 1 radii, 30 boxes; cell tiles against the
    // packed all-pairs test and the tiled fill; pair test, scan and fill in ms):
    // one graph, 2D: 8192 nodes 0.054 against 0.046, 12000 0.059 against 0.065;
    // 3D: 12000 0.093 against 0.076, 16384 0.099 against 0.117.  In a batch the
    // cell stages' short launches overlap other queries' work, and they pay
    // sooner (builds of 400k nodes in all): 2D: 2500 nodes a query 0.58 against
    // 0.51, 4000 0.54 against 0.68; 3D: 4000 0.93 against 0.86, 6000 1.01
    // against 1.11.
    *pays = frac <= 0.3 && N >= (d == 2 ? (batched ? 3200 : 10500) : (batched ? 5000 : 14000));
    // Cells that replace the all-pairs tiles form their sum, which rounds fewer
    // squares than sq_dist, so that a graph does not depend on which of the two
    // builds it.  Cells have formed sq_dist's from these lines on.
    cg->pairs_sum = !(frac <= 0.25 && N >= (d == 2 ? (batched ? 4096 : 12000) : 32768));
    return true;
}

namespace {
template <int D>
cudaError_t rows_t(const SpaceArgs& s, const float* X, const CellGrid& cg, const int* start, const int* sorted,
                   bool fill, int* out_count, int* max_deg, const int* row, int* col, float* cost, int* overflow, long long cap,
                   cudaStream_t st) {
    const int words = fill ? cell_fill_words(cg, s.N) : 0, rank = fill ? cell_rank_words(cg, s.N) : 0;
    const size_t smem = cell_tile_smem(D, fill, words, rank);
    auto launch = [&](auto kern) {
        const cudaError_t e = allow_full_smem((const void*)kern);
        if (e != cudaSuccess) return e;
        kern<<<cg.ncells, kCellWarps * 32, smem, st>>>(s, X, cg, start, sorted, out_count, max_deg, row, col, cost,
                                                       overflow, words, rank, cap);
        return cudaSuccess;
    };
    const cudaError_t e = fill ? launch(cells_tile_kernel<D, true>) : launch(cells_tile_kernel<D, false>);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}
}  // namespace

cudaError_t launch_cells_count(const SpaceArgs& s, const float* X, const CellGrid& cg, int* cell_of, int* cell_cnt,
                               cudaStream_t st) {
    const int blocks = (s.N + 255) / 256;
    if (s.d == 2) cells_count_kernel<2><<<blocks, 256, 0, st>>>(s, X, cg, cell_of, cell_cnt);
    else if (s.d == 3) cells_count_kernel<3><<<blocks, 256, 0, st>>>(s, X, cg, cell_of, cell_cnt);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
}

cudaError_t launch_cells_scatter(int N, const int* cell_of, const int* cell_start, int* cell_cnt, int* sorted,
                                 cudaStream_t st) {
    cells_scatter_kernel<<<(N + 255) / 256, 256, 0, st>>>(N, cell_of, cell_start, cell_cnt, sorted);
    return cudaGetLastError();
}

cudaError_t launch_cells_rows(const SpaceArgs& s, const float* X, const CellGrid& cg, const int* cell_of,
                              const int* cell_start, const int* sorted, bool fill, int* out_count, int* max_deg,
                              const int* row, int* col, float* cost, int* overflow, cudaStream_t st, long long cap) {
    (void)cell_of;
    if (s.d == 2) return rows_t<2>(s, X, cg, cell_start, sorted, fill, out_count, max_deg, row, col, cost, overflow, cap, st);
    if (s.d == 3) return rows_t<3>(s, X, cg, cell_start, sorted, fill, out_count, max_deg, row, col, cost, overflow, cap, st);
    return cudaErrorInvalidValue;
}

}  // namespace gmtk
