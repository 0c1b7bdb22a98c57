// Cell-list neighbour search for geometric graphs in 2 and 3 dimensions: a
// faster way to the same neighbour sets (Section III-A's r-disk neighbours,
// precomputed in Section V-A), not a change of the method.  Nodes are
// counting-sorted by grid cell; a row's candidates are the nodes of the 3^d
// cells around its own, which lie in 3^(d-1) runs of consecutive cells along
// axis 0.  Every candidate takes an FP32 edge predicate, and each row's columns
// come out in ascending order.  With pairs_sum the predicate is the all-pairs
// tiles' and the CSR is the same bits as theirs; without it every square is
// rounded (sq_dist), and a pair within one rounding of the radius may differ.
//
// One CTA per cell (a cell tile): the cell's candidates (the same for every
// row of the cell) are loaded into shared memory once, with their coordinates,
// two to a float4; for the fill they are ordered by node index through a bitmap
// of the graph's nodes (a candidate's rank is the number of bits below its
// own).  Then 32 rows at a time, a lane per row: a warp tests its rows against
// 32 candidates with packed FP32 arithmetic (two candidates per instruction),
// which gives each row a word of verdicts.  The count pass adds up their bits;
// the fill compacts a row's verdicts into a list and writes the row's columns
// and costs from it, all lanes busy and consecutive.  A cell with more than
// tile_cand candidates takes the row-by-row path instead (one warp per row,
// candidates gathered from global memory, columns ordered through a bitmap of
// the row or a sorted list).
// Measured on one GB300 against candidates sorted bitonically and one row per
// warp tested lane by lane (3D, 65537 nodes, 15 M edges): count 113 -> 57 us
// (51 with the squares not rounded on their own), fill 365 -> 132 us.
#pragma once

#include "graph_body.cuh"

namespace gmtk {

constexpr int kCellWarps = 8;  // warps per cell tile
// Candidates a cell tile holds in shared memory, and how many of a row's
// verdicts the fill compacts at a time (a u16 list per warp).
__host__ __device__ constexpr int tile_cand(int D) { return D == 3 ? 2048 : 1024; }
constexpr int kTileChunk = 1024;
// Nodes up to which candidates are ordered through a bitmap of the nodes (24
// KB of shared memory); larger graphs sort them (bitonic).
constexpr int kTileRankNodes = 131072;

template <int D>
__device__ __forceinline__ int cell_index(const CellGrid& cg, const float* x) {
    int idx = 0;
#pragma unroll
    for (int a = D - 1; a >= 0; --a) {
        int k = (int)floorf((x[a] - cg.lo[a]) * cg.inv_h);
        k = min(max(k, 0), cg.g[a] - 1);
        idx = idx * cg.g[a] + k;
    }
    return idx;
}

template <int D>
__device__ __forceinline__ void cell_count_node(const SpaceArgs& s, const float* __restrict__ X, const CellGrid& cg,
                                                int* __restrict__ cell_of, int* __restrict__ cnt, int v) {
    if (v >= s.N) return;
    float x[D];
#pragma unroll
    for (int a = 0; a < D; ++a) x[a] = X[(size_t)a * s.pitch + v];
    const int c = cell_index<D>(cg, x);
    cell_of[v] = c;
    atomicAdd(&cnt[c], 1);
}

__device__ __forceinline__ void cell_scatter_node(int N, const int* __restrict__ cell_of,
                                                  const int* __restrict__ start, int* __restrict__ cnt,
                                                  int* __restrict__ sorted, int v) {
    if (v >= N) return;
    const int c = cell_of[v];
    sorted[start[c] + atomicSub(&cnt[c], 1) - 1] = v;
}

// Words of the row-by-row fill's per-warp buffer for a graph of N nodes.
__host__ __device__ inline int cell_fill_words(const CellGrid& cg, int N) {
    const int W = (N + 31) / 32;
    return !cg.list_only && W <= kCellList ? W : kCellList;
}

// Words of the bitmap that orders the fill's candidates (0: they are sorted).
__host__ __device__ inline int cell_rank_words(const CellGrid& cg, int N) {
    return !cg.list_only && N <= kTileRankNodes ? (N + 31) / 32 : 0;
}

// Byte offsets of a cell tile's shared memory: coordinates in pairs (x0 x1 y0
// y1, then z0 z1), candidates, the row group's verdict words (fill) or counts,
// then the ordering bitmap with its prefixes, whose place the warps' lists take.
struct CellTileLayout {
    unsigned z, cand, mask, lists, total;
};
__host__ __device__ inline CellTileLayout cell_tile_layout(int D, bool fill, int rank_words) {
    const unsigned T = (unsigned)tile_cand(D);
    CellTileLayout L;
    L.z = 8u * T;
    L.cand = L.z + (D == 3 ? 4u * T : 0u);
    L.mask = L.cand + 4u * T;
    L.lists = L.mask + (fill ? 32u * (T / 32 + 1) * 4u : 32u * 4u);
    const unsigned rank = 6u * (unsigned)rank_words, lists = kCellWarps * kTileChunk * 2u;
    L.total = L.lists + (fill ? (rank > lists ? rank : lists) : 0u);
    return L;
}

// Dynamic shared memory of a cell tile: the candidate tile or, for a cell
// with too many candidates, the row-by-row buffers of its warps.
__host__ __device__ inline size_t cell_tile_smem(int D, bool fill, int words, int rank_words) {
    const size_t tile = cell_tile_layout(D, fill, rank_words).total;
    const size_t rows = (size_t)kCellWarps * words * sizeof(int);
    return tile > rows ? tile : rows;
}

// The candidate runs of cell `cell`: up to 3^(d-1) runs of consecutive cells
// along axis 0 ([rs, re) in the cell-sorted node order).  Returns their total.
template <int D>
__device__ __forceinline__ int cell_runs(const CellGrid& cg, const int* __restrict__ start, int cell, int* rs,
                                         int* re) {
    constexpr int NR = D == 3 ? 9 : 3;
    int c[3] = {0, 0, 0};
#pragma unroll
    for (int a = 0; a < D; ++a) {
        c[a] = cell % cg.g[a];
        cell /= cg.g[a];
    }
    int T = 0;
#pragma unroll
    for (int k = 0; k < NR; ++k) {
        const int y = c[1] + (k % 3) - 1, z = D == 3 ? c[2] + (k / 3) - 1 : 0;
        const bool ok = y >= 0 && y < cg.g[1] && z >= 0 && z < cg.g[2];
        const int base = (z * cg.g[1] + y) * cg.g[0];
        const int x0 = max(c[0] - 1, 0), x1 = min(c[0] + 1, cg.g[0] - 1);
        rs[k] = ok ? start[base + x0] : 0;
        re[k] = ok ? start[base + x1 + 1] : 0;
        T += re[k] - rs[k];
    }
    return T;
}

// Candidate t of the runs (t < their total).
template <int D>
__device__ __forceinline__ int run_candidate(const int* __restrict__ sorted, const int* rs, const int* re, int t) {
    constexpr int NR = D == 3 ? 9 : 3;
    int j = -1, off = t;
#pragma unroll
    for (int k = 0; k < NR; ++k) {
        const int len = re[k] - rs[k];
        if (j < 0 && off >= 0 && off < len) j = sorted[rs[k] + off];
        off -= len;
    }
    return j;
}

// Row-by-row path, one warp: row v with candidates in the given runs.  Count
// pass (FILL = false) or fill pass, whose warp buffer `list` holds
// cell_fill_words(cg, N) words.
template <int D, bool FILL>
__device__ __forceinline__ void cell_row(const SpaceArgs& s, const float* __restrict__ X, const CellGrid& cg,
                                         const int* __restrict__ sorted, const int* rs, const int* re, int T,
                                         int* __restrict__ out_count, int* __restrict__ max_deg,
                                         const int* __restrict__ row, int* __restrict__ col, float* __restrict__ cost,
                                         int* __restrict__ overflow, int* list, int v) {
    const int lane = threadIdx.x & 31;
    float xv[D];
#pragma unroll
    for (int a = 0; a < D; ++a) xv[a] = X[(size_t)a * s.pitch + v];
    // Fill: with N <= 32 kCellList the warp's buffer holds a bitmap of the
    // row's columns, which yields them in ascending order; larger graphs keep
    // a list of columns and sort it (bitonic).
    const int W = (s.N + 31) / 32;
    const bool bitmap = FILL && W <= kCellList && !cg.list_only;
    if (bitmap) {
        for (int q = lane; q < W; q += 32) list[q] = 0;
        __syncwarp();
    }
    int n = 0;
    for (int t0 = 0; t0 < T; t0 += 32) {
        const int t = t0 + lane;
        const int j = t < T ? run_candidate<D>(sorted, rs, re, t) : -1;
        bool pass = false;
        if (j >= 0 && j != v) {
            float xj[D];
#pragma unroll
            for (int a = 0; a < D; ++a) xj[a] = X[(size_t)a * s.pitch + j];
            pass = cg.pairs_sum ? sq_dist_pairs<D>(xv, xj) < s.r2_threshold : connects<GMT_COST_EUCLID, D>(s, xv, xj);
        }
        const unsigned m = __ballot_sync(0xffffffffu, pass);
        if (bitmap) {
            if (pass) atomicOr((unsigned*)&list[j >> 5], 1u << (j & 31));
        } else if (FILL) {
            const int pos = n + __popc(m & ((1u << lane) - 1u));
            if (pass && pos < kCellList) list[pos] = j;
        }
        n += __popc(m);
    }
    if (!FILL) {
        if (lane == 0) {
            out_count[v] = n;
            atomicMax(max_deg, n);
        }
        return;
    }
    const int b = row[v];
    if (bitmap) {
        __syncwarp();
        int done = 0;
        for (int c0 = 0; c0 < W; c0 += 32) {
            const int wd = c0 + lane;
            unsigned bits = wd < W ? (unsigned)list[wd] : 0u;
            const int cnt = __popc(bits);
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            int pos = b + done + incl - cnt;
            while (bits) {
                const int j = 32 * wd + __ffs(bits) - 1;
                bits &= bits - 1;
                float xj[D];
#pragma unroll
                for (int a = 0; a < D; ++a) xj[a] = X[(size_t)a * s.pitch + j];
                col[pos] = j;
                cost[pos] = edge_cost<GMT_COST_EUCLID, D>(s, xv, xj);
                ++pos;
            }
            done += __shfl_sync(0xffffffffu, incl, 31);
        }
        __syncwarp();
        return;
    }
    if (n > kCellList) {
        if (lane == 0) atomicExch(overflow, 1);
        return;
    }
    // bitonic sort of the row's columns (padded to a power of two with INT_MAX)
    int L = 1;
    while (L < n) L <<= 1;
    for (int t = n + lane; t < L; t += 32) list[t] = INT_MAX;
    __syncwarp();
    for (int k = 2; k <= L; k <<= 1) {
        for (int jj = k >> 1; jj > 0; jj >>= 1) {
            for (int i = lane; i < L; i += 32) {
                const int ix = i ^ jj;
                if (ix > i) {
                    const int a = list[i], b2 = list[ix];
                    if ((a > b2) == ((i & k) == 0)) {
                        list[i] = b2;
                        list[ix] = a;
                    }
                }
            }
            __syncwarp();
        }
    }
    for (int t = lane; t < n; t += 32) {
        const int j = list[t];
        float xj[D];
#pragma unroll
        for (int a = 0; a < D; ++a) xj[a] = X[(size_t)a * s.pitch + j];
        col[b + t] = j;
        cost[b + t] = edge_cost<GMT_COST_EUCLID, D>(s, xv, xj);
    }
    __syncwarp();
}

// Verdicts of a row (its coordinates in both halves of xi) on candidates
// 32 w to 32 w + 31.  PAIRS: the all-pairs tiles' sum, else sq_dist's.
template <int D, bool PAIRS>
__device__ __forceinline__ unsigned cell_verdicts(const float* xy, const float* zz, const unsigned long long* xi, int w,
                                                  float thr) {
    unsigned bits = 0u;
#pragma unroll
    for (int b = 0; b < 32; b += 2) {
        const float4 q = reinterpret_cast<const float4*>(xy)[w * 16 + (b >> 1)];
        const unsigned long long t0 = f2_sub(f2_pack(q.x, q.y), xi[0]);
        const unsigned long long t1 = f2_sub(f2_pack(q.z, q.w), xi[1]);
        unsigned long long d2 = PAIRS ? f2_sqr_add(t0, f2_mul(t1, t1)) : f2_add(f2_sqr(t0), f2_sqr(t1));
        if (D == 3) {
            const float2 z = reinterpret_cast<const float2*>(zz)[w * 16 + (b >> 1)];
            const unsigned long long t2 = f2_sub(f2_pack(z.x, z.y), xi[2]);
            d2 = PAIRS ? f2_sqr_add(t2, d2) : f2_add(d2, f2_sqr(t2));
        }
        float da, db;
        f2_unpack(d2, da, db);
        bits |= (da < thr ? 1u : 0u) << b;
        bits |= (db < thr ? 1u : 0u) << (b + 1);
    }
    return bits;
}

// One CTA of kCellWarps warps: every row of cell `cell`.  smem:
// cell_tile_smem(D, FILL, words, rank_words) bytes, 16-byte aligned; words =
// cell_fill_words(cg, N) and rank_words = cell_rank_words(cg, N) for the fill.
template <int D, bool FILL>
__device__ __forceinline__ void cell_tile(const SpaceArgs& s, const float* __restrict__ X, const CellGrid& cg,
                                          const int* __restrict__ start, const int* __restrict__ sorted,
                                          int* __restrict__ out_count, int* __restrict__ max_deg,
                                          const int* __restrict__ row, int* __restrict__ col,
                                          float* __restrict__ cost, int* __restrict__ overflow, int* smem, int words,
                                          int rank_words, int cell) {
    constexpr int NR = D == 3 ? 9 : 3;
    constexpr int kCand = tile_cand(D), kPitch = kCand / 32 + 1;
    const int r0 = start[cell], R = start[cell + 1] - r0;
    if (R <= 0) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
    const float INF = f_inf();
    int rs[NR], re[NR];
    const int T = cell_runs<D>(cg, start, cell, rs, re);
    if (T > kCand) {
        for (int r = warp; r < R; r += kCellWarps)
            cell_row<D, FILL>(s, X, cg, sorted, rs, re, T, out_count, max_deg, row, col, cost, overflow,
                              smem + warp * words, sorted[r0 + r]);
        return;
    }
    const CellTileLayout L = cell_tile_layout(D, FILL, rank_words);
    unsigned char* const base = reinterpret_cast<unsigned char*>(smem);
    float* const xy = reinterpret_cast<float*>(base);
    float* const zz = reinterpret_cast<float*>(base + L.z);
    int* const cand = reinterpret_cast<int*>(base + L.cand);
    unsigned* const mask = reinterpret_cast<unsigned*>(base + L.mask);  // [32][kPitch]
    int* const counts = reinterpret_cast<int*>(base + L.mask);
    unsigned* const bitmap = reinterpret_cast<unsigned*>(base + L.lists);
    unsigned short* const prefix = reinterpret_cast<unsigned short*>(bitmap + rank_words);
    unsigned short* const list = reinterpret_cast<unsigned short*>(base + L.lists) + warp * kTileChunk;
    auto place = [&](int t, int j) {  // candidate t is node j (-1: none, infinitely far)
        const int p = t >> 1, h = t & 1;
        xy[4 * p + h] = j >= 0 ? X[j] : INF;
        xy[4 * p + 2 + h] = j >= 0 ? X[(size_t)s.pitch + j] : INF;
        if (D == 3) zz[2 * p + h] = j >= 0 ? X[(size_t)2 * s.pitch + j] : INF;
    };
    const int nw = (T + 31) / 32;  // words of verdicts per row
    if (!FILL) {
        for (int t = tid; t < nw * 32; t += blockDim.x) place(t, t < T ? run_candidate<D>(sorted, rs, re, t) : -1);
    } else if (rank_words > 0) {
        __shared__ int warp_sum[kCellWarps];
        for (int w = tid; w < rank_words; w += blockDim.x) bitmap[w] = 0u;
        __syncthreads();
        for (int t = tid; t < T; t += blockDim.x) {
            const int j = run_candidate<D>(sorted, rs, re, t);
            atomicOr(&bitmap[j >> 5], 1u << (j & 31));
        }
        __syncthreads();
        // exclusive prefix of the words' bits, a run of words per thread
        const int per = (rank_words + (int)blockDim.x - 1) / (int)blockDim.x;
        const int w0 = min(rank_words, tid * per), w1 = min(rank_words, w0 + per);
        int sum = 0;
        for (int w = w0; w < w1; ++w) sum += __popc(bitmap[w]);
        int incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) warp_sum[warp] = incl;
        __syncthreads();
        int at = incl - sum;
        for (int w = 0; w < warp; ++w) at += warp_sum[w];
        // the run's candidates, in order
        for (int w = w0; w < w1; ++w) {
            prefix[w] = (unsigned short)at;
            at += __popc(bitmap[w]);
        }
        __syncthreads();
        for (int t = tid; t < nw * 32; t += blockDim.x) {
            if (t < T) {
                const int j = run_candidate<D>(sorted, rs, re, t);
                const int k = prefix[j >> 5] + __popc(bitmap[j >> 5] & ((1u << (j & 31)) - 1u));
                cand[k] = j;
                place(k, j);
            } else {
                place(t, -1);
            }
        }
    } else {
        int P2 = 1;  // sort the candidates by node index (bitonic, padded with INT_MAX)
        while (P2 < T) P2 <<= 1;
        for (int t = tid; t < P2; t += blockDim.x) cand[t] = t < T ? run_candidate<D>(sorted, rs, re, t) : INT_MAX;
        __syncthreads();
        for (int k = 2; k <= P2; k <<= 1) {
            for (int jj = k >> 1; jj > 0; jj >>= 1) {
                for (int i = tid; i < P2; i += blockDim.x) {
                    const int ix = i ^ jj;
                    if (ix > i) {
                        const int a = cand[i], b2 = cand[ix];
                        if ((a > b2) == ((i & k) == 0)) {
                            cand[i] = b2;
                            cand[ix] = a;
                        }
                    }
                }
                __syncthreads();
            }
        }
        for (int t = tid; t < nw * 32; t += blockDim.x) place(t, t < T ? cand[t] : -1);
    }
    const float thr = s.r2_threshold;
    for (int g0 = 0; g0 < R; g0 += 32) {
        if (!FILL && tid < 32) counts[tid] = 0;
        __syncthreads();  // the candidates; the previous rows' verdicts are used
        // verdicts of 32 rows, a lane per row
        const bool has = g0 + lane < R;
        const int v = has ? sorted[r0 + g0 + lane] : 0;
        unsigned long long xi[3];
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const float c = X[(size_t)a * s.pitch + v];
            xi[a] = f2_pack(c, c);
        }
        int self = 0;  // the row's own place among the candidates (its distance, 0, passes the test)
        if (FILL) {
            int hi = T - 1;
            while (self < hi) {
                const int mid = (self + hi) >> 1;
                if (cand[mid] < v) self = mid + 1;
                else hi = mid;
            }
        }
        int cnt = 0;
        for (int w = warp; w < nw; w += kCellWarps) {
            unsigned bits = cg.pairs_sum ? cell_verdicts<D, true>(xy, zz, xi, w, thr) : cell_verdicts<D, false>(xy, zz, xi, w, thr);
            if (!has) bits = 0u;
            if (FILL) {
                if ((self >> 5) == w) bits &= ~(1u << (self & 31));
                mask[lane * kPitch + w] = bits;
            } else {
                cnt += __popc(bits);
            }
        }
        if (!FILL) {
            if (has && cnt) atomicAdd(&counts[lane], cnt);
            __syncthreads();
            if (warp == 0 && has) {
                // without the node itself, which passes the test only if its
                // coordinates are finite (a bad start or appended sample, which
                // the build reports, may not be: a count is never negative)
                float x[D];
#pragma unroll
                for (int a = 0; a < D; ++a) x[a] = X[(size_t)a * s.pitch + v];
                out_count[v] = counts[lane] - (sq_dist_pairs<D>(x, x) < thr ? 1 : 0);
            }
            __syncthreads();
            continue;
        }
        __syncthreads();
        // columns and costs, a warp per row
        for (int r = warp; r < min(32, R - g0); r += kCellWarps) {
            const int u = __shfl_sync(0xffffffffu, v, r);
            float xu[D];
#pragma unroll
            for (int a = 0; a < D; ++a) xu[a] = X[(size_t)a * s.pitch + u];
            int pos = row[u];
            const int end = row[u + 1];
            for (int w0 = 0; w0 < nw; w0 += kTileChunk / 32) {
                const int w = w0 + lane;
                unsigned bits = w < nw ? mask[r * kPitch + w] : 0u;
                const int n = __popc(bits);
                int incl = n;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                const int total = __shfl_sync(0xffffffffu, incl, 31);
                for (int k = incl - n; bits; bits &= bits - 1) list[k++] = (unsigned short)(32 * w + __ffs(bits) - 1);
                __syncwarp();
                for (int e = lane; e < total; e += 32) {
                    const int t = list[e], p = t >> 1, h = t & 1;
                    float xj[3] = {xy[4 * p + h], xy[4 * p + 2 + h], D == 3 ? zz[2 * p + h] : 0.0f};
                    if (pos + e < end) {
                        col[pos + e] = cand[t];
                        cost[pos + e] = edge_cost<GMT_COST_EUCLID, D>(s, xu, xj);
                    }
                }
                pos += total;
                __syncwarp();
            }
        }
    }
}

}  // namespace gmtk
