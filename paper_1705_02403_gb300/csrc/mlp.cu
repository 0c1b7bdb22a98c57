// Learned sampling proposal: the BF16 tensor-core GEMM launcher and the C ABI
// entry point that exposes it (gmt_gemm_bf16).  The network, its training and
// the proposal sampler build on these (proposal.cu).
#include <algorithm>
#include <atomic>
#include <climits>
#include <cstring>
#include <mutex>
#include <string>

#include "gemm_tc.cuh"
#include "internal.h"

namespace gmtk {

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    });
    return fn;
}

// Tensor map of a row-major BF16 matrix [rows, cols] (cols contiguous) read in
// boxes of 64 columns x box_rows rows, 128-byte swizzle, zero fill out of range.
cudaError_t make_map(CUtensorMap* map, const void* ptr, int rows, int cols, int box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return cudaErrorNotSupported;
    if (((uintptr_t)ptr & 15) != 0 || (cols * 2) % 16 != 0) return cudaErrorInvalidValue;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kGemmBK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// Tensor map of an FP32 output [slices][rows][cols] (cols contiguous, row
// stride ld floats) written in boxes of 32 x 32, 128-byte swizzle.
cudaError_t make_out_map(CUtensorMap* map, float* ptr, int slices, int rows, int cols, int ld) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return cudaErrorNotSupported;
    const cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)slices};
    const cuuint64_t strides[2] = {(cuuint64_t)ld * 4, (cuuint64_t)ld * 4 * (cuuint64_t)rows};
    const cuuint32_t box[3] = {32, 32, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, ptr, dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

int device_sms() {
    static std::atomic<int> cached{0};
    int sms = cached.load(std::memory_order_relaxed);
    if (sms <= 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
            sms = 148;
        cached.store(sms, std::memory_order_relaxed);
    }
    return sms;
}

// Columns of a CTA pair's tile: the width that finishes soonest, taking a
// tile's time as its columns (at least 64: below, the loads of A's 256 rows
// set the pace) plus 24 columns' worth of pipeline fill and epilogue tail,
// times the waves of items over the pairs.  4096^3 takes 224 (304 items, four
// full waves of 76) where 256 (256 items) would leave the fourth a third full.
int pair_tile_n(int M, int N, int splits, int pairs, bool b_mn) {
    int best = 256;
    long long best_cost = LLONG_MAX;
    for (int t = 256; t >= 32; t -= 32) {
        if (b_mn && t % 128) continue;  // each CTA's half is read in boxes of 64 rows
        const long long items = (long long)((M + 255) / 256) * ((N + t - 1) / t) * splits;
        const long long cost = (items + pairs - 1) / pairs * (std::max(t, 64) + 24);
        if (cost < best_cost) { best_cost = cost; best = t; }
    }
    return best;
}

// Does a product of more than 128 rows run on single CTAs all the same?  per:
// the K-blocks of a slice; rowwise: the output leaves row by row (BF16, or FP32
// rows that do not start on 16 bytes), which costs a pair's two epilogues more
// than four of a single CTA's tiles cost theirs.  With one wave of 128 x 128
// tiles or less and deep K both kernels wait for the same loads, and a pair's
// tiles only split them more finely.  One GB300, single CTAs against pairs, us:
// BF16 513 x 20000 x 64 28 and 36, 8192 x 8192 x 64 141 and 170, 4096 x 4096 x 128
// 38 and 45, 4096 x 512 x 512 94% of the pairs', FP32 2048 x 1003 x 256 the same,
// 2048 x 128 x 8192 43 and 46; the other way BF16 8192 x 8192 x 512 61% faster on
// pairs, 513 x 4096 x 512 8%, 1000 x 1003 x 256 29%, FP32 256 x 4096 x 1024 10%.
// (Bits are equal.)
bool single_ctas(int M, int N, int splits, int per, bool rowwise) {
    const long long tiles_n = (N + kGemmBN - 1) / kGemmBN, tiles = (M + kGemmBM - 1) / kGemmBM * tiles_n * splits;
    const int sms = device_sms();
    if (tiles_n > 65535) return false;  // the grid's limit
    if (tiles <= sms && per > 2048 / kGemmBK) return true;
    return rowwise && 2 * tiles > sms && (tiles <= sms || per < 512 / kGemmBK);
}

// Sum of split-K partials [splits][M][N] plus the epilogue.
__global__ void splitk_reduce_kernel(const float* __restrict__ part, int splits, int M, int N, int epilogue,
                                     const float* __restrict__ bias, float* __restrict__ C,
                                     __nv_bfloat16* __restrict__ Cb, int ldc) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)M * N) return;
    const int row = (int)(t / N), col = (int)(t % N);
    float s = 0.0f;
    for (int k = 0; k < splits; ++k) s += part[(size_t)k * M * N + t];
    if (epilogue == kEpiBiasReluBF16) {
        const float x = fmaxf(s + (bias ? bias[col] : 0.0f), 0.0f);
        Cb[(size_t)row * ldc + col] = __float2bfloat16_rn(x);
    } else {
        C[(size_t)row * ldc + col] = s + ((epilogue == kEpiBiasF32 && bias) ? bias[col] : 0.0f);
    }
}

}  // namespace

// C = A . B^T with A [M, K], B [N, K] BF16 row-major (a_mn, b_mn: the operand is
// stored [K, M] or [K, N] instead; M > 128 only); epilogue as GemmEpilogue.
// splits > 1 splits K into `partial` ([splits][M][N] FP32) and reduces
// deterministically.
cudaError_t gemm_bf16_tn(int M, int N, int K, const __nv_bfloat16* A, const __nv_bfloat16* B, int epilogue,
                         const float* bias, float* C, __nv_bfloat16* Cb, int ldc, int splits, float* partial,
                         int* error, cudaStream_t st, bool a_mn, bool b_mn, int* partials_left) {
    if (M <= 0 || N <= 0 || K <= 0 || (K % 8 != 0 && !(a_mn && b_mn))) return cudaErrorInvalidValue;
    static std::atomic<bool> attr_set{false};  // setting it twice is harmless
    if (!attr_set.load(std::memory_order_relaxed)) {
        cudaError_t e = cudaFuncSetAttribute(gemm_tn_bf16_kernel<kGemmStagesDeep>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             gemm_smem_bytes(kGemmStagesDeep));
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(gemm_tn_bf16_kernel<kGemmStagesShort>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, gemm_smem_bytes(kGemmStagesShort));
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(gemm_pair_bf16_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmem);
        if (e != cudaSuccess) return e;
        attr_set.store(true, std::memory_order_relaxed);
    }
    const int kb = (K + kGemmBK - 1) / kGemmBK;
    if (splits < 1) splits = 1;
    if (splits > kb) splits = kb;
    const int per = (kb + splits - 1) / splits;
    splits = (kb + per - 1) / per;  // every split gets at least one K-block
    if (splits > 1 && !partial) return cudaErrorInvalidValue;
    PairArgs p;
    std::memset(&p, 0, sizeof(p));
    GemmArgs& g = p.g;
    g.M = M; g.N = N; g.K = K; g.k_blocks_per_split = per; g.error = error; g.bias = bias; g.ldc = ldc;
    g.epilogue = epilogue; g.C = C; g.Cb = Cb;
    if (splits > 1) { g.epilogue = kEpiPartialF32; g.C = partial; g.ldc = N; }
    CUtensorMap ta, tb;
    cudaError_t e;
    // More than half a pair's rows: CTA pairs.  (M <= 128 would leave the
    // second CTA of every pair without rows: 4096 x 4096 x 128 rows.)
    // FP32 outputs leave a pair by TMA where their rows start on 16 bytes
    const bool tma = g.epilogue != kEpiBiasReluBF16 && g.ldc % 4 == 0 && ((uintptr_t)g.C & 15) == 0;
    if (a_mn || b_mn || (M > kGemmBM && !single_ctas(M, N, splits, per, !tma))) {
        const int pairs = std::max(1, device_sms() / 2);
        p.splits = splits; p.a_mn = a_mn; p.b_mn = b_mn;
        p.tile_n = pair_tile_n(M, N, splits, pairs, b_mn);
        p.tiles_m = (M + 255) / 256;
        p.tiles_n = (N + p.tile_n - 1) / p.tile_n;
        e = a_mn ? make_map(&ta, A, K, M, kGemmBK) : make_map(&ta, A, M, K, kGemmBM);
        if (e == cudaSuccess) e = b_mn ? make_map(&tb, B, K, N, kGemmBK) : make_map(&tb, B, N, K, p.tile_n / 2);
        if (e != cudaSuccess) return e;
        const long long items = (long long)p.tiles_m * p.tiles_n * splits;
        if (items > INT_MAX) return cudaErrorInvalidValue;
        CUtensorMap tc;
        std::memset(&tc, 0, sizeof(tc));
        p.tma_store = tma && make_out_map(&tc, g.C, g.epilogue == kEpiPartialF32 ? splits : 1, M, N, g.ldc) == cudaSuccess;
        gemm_pair_bf16_kernel<<<2 * (int)std::min<long long>(items, pairs), kPairThreads, kPairSmem, st>>>(ta, tb, tc, p);
    } else {
        e = make_map(&ta, A, M, K, kGemmBM);
        if (e == cudaSuccess) e = make_map(&tb, B, N, K, kGemmBN);
        if (e != cudaSuccess) return e;
        const dim3 grid((M + kGemmBM - 1) / kGemmBM, (N + kGemmBN - 1) / kGemmBN, splits);
        // short K: a shallow ring, two CTAs per SM
        if (per <= 2 * kGemmStagesShort)
            gemm_tn_bf16_kernel<kGemmStagesShort><<<grid, 128, gemm_smem_bytes(kGemmStagesShort), st>>>(ta, tb, g);
        else
            gemm_tn_bf16_kernel<kGemmStagesDeep><<<grid, 128, gemm_smem_bytes(kGemmStagesDeep), st>>>(ta, tb, g);
    }
    e = cudaGetLastError();
    if (partials_left) *partials_left = splits;
    if (e != cudaSuccess || splits == 1 || partials_left) return e;
    const long long total = (long long)M * N;
    splitk_reduce_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(partial, splits, M, N, epilogue, bias, C, Cb,
                                                                          ldc);
    return cudaGetLastError();
}

}  // namespace gmtk

extern "C" gmt_status gmt_gemm_bf16(int32_t M, int32_t N, int32_t K, const void* A, const void* B, int32_t epilogue,
                                    const float* bias, float* C, void* C_bf16, int32_t splits, float* workspace,
                                    int32_t* error_flag, gmt_stream stream) {
    if (M <= 0 || N <= 0 || K <= 0 || K % 8 != 0 || !A || !B || !error_flag) {
        gmtk::record_error("gmt_gemm_bf16: need M, N, K > 0, K % 8 == 0, non-NULL A, B, error_flag");
        return GMT_ERR_INVALID;
    }
    if (epilogue < 0 || epilogue > 2 || (epilogue == 1 ? !C_bf16 : !C)) {
        gmtk::record_error("gmt_gemm_bf16: bad epilogue or missing output");
        return GMT_ERR_INVALID;
    }
    if (splits > 1 && !workspace) {
        gmtk::record_error("gmt_gemm_bf16: split-K needs a workspace of splits*M*N floats");
        return GMT_ERR_INVALID;
    }
    cudaError_t e = gmtk::gemm_bf16_tn(M, N, K, (const __nv_bfloat16*)A, (const __nv_bfloat16*)B, epilogue, bias, C,
                                       (__nv_bfloat16*)C_bf16, N, splits, workspace, error_flag, (cudaStream_t)stream);
    if (e != cudaSuccess) {
        gmtk::record_error((std::string("gmt_gemm_bf16: ") + cudaGetErrorString(e)).c_str());
        return GMT_ERR_CUDA;
    }
    return GMT_OK;
}
