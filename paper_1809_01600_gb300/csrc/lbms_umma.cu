// BF16 matrix product of the pointwise warm-start network on the
// fifth-generation tensor cores: P[z][M][N] = sum_{k in chunk z} A[m][k]
// B[n][k] with A [M][K] and B [N][K] both K-contiguous ("TN"), FP32
// accumulation.  (The U-Net's products are in lbms_conv.cu.)
//
// One CTA of 128 threads per 128 x 64 output tile and K chunk.  Operand
// tiles of 64 K-elements (one 128-byte swizzle span of BF16) are staged in
// shared memory by TMA (cp.async.bulk.tensor, 128-byte swizzle) through a
// four-stage ring of mbarriers; one thread issues tcgen05.mma (M = 128,
// N = 64, K = 16 per instruction) into a TMEM accumulator of 64 columns, and
// tcgen05.commit releases each stage when the products reading it are done.
// The four warps then read their 32 TMEM lanes (rows) with tcgen05.ld and
// store FP32.  Rows and K beyond the operands' extents are zero-filled by
// TMA, so M and K need no padding; N is a multiple of 64.
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <mutex>

#include "lbms_internal.h"
#include "lbms_umma.cuh"

namespace lbms {
namespace {

constexpr int kUM = 128;                       // output rows per CTA (UMMA M)
constexpr int kUN = 64;                        // output columns per CTA (UMMA N)
constexpr int kUK = 64;                        // K per stage: 64 BF16 = one 128-byte swizzle row
constexpr int kStages = 4;
constexpr int kABytes = kUM * kUK * 2;         // 16 KiB
constexpr int kBBytes = kUN * kUK * 2;         // 8 KiB
constexpr int kStageBytes = kABytes + kBBytes;
constexpr int kTmemCols = 64;                  // FP32 accumulator: 128 lanes x 64 columns
constexpr size_t kSmemBytes = 1024 + (size_t)kStages * kStageBytes + 256;

__global__ void __launch_bounds__(128, 1) umma_gemm_kernel(const __grid_constant__ CUtensorMap mapA,
                                                           const __grid_constant__ CUtensorMap mapB,
                                                           float* __restrict__ P, int M, int N, int kchunk,
                                                           unsigned int* __restrict__ err) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* full = reinterpret_cast<uint64_t*>(base + (size_t)kStages * kStageBytes);
    uint64_t* empty = full + kStages;
    uint64_t* done = empty + kStages;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n0 = blockIdx.x * kUN, m0 = blockIdx.y * kUM, k0 = blockIdx.z * kchunk;
    const int nk = kchunk / kUK;
    constexpr uint32_t idesc = umma_idesc(kUM, kUN, false);

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(tmem_slot, kTmemCols);
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;

    if (threadIdx.x == 0) {
        bool ok = true;
        int issued = 0;                        // stages whose loads were issued
        auto load = [&](int kt) {
            const int s = kt % kStages;
            uint8_t* sa = base + (size_t)s * kStageBytes;
            mbar_expect_tx(&full[s], kStageBytes);
            tma_load_2d(sa, &mapA, k0 + kt * kUK, m0, &full[s]);
            tma_load_2d(sa + kABytes, &mapB, k0 + kt * kUK, n0, &full[s]);
            ++issued;
        };
        for (int kt = 0; kt < nk && kt < kStages; ++kt) load(kt);
        int consumed = 0;
        for (int kt = 0; kt < nk; ++kt) {
            const int s = kt % kStages;
            const uint32_t ph = (uint32_t)(kt / kStages) & 1u;
            if (!mbar_wait(&full[s], ph)) {
                ok = false;
                break;
            }
            ++consumed;
            fence_after();
            const uint32_t a = smem_u32(base + (size_t)s * kStageBytes);
            const uint32_t b = a + kABytes;
#pragma unroll
            for (int j = 0; j < kUK / 16; ++j)
                umma_f16(tmem, kmajor_desc(a + 32 * j, 128), kmajor_desc(b + 32 * j, 128), idesc, (kt | j) != 0);
            umma_commit(&empty[s]);
            if (kt + kStages < nk) {
                if (!mbar_wait(&empty[s], ph)) {
                    ok = false;
                    break;
                }
                load(kt + kStages);
            }
        }
        umma_commit(done);                     // arrives once every product issued above is complete
        if (!ok) {
            atomicOr(err, 1u);
            // copies still in flight land in their stages before the CTA exits
            for (int kt = consumed; kt < issued; ++kt) mbar_wait(&full[kt % kStages], (uint32_t)(kt / kStages) & 1u);
        }
    }
    __syncwarp();
    const bool got = mbar_wait(done, 0);
    fence_after();
    if (!got) {
        if (lane == 0) atomicOr(err, 2u);
    } else {
        // warp w holds TMEM lanes (rows) 32 w .. 32 w + 31: row m0 + 32 w + lane, 64 columns
        const uint32_t taddr = tmem + ((uint32_t)(32 * warp) << 16);
        uint32_t v0[32], v1[32];
        tmem_ld32(taddr, v0);
        tmem_ld32(taddr + 32, v1);
        tmem_wait_ld();
        const int row = m0 + 32 * warp + lane;
        if (row < M) {
            float4* dst = reinterpret_cast<float4*>(P + (int64_t)blockIdx.z * M * N + (int64_t)row * N + n0);
#pragma unroll
            for (int q = 0; q < 8; ++q)
                dst[q] = make_float4(__uint_as_float(v0[4 * q]), __uint_as_float(v0[4 * q + 1]),
                                     __uint_as_float(v0[4 * q + 2]), __uint_as_float(v0[4 * q + 3]));
#pragma unroll
            for (int q = 0; q < 8; ++q)
                dst[8 + q] = make_float4(__uint_as_float(v1[4 * q]), __uint_as_float(v1[4 * q + 1]),
                                         __uint_as_float(v1[4 * q + 2]), __uint_as_float(v1[4 * q + 3]));
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
std::once_flag g_once;
cudaError_t g_init = cudaErrorNotReady;

void init_once() {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn) {
        g_init = e != cudaSuccess ? e : cudaErrorNotSupported;
        return;
    }
    g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    g_init = cudaFuncSetAttribute(umma_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
    if (g_init == cudaSuccess) g_init = conv_init();
}

}  // namespace

bool make_map(CUtensorMap* map, const void* base, int inner, int rows, int ld, int row_bytes, int box_rows) {
    const cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {(cuuint32_t)(row_bytes / 2), (cuuint32_t)box_rows};
    const cuuint32_t es[2] = {1, 1};
    return g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE,
                    row_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

cudaError_t umma_gemm_init() {
    std::call_once(g_once, init_once);
    return g_init;
}

bool umma_gemm_supported(const void* A, int lda, const void* B, int ldb, int M, int N, int K, int S) {
    if (M < 1 || N < kUN || N % kUN || K < 1 || S < 1 || K % S || (K / S) % kUK) return false;
    if (lda % 8 || ldb % 8 || lda < K || ldb < K) return false;
    if ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15u) return false;
    return (M + kUM - 1) / kUM <= 65535 && S <= 65535;
}

cudaError_t umma_gemm_tn(const void* A, int lda, const void* B, int ldb, float* P, int M, int N, int K, int S,
                         unsigned int* err, cudaStream_t st) {
    cudaError_t e = umma_gemm_init();
    if (e != cudaSuccess) return e;
    if (!umma_gemm_supported(A, lda, B, ldb, M, N, K, S)) return cudaErrorInvalidValue;
    CUtensorMap ma, mb;
    if (!make_map(&ma, A, K, M, lda, 128, kUM) || !make_map(&mb, B, K, N, ldb, 128, kUN)) return cudaErrorInvalidValue;
    const dim3 grid(N / kUN, (M + kUM - 1) / kUM, S);
    umma_gemm_kernel<<<grid, 128, kSmemBytes, st>>>(ma, mb, P, M, N, K / S, err);
    return cudaGetLastError();
}

}  // namespace lbms
