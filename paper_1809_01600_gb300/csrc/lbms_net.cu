// Learned warm start (declared in include/lbms_net.h): feature rows of an
// anode's fluid cells, a pointwise MLP with BF16 tensor-core matrix products
// and FP32 accumulation, its backward pass and Adam.
//
// The products run on the tcgen05 kernels of lbms_conv.cu.  At 8192 rows and
// width 704 they are small (11 products of 8 GFLOP at most), so what bounds a
// step is everything around them: bias, ReLU and its gradient, the loss and the
// bias gradients are taken on a product's accumulators, the weight gradients
// read both operands as they lie, and Adam is one launch.  A step with its
// transfers and the gradients: 0.771 ms with a kernel for each of these, 0.376.
//
// The mma.sync kernel here (m16n8k16) is what remains when it is forced or
// tcgen05 is missing: P = A . B^T with A [M][K] and B [N][K] both K-contiguous
// BF16 ("TN"), M and N multiples of 64, K a multiple of 32 per split; the
// weight gradients get that form from transposed copies of the activations.
// Every size is padded at allocation so that no tile crosses a buffer's end:
// the kernels need no bounds checks, and the host checks the divisibility
// before every launch.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/lbms.h"
#include "../../include/lbms_net.h"
#include "lbms_internal.h"

namespace {

using bf16 = __nv_bfloat16;

constexpr int kF = LBMS_NET_FEATURES;   // feature row width
constexpr int kFUsed = 16;              // features actually set
constexpr int kOutPad = 64;             // output layer rows (3 used)
constexpr int kOut = 3;
constexpr float kTargetScale = 100.0f;  // network output = 100 (X - X_profile)
constexpr int kZeroHead = 10;           // floats before the bias gradients: loss and sums (4 FP64), a counter
constexpr int kMaxRows = 32768;         // rows per forward / training batch
constexpr int kTM = 64, kTN = 64, kTK = 32;

// ---------------------------------------------------------------- generator
// SplitMix64 (Steele, Lea, Flood 2014): a counter-based generator, one
// 64-bit output per key.
__host__ __device__ inline uint64_t splitmix64(uint64_t x) {
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}
inline double unit_double(uint64_t x) { return (double)(splitmix64(x) >> 11) * (1.0 / 9007199254740992.0); }

// ------------------------------------------------------------------- GEMM
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned sa = static_cast<unsigned>(__cvta_generic_to_shared(smem));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem));
}
// Four 8x8 BF16 matrices from shared memory; lane l supplies the address of
// row (l % 8) of matrix l / 8.
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], const void* smem) {
    const unsigned sa = static_cast<unsigned>(__cvta_generic_to_shared(smem));
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(sa));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}

// P[z][M][N] = sum over k in [z kchunk, (z+1) kchunk) of A[m][k] B[n][k].
// Block: 64 x 64 output tile, 4 warps of 32 x 32; K in steps of 32 staged in
// shared memory by cp.async, two stages (the next step loads while this one
// is multiplied); rows padded to 40 elements for conflict-free fragment
// reads.
__global__ void __launch_bounds__(128) gemm_tn_kernel(const bf16* __restrict__ A, int lda, const bf16* __restrict__ B,
                                                      int ldb, float* __restrict__ P, int M, int N, int kchunk) {
    __shared__ __align__(16) bf16 sA[2][kTM][kTK + 8];
    __shared__ __align__(16) bf16 sB[2][kTN][kTK + 8];
    const int m0 = blockIdx.y * kTM, n0 = blockIdx.x * kTN;
    const int k0 = blockIdx.z * kchunk;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
    const int g = lane >> 2, t = lane & 3;
    float acc[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[i][j][r] = 0.0f;

    // 64 rows x 32 elements = 256 chunks of 16 bytes per operand and stage
    auto stage = [&](int buf, int kk) {
        for (int c = threadIdx.x; c < kTM * kTK / 8; c += 128) {
            const int r = c >> 2, q = (c & 3) * 8;
            cp_async16(&sA[buf][r][q], A + (int64_t)(m0 + r) * lda + kk + q);
            cp_async16(&sB[buf][r][q], B + (int64_t)(n0 + r) * ldb + kk + q);
        }
        cp_async_commit();
    };
    const int nk = kchunk / kTK;
    stage(0, k0);
    for (int it = 0; it < nk; ++it) {
        const int buf = it & 1;
        if (it + 1 < nk) {
            stage(buf ^ 1, k0 + (it + 1) * kTK);
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        __syncthreads();
#pragma unroll
        for (int ks = 0; ks < kTK; ks += 16) {
            // A fragments (16 x 16, rows m): matrices (rows 0-7 | 8-15) x (k 0-7 | 8-15);
            // B fragments of two n-blocks of 8: matrices (n 0-7, k 0-7), (n 0-7, k 8-15),
            // (n 8-15, k 0-7), (n 8-15, k 8-15), i.e. b[j][0], b[j][1], b[j+1][0], b[j+1][1]
            uint32_t a[2][4], b[4][2];
#pragma unroll
            for (int i = 0; i < 2; ++i) ldsm_x4(a[i], &sA[buf][wm + i * 16 + (lane & 15)][ks + (lane >> 4) * 8]);
#pragma unroll
            for (int jj = 0; jj < 2; ++jj) {
                uint32_t r[4];
                ldsm_x4(r, &sB[buf][wn + jj * 16 + (lane & 7) + ((lane >> 4) << 3)][ks + ((lane >> 3) & 1) * 8]);
                b[2 * jj][0] = r[0];
                b[2 * jj][1] = r[1];
                b[2 * jj + 1][0] = r[2];
                b[2 * jj + 1][1] = r[3];
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], a[i], b[j]);
        }
        __syncthreads();   // the stage just read is refilled two steps later
    }
    float* Pz = P + (int64_t)blockIdx.z * M * N;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int r = m0 + wm + i * 16 + g;
            const int c = n0 + wn + j * 8 + 2 * t;
            *reinterpret_cast<float2*>(Pz + (int64_t)r * N + c) = make_float2(acc[i][j][0], acc[i][j][1]);
            *reinterpret_cast<float2*>(Pz + (int64_t)(r + 8) * N + c) = make_float2(acc[i][j][2], acc[i][j][3]);
        }
}

// ---------------------------------------------------------- elementwise
// Z = P + b (one row per thread block row); hidden layers store relu(Z) as
// BF16 [R][C], the output layer stores Z as FP32.
__global__ void bias_act_kernel(const float* __restrict__ P, const float* __restrict__ b, int R, int C, int relu,
                                bf16* __restrict__ act, float* __restrict__ Y) {
    const int64_t n = (int64_t)R * C;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const float z = P[e] + b[e % C];
        if (relu)
            act[e] = __float2bfloat16_rn(z > 0.0f ? z : 0.0f);
        else
            Y[e] = z;
    }
}

// out[c][r] = in[r][c]; R and C multiples of 32.
__global__ void transpose_kernel(const bf16* __restrict__ in, bf16* __restrict__ out, int R, int C) {
    __shared__ bf16 tile[32][33];
    const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
    for (int y = threadIdx.y; y < 32; y += 8) tile[y][threadIdx.x] = in[(int64_t)(r0 + y) * C + c0 + threadIdx.x];
    __syncthreads();
    for (int y = threadIdx.y; y < 32; y += 8) out[(int64_t)(c0 + y) * R + r0 + threadIdx.x] = tile[threadIdx.x][y];
}

// Mean-square error over the 3 used outputs and its gradient dY (BF16,
// zero in the padded columns); bias gradient of the output layer and the
// loss summed with atomics.  One block of 256 threads per 64 rows.
__global__ void loss_grad_kernel(const float* __restrict__ Y, const float* __restrict__ T, int R,
                                 bf16* __restrict__ dY, float* __restrict__ gb, double* __restrict__ loss) {
    __shared__ float colsum[kOutPad];
    __shared__ double lsum[256];
    if (threadIdx.x < kOutPad) colsum[threadIdx.x] = 0.0f;
    __syncthreads();
    const float scale = 2.0f / (float)(R * kOut);
    double l = 0.0;
    const int r0 = blockIdx.x * 64;
    for (int e = threadIdx.x; e < 64 * kOutPad; e += 256) {
        const int r = r0 + e / kOutPad, c = e % kOutPad;
        float gval = 0.0f;
        if (c < kOut) {
            const float d = Y[(int64_t)r * kOutPad + c] - T[(int64_t)r * 4 + c];
            l += (double)d * d;
            gval = scale * d;
            atomicAdd(&colsum[c], gval);
        }
        dY[(int64_t)r * kOutPad + c] = __float2bfloat16_rn(gval);
    }
    lsum[threadIdx.x] = l;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s) lsum[threadIdx.x] += lsum[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(loss, lsum[0] / (double)(R * kOut));
    if (threadIdx.x < kOut) atomicAdd(&gb[threadIdx.x], colsum[threadIdx.x]);
}

// dZ = dA * (layer input > 0) as BF16 [R][C]; bias gradient column sums.
// One block of 256 threads per 32 rows x C columns (C a multiple of 64).
__global__ void relu_back_kernel(const float* __restrict__ dA, const bf16* __restrict__ act, int R, int C,
                                 bf16* __restrict__ dZ, float* __restrict__ gb) {
    const int r0 = blockIdx.x * 32;
    for (int c = threadIdx.x; c < C; c += blockDim.x) {
        float s = 0.0f;
        for (int r = r0; r < r0 + 32; ++r) {
            const int64_t e = (int64_t)r * C + c;
            const float v = __bfloat162float(act[e]) > 0.0f ? dA[e] : 0.0f;
            dZ[e] = __float2bfloat16_rn(v);
            s += v;
        }
        atomicAdd(&gb[c], s);
    }
}

// G[e] = sum_z P[z][e]
__global__ void splitk_sum_kernel(const float* __restrict__ P, int S, int64_t n, float* __restrict__ G) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        float s = 0.0f;
        for (int z = 0; z < S; ++z) s += P[(int64_t)z * n + e];
        G[e] = s;
    }
}

// One Adam step (betas 0.9 / 0.999, eps 1e-8) over all parameter arrays of a
// network in one launch (blockIdx.y: the array), with the BF16 copies of the
// weights: Wb as stored [O][I]; Wt its transpose [I][O], or for 3x3x3
// convolutions (ci != 0, I = 27 ci) the flipped weights [ci][27 O].  Launched
// per array this took 39 launches and 230 us of a U-Net step.
struct AdamItem {
    float *p, *m, *v;
    const float* g;
    int64_t n;
    bf16 *Wb, *Wt;
    int O, I, ci;
};
struct AdamList {
    AdamItem it[26];
};

__global__ void adam_all_kernel(const __grid_constant__ AdamList list, float lr, float c1, float c2) {
    const AdamItem& a = list.it[blockIdx.y];
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < a.n; e += (int64_t)gridDim.x * blockDim.x) {
        const float gr = a.g[e];
        const float mm = 0.9f * a.m[e] + 0.1f * gr;
        const float vv = 0.999f * a.v[e] + 0.001f * gr * gr;
        a.m[e] = mm;
        a.v[e] = vv;
        const float w = a.p[e] - lr * (mm * c1) / (sqrtf(vv * c2) + 1e-8f);
        a.p[e] = w;
        if (a.Wb) {
            const int o = (int)(e / a.I), i = (int)(e % a.I);
            const bf16 wb = __float2bfloat16_rn(w);
            a.Wb[e] = wb;
            if (a.ci)
                a.Wt[(int64_t)(i % a.ci) * 27 * a.O + (int64_t)(i / a.ci) * a.O + o] = wb;
            else
                a.Wt[(int64_t)i * a.O + o] = wb;
        }
    }
}

// BF16 copy of the FP32 weights [O][I] and its transpose.
__global__ void cast_weights_kernel(const float* __restrict__ W, int O, int I, bf16* __restrict__ Wb,
                                    bf16* __restrict__ WbT) {
    const int64_t n = (int64_t)O * I;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int o = (int)(e / I), i = (int)(e % I);
        const bf16 wb = __float2bfloat16_rn(W[e]);
        Wb[e] = wb;
        WbT[(int64_t)i * O + o] = wb;
    }
}

// A training batch: row r takes training row splitmix64(key + r) mod n.
__global__ void sample_kernel(const bf16* __restrict__ feat, const float* __restrict__ targ, int64_t n, uint64_t key,
                              int R, bf16* __restrict__ X, float* __restrict__ T) {
    const int r = blockIdx.x;
    const int64_t src = (int64_t)(splitmix64(key + (uint64_t)r) % (uint64_t)n);
    for (int c = threadIdx.x; c < kF; c += blockDim.x) X[(int64_t)r * kF + c] = feat[src * kF + c];
    if (threadIdx.x < 4) T[(int64_t)r * 4 + threadIdx.x] = targ[src * 4 + threadIdx.x];
}

// ------------------------------------------------------------- features
// Dense index of every fluid cell from its coordinate word.
__global__ void cell_index_kernel(const uint32_t* __restrict__ code, int nf, int nx, int ny,
                                  int64_t* __restrict__ cell) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= nf) return;
    const uint32_t c = code[j];
    cell[j] = ((int64_t)(c >> 21) * ny + ((c >> 11) & 1023u)) * nx + (c & 2047u);
}

// Fluid mask on the dense grid (cleared before) and fluid cells per x-plane.
__global__ void mask_kernel(const int64_t* __restrict__ cell, int nf, int nx, uint8_t* __restrict__ mask,
                            int* __restrict__ plane) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= nf) return;
    mask[cell[j]] = 1;
    atomicAdd(&plane[cell[j] % nx], 1);
}

// Fluid voxels in the windows of half-width 1, 3 and 7 around each voxel, one
// axis after the other (x clamped, y and z periodic).  The counts are whole
// numbers: at most 15, then 225, then 3375.
struct Windows {
    uint8_t* v[3];
};
__device__ constexpr int half_width(int q) { return q == 0 ? 1 : (q == 1 ? 3 : 7); }

__global__ void window_x_kernel(const uint8_t* __restrict__ mask, int64_t N, int nx, Windows out) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < N; e += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(e % nx);
        int s[3] = {0, 0, 0};
#pragma unroll
        for (int d = -7; d <= 7; ++d) {
            const int v = x + d >= 0 && x + d < nx ? mask[e + d] : 0;
#pragma unroll
            for (int q = 0; q < 3; ++q)
                if (d >= -half_width(q) && d <= half_width(q)) s[q] += v;
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) out.v[q][e] = (uint8_t)s[q];
    }
}

__device__ __forceinline__ int wrap(int a, int n) {   // a in [-7, n + 7)
    if (n >= 7) return a < 0 ? a + n : (a >= n ? a - n : a);
    a %= n;
    return a < 0 ? a + n : a;
}

__global__ void window_y_kernel(Windows in, int64_t N, int nx, int ny, Windows out) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < N; e += (int64_t)gridDim.x * blockDim.x) {
        const int y = (int)((e / nx) % ny);
        int s[3] = {0, 0, 0};
#pragma unroll
        for (int d = -7; d <= 7; ++d) {
            const int64_t j = e + (int64_t)(wrap(y + d, ny) - y) * nx;
#pragma unroll
            for (int q = 0; q < 3; ++q)
                if (d >= -half_width(q) && d <= half_width(q)) s[q] += in.v[q][j];
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) out.v[q][e] = (uint8_t)s[q];
    }
}

// The last axis, and the counts over the windows' sizes: w[q][e].
__global__ void window_z_kernel(Windows in, int64_t N, int nx, int ny, int nz, float* __restrict__ w) {
    const int64_t plane = (int64_t)nx * ny;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < N; e += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(e % nx), z = (int)(e / plane);
        int s[3] = {0, 0, 0};
#pragma unroll
        for (int d = -7; d <= 7; ++d) {
            if (nz == 1 && d != 0) continue;
            const int64_t j = e + (int64_t)(wrap(z + d, nz) - z) * plane;
#pragma unroll
            for (int q = 0; q < 3; ++q)
                if (d >= -half_width(q) && d <= half_width(q)) s[q] += in.v[q][j];
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int h = half_width(q), t = 2 * h + 1;
            const int wide = min(x + h, nx - 1) - max(x - h, 0) + 1;
            w[q * N + e] = (float)s[q] / (float)(wide * t * (nz > 1 ? t : 1));
        }
    }
}

// dense[s][cell[j]] = v[s][j] (dense cleared before).
__global__ void scatter_kernel(const double* __restrict__ v, const int64_t* __restrict__ cell, int nf, int64_t N,
                               double* __restrict__ dense) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= nf) return;
    for (int s = 0; s < 3; ++s) dense[s * N + cell[j]] = v[(int64_t)s * nf + j];
}

// Feature row of fluid cell j (dense index cell[j]), one thread per column:
//  0-2 profile X at x, 3 x / (nx - 1), 4-6 fluid fraction of the windows,
//  7 current / 2, 8-10 inlet X, 11 (x / (nx - 1)) current / 2,
//  12 cross-section porosity at x, 13 normalised cumulative resistance,
//  14 1 / (4 cross-section porosity), 15 one; 16-63 zero.
__global__ void assemble_kernel(const int64_t* __restrict__ cell, int nf, int nx, const float* __restrict__ xtab,
                                const float* __restrict__ w1, const float* __restrict__ w3,
                                const float* __restrict__ w7, float cur, float xi0, float xi1, float xi2,
                                bf16* __restrict__ out) {
    const int j = blockIdx.x * blockDim.y + threadIdx.y;
    if (j >= nf) return;
    const int64_t e = cell[j];
    const int x = (int)(e % nx);
    const float* tx = xtab + (int64_t)x * 8;
    const float xr = tx[3];
    float f = 0.0f;
    switch (threadIdx.x) {
        case 0: f = tx[0]; break;
        case 1: f = tx[1]; break;
        case 2: f = tx[2]; break;
        case 3: f = xr; break;
        case 4: f = w1[e]; break;
        case 5: f = w3[e]; break;
        case 6: f = w7[e]; break;
        case 7: f = 0.5f * cur; break;
        case 8: f = xi0; break;
        case 9: f = xi1; break;
        case 10: f = xi2; break;
        case 11: f = 0.5f * cur * xr; break;
        case 12: f = tx[4]; break;
        case 13: f = tx[5]; break;
        case 14: f = tx[6]; break;
        case 15: f = 1.0f; break;
        default: f = 0.0f;
    }
    out[(int64_t)j * kF + threadIdx.x] = __float2bfloat16_rn(f);
}

// X_s = profile_s(x) + Y[j][s] / 100, clamped at 1e-6 and renormalised;
// out [3][nf] in FP64.
__global__ void predict_post_kernel(const float* __restrict__ Y, int ld, const int64_t* __restrict__ cell, int j0, int rows,
                                    int nf, int nx, const float* __restrict__ xtab, double* __restrict__ out) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = j0 + r;
    if (r >= rows || j >= nf) return;
    const int x = (int)(cell[j] % nx);
    double X[3], s = 0.0;
    for (int q = 0; q < 3; ++q) {
        double v = (double)xtab[(int64_t)x * 8 + q] + (double)Y[(int64_t)r * ld + q] / kTargetScale;
        v = v < 1e-6 ? 1e-6 : v;
        X[q] = v;
        s += v;
    }
    for (int q = 0; q < 3; ++q) out[(int64_t)q * nf + j] = X[q] / s;
}

}  // namespace

// ------------------------------------------------------------------ host
struct lbms_net {
    int width = 0, depth = 0, layers = 0;
    std::vector<int> in, out;               // padded sizes per layer
    std::vector<float*> W, b, mW, vW, mb, vb, gW, gb;
    std::vector<bf16*> Wb, WbT;
    std::vector<bf16*> act, actT;           // act[l] = input of layer l, [kMaxRows][in_l]
    bf16* dz[2] = {nullptr, nullptr};       // [kMaxRows][max width] ping-pong
    bf16* dzT = nullptr;                    // [max width][kMaxRows]
    float* P = nullptr;                     // GEMM partials
    size_t P_floats = 0;
    float* Y = nullptr;                     // output rows, y_ld apart
    int y_ld = kOutPad;
    float* T = nullptr;                     // [kMaxRows][4]: targets, 1
    float* zero = nullptr;                  // the loss and all bias gradients, cleared together
    size_t zero_bytes = 0;
    float* flat = nullptr;                  // parameters or gradients in the caller's order
    std::mutex flat_use;
    double* loss = nullptr;
    bf16* feat = nullptr;                   // training rows [cap][kF]
    float* targ = nullptr;                  // [cap][4]
    int64_t n_rows = 0, cap = 0;
    int64_t step = 0;
    uint64_t seed = 0;
    unsigned int* gemm_err = nullptr;       // raised by the tensor-core GEMM on a timed-out wait
    int gemm_kind = LBMS_NET_GEMM_AUTO;
    int64_t tcgen05_calls = 0, mma_sync_calls = 0;
    std::vector<void*> allocs;
    char* room = nullptr;                   // working memory of the case at hand, grown on demand and kept
    size_t room_bytes = 0;                  //   up to kRoomKept bytes
    std::string err;
};

namespace {

lbms_status nfail(lbms_net* n, lbms_status s, const char* fmt, ...) {
    if (n) {
        char buf[512];
        va_list ap;
        va_start(ap, fmt);
        std::vsnprintf(buf, sizeof(buf), fmt, ap);
        va_end(ap);
        n->err = buf;
    }
    return s;
}

#define NCK(expr, what)                                                                               \
    do {                                                                                             \
        cudaError_t e_ = (expr);                                                                     \
        if (e_ != cudaSuccess) return nfail(n, LBMS_ECUDA, "%s: %s", what, cudaGetErrorString(e_)); \
    } while (0)

// Every request is recorded, failed ones as null, so that one scan of
// `allocs` finds a failure.
template <typename T>
T* nalloc(lbms_net* n, size_t count) {
    void* p = nullptr;
    lbms::dev_malloc(&p, std::max<size_t>(count, 1) * sizeof(T));
    n->allocs.push_back(p);
    return static_cast<T*>(p);
}

int grid_for(int64_t n) { return (int)std::min<int64_t>((n + 255) / 256, 152 * 16); }

int64_t n_params(const lbms_net* n) {
    int64_t s = 0;
    for (int l = 0; l < n->layers; ++l) {
        const int o = l == n->layers - 1 ? kOut : n->out[l];
        s += (int64_t)o * n->in[l] + o;
    }
    return s;
}

// P[z] = A . B^T on the mma.sync kernel, with the checks the kernel relies on.
lbms_status gemm(lbms_net* n, const bf16* A, int lda, const bf16* B, int ldb, int M, int N, int K, int S) {
    if ((size_t)S * M * N > n->P_floats)
        return nfail(n, LBMS_EINVAL, "internal GEMM shape %d x %d x %d (split %d) exceeds the partials", M, N, K, S);
    if (n->gemm_kind == LBMS_NET_GEMM_TCGEN05)
        return nfail(n, LBMS_ECUDA, "the tcgen05 kernels are unavailable: %s", cudaGetErrorString(lbms::umma_init()));
    if (M % kTM || N % kTN || K % (kTK * S) || lda % 8 || ldb % 8)
        return nfail(n, LBMS_EINVAL, "internal GEMM shape %d x %d x %d (split %d) not tileable", M, N, K, S);
    gemm_tn_kernel<<<dim3(N / kTN, M / kTM, S), 128>>>(A, lda, B, ldb, n->P, M, N, K / S);
    NCK(cudaGetLastError(), "gemm");
    ++n->mma_sync_calls;
    return LBMS_OK;
}

// Reads and clears the tensor-core GEMM's error flag (after the device work).
lbms_status check_gemm(lbms_net* n) {
    unsigned int f = 0;
    NCK(cudaMemcpy(&f, n->gemm_err, sizeof(f), cudaMemcpyDeviceToHost), "GEMM flag");
    if (!f) return LBMS_OK;
    NCK(cudaMemset(n->gemm_err, 0, sizeof(f)), "GEMM flag");
    return nfail(n, LBMS_ECUDA, "tensor-core GEMM: an mbarrier wait timed out (flag %u)", f);
}

lbms_status transpose(lbms_net* n, const bf16* in, bf16* out, int R, int C) {
    transpose_kernel<<<dim3(C / 32, R / 32), dim3(32, 8)>>>(in, out, R, C);
    NCK(cudaGetLastError(), "transpose");
    return LBMS_OK;
}

// Whether the passes run on the tensor-core kernels with the work after each
// product on its accumulators (lbms_conv.cu), which take every shape of the
// network; the mma.sync kernel, when forced, runs the passes below it one
// kernel at a time.
bool fused(const lbms_net* n) { return n->gemm_kind != LBMS_NET_GEMM_MMA_SYNC && lbms::umma_init() == cudaSuccess; }

// A layer's product over R rows: x [R][C] . W [N][C]^T.
lbms::ConvJob layer_job(const bf16* x, int R, int C, const bf16* W, int N, lbms::ConvOut kind) {
    lbms::ConvJob j;
    j.x = x;
    j.W = W;
    j.rows = R;
    j.C = C;
    j.N = N;
    j.taps = 1;
    j.kind = kind;
    return j;
}

// Forward pass of R rows already in act[0].  With `train`, what the backward
// pass needs is kept: fused, the output gradient (dz[0]), its bias gradient
// and the loss against n->T; else the transposed activations.  Without it the
// output is in n->Y, y_ld apart.
lbms_status forward(lbms_net* n, int R, bool train) {
    lbms_status st;
    if (train) NCK(cudaMemsetAsync(n->zero, 0, n->zero_bytes, 0), "loss and bias grads");
    if (fused(n)) {
        for (int l = 0; l < n->layers; ++l) {
            const bool last = l == n->layers - 1;
            lbms::ConvJob j = layer_job(n->act[l], R, n->in[l], n->Wb[l], n->out[l], last ? lbms::kOutHead : lbms::kOutRelu);
            j.ep.bias = n->b[l];
            if (!last) {
                j.ep.out = n->act[l + 1];
            } else if (train) {
                j.ep.T = n->T;
                j.ep.grad_scale = 2.0f / (float)(R * kOut);
                j.ep.loss_scale = 1.0 / (double)(R * kOut);
                j.ep.out = n->dz[0];
                j.ep.gb = n->gb[l];
                j.ep.loss = n->loss;
                j.ep.done = reinterpret_cast<unsigned int*>(n->loss + 4);
            } else {
                j.ep.Y = n->Y;
                n->y_ld = 4;
            }
            NCK(lbms::umma_conv(j, n->gemm_err, 0), "layer");
            ++n->tcgen05_calls;
        }
        return LBMS_OK;
    }
    n->y_ld = kOutPad;
    for (int l = 0; l < n->layers; ++l) {
        const bool last = l == n->layers - 1;
        if (train) {
            st = transpose(n, n->act[l], n->actT[l], R, n->in[l]);
            if (st != LBMS_OK) return st;
        }
        st = gemm(n, n->act[l], n->in[l], n->Wb[l], n->in[l], R, n->out[l], n->in[l], 1);
        if (st != LBMS_OK) return st;
        bias_act_kernel<<<grid_for((int64_t)R * n->out[l]), 256>>>(n->P, n->b[l], R, n->out[l], last ? 0 : 1,
                                                                   last ? nullptr : n->act[l + 1],
                                                                   last ? n->Y : nullptr);
        NCK(cudaGetLastError(), "bias/activation");
    }
    return LBMS_OK;
}

// Backward pass and (lr > 0) Adam step for the R rows of the last forward
// pass (train) with targets in n->T.  Gradients stay in gW / gb.
lbms_status backward_step(lbms_net* n, int R, double lr, double* loss) {
    lbms_status st;
    const int L = n->layers;
    const bool fast = fused(n);
    if (!fast) {
        loss_grad_kernel<<<R / 64, 256>>>(n->Y, n->T, R, n->dz[0], n->gb[L - 1], n->loss);
        NCK(cudaGetLastError(), "loss");
    }
    int cur = 0;
    // split of the R-long reduction of the weight gradients: chunks of >= 512
    // rows, a divisor of R / 64 so that every chunk is whole 64-row steps (the
    // K step of the tcgen05 kernel; two of the mma.sync kernel's)
    int S = std::max(1, std::min(16, R / 512));
    while (S > 1 && (R / 64) % S) --S;
    for (int l = L - 1; l >= 0; --l) {
        const int O = n->out[l], I = n->in[l];
        // weight gradient: dZ^T [O][R] . act^T [I][R]
        if (fast) {
            lbms::WgradJob j;
            j.x = n->dz[cur];
            j.C = O;
            j.dz = n->act[l];
            j.N = I;
            j.rows = R;
            j.S = S;
            j.taps = 1;
            j.P = n->P;
            NCK(lbms::umma_wgrad(j, n->gemm_err, 0), "weight gradient");
            ++n->tcgen05_calls;
        } else {
            st = transpose(n, n->dz[cur], n->dzT, R, O);
            if (st != LBMS_OK) return st;
            st = gemm(n, n->dzT, R, n->actT[l], R, O, I, R, S);
            if (st != LBMS_OK) return st;
        }
        splitk_sum_kernel<<<grid_for((int64_t)O * I), 256>>>(n->P, S, (int64_t)O * I, n->gW[l]);
        NCK(cudaGetLastError(), "split-k sum");
        if (l > 0) {
            // input gradient: dZ [R][O] . W^T -> [R][I], then through the ReLU of layer l - 1
            if (fast) {
                lbms::ConvJob j = layer_job(n->dz[cur], R, O, n->WbT[l], I, lbms::kOutReluBack);
                j.ep.act = n->act[l];
                j.ep.out = n->dz[cur ^ 1];
                j.ep.gb = n->gb[l - 1];
                NCK(lbms::umma_conv(j, n->gemm_err, 0), "input gradient");
                ++n->tcgen05_calls;
            } else {
                st = gemm(n, n->dz[cur], O, n->WbT[l], O, R, I, O, 1);
                if (st != LBMS_OK) return st;
                relu_back_kernel<<<R / 32, 256>>>(n->P, n->act[l], R, I, n->dz[cur ^ 1], n->gb[l - 1]);
                NCK(cudaGetLastError(), "relu backward");
            }
            cur ^= 1;
        }
    }
    if (lr > 0.0) {
        ++n->step;
        const float c1 = (float)(1.0 / (1.0 - std::pow(0.9, (double)n->step)));
        const float c2 = (float)(1.0 / (1.0 - std::pow(0.999, (double)n->step)));
        AdamList list = {};
        for (int l = 0; l < L; ++l) {
            const int O = n->out[l], I = n->in[l];
            list.it[2 * l] = {n->W[l], n->mW[l], n->vW[l], n->gW[l], (int64_t)O * I, n->Wb[l], n->WbT[l], O, I, 0};
            list.it[2 * l + 1] = {n->b[l], n->mb[l], n->vb[l], n->gb[l], O, nullptr, nullptr, O, 1, 0};
        }
        adam_all_kernel<<<dim3(152, 2 * L), 256>>>(list, (float)lr, c1, c2);
        NCK(cudaGetLastError(), "adam");
    }
    if (loss) NCK(cudaMemcpy(loss, n->loss, sizeof(double), cudaMemcpyDeviceToHost), "read loss");
    return LBMS_OK;
}

// Working memory that a network keeps between calls (about 43 bytes a voxel and
// 168 a fluid cell: grids of 5 M voxels); what a larger case took goes back at
// the end of its call, which takes ten milliseconds or more.
constexpr size_t kRoomKept = (size_t)512 << 20;

// Feature rows (device, [rows_pad][kF], zero padded) and the per-x table of
// one case, with room for a prediction; rows_pad = nf rounded up to 64.  All
// of it lies in the net's working memory, valid until its next case.
struct CaseFeatures {
    explicit CaseFeatures(lbms_net* n) : net(n) {}
    CaseFeatures(const CaseFeatures&) = delete;
    ~CaseFeatures() {
        if (net->room_bytes <= kRoomKept) return;
        cudaFree(net->room);                // waits for the device
        net->room = nullptr;
        net->room_bytes = 0;
    }
    lbms_net* net;
    bf16* rows = nullptr;
    float* xtab = nullptr;
    int64_t* cell = nullptr;         // dense index of each fluid cell
    int64_t* row = nullptr;          // [nf], for the caller
    double* pred = nullptr;          // [3][nf], for the caller
    double* dense = nullptr;         // [3][N], for the caller
    int nf = 0, nx = 0, rows_pad = 0;
    std::vector<double> prof;
};

lbms_status case_features(lbms_net* n, lbms_ctx* ctx, int k, CaseFeatures& F) {
    lbms::CaseView v;
    if (!lbms::case_view(ctx, k, &v)) return nfail(n, LBMS_EINVAL, "case index %d out of range", k);
    if (!v.has_bc) return nfail(n, LBMS_ESTATE, "case %d has no boundary data yet", k);
    if (v.periodic_x) return nfail(n, LBMS_EINVAL, "case %d is periodic in x (no inlet / outlet)", k);
    if (!lbms::case_profile_1d(ctx, k, F.prof))
        return nfail(n, LBMS_EDEPLETED, "the 1-D profile of case %d drives a mole fraction below zero", k);
    const int nx = v.nx, ny = v.ny, nz = v.nz;
    const int64_t N = v.N;
    F.nf = v.nf;
    F.nx = nx;
    F.rows_pad = (v.nf + 63) / 64 * 64;
    uint8_t *mask = nullptr, *b[6] = {};
    float* w = nullptr;
    int* plane = nullptr;
    auto lay_out = [&](char* p) {
        auto take = [&](auto*& ptr, size_t count) {
            ptr = reinterpret_cast<std::remove_reference_t<decltype(ptr)>>(p);
            p += (count * sizeof(*ptr) + 255) / 256 * 256;
        };
        take(F.rows, (size_t)F.rows_pad * kF);
        take(F.cell, v.nf);
        take(F.row, v.nf);
        take(F.pred, (size_t)3 * v.nf);
        take(F.dense, (size_t)3 * N);
        take(F.xtab, (size_t)nx * 8);
        take(w, (size_t)3 * N);
        take(plane, nx);
        take(mask, N);
        for (auto& q : b) take(q, N);
        return p;
    };
    const size_t need = (size_t)(lay_out(nullptr) - (char*)nullptr);
    if (need > n->room_bytes) {
        NCK(cudaDeviceSynchronize(), "feature buffers");
        cudaFree(n->room);
        n->room = nullptr;
        n->room_bytes = 0;
        if (lbms::dev_malloc(&n->room, need) != cudaSuccess) return nfail(n, LBMS_ENOMEM, "feature buffers");
        n->room_bytes = need;
    }
    lay_out(n->room);
    const int gc = (v.nf + 255) / 256, g = grid_for(N);
    if (v.cell_code) {
        cell_index_kernel<<<gc, 256>>>(v.cell_code, v.nf, nx, ny, F.cell);
        NCK(cudaGetLastError(), "cells");
    } else {
        NCK(cudaMemcpy(F.cell, v.fluid_cell, v.nf * sizeof(int64_t), cudaMemcpyHostToDevice), "cells");
    }
    NCK(cudaMemsetAsync(mask, 0, N, 0), "mask");
    NCK(cudaMemsetAsync(plane, 0, nx * sizeof(int), 0), "mask");
    mask_kernel<<<gc, 256>>>(F.cell, v.nf, nx, mask, plane);
    NCK(cudaGetLastError(), "mask");
    const Windows wx{{b[0], b[1], b[2]}}, wy{{b[3], b[4], b[5]}};
    window_x_kernel<<<g, 256>>>(mask, N, nx, wx);
    window_y_kernel<<<g, 256>>>(wx, N, nx, ny, wy);
    window_z_kernel<<<g, 256>>>(wy, N, nx, ny, nz, w);
    NCK(cudaGetLastError(), "box filter");
    // host: per-x table (profile, x / (nx - 1), plane porosity, normalised
    // cumulative resistance, inverse porosity)
    std::vector<int> count(nx);
    NCK(cudaMemcpy(count.data(), plane, nx * sizeof(int), cudaMemcpyDeviceToHost), "plane porosity");
    std::vector<double> phi(nx, 0.0);
    for (int x = 0; x < nx; ++x) phi[x] = std::max(count[x] / ((double)ny * nz), 1.0 / ((double)ny * nz));
    std::vector<double> res(nx, 0.0);
    for (int x = 1; x < nx; ++x) res[x] = res[x - 1] + 0.5 * (1.0 / phi[x - 1] + 1.0 / phi[x]);
    std::vector<float> xtab((size_t)nx * 8, 0.0f);
    for (int x = 0; x < nx; ++x) {
        for (int s = 0; s < 3; ++s) xtab[(size_t)x * 8 + s] = (float)F.prof[(size_t)s * nx + x];
        xtab[(size_t)x * 8 + 3] = (float)x / (float)(nx - 1);
        xtab[(size_t)x * 8 + 4] = (float)phi[x];
        xtab[(size_t)x * 8 + 5] = (float)(res[nx - 1] > 0 ? res[x] / res[nx - 1] : 0.0);
        xtab[(size_t)x * 8 + 6] = (float)(0.25 / phi[x]);
    }
    NCK(cudaMemcpy(F.xtab, xtab.data(), xtab.size() * sizeof(float), cudaMemcpyHostToDevice), "x table");
    NCK(cudaMemsetAsync(F.rows + (size_t)v.nf * kF, 0, (size_t)(F.rows_pad - v.nf) * kF * sizeof(bf16), 0), "rows");
    const dim3 blk(kF, 4);
    assemble_kernel<<<(v.nf + 3) / 4, blk>>>(F.cell, v.nf, nx, F.xtab, w, w + N, w + 2 * N, (float)v.current,
                                             (float)v.x_in[0], (float)v.x_in[1], (float)v.x_in[2], F.rows);
    NCK(cudaGetLastError(), "features");
    return LBMS_OK;
}

// The prediction F.pred becomes case k's state and, with Xout, the caller's
// dense field.
lbms_status take_prediction(lbms_net* n, lbms_ctx* ctx, int k, const CaseFeatures& F, double* Xout) {
    lbms::CaseView v;
    lbms::case_view(ctx, k, &v);
    if (Xout) {
        NCK(cudaMemsetAsync(F.dense, 0, (size_t)3 * v.N * sizeof(double), 0), "prediction");
        scatter_kernel<<<(F.nf + 255) / 256, 256>>>(F.pred, F.cell, F.nf, v.N, F.dense);
        NCK(cudaGetLastError(), "prediction");
        lbms::touch_pages(Xout, 3 * v.N);
        NCK(cudaMemcpy(Xout, F.dense, (size_t)3 * v.N * sizeof(double), cudaMemcpyDeviceToHost), "read prediction");
    }
    NCK(cudaStreamSynchronize(0), "prediction");   // the handle may work on another stream
    const lbms_status st = (lbms_status)lbms::case_restart_device(ctx, k, F.pred);
    if (st != LBMS_OK) return nfail(n, st, "restarting case %d: %s", k, lbms_last_error(ctx));
    return LBMS_OK;
}

lbms_status grow(lbms_net* n, int64_t need) {
    if (need <= n->cap) return LBMS_OK;
    int64_t cap = std::max<int64_t>(need, 2 * n->cap);
    bf16* f = nullptr;
    float* t = nullptr;
    NCK(lbms::dev_malloc(&f, (size_t)cap * kF * sizeof(bf16)), "training rows");
    if (lbms::dev_malloc(&t, (size_t)cap * 4 * sizeof(float)) != cudaSuccess) {
        cudaFree(f);
        return nfail(n, LBMS_ENOMEM, "training targets");
    }
    if (n->n_rows) {
        NCK(cudaMemcpy(f, n->feat, (size_t)n->n_rows * kF * sizeof(bf16), cudaMemcpyDeviceToDevice), "grow");
        NCK(cudaMemcpy(t, n->targ, (size_t)n->n_rows * 4 * sizeof(float), cudaMemcpyDeviceToDevice), "grow");
    }
    cudaFree(n->feat);
    cudaFree(n->targ);
    n->feat = f;
    n->targ = t;
    n->cap = cap;
    return LBMS_OK;
}

lbms_status upload_rows(lbms_net* n, const uint16_t* features, int rows) {
    if (!features || rows < 64 || rows > kMaxRows || rows % 64)
        return nfail(n, LBMS_EINVAL, "rows must be a multiple of 64 in [64, %d]", kMaxRows);
    NCK(cudaMemcpy(n->act[0], features, (size_t)rows * kF * sizeof(bf16), cudaMemcpyHostToDevice), "features");
    return LBMS_OK;
}

}  // namespace

extern "C" {

lbms_status lbms_net_create(int width, int depth, uint64_t seed, lbms_net** out) {
    if (!out) return LBMS_EINVAL;
    *out = nullptr;
    if (width < 64 || width > 2048 || width % 64 || depth < 1 || depth > 8) return LBMS_EINVAL;
    lbms_net* n = new (std::nothrow) lbms_net;
    if (!n) return LBMS_ENOMEM;
    n->width = width;
    n->depth = depth;
    n->layers = depth + 1;
    n->seed = seed;
    for (int l = 0; l < n->layers; ++l) {
        n->in.push_back(l == 0 ? kF : width);
        n->out.push_back(l == n->layers - 1 ? kOutPad : width);
    }
    bool ok = true;
    size_t pmax = (size_t)kMaxRows * std::max(width, kF);
    for (int l = 0; l < n->layers; ++l) {
        const size_t nw = (size_t)n->out[l] * n->in[l];
        pmax = std::max(pmax, (size_t)16 * nw);
        n->W.push_back(nalloc<float>(n, nw));
        n->mW.push_back(nalloc<float>(n, nw));
        n->vW.push_back(nalloc<float>(n, nw));
        n->gW.push_back(nalloc<float>(n, nw));
        n->b.push_back(nalloc<float>(n, n->out[l]));
        n->mb.push_back(nalloc<float>(n, n->out[l]));
        n->vb.push_back(nalloc<float>(n, n->out[l]));
        n->Wb.push_back(nalloc<bf16>(n, nw));
        n->WbT.push_back(nalloc<bf16>(n, nw));
        n->act.push_back(nalloc<bf16>(n, (size_t)kMaxRows * n->in[l]));
        n->actT.push_back(nalloc<bf16>(n, (size_t)kMaxRows * n->in[l]));
    }
    const size_t wmax = std::max(width, kOutPad);
    n->dz[0] = nalloc<bf16>(n, (size_t)kMaxRows * wmax);
    n->dz[1] = nalloc<bf16>(n, (size_t)kMaxRows * wmax);
    n->dzT = nalloc<bf16>(n, (size_t)kMaxRows * wmax);
    n->P = nalloc<float>(n, pmax);
    n->P_floats = pmax;
    n->Y = nalloc<float>(n, (size_t)kMaxRows * kOutPad);
    n->T = nalloc<float>(n, (size_t)kMaxRows * 4);
    size_t biases = 0;
    for (int l = 0; l < n->layers; ++l) biases += n->out[l];
    n->zero_bytes = kZeroHead * sizeof(float) + biases * sizeof(float);
    n->zero = nalloc<float>(n, kZeroHead + biases);
    n->loss = reinterpret_cast<double*>(n->zero);
    for (int l = 0, o = kZeroHead; l < n->layers; o += n->out[l++]) n->gb.push_back(n->zero ? n->zero + o : nullptr);
    n->flat = nalloc<float>(n, n_params(n));
    n->gemm_err = nalloc<unsigned int>(n, 1);
    for (void* p : n->allocs) ok = ok && p;
    if (!ok) {
        lbms_net_destroy(n);
        return LBMS_ENOMEM;
    }
    // He-uniform hidden layers, zero output layer and biases; moments zero
    for (int l = 0; l < n->layers; ++l) {
        const size_t nw = (size_t)n->out[l] * n->in[l];
        std::vector<float> w(nw, 0.0f);
        if (l < n->layers - 1) {
            const double a = std::sqrt(6.0 / (l == 0 ? kFUsed : n->in[l]));
            for (size_t e = 0; e < nw; ++e)
                w[e] = (float)(a * (2.0 * unit_double(seed * 0x100000001ull + (uint64_t)l * 0x1000000000ull + e) - 1.0));
        }
        if (cudaMemcpy(n->W[l], w.data(), nw * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess) ok = false;
        cudaMemset(n->gemm_err, 0, sizeof(unsigned int));
        cudaMemset(n->mW[l], 0, nw * sizeof(float));
        cudaMemset(n->vW[l], 0, nw * sizeof(float));
        cudaMemset(n->gW[l], 0, nw * sizeof(float));
        cudaMemset(n->b[l], 0, n->out[l] * sizeof(float));
        cudaMemset(n->mb[l], 0, n->out[l] * sizeof(float));
        cudaMemset(n->vb[l], 0, n->out[l] * sizeof(float));
        cudaMemset(n->gb[l], 0, n->out[l] * sizeof(float));
        cast_weights_kernel<<<grid_for((int64_t)nw), 256>>>(n->W[l], n->out[l], n->in[l], n->Wb[l], n->WbT[l]);
    }
    for (int l = 0; l < n->layers; ++l)
        cudaMemset(n->act[l], 0, (size_t)kMaxRows * n->in[l] * sizeof(bf16));
    if (!ok || cudaDeviceSynchronize() != cudaSuccess) {
        lbms_net_destroy(n);
        return LBMS_ECUDA;
    }
    *out = n;
    return LBMS_OK;
}

void lbms_net_destroy(lbms_net* n) {
    if (!n) return;
    for (void* p : n->allocs) cudaFree(p);
    cudaFree(n->room);
    cudaFree(n->feat);
    cudaFree(n->targ);
    delete n;
}

const char* lbms_net_last_error(const lbms_net* n) { return n ? n->err.c_str() : ""; }

lbms_status lbms_net_info(const lbms_net* n, int64_t* np, int64_t* ns) {
    if (!n) return LBMS_EINVAL;
    if (np) *np = n_params(n);
    if (ns) *ns = n->n_rows;
    return LBMS_OK;
}

lbms_status lbms_net_features(lbms_net* n, lbms_ctx* ctx, int k, uint16_t* rows, int64_t n_rows) {
    if (!n || !ctx || !rows) return LBMS_EINVAL;
    lbms::CaseView v;
    if (!lbms::case_view(ctx, k, &v)) return nfail(n, LBMS_EINVAL, "case index %d out of range", k);
    if (n_rows != v.nf) return nfail(n, LBMS_EINVAL, "case %d has %d fluid cells, the buffer holds %lld rows", k, v.nf,
                                     (long long)n_rows);
    CaseFeatures F(n);
    lbms_status st = case_features(n, ctx, k, F);
    if (st != LBMS_OK) return st;
    NCK(cudaMemcpy(rows, F.rows, (size_t)v.nf * kF * sizeof(bf16), cudaMemcpyDeviceToHost), "feature rows");
    return LBMS_OK;
}

lbms_status lbms_net_add_sample(lbms_net* n, lbms_ctx* ctx, int k) {
    if (!n || !ctx) return LBMS_EINVAL;
    CaseFeatures F(n);
    lbms_status st = case_features(n, ctx, k, F);
    if (st != LBMS_OK) return st;
    lbms::CaseView v;
    lbms::case_view(ctx, k, &v);
    std::vector<double> X((size_t)3 * v.N);
    st = lbms_batch_get_fields(ctx, k, X.data(), nullptr, nullptr);
    if (st != LBMS_OK) return nfail(n, st, "reading the fields of case %d: %s", k, lbms_last_error(ctx));
    std::vector<float> t((size_t)v.nf * 4, 0.0f);
    for (int j = 0; j < v.nf; ++j) {
        const int64_t e = v.fluid_cell[j];
        const int x = (int)(e % v.nx);
        for (int s = 0; s < 3; ++s)
            t[(size_t)j * 4 + s] = (float)(kTargetScale * (X[(size_t)s * v.N + e] - F.prof[(size_t)s * v.nx + x]));
        t[(size_t)j * 4 + 3] = 1.0f;
    }
    st = grow(n, n->n_rows + v.nf);
    if (st != LBMS_OK) return st;
    NCK(cudaMemcpy(n->feat + n->n_rows * kF, F.rows, (size_t)v.nf * kF * sizeof(bf16), cudaMemcpyDeviceToDevice),
        "append rows");
    NCK(cudaMemcpy(n->targ + n->n_rows * 4, t.data(), t.size() * sizeof(float), cudaMemcpyHostToDevice),
        "append targets");
    n->n_rows += v.nf;
    return LBMS_OK;
}

lbms_status lbms_net_train(lbms_net* n, int iters, int batch, double lr, double* last_loss) {
    if (!n) return LBMS_EINVAL;
    if (iters < 0 || batch < 64 || batch > kMaxRows || batch % 64 || !(lr > 0.0))
        return nfail(n, LBMS_EINVAL, "need iters >= 0, batch a multiple of 64 in [64, %d], lr > 0", kMaxRows);
    if (n->n_rows < 1) return nfail(n, LBMS_ESTATE, "no training rows (call lbms_net_add_sample first)");
    double tail = 0.0;
    int nt = 0;
    for (int it = 0; it < iters; ++it) {
        const double cw = 0.5 * (1.0 + std::cos(3.14159265358979323846 * (double)it / std::max(1, iters)));
        const double lr_it = lr / 20.0 + (lr - lr / 20.0) * cw;
        const uint64_t key = splitmix64(n->seed ^ 0xA5A5A5A5ull) + (uint64_t)n->step * (uint64_t)kMaxRows;
        sample_kernel<<<batch, 64>>>(n->feat, n->targ, n->n_rows, key, batch, n->act[0], n->T);
        NCK(cudaGetLastError(), "sample");
        lbms_status st = forward(n, batch, true);
        if (st != LBMS_OK) return st;
        const bool want = it >= iters - 10;
        double l = 0.0;
        st = backward_step(n, batch, lr_it, want ? &l : nullptr);
        if (st != LBMS_OK) return st;
        if (want) {
            tail += l;
            ++nt;
        }
    }
    NCK(cudaDeviceSynchronize(), "train");
    lbms_status gst = check_gemm(n);
    if (gst != LBMS_OK) return gst;
    if (last_loss) *last_loss = nt ? tail / nt : 0.0;
    return LBMS_OK;
}

lbms_status lbms_net_forward(lbms_net* n, const uint16_t* features, int rows, float* out) {
    if (!n || !out) return LBMS_EINVAL;
    lbms_status st = upload_rows(n, features, rows);
    if (st != LBMS_OK) return st;
    st = forward(n, rows, false);
    if (st != LBMS_OK) return st;
    std::vector<float> y((size_t)rows * n->y_ld);
    NCK(cudaMemcpy(y.data(), n->Y, y.size() * sizeof(float), cudaMemcpyDeviceToHost), "read output");
    st = check_gemm(n);
    if (st != LBMS_OK) return st;
    for (int r = 0; r < rows; ++r)
        for (int s = 0; s < kOut; ++s) out[(size_t)r * kOut + s] = y[(size_t)r * n->y_ld + s];
    return LBMS_OK;
}

lbms_status lbms_net_train_batch(lbms_net* n, const uint16_t* features, const float* targets, int rows, double lr,
                                 double* loss) {
    if (!n || !targets || !(lr >= 0.0)) return LBMS_EINVAL;
    lbms_status st = upload_rows(n, features, rows);
    if (st != LBMS_OK) return st;
    std::vector<float> t((size_t)rows * 4, 0.0f);
    for (int r = 0; r < rows; ++r) {
        for (int s = 0; s < kOut; ++s) t[(size_t)r * 4 + s] = targets[(size_t)r * kOut + s];
        t[(size_t)r * 4 + 3] = 1.0f;
    }
    NCK(cudaMemcpy(n->T, t.data(), t.size() * sizeof(float), cudaMemcpyHostToDevice), "targets");
    st = forward(n, rows, true);
    if (st != LBMS_OK) return st;
    st = backward_step(n, rows, lr, loss);
    if (st != LBMS_OK) return st;
    NCK(cudaDeviceSynchronize(), "train batch");
    return check_gemm(n);
}

lbms_status lbms_net_set_gemm(lbms_net* n, int kind) {
    if (!n || (kind != LBMS_NET_GEMM_AUTO && kind != LBMS_NET_GEMM_TCGEN05 && kind != LBMS_NET_GEMM_MMA_SYNC))
        return LBMS_EINVAL;
    if (kind == LBMS_NET_GEMM_TCGEN05) {
        const cudaError_t e = lbms::umma_init();
        if (e != cudaSuccess) return nfail(n, LBMS_ECUDA, "tcgen05 GEMM unavailable: %s", cudaGetErrorString(e));
    }
    n->gemm_kind = kind;
    return LBMS_OK;
}

lbms_status lbms_net_gemm_calls(const lbms_net* n, int64_t* tcgen05, int64_t* mma_sync) {
    if (!n) return LBMS_EINVAL;
    if (tcgen05) *tcgen05 = n->tcgen05_calls;
    if (mma_sync) *mma_sync = n->mma_sync_calls;
    return LBMS_OK;
}

lbms_status lbms_net_get(const lbms_net* cn, int what, float* buf, int64_t count) {
    lbms_net* n = const_cast<lbms_net*>(cn);
    if (!n || !buf || (what != 0 && what != 1)) return LBMS_EINVAL;
    if (count < n_params(n)) return nfail(n, LBMS_EINVAL, "buffer holds %lld floats, need %lld", (long long)count,
                                          (long long)n_params(n));
    // gathered on the device, one copy to the host
    const std::lock_guard<std::mutex> hold(n->flat_use);
    int64_t off = 0;
    auto take = [&](const float* p, size_t count) {
        const cudaError_t e =
            cudaMemcpyAsync(n->flat + off, p, count * sizeof(float), cudaMemcpyDeviceToDevice, 0);
        off += (int64_t)count;
        return e;
    };
    for (int l = 0; l < n->layers; ++l) {
        const int o = l == n->layers - 1 ? kOut : n->out[l];
        NCK(take(what ? n->gW[l] : n->W[l], (size_t)o * n->in[l]), "get");   // the first o rows of [out][in]
        NCK(take(what ? n->gb[l] : n->b[l], o), "get");
    }
    NCK(cudaMemcpy(buf, n->flat, (size_t)off * sizeof(float), cudaMemcpyDeviceToHost), "get");
    return LBMS_OK;
}

lbms_status lbms_net_set(lbms_net* n, const float* buf, int64_t count) {
    if (!n || !buf) return LBMS_EINVAL;
    if (count < n_params(n)) return nfail(n, LBMS_EINVAL, "buffer holds %lld floats, need %lld", (long long)count,
                                          (long long)n_params(n));
    int64_t off = 0;
    for (int l = 0; l < n->layers; ++l) {
        const int o = l == n->layers - 1 ? kOut : n->out[l];
        const size_t nw = (size_t)o * n->in[l];
        NCK(cudaMemcpy(n->W[l], buf + off, nw * sizeof(float), cudaMemcpyHostToDevice), "set");
        off += nw;
        NCK(cudaMemcpy(n->b[l], buf + off, o * sizeof(float), cudaMemcpyHostToDevice), "set");
        off += o;
        cast_weights_kernel<<<grid_for((int64_t)n->out[l] * n->in[l]), 256>>>(n->W[l], n->out[l], n->in[l],
                                                                              n->Wb[l], n->WbT[l]);
        NCK(cudaGetLastError(), "cast");
    }
    NCK(cudaDeviceSynchronize(), "set");
    return LBMS_OK;
}

lbms_status lbms_net_warm_start(lbms_net* n, lbms_ctx* ctx, int k, double* Xout) {
    if (!n || !ctx) return LBMS_EINVAL;
    CaseFeatures F(n);
    lbms_status st = case_features(n, ctx, k, F);
    if (st != LBMS_OK) return st;
    lbms::CaseView v;
    lbms::case_view(ctx, k, &v);
    for (int j0 = 0; j0 < F.rows_pad; j0 += kMaxRows) {
        const int rows = std::min(kMaxRows, F.rows_pad - j0);
        NCK(cudaMemcpy(n->act[0], F.rows + (size_t)j0 * kF, (size_t)rows * kF * sizeof(bf16),
                       cudaMemcpyDeviceToDevice),
            "rows");
        st = forward(n, rows, false);
        if (st != LBMS_OK) return st;
        predict_post_kernel<<<(rows + 255) / 256, 256>>>(n->Y, n->y_ld, F.cell, j0, rows, v.nf, v.nx, F.xtab, F.pred);
        NCK(cudaGetLastError(), "prediction");
    }
    st = check_gemm(n);   // before the handle's state is replaced
    if (st != LBMS_OK) return st;
    return take_prediction(n, ctx, k, F, Xout);
}

// For tests: leaves the network as a product whose wait ran out does.
int lbms_internal_net_timeout(lbms_net* n) {
    const unsigned int f = 1u;
    return cudaMemcpy(n->gemm_err, &f, sizeof(f), cudaMemcpyHostToDevice);
}

}  // extern "C"

#include "lbms_unet.cuh"
