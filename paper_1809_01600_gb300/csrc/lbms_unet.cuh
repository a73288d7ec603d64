// The convolutional warm start (declared in include/lbms_net.h): a 3-D U-Net
// over the anode's voxels, trained and run with this file's kernels and the
// tcgen05 kernels of lbms_conv.cu.  Included at the end of lbms_net.cu, whose
// feature builder, split-K sum, Adam and weight-cast kernels it shares.
//
// Layout.  Activations are channels-last BF16 rows [row][C] (C = 32, 64 or
// 128 at the three levels, the smallest that holds the real channels; the
// real channels first, zeros after).  Each volume of X x Y x Z voxels is
// stored with a zero halo of one voxel in front of each row, plane and volume,
// in Xp x Yp x Zp = (X + 1) x (Y + 1) x (Z + 1) rows, volumes one after the other:
// the halo behind a row is the one in front of the next, and behind the last
// volume come padding rows (zeros) and what TMA fills in (zeros).  A halo on
// both sides and rows of a multiple of 8 took 9 % more rows at 96^3 and 18 % at
// 64x32x32.  The row count is padded to a multiple of 64 S (S chunks of the
// reductions over rows).  The neighbour of a voxel at tap (dz, dy, dx) is
// then off = (dz Yp + dy) Xp + dx rows away, so a 3x3x3 convolution is an
// implicit GEMM on the tensor cores (lbms_conv.cu).  What follows a product
// is done on its accumulators: bias, ReLU, zero halo and the copy into the
// concatenation's buffer (forward); the ReLU mask of the next layer down, its
// BF16 gradient and the bias-gradient sums (backward); the split of a
// concatenation's gradient; the transposed convolution's scatter to the 8
// children of a voxel; the head's loss.  Weight gradients are products over
// rows that read both operands as they lie in memory.  Every kernel that
// writes an activation or a gradient writes all its rows, zeros outside the
// volumes, so the halo reads as zero padding whatever batch used the buffers
// before (the gathered gradients G are cleared when the layout changes).
namespace {

constexpr int kUInC = 32;      // stored input channels: the 16 feature columns, the fluid mask, zeros
constexpr int kUInReal = 17;
constexpr int kUOutC = 32;     // stored output channels of the 1x1 head (3 used)
constexpr int kULayers = 13;

// Layout of one resolution level of a batch (all row counts below 2^31).
struct Geo {
    int B = 0, X = 0, Y = 0, Z = 0;   // volumes; interior extents of one volume
    int Xp = 0, Yp = 0, Zp = 0;       // extents with the halo
    int64_t V = 0;                    // interior voxels of the batch
    int64_t R = 0;                    // rows of the layout, B Xp Yp Zp
    int64_t Rp = 0;                   // rows processed: R + 2 or more, a multiple of 64 S
    int S = 1;                        // chunks of the reductions over rows
};

// Interior coordinates of row r; false for halo and padding rows.
__device__ __forceinline__ bool row_voxel(const Geo& g, int64_t r, int& x, int& y, int& z, int& b) {
    if (r >= g.R) return false;
    unsigned q = (unsigned)r;
    x = (int)(q % (unsigned)g.Xp) - 1;
    q /= (unsigned)g.Xp;
    y = (int)(q % (unsigned)g.Yp) - 1;
    q /= (unsigned)g.Yp;
    z = (int)(q % (unsigned)g.Zp) - 1;
    b = (int)(q / (unsigned)g.Zp);
    return x >= 0 && x < g.X && y >= 0 && y < g.Y && z >= 0 && z < g.Z;
}

__device__ __forceinline__ int64_t voxel_row(const Geo& g, int b, int x, int y, int z) {
    return (((int64_t)b * g.Zp + z + 1) * g.Yp + y + 1) * g.Xp + x + 1;
}

// One warp per row: the global warp index and the warp count of the grid.
__device__ __forceinline__ int64_t warp_id() { return ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; }
__device__ __forceinline__ int64_t warp_count() { return ((int64_t)gridDim.x * blockDim.x) >> 5; }

// 2x2x2 max pooling from level `hi` to level `lo` (C channels): every row
// of lo, the maximum of the 8 children and the child (dz 4 + dy 2 + dx) of
// the first maximum on interior rows, 0 elsewhere.  A thread takes 8 channels
// of a row (16-byte loads).
__global__ void __launch_bounds__(256) pool_rows_kernel(const bf16* __restrict__ x, Geo hi, Geo lo, int C,
                                                        bf16* __restrict__ y, uint8_t* __restrict__ arg) {
    const int per = C / 8;
    const int64_t n = lo.Rp * per;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = e / per;
        const int c = (int)(e - r * per) * 8;
        int xl, yl, zl, b;
        const bool in = row_voxel(lo, r, xl, yl, zl, b);
        __align__(16) bf16 best[8];
        __align__(8) uint8_t at[8];
        for (int q = 0; q < 8; ++q) {
            best[q] = __float2bfloat16_rn(0.0f);
            at[q] = 0;
        }
        if (in) {
            const int64_t c0 = voxel_row(hi, b, 2 * xl, 2 * yl, 2 * zl);
            float m[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const int64_t w = c0 + ((int64_t)(t >> 2) * hi.Yp + ((t >> 1) & 1)) * hi.Xp + (t & 1);
                __align__(16) bf16 v[8];
                *reinterpret_cast<uint4*>(v) = __ldg(reinterpret_cast<const uint4*>(x + w * C + c));
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const float f = __bfloat162float(v[q]);
                    if (t == 0 || f > m[q]) {
                        m[q] = f;
                        best[q] = v[q];
                        at[q] = (uint8_t)t;
                    }
                }
            }
        }
        *reinterpret_cast<uint4*>(y + r * C + c) = *reinterpret_cast<const uint4*>(best);
        *reinterpret_cast<uint2*>(arg + r * C + c) = *reinterpret_cast<const uint2*>(at);
    }
}

// The gradient through a pooling, a skip connection and the ReLU below both:
// dz[r][c] = BF16(act > 0 ? skip[r][c] + (dp of the parent where r holds its
// maximum) : 0) on every row of hi (act is 0 outside the volumes), and the
// column sums of the unrounded values added into gb.  C is 32 or 64; a thread
// takes 8 channels of a row.  Bound by memory: 9 C bytes a row read (skip
// FP32, act, arg of the parent) and 2 C written.
__global__ void __launch_bounds__(256) pool_relu_back_kernel(const float* __restrict__ dp, const uint8_t* __restrict__ arg,
                                                             const float* __restrict__ skip,
                                                             const bf16* __restrict__ act, Geo hi, Geo lo, int C,
                                                             bf16* __restrict__ dz, float* __restrict__ gb) {
    __shared__ float part[256 * 8];
    const int per = C / 8;
    const int c = (threadIdx.x % per) * 8;
    float sum[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) sum[q] = 0.0f;
    const int rows = 256 / per;
    for (int64_t r = (int64_t)blockIdx.x * rows + threadIdx.x / per; r < hi.Rp; r += (int64_t)gridDim.x * rows) {
        const uint4 av = __ldg(reinterpret_cast<const uint4*>(act + r * C + c));
        __align__(16) bf16 o[8];
        if (av.x | av.y | av.z | av.w) {
            __align__(16) bf16 a[8];
            *reinterpret_cast<uint4*>(a) = av;
            float v[8];
            *reinterpret_cast<float4*>(v) = __ldg(reinterpret_cast<const float4*>(skip + r * C + c));
            *reinterpret_cast<float4*>(v + 4) = __ldg(reinterpret_cast<const float4*>(skip + r * C + c + 4));
            int x, y, z, b;
            if (row_voxel(hi, r, x, y, z, b)) {
                const int64_t p = voxel_row(lo, b, x >> 1, y >> 1, z >> 1);
                const int t = (z & 1) * 4 + (y & 1) * 2 + (x & 1);
                __align__(8) uint8_t at[8];
                *reinterpret_cast<uint2*>(at) = __ldg(reinterpret_cast<const uint2*>(arg + p * C + c));
                float d[8];
                *reinterpret_cast<float4*>(d) = __ldg(reinterpret_cast<const float4*>(dp + p * C + c));
                *reinterpret_cast<float4*>(d + 4) = __ldg(reinterpret_cast<const float4*>(dp + p * C + c + 4));
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (at[q] == t) v[q] += d[q];
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float w = __bfloat162float(a[q]) > 0.0f ? v[q] : 0.0f;
                o[q] = __float2bfloat16_rn(w);
                sum[q] += w;
            }
        } else {
            *reinterpret_cast<uint4*>(o) = make_uint4(0u, 0u, 0u, 0u);
        }
        *reinterpret_cast<uint4*>(dz + r * C + c) = *reinterpret_cast<const uint4*>(o);
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) part[threadIdx.x * 8 + q] = sum[q];
    __syncthreads();
    if (threadIdx.x < C) {   // column threadIdx.x: threads of channel group threadIdx.x / 8
        float t = 0.0f;
        for (int g = threadIdx.x / 8; g < 256; g += per) t += part[g * 8 + threadIdx.x % 8];
        atomicAdd(&gb[threadIdx.x], t);
    }
}

// G[o][i] = sum_z P[z][i][o] (split-K partials of a transposed product), in
// the order of z; threads walk P's order, 8 chunks in flight.
__global__ void splitk_sum_t_kernel(const float* __restrict__ P, int S, int I, int O, float* __restrict__ G) {
    const int64_t n = (int64_t)O * I;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        float acc = 0.0f;
        int z = 0;
        for (; z + 8 <= S; z += 8) {
            float v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = __ldg(P + (int64_t)(z + q) * n + e);
#pragma unroll
            for (int q = 0; q < 8; ++q) acc += v[q];
        }
        for (; z < S; ++z) acc += __ldg(P + (int64_t)z * n + e);
        const int i = (int)(e / O), o = (int)(e % O);
        G[(int64_t)o * I + i] = acc;
    }
}

// BF16 copies of a 3x3x3 convolution's FP32 weights W [co_s][27 ci_s]
// (entry (co, tap ci_s + ci)): Wb, the same layout, and Wf [ci_s][27 co_s],
// the flipped weights of the input gradient, entry (ci, tap co_s + co).
__global__ void conv_cast_kernel(const float* __restrict__ W, int co_s, int ci_s, bf16* __restrict__ Wb,
                                 bf16* __restrict__ Wf) {
    const int K = 27 * ci_s;
    const int64_t n = (int64_t)co_s * K;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int co = (int)(e / K), k = (int)(e % K);
        const int tap = k / ci_s, ci = k - tap * ci_s;
        const bf16 wb = __float2bfloat16_rn(W[e]);
        Wb[e] = wb;
        Wf[(int64_t)ci * 27 * co_s + tap * co_s + co] = wb;
    }
}

// A batch given as FP32 [B][17][Z][Y][X] (channel 16 the fluid mask) into
// the interior rows of x0 [rows][kUInC] (BF16) and the mask column of T [rows][4]
// (both cleared before); one warp per voxel.
__global__ void vol_in_kernel(const float* __restrict__ in, Geo g, bf16* __restrict__ x0, float* __restrict__ T) {
    const int lane = threadIdx.x & 31;
    const int64_t S = (int64_t)g.X * g.Y * g.Z;
    for (int64_t v = warp_id(); v < g.V; v += warp_count()) {
        const int b = (int)(v / S);
        const int64_t s = v - b * S;
        const int x = (int)(s % g.X), y = (int)((s / g.X) % g.Y), z = (int)(s / ((int64_t)g.X * g.Y));
        const int64_t r = voxel_row(g, b, x, y, z);
        for (int c = lane; c < kUInC; c += 32) {
            const float val = c < kUInReal ? in[((int64_t)b * kUInReal + c) * S + s] : 0.0f;
            x0[r * kUInC + c] = __float2bfloat16_rn(val);
            if (c == kUInReal - 1) T[r * 4 + 3] = val;
        }
    }
}

// Targets given as FP32 [B][3][Z][Y][X] into T[row][0:3] of the interior rows.
__global__ void vol_target_kernel(const float* __restrict__ t, Geo g, float* __restrict__ T) {
    const int64_t S = (int64_t)g.X * g.Y * g.Z;
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < g.V; v += (int64_t)gridDim.x * blockDim.x) {
        const int b = (int)(v / S);
        const int64_t s = v - b * S;
        const int x = (int)(s % g.X), y = (int)((s / g.X) % g.Y), z = (int)(s / ((int64_t)g.X * g.Y));
        const int64_t r = voxel_row(g, b, x, y, z);
        for (int c = 0; c < 3; ++c) T[r * 4 + c] = t[((int64_t)b * 3 + c) * S + s];
    }
}

// Input rows of one case: vol[row[j]][c] = rows[j][c] (c < 16), the fluid
// mask in channel 16; every other row stays zero (cleared before).
__global__ void unet_inputs_kernel(const bf16* __restrict__ rows, const int64_t* __restrict__ row, int nf,
                                   bf16* __restrict__ vol) {
    const int64_t n = (int64_t)nf * kUInC;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int j = (int)(e / kUInC), c = (int)(e % kUInC);
        bf16 val = __float2bfloat16_rn(0.0f);
        if (c < kFUsed) val = rows[(int64_t)j * kF + c];
        else if (c == kFUsed) val = __float2bfloat16_rn(1.0f);
        vol[row[j] * kUInC + c] = val;
    }
}

// Row of every fluid cell of a case (dense index cell[j]) in the layout of
// its volume.
__global__ void cell_row_kernel(const int64_t* __restrict__ cell, int nf, int nx, int ny, Geo g,
                                int64_t* __restrict__ row) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= nf) return;
    const int64_t e = cell[j];
    row[j] = voxel_row(g, 0, (int)(e % nx), (int)((e / nx) % ny), (int)(e / ((int64_t)nx * ny)));
}

// The prediction of one case from the head's output Y [r][4] at its row
// row[j]: X_s = profile_s(x) + Y[row][s] / 100, clamped at 1e-6 and
// renormalised; out [3][nf] FP64.  Xp: the padded x extent (x = row mod Xp - 1).
__global__ void unet_post_kernel(const float* __restrict__ Y, const int64_t* __restrict__ row, int nf, int Xp,
                                 const float* __restrict__ xtab, double* __restrict__ out) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= nf) return;
    const int64_t r = row[j];
    const int x = (int)(r % Xp) - 1;
    double X[3], s = 0.0;
    for (int q = 0; q < 3; ++q) {
        double val = (double)xtab[(int64_t)x * 8 + q] + (double)Y[r * 4 + q] / kTargetScale;
        val = val < 1e-6 ? 1e-6 : val;
        X[q] = val;
        s += val;
    }
    for (int q = 0; q < 3; ++q) out[(int64_t)q * nf + j] = X[q] / s;
}

}  // namespace

// ------------------------------------------------------------------ host
struct lbms_unet {
    struct Layer {
        int kind = 3;            // 3: 3x3x3 conv + ReLU, 2: 2x2x2 transposed conv (stride 2), 1: 1x1 head
        int level = 0;           // resolution level of the output (0 full, 1 half, 2 quarter)
        int ci = 0, ci_s = 0, co = 0, co_s = 0;   // real / stored channels
        int rows = 0, K = 0;     // FP32 master weights W [rows][K]
        float *W = nullptr, *m = nullptr, *v = nullptr, *g = nullptr;
        float *b = nullptr, *mb = nullptr, *vb = nullptr, *gb = nullptr;   // [co_s]
        bf16* Wb = nullptr;      // BF16 copy of W
        bf16* Wt = nullptr;      // kind 3: flipped weights [ci_s][27 co_s]; kinds 1, 2: transpose of Wb [K][rows]
    };
    int width = 0;
    Layer L[kULayers];           // e1a e1b e2a e2b e3a e3b u2 d2a d2b u1 d1a d1b head
    int64_t vcap = 0;            // interior voxels of one batch at most
    // activations and scratch, sized for the largest batch layout so far (grown on demand)
    int64_t cap[3] = {0, 0, 0};  // rows per level the buffers hold
    size_t splits[3] = {0, 0, 0};   // and chunks of the reductions the partials hold
    bf16 *x0 = nullptr, *e1a = nullptr, *e1 = nullptr, *c1 = nullptr, *d1a = nullptr, *d1 = nullptr;
    bf16 *p1 = nullptr, *e2a = nullptr, *e2 = nullptr, *c2 = nullptr, *d2a = nullptr, *d2 = nullptr;
    bf16 *p2 = nullptr, *e3a = nullptr, *e3 = nullptr;
    uint8_t *arg1 = nullptr, *arg2 = nullptr;
    bf16 *za[3] = {nullptr, nullptr, nullptr}, *zb[3] = {nullptr, nullptr, nullptr};   // pre-activation gradients per level
    bf16 *G1 = nullptr, *G2 = nullptr;            // transposed convolutions' output gradients, gathered by parent
    float *skip0 = nullptr, *skip1 = nullptr;     // skip connections' gradients
    float *dp1 = nullptr, *dp2 = nullptr;         // pooled activations' gradients
    float *P = nullptr, *Y = nullptr, *T = nullptr;
    size_t P_floats = 0;
    int last[4] = {0, 0, 0, 0};  // B, X, Y, Z of the layout the buffers held last
    std::vector<void*> bufs;     // the grown buffers
    float* zero = nullptr;       // the loss and all bias gradients, cleared together
    size_t zero_bytes = 0;
    double* loss = nullptr;
    float* flat = nullptr;       // parameters or gradients in the caller's order
    std::mutex flat_use;
    unsigned int* gemm_err = nullptr;
    struct Sample {
        int X = 0, Y = 0, Z = 0;                // interior extents (multiples of 4)
        int64_t rows = 0, nfluid = 0;           // rows of its layout; fluid voxels
        bf16* in = nullptr;                     // [rows][kUInC]
        float* tg = nullptr;                    // [rows][4]: 100 (X - profile), fluid mask
    };
    std::vector<Sample> samples;
    int64_t step = 0, tcgen05_calls = 0;
    uint64_t seed = 0;
    std::vector<void*> allocs;   // weights and the small fixed buffers
    std::string msg;
    lbms_net feat;               // error messages and working memory of the shared feature builder
};

namespace {

lbms_status ufail(lbms_unet* u, lbms_status s, const char* fmt, ...) {
    if (u) {
        char buf[512];
        va_list ap;
        va_start(ap, fmt);
        std::vsnprintf(buf, sizeof(buf), fmt, ap);
        va_end(ap);
        u->msg = buf;
    }
    return s;
}

#define UCK(expr, what)                                                                               \
    do {                                                                                             \
        cudaError_t e_ = (expr);                                                                     \
        if (e_ != cudaSuccess) return ufail(u, LBMS_ECUDA, "%s: %s", what, cudaGetErrorString(e_)); \
    } while (0)

#define UST(call)                     \
    do {                              \
        lbms_status s_ = (call);      \
        if (s_ != LBMS_OK) return s_; \
    } while (0)

template <typename T>
T* ualloc(lbms_unet* u, size_t count) {
    void* p = nullptr;
    lbms::dev_malloc(&p, std::max<size_t>(count, 1) * sizeof(T));
    u->allocs.push_back(p);
    return static_cast<T*>(p);
}

// The reductions over rows (weight gradients) are split in S chunks, of as many
// voxels as 16384 rows hold where the halo lies on both sides of a row (of a
// multiple of 8), a plane and a volume.  The tensor cores' FP32 accumulators
// truncate, so a chunk's length is its error: 2e-5 to 3e-5 of a gradient at this
// length, and 3.5e-5 more with chunks 2.4 times as long.
constexpr int64_t kChunkRows = 16384;
// Rows of a level at most: what batches were always limited to (the kernels'
// row numbers are 32-bit, and rows times channels fit 63 bits far beyond it).
constexpr int64_t kGemmMaxRows = 65535ll * 128;

// Zero rows behind the last volume that the weight gradients of the 3x3x3
// convolutions need (they reach dz up to two rows late).
constexpr int64_t kTailRows = 2;

int64_t splits_for(int B, int X, int Y, int Z) {
    const int64_t R = (int64_t)B * ((X + 9) / 8 * 8) * (Y + 2) * (Z + 2);
    return std::max<int64_t>(1, (R + kChunkRows - 1) / kChunkRows);
}

Geo make_geo(int B, int X, int Y, int Z) {
    Geo g;
    g.B = B;
    g.X = X;
    g.Y = Y;
    g.Z = Z;
    g.Xp = X + 1;
    g.Yp = Y + 1;
    g.Zp = Z + 1;
    g.V = (int64_t)B * X * Y * Z;
    g.R = (int64_t)B * g.Xp * g.Yp * g.Zp;
    g.S = (int)splits_for(B, X, Y, Z);
    const int64_t q = 64 * (int64_t)g.S;
    g.Rp = (g.R + kTailRows + q - 1) / q * q;
    return g;
}

// The three levels of a batch of B volumes of X x Y x Z voxels.
struct Levels {
    Geo g[3];
};

Levels levels_of(int B, int X, int Y, int Z) {
    Levels v;
    for (int l = 0; l < 3; ++l) v.g[l] = make_geo(B, X >> l, Y >> l, Z >> l);
    return v;
}

bool levels_fit(const Levels& v) {
    for (const auto& g : v.g)
        if (g.Rp > kGemmMaxRows) return false;
    return true;
}

// Grows the activation and scratch buffers to hold the layout of `v`.
lbms_status ensure_buffers(lbms_unet* u, const Levels& v) {
    int64_t c[3];
    size_t sp[3];
    bool grow = false;
    for (int l = 0; l < 3; ++l) {
        c[l] = std::max(u->cap[l], v.g[l].Rp);
        sp[l] = std::max<size_t>(u->splits[l], v.g[l].S);
        grow = grow || c[l] > u->cap[l] || sp[l] > u->splits[l];
    }
    if (!grow) return LBMS_OK;
    UCK(cudaDeviceSynchronize(), "U-Net buffers");
    for (void* p : u->bufs) cudaFree(p);
    u->bufs.clear();
    for (int l = 0; l < 3; ++l) u->cap[l] = u->splits[l] = 0;
    const size_t c0 = c[0], c1 = c[1], c2 = c[2];
    const size_t s0 = sp[0], s1 = sp[1], s2 = sp[2];
    u->P_floats = std::max({s0 * 64 * 864, s1 * 128 * 1728, s2 * 128 * 3456, s1 * 256 * 64, s2 * 512 * 128});
    bool ok = true;
    auto get = [&](size_t bytes) {
        void* p = nullptr;
        if (ok && lbms::dev_malloc(&p, std::max<size_t>(bytes, 16)) == cudaSuccess) {
            u->bufs.push_back(p);
            ok = cudaMemset(p, 0, std::max<size_t>(bytes, 16)) == cudaSuccess;
        } else {
            ok = false;
        }
        return p;
    };
    auto act = [&](size_t rows, int C) { return static_cast<bf16*>(get(rows * C * sizeof(bf16))); };
    auto f32 = [&](size_t count) { return static_cast<float*>(get(count * sizeof(float))); };
    u->x0 = act(c0, kUInC);
    u->e1a = act(c0, 32);
    u->e1 = act(c0, 32);
    u->c1 = act(c0, 64);
    u->d1a = act(c0, 32);
    u->d1 = act(c0, 32);
    u->p1 = act(c1, 32);
    u->e2a = act(c1, 64);
    u->e2 = act(c1, 64);
    u->c2 = act(c1, 128);
    u->d2a = act(c1, 64);
    u->d2 = act(c1, 64);
    u->p2 = act(c2, 64);
    u->e3a = act(c2, 128);
    u->e3 = act(c2, 128);
    u->arg1 = static_cast<uint8_t*>(get(c1 * 32));
    u->arg2 = static_cast<uint8_t*>(get(c2 * 64));
    for (int l = 0; l < 3; ++l) {
        u->za[l] = act(l == 0 ? c0 : l == 1 ? c1 : c2, 32 << l);
        u->zb[l] = act(l == 0 ? c0 : l == 1 ? c1 : c2, 32 << l);
    }
    u->G1 = act(c1, 256);
    u->G2 = act(c2, 512);
    u->skip0 = f32(c0 * 32);
    u->skip1 = f32(c1 * 64);
    u->dp1 = f32(c1 * 32);
    u->dp2 = f32(c2 * 64);
    u->P = f32(u->P_floats);
    u->Y = f32(c0 * 4);
    u->T = f32(c0 * 4);
    for (int& d : u->last) d = 0;
    if (!ok) {
        for (void* p : u->bufs) cudaFree(p);
        u->bufs.clear();
        return ufail(u, LBMS_ENOMEM, "U-Net buffers for %lld rows", (long long)c0);
    }
    for (int l = 0; l < 3; ++l) {
        u->cap[l] = c[l];
        u->splits[l] = sp[l];
    }
    return LBMS_OK;
}

// Blocks of 256 threads for one warp per row over R rows (grid-stride beyond 152 x 16 blocks).
int warp_grid(int64_t R) { return (int)std::max<int64_t>(1, std::min<int64_t>((R + 7) / 8, 152 * 16)); }

lbms::RowLayout layout_of(const Geo& g) {
    lbms::RowLayout l;
    l.X = g.X;
    l.Y = g.Y;
    l.Z = g.Z;
    l.Xp = g.Xp;
    l.Yp = g.Yp;
    l.Zp = g.Zp;
    l.R = g.R;
    return l;
}

// Row offsets of the 27 taps on layout g, times sign.
void set_taps(const Geo& g, int sign, int (&off)[27]) {
    for (int k = 0; k < 27; ++k) {
        const int dx = k % 3 - 1, dy = (k / 3) % 3 - 1, dz = k / 9 - 1;
        off[k] = sign * ((dz * g.Yp + dy) * g.Xp + dx);
    }
}

// A product over the rows of g: x [Rp][C] with the layer's weights W [N][taps C].
lbms::ConvJob conv_job(const Geo& g, const bf16* x, int C, const bf16* W, int N, int taps, int sign,
                       lbms::ConvOut kind) {
    lbms::ConvJob j;
    j.x = x;
    j.W = W;
    j.rows = (int)g.Rp;
    j.C = C;
    j.N = N;
    j.taps = taps;
    if (taps == 27) set_taps(g, sign, j.off);
    j.kind = kind;
    j.ep.g = layout_of(g);
    return j;
}

lbms_status run_conv(lbms_unet* u, const lbms::ConvJob& j, const char* what) {
    UCK(lbms::umma_conv(j, u->gemm_err, 0), what);
    ++u->tcgen05_calls;
    return LBMS_OK;
}

// ------------------------------------------------------ layer passes
// relu(conv3(x) + b) -> out; with cat, the first w columns also to cat[r][off ...] (stride ld)
lbms_status conv_fwd(lbms_unet* u, const lbms_unet::Layer& l, const bf16* x, const Geo& g, bf16* out,
                     bf16* cat = nullptr, int ld = 0, int off = 0, int w = 0) {
    lbms::ConvJob j = conv_job(g, x, l.ci_s, l.Wb, l.co_s, 27, 1, lbms::kOutRelu);
    j.ep.bias = l.b;
    j.ep.out = out;
    j.ep.cat = cat;
    j.ep.cat_ld = ld;
    j.ep.cat_off = off;
    j.ep.w = w;
    return run_conv(u, j, "convolution");
}

// transposed 2x2x2 convolution of x [lo.Rp][ci_s] into the first w columns of cat [hi.Rp][2 co_s]
lbms_status up_fwd(lbms_unet* u, const lbms_unet::Layer& l, const bf16* x, const Geo& lo, const Geo& hi, bf16* cat) {
    lbms::ConvJob j = conv_job(lo, x, l.ci_s, l.Wb, l.rows, 1, 1, lbms::kOutUp);
    j.ep.bias = l.b;
    j.ep.cat = cat;
    j.ep.cat_ld = 2 * l.co_s;
    j.ep.Cg = l.co_s;
    j.ep.w = l.co;
    j.ep.other = layout_of(hi);
    return run_conv(u, j, "up convolution");
}

// Weight gradient from the pre-activation gradient dz (kind 3: dz [Rp][co_s]
// against the taps of x [Rp][ci_s]; kinds 1, 2: of [rows] = dz's or G's columns)
lbms_status layer_wgrad(lbms_unet* u, const lbms_unet::Layer& l, const bf16* x, const bf16* dz, const Geo& g) {
    if ((size_t)g.S * l.rows * l.K > u->P_floats) return ufail(u, LBMS_EINVAL, "U-Net weight gradient too large");
    lbms::WgradJob j;
    j.rows = (int)g.Rp;
    j.S = g.S;
    j.P = u->P;
    const int64_t n = (int64_t)l.rows * l.K;
    if (l.kind == 3) {   // P [S][27 ci_s][co_s]
        j.x = x;
        j.C = l.ci_s;
        j.dz = dz;
        j.N = l.co_s;
        set_taps(g, 1, j.off);
    } else {             // P [S][rows][K]
        j.x = dz;
        j.C = l.rows;
        j.dz = x;
        j.N = l.K;
        j.taps = 1;
    }
    UCK(lbms::umma_wgrad(j, u->gemm_err, 0), "weight gradient");
    ++u->tcgen05_calls;
    if (l.kind == 3)
        splitk_sum_t_kernel<<<grid_for(n), 256>>>(u->P, g.S, l.K, l.co_s, l.g);
    else
        splitk_sum_kernel<<<grid_for(n), 256>>>(u->P, g.S, n, l.g);
    UCK(cudaGetLastError(), "split-k sum");
    return LBMS_OK;
}

// The gradient of a layer's input through the ReLU of the layer `prev` that
// made it (activation act): prev's pre-activation gradient into out, its bias
// gradient into prev.gb.
lbms_status dgrad_relu(lbms_unet* u, const lbms_unet::Layer& l, const bf16* dz, const Geo& g, const bf16* act,
                       const lbms_unet::Layer& prev, bf16* out) {
    const bool conv = l.kind == 3;
    lbms::ConvJob j = conv_job(g, dz, conv ? l.co_s : l.rows, l.Wt, l.ci_s, conv ? 27 : 1, -1, lbms::kOutReluBack);
    j.ep.act = act;
    j.ep.out = out;
    j.ep.gb = prev.gb;
    return run_conv(u, j, "input gradient");
}

// The gradient of a concatenation (up-sampled half, skip half) read by l: the
// first gathered into G for the transposed convolution `up`, the second into
// skip.
lbms_status dgrad_split(lbms_unet* u, const lbms_unet::Layer& l, const bf16* dz, const Geo& g, const Geo& lo,
                        const lbms_unet::Layer& up, bf16* G, float* skip) {
    lbms::ConvJob j = conv_job(g, dz, l.co_s, l.Wt, l.ci_s, 27, -1, lbms::kOutSplit);
    j.ep.G = G;
    j.ep.Cg = up.co_s;
    j.ep.w = up.co;
    j.ep.gb = up.gb;
    j.ep.P = skip;
    j.ep.other = layout_of(lo);
    return run_conv(u, j, "input gradient");
}

// The gradient of a pooled activation, FP32 [Rp][ci_s].
lbms_status dgrad_store(lbms_unet* u, const lbms_unet::Layer& l, const bf16* dz, const Geo& g, float* out) {
    lbms::ConvJob j = conv_job(g, dz, l.co_s, l.Wt, l.ci_s, 27, -1, lbms::kOutStore);
    j.ep.P = out;
    return run_conv(u, j, "input gradient");
}

// ------------------------------------------------------ network passes
// Forward pass of a batch already in u->x0 (layout v.g[0]).  With `train`,
// against u->T: the loss, the head's output gradient (za[0]) and its bias
// gradient; otherwise the head's output in u->Y [Rp][4].
lbms_status unet_forward(lbms_unet* u, const Levels& v, bool train, float inv_n) {
    const Geo &g0 = v.g[0], &g1 = v.g[1], &g2 = v.g[2];
    const int w = u->width;
    auto& L = u->L;
    if (u->last[0] != g0.B || u->last[1] != g0.X || u->last[2] != g0.Y || u->last[3] != g0.Z) {
        UCK(cudaMemsetAsync(u->G1, 0, (size_t)u->cap[1] * 256 * sizeof(bf16), 0), "clear gradients");
        UCK(cudaMemsetAsync(u->G2, 0, (size_t)u->cap[2] * 512 * sizeof(bf16), 0), "clear gradients");
        u->last[0] = g0.B;
        u->last[1] = g0.X;
        u->last[2] = g0.Y;
        u->last[3] = g0.Z;
    }
    UST(conv_fwd(u, L[0], u->x0, g0, u->e1a));
    UST(conv_fwd(u, L[1], u->e1a, g0, u->e1, u->c1, 64, w, w));
    pool_rows_kernel<<<grid_for(g1.Rp * 4), 256>>>(u->e1, g0, g1, 32, u->p1, u->arg1);
    UCK(cudaGetLastError(), "pool");
    UST(conv_fwd(u, L[2], u->p1, g1, u->e2a));
    UST(conv_fwd(u, L[3], u->e2a, g1, u->e2, u->c2, 128, 2 * w, 2 * w));
    pool_rows_kernel<<<grid_for(g2.Rp * 8), 256>>>(u->e2, g1, g2, 64, u->p2, u->arg2);
    UCK(cudaGetLastError(), "pool");
    UST(conv_fwd(u, L[4], u->p2, g2, u->e3a));
    UST(conv_fwd(u, L[5], u->e3a, g2, u->e3));
    UST(up_fwd(u, L[6], u->e3, g2, g1, u->c2));
    UST(conv_fwd(u, L[7], u->c2, g1, u->d2a));
    UST(conv_fwd(u, L[8], u->d2a, g1, u->d2));
    UST(up_fwd(u, L[9], u->d2, g1, g0, u->c1));
    UST(conv_fwd(u, L[10], u->c1, g0, u->d1a));
    UST(conv_fwd(u, L[11], u->d1a, g0, u->d1));
    const lbms_unet::Layer& h = L[12];
    lbms::ConvJob j = conv_job(g0, u->d1, h.ci_s, h.Wb, h.rows, 1, 1, lbms::kOutHead);
    j.ep.bias = h.b;
    if (train) {
        UCK(cudaMemsetAsync(u->zero, 0, u->zero_bytes, 0), "loss and bias gradients");
        j.ep.T = u->T;
        j.ep.grad_scale = 2.0f * inv_n;
        j.ep.loss_scale = (double)inv_n;
        j.ep.out = u->za[0];
        j.ep.gb = h.gb;
        j.ep.loss = u->loss;
        j.ep.done = reinterpret_cast<unsigned int*>(u->loss + 4);
    } else {
        j.ep.Y = u->Y;
    }
    return run_conv(u, j, "head");
}

// The backward pass through every layer after unet_forward(train); gradients
// in each layer's g / gb.
lbms_status unet_backward(lbms_unet* u, const Levels& v) {
    const Geo &g0 = v.g[0], &g1 = v.g[1], &g2 = v.g[2];
    auto& L = u->L;
    bf16 **za = u->za, **zb = u->zb;
    UST(layer_wgrad(u, L[12], u->d1, za[0], g0));
    UST(dgrad_relu(u, L[12], za[0], g0, u->d1, L[11], zb[0]));
    // decoder, level 0
    UST(layer_wgrad(u, L[11], u->d1a, zb[0], g0));
    UST(dgrad_relu(u, L[11], zb[0], g0, u->d1a, L[10], za[0]));
    UST(layer_wgrad(u, L[10], u->c1, za[0], g0));
    UST(dgrad_split(u, L[10], za[0], g0, g1, L[9], u->G1, u->skip0));
    UST(layer_wgrad(u, L[9], u->d2, u->G1, g1));
    UST(dgrad_relu(u, L[9], u->G1, g1, u->d2, L[8], za[1]));
    // decoder, level 1
    UST(layer_wgrad(u, L[8], u->d2a, za[1], g1));
    UST(dgrad_relu(u, L[8], za[1], g1, u->d2a, L[7], zb[1]));
    UST(layer_wgrad(u, L[7], u->c2, zb[1], g1));
    UST(dgrad_split(u, L[7], zb[1], g1, g2, L[6], u->G2, u->skip1));
    UST(layer_wgrad(u, L[6], u->e3, u->G2, g2));
    UST(dgrad_relu(u, L[6], u->G2, g2, u->e3, L[5], za[2]));
    // bottom, level 2
    UST(layer_wgrad(u, L[5], u->e3a, za[2], g2));
    UST(dgrad_relu(u, L[5], za[2], g2, u->e3a, L[4], zb[2]));
    UST(layer_wgrad(u, L[4], u->p2, zb[2], g2));
    UST(dgrad_store(u, L[4], zb[2], g2, u->dp2));
    // encoder, level 1
    pool_relu_back_kernel<<<152 * 4, 256>>>(u->dp2, u->arg2, u->skip1, u->e2, g1, g2, 64, za[1], L[3].gb);
    UCK(cudaGetLastError(), "pool backward");
    UST(layer_wgrad(u, L[3], u->e2a, za[1], g1));
    UST(dgrad_relu(u, L[3], za[1], g1, u->e2a, L[2], zb[1]));
    UST(layer_wgrad(u, L[2], u->p1, zb[1], g1));
    UST(dgrad_store(u, L[2], zb[1], g1, u->dp1));
    // encoder, level 0
    pool_relu_back_kernel<<<152 * 4, 256>>>(u->dp1, u->arg1, u->skip0, u->e1, g0, g1, 32, za[0], L[1].gb);
    UCK(cudaGetLastError(), "pool backward");
    UST(layer_wgrad(u, L[1], u->e1a, za[0], g0));
    UST(dgrad_relu(u, L[1], za[0], g0, u->e1a, L[0], zb[0]));
    return layer_wgrad(u, L[0], u->x0, zb[0], g0);
}

// The BF16 copies of one layer's weights from its FP32 master copy.
lbms_status cast_layer(lbms_unet* u, const lbms_unet::Layer& l) {
    if (l.kind == 3)
        conv_cast_kernel<<<grid_for((int64_t)l.rows * l.K), 256>>>(l.W, l.co_s, l.ci_s, l.Wb, l.Wt);
    else
        cast_weights_kernel<<<grid_for((int64_t)l.rows * l.K), 256>>>(l.W, l.rows, l.K, l.Wb, l.Wt);
    UCK(cudaGetLastError(), "weight cast");
    return LBMS_OK;
}

// One Adam step (betas 0.9 / 0.999, eps 1e-8) on every layer.
lbms_status unet_adam(lbms_unet* u, double lr) {
    ++u->step;
    const float c1 = (float)(1.0 / (1.0 - std::pow(0.9, (double)u->step)));
    const float c2 = (float)(1.0 / (1.0 - std::pow(0.999, (double)u->step)));
    AdamList list = {};
    for (int i = 0; i < kULayers; ++i) {
        const auto& l = u->L[i];
        list.it[2 * i] = {l.W, l.m, l.v, l.g, (int64_t)l.rows * l.K, l.Wb, l.Wt, l.rows, l.K, l.kind == 3 ? l.ci_s : 0};
        list.it[2 * i + 1] = {l.b, l.mb, l.vb, l.gb, l.co_s, nullptr, nullptr, l.co_s, 1, 0};
    }
    adam_all_kernel<<<dim3(152, 2 * kULayers), 256>>>(list, (float)lr, c1, c2);
    UCK(cudaGetLastError(), "adam");
    return LBMS_OK;
}

lbms_status unet_check_gemm(lbms_unet* u) {
    unsigned int f = 0;
    UCK(cudaMemcpy(&f, u->gemm_err, sizeof(f), cudaMemcpyDeviceToHost), "GEMM flag");
    if (!f) return LBMS_OK;
    UCK(cudaMemset(u->gemm_err, 0, sizeof(f)), "GEMM flag");
    return ufail(u, LBMS_ECUDA, "tensor-core GEMM: an mbarrier wait timed out (flag %u)", f);
}

int64_t layer_weights(const lbms_unet::Layer& l) {
    return (int64_t)l.co * l.ci * (l.kind == 3 ? 27 : l.kind == 2 ? 8 : 1);
}

int64_t unet_params(const lbms_unet* u) {
    int64_t s = 0;
    for (const auto& l : u->L) s += layer_weights(l) + l.co;
    return s;
}

// Flat index in W of the real weight number e of a layer, in PyTorch's
// order: Conv3d [co][ci][kz][ky][kx], ConvTranspose3d [ci][co][kz][ky][kx].
__host__ __device__ size_t weight_slot(const lbms_unet::Layer& l, int64_t e) {
    if (l.kind == 3) {
        const int tap = (int)(e % 27), ci = (int)((e / 27) % l.ci), co = (int)(e / (27 * (int64_t)l.ci));
        return (size_t)co * l.K + (size_t)tap * l.ci_s + ci;
    }
    if (l.kind == 2) {
        const int t = (int)(e % 8), co = (int)((e / 8) % l.co), ci = (int)(e / (8 * (int64_t)l.co));
        return (size_t)(t * l.co_s + co) * l.K + ci;
    }
    const int ci = (int)(e % l.ci), co = (int)(e / l.ci);
    return (size_t)co * l.K + ci;
}

// The n real weights and then the biases of a layer between its storage
// (W, b) and a flat array in PyTorch's order: flat <- storage, or back.
__global__ void layer_flat_kernel(const __grid_constant__ lbms_unet::Layer l, float* __restrict__ W,
                                  float* __restrict__ b, int64_t n, float* __restrict__ flat, bool back) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n + l.co; e += (int64_t)gridDim.x * blockDim.x) {
        float* p = e < n ? W + weight_slot(l, e) : b + (e - n);
        if (back)
            *p = flat[e];
        else
            flat[e] = *p;
    }
}

// A case on the network's grid: interior extents rounded up to multiples
// of 4 (the added voxels solid), each fluid cell's row in the layout of one volume.
struct CaseVolume {
    Geo g;
    std::vector<int64_t> row;
};

void case_volume(const lbms::CaseView& v, CaseVolume& cv) {
    cv.g = make_geo(1, (v.nx + 3) / 4 * 4, (v.ny + 3) / 4 * 4, (v.nz + 3) / 4 * 4);
    cv.row.resize(v.nf);
    for (int j = 0; j < v.nf; ++j) {
        const int64_t e = v.fluid_cell[j];
        const int x = (int)(e % v.nx), y = (int)((e / v.nx) % v.ny), z = (int)(e / ((int64_t)v.nx * v.ny));
        cv.row[j] = (((int64_t)z + 1) * cv.g.Yp + y + 1) * cv.g.Xp + x + 1;
    }
}

}  // namespace

extern "C" {

void lbms_unet_destroy(lbms_unet* u) {
    if (!u) return;
    cudaDeviceSynchronize();
    for (void* p : u->allocs) cudaFree(p);
    for (void* p : u->bufs) cudaFree(p);
    cudaFree(u->feat.room);
    for (auto& s : u->samples) {
        cudaFree(s.in);
        cudaFree(s.tg);
    }
    delete u;
}

lbms_status lbms_unet_create(int width, int64_t max_voxels, uint64_t seed, lbms_unet** out) {
    if (!out) return LBMS_EINVAL;
    *out = nullptr;
    if (width < 4 || width > 32 || max_voxels < 64 || max_voxels > LBMS_UNET_MAX_VOXELS) return LBMS_EINVAL;
    lbms_unet* u = new (std::nothrow) lbms_unet;
    if (!u) return LBMS_ENOMEM;
    u->width = width;
    u->seed = seed;
    u->vcap = max_voxels;
    const int w = width;
    // kind, output level, real / stored input channels, real / stored output channels
    const int spec[kULayers][6] = {{3, 0, kUInReal, kUInC, w, 32}, {3, 0, w, 32, w, 32},
                                   {3, 1, w, 32, 2 * w, 64},       {3, 1, 2 * w, 64, 2 * w, 64},
                                   {3, 2, 2 * w, 64, 4 * w, 128},  {3, 2, 4 * w, 128, 4 * w, 128},
                                   {2, 1, 4 * w, 128, 2 * w, 64},  {3, 1, 4 * w, 128, 2 * w, 64},
                                   {3, 1, 2 * w, 64, 2 * w, 64},   {2, 0, 2 * w, 64, w, 32},
                                   {3, 0, 2 * w, 64, w, 32},       {3, 0, w, 32, w, 32},
                                   {1, 0, w, 32, 3, kUOutC}};
    for (int i = 0; i < kULayers; ++i) {
        auto& l = u->L[i];
        l.kind = spec[i][0];
        l.level = spec[i][1];
        l.ci = spec[i][2];
        l.ci_s = spec[i][3];
        l.co = spec[i][4];
        l.co_s = spec[i][5];
        l.rows = l.kind == 2 ? 8 * l.co_s : l.co_s;
        l.K = l.kind == 3 ? 27 * l.ci_s : l.ci_s;
        const size_t nw = (size_t)l.rows * l.K;
        l.W = ualloc<float>(u, nw);
        l.m = ualloc<float>(u, nw);
        l.v = ualloc<float>(u, nw);
        l.g = ualloc<float>(u, nw);
        l.b = ualloc<float>(u, l.co_s);
        l.mb = ualloc<float>(u, l.co_s);
        l.vb = ualloc<float>(u, l.co_s);
        l.Wb = ualloc<bf16>(u, nw);
        l.Wt = ualloc<bf16>(u, l.kind == 3 ? (size_t)l.ci_s * 27 * l.co_s : nw);
    }
    size_t biases = 0;
    for (const auto& l : u->L) biases += l.co_s;
    u->zero_bytes = kZeroHead * sizeof(float) + biases * sizeof(float);
    u->zero = ualloc<float>(u, kZeroHead + biases);
    u->loss = reinterpret_cast<double*>(u->zero);
    float* gb = u->zero ? u->zero + kZeroHead : nullptr;
    for (auto& l : u->L) {
        l.gb = gb;
        if (gb) gb += l.co_s;
    }
    u->flat = ualloc<float>(u, unet_params(u));
    u->gemm_err = ualloc<unsigned int>(u, 1);
    bool ok = true;
    for (void* p : u->allocs) ok = ok && p;
    if (!ok) {
        lbms_unet_destroy(u);
        return LBMS_ENOMEM;
    }
    ok = lbms::umma_init() == cudaSuccess;
    ok = ok && cudaMemset(u->gemm_err, 0, sizeof(unsigned int)) == cudaSuccess;
    // He-uniform weights on the real entries (fan-in 27 ci for the 3x3x3
    // convolutions, ci for the transposed ones), zero head, zero biases
    for (int i = 0; i < kULayers && ok; ++i) {
        auto& l = u->L[i];
        const size_t nw = (size_t)l.rows * l.K;
        std::vector<float> W(nw, 0.0f);
        if (l.kind != 1) {
            const int64_t taps = l.kind == 3 ? 27 : 8;
            const double a = std::sqrt(6.0 / (double)((l.kind == 3 ? 27 : 1) * l.ci));
            const int64_t n = (int64_t)l.co * l.ci * taps;
            for (int64_t e = 0; e < n; ++e)
                W[weight_slot(l, e)] =
                    (float)(a * (2.0 * unit_double(seed * 0x100000001ull + (uint64_t)(i + 1) * 0x1000000000ull + e) - 1.0));
        }
        ok = ok && cudaMemcpy(l.W, W.data(), nw * sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess;
        for (float* p : {l.m, l.v, l.g}) ok = ok && cudaMemset(p, 0, nw * sizeof(float)) == cudaSuccess;
        for (float* p : {l.b, l.mb, l.vb, l.gb}) ok = ok && cudaMemset(p, 0, l.co_s * sizeof(float)) == cudaSuccess;
        ok = ok && cast_layer(u, l) == LBMS_OK;
    }
    if (!ok || cudaDeviceSynchronize() != cudaSuccess) {
        lbms_unet_destroy(u);
        return LBMS_ECUDA;
    }
    *out = u;
    return LBMS_OK;
}

const char* lbms_unet_last_error(const lbms_unet* u) { return u ? u->msg.c_str() : ""; }

lbms_status lbms_unet_info(const lbms_unet* u, int64_t* n_params, int64_t* n_samples) {
    if (!u) return LBMS_EINVAL;
    if (n_params) *n_params = unet_params(u);
    if (n_samples) *n_samples = (int64_t)u->samples.size();
    return LBMS_OK;
}

lbms_status lbms_unet_gemm_calls(const lbms_unet* u, int64_t* tcgen05_calls) {
    if (!u) return LBMS_EINVAL;
    if (tcgen05_calls) *tcgen05_calls = u->tcgen05_calls;
    return LBMS_OK;
}

lbms_status lbms_unet_add_sample(lbms_unet* u, lbms_ctx* ctx, int k) {
    if (!u || !ctx) return LBMS_EINVAL;
    CaseFeatures F(&u->feat);
    lbms_status st = case_features(&u->feat, ctx, k, F);
    if (st != LBMS_OK) return ufail(u, st, "%s", u->feat.err.c_str());
    lbms::CaseView v;
    lbms::case_view(ctx, k, &v);
    CaseVolume cv;
    case_volume(v, cv);
    if (cv.g.V > u->vcap || !levels_fit(levels_of(1, cv.g.X, cv.g.Y, cv.g.Z)))
        return ufail(u, LBMS_EINVAL, "case %d needs %lld voxels, the network was made for %lld", k, (long long)cv.g.V,
                     (long long)u->vcap);
    std::vector<double> X((size_t)3 * v.N);
    st = lbms_batch_get_fields(ctx, k, X.data(), nullptr, nullptr);
    if (st != LBMS_OK) return ufail(u, st, "reading the fields of case %d: %s", k, lbms_last_error(ctx));
    const int64_t R = cv.g.R;
    std::vector<float> t((size_t)R * 4, 0.0f);
    for (int j = 0; j < v.nf; ++j) {
        const int64_t e = v.fluid_cell[j];
        const int x = (int)(e % v.nx);
        float* r = &t[(size_t)cv.row[j] * 4];
        for (int s = 0; s < 3; ++s) r[s] = (float)(kTargetScale * (X[(size_t)s * v.N + e] - F.prof[(size_t)s * v.nx + x]));
        r[3] = 1.0f;
    }
    lbms_unet::Sample s;
    s.X = cv.g.X;
    s.Y = cv.g.Y;
    s.Z = cv.g.Z;
    s.rows = R;
    s.nfluid = v.nf;
    int64_t* prow = F.row;
    if (lbms::dev_malloc(&s.in, (size_t)R * kUInC * sizeof(bf16)) != cudaSuccess) return ufail(u, LBMS_ENOMEM, "sample");
    if (lbms::dev_malloc(&s.tg, (size_t)R * 4 * sizeof(float)) != cudaSuccess) {
        cudaFree(s.in);
        return ufail(u, LBMS_ENOMEM, "sample");
    }
    cudaError_t e = cudaMemcpy(prow, cv.row.data(), v.nf * sizeof(int64_t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(s.in, 0, (size_t)R * kUInC * sizeof(bf16));
    if (e == cudaSuccess) {
        unet_inputs_kernel<<<grid_for((int64_t)v.nf * kUInC), 256>>>(F.rows, prow, v.nf, s.in);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(s.tg, t.data(), t.size() * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        cudaFree(s.in);
        cudaFree(s.tg);
        return ufail(u, LBMS_ECUDA, "sample: %s", cudaGetErrorString(e));
    }
    u->samples.push_back(s);   // owned from here on (freed by destroy)
    return LBMS_OK;
}

lbms_status lbms_unet_add_volume(lbms_unet* u, const float* x, const float* t, int X, int Y, int Z) {
    if (!u || !x || !t) return LBMS_EINVAL;
    if (X < 4 || Y < 4 || Z < 4 || X % 4 || Y % 4 || Z % 4)
        return ufail(u, LBMS_EINVAL, "volume extents must be multiples of 4");
    const Geo g = make_geo(1, X, Y, Z);
    if (g.V > u->vcap || !levels_fit(levels_of(1, X, Y, Z)))
        return ufail(u, LBMS_EINVAL, "the volume holds %lld voxels, the network was made for %lld", (long long)g.V,
                     (long long)u->vcap);
    double nf = 0.0;
    for (int64_t s = 0; s < g.V; ++s) nf += x[(int64_t)(kUInReal - 1) * g.V + s];
    lbms_unet::Sample s;
    s.X = X;
    s.Y = Y;
    s.Z = Z;
    s.rows = g.R;
    s.nfluid = (int64_t)std::llround(nf);
    float* dev = nullptr;
    const size_t nin = (size_t)g.V * kUInReal, ntg = (size_t)g.V * 3;
    if (lbms::dev_malloc(&dev, (nin + ntg) * sizeof(float)) != cudaSuccess) return ufail(u, LBMS_ENOMEM, "volume upload");
    cudaError_t e = lbms::dev_malloc(&s.in, (size_t)g.R * kUInC * sizeof(bf16));
    if (e == cudaSuccess) e = lbms::dev_malloc(&s.tg, (size_t)g.R * 4 * sizeof(float));
    if (e == cudaSuccess) e = cudaMemcpy(dev, x, nin * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(dev + nin, t, ntg * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(s.in, 0, (size_t)g.R * kUInC * sizeof(bf16));
    if (e == cudaSuccess) e = cudaMemset(s.tg, 0, (size_t)g.R * 4 * sizeof(float));
    if (e == cudaSuccess) {
        vol_in_kernel<<<warp_grid(g.V), 256>>>(dev, g, s.in, s.tg);
        vol_target_kernel<<<grid_for(g.V), 256>>>(dev + nin, g, s.tg);
        e = cudaDeviceSynchronize();
    }
    cudaFree(dev);
    if (e != cudaSuccess) {
        cudaFree(s.in);
        cudaFree(s.tg);
        return ufail(u, LBMS_ECUDA, "volume upload: %s", cudaGetErrorString(e));
    }
    u->samples.push_back(s);
    return LBMS_OK;
}

lbms_status lbms_unet_train(lbms_unet* u, int iters, int max_batch, double lr, double* last_loss) {
    if (!u) return LBMS_EINVAL;
    if (iters < 0 || max_batch < 1 || !(lr > 0.0))
        return ufail(u, LBMS_EINVAL, "need iters >= 0, max_batch >= 1, lr > 0");
    if (u->samples.empty()) return ufail(u, LBMS_ESTATE, "no training volumes (call lbms_unet_add_sample first)");
    // groups of equal volume extents, in order of first appearance, and the batch size of each
    std::vector<std::vector<int>> groups;
    for (int i = 0; i < (int)u->samples.size(); ++i) {
        const auto& s = u->samples[i];
        bool placed = false;
        for (auto& g : groups) {
            const auto& f = u->samples[g[0]];
            if (f.X == s.X && f.Y == s.Y && f.Z == s.Z) {
                g.push_back(i);
                placed = true;
                break;
            }
        }
        if (!placed) groups.push_back({i});
    }
    std::vector<int> Bg(groups.size());
    for (size_t gi = 0; gi < groups.size(); ++gi) {
        const auto& s0 = u->samples[groups[gi][0]];
        const int64_t Vs = (int64_t)s0.X * s0.Y * s0.Z;
        int B = (int)std::min<int64_t>({(int64_t)max_batch, (int64_t)groups[gi].size(), u->vcap / Vs});
        while (B > 1 && !levels_fit(levels_of(B, s0.X, s0.Y, s0.Z))) --B;
        Bg[gi] = B;
        UST(ensure_buffers(u, levels_of(B, s0.X, s0.Y, s0.Z)));
    }
    double tail = 0.0;
    int nt = 0;
    for (int it = 0; it < iters; ++it) {
        const size_t gi = it % groups.size();
        const auto& g = groups[gi];
        const auto& s0 = u->samples[g[0]];
        const int B = Bg[gi];
        const Levels lv = levels_of(B, s0.X, s0.Y, s0.Z);
        const uint64_t key = splitmix64(u->seed ^ 0x5A5A5A5Aull) + (uint64_t)u->step * 64ull;
        int64_t nfl = 0;
        for (int i = 0; i < B; ++i) {
            const auto& s = u->samples[g[splitmix64(key + (uint64_t)i) % g.size()]];
            UCK(cudaMemcpyAsync(u->x0 + i * s.rows * kUInC, s.in, s.rows * kUInC * sizeof(bf16),
                                cudaMemcpyDeviceToDevice, 0),
                "batch");
            UCK(cudaMemcpyAsync(u->T + i * s.rows * 4, s.tg, s.rows * 4 * sizeof(float), cudaMemcpyDeviceToDevice, 0),
                "batch");
            nfl += s.nfluid;
        }
        const Geo& g0 = lv.g[0];
        UCK(cudaMemsetAsync(u->x0 + g0.R * kUInC, 0, (g0.Rp - g0.R) * kUInC * sizeof(bf16), 0), "batch");
        UCK(cudaMemsetAsync(u->T + g0.R * 4, 0, (g0.Rp - g0.R) * 4 * sizeof(float), 0), "batch");
        const double cw = 0.5 * (1.0 + std::cos(3.14159265358979323846 * (double)it / std::max(1, iters)));
        const double lr_it = lr / 20.0 + (lr - lr / 20.0) * cw;
        UST(unet_forward(u, lv, true, (float)(1.0 / (3.0 * (double)std::max<int64_t>(nfl, 1)))));
        UST(unet_backward(u, lv));
        UST(unet_adam(u, lr_it));
        if (it >= iters - 10) {
            double l = 0.0;
            UCK(cudaMemcpy(&l, u->loss, sizeof(double), cudaMemcpyDeviceToHost), "read loss");
            tail += l;
            ++nt;
        }
    }
    UCK(cudaDeviceSynchronize(), "train");
    UST(unet_check_gemm(u));
    if (last_loss) *last_loss = nt ? tail / nt : 0.0;
    return LBMS_OK;
}

lbms_status lbms_unet_warm_start(lbms_unet* u, lbms_ctx* ctx, int k, double* Xout) {
    if (!u || !ctx) return LBMS_EINVAL;
    CaseFeatures F(&u->feat);
    lbms_status st = case_features(&u->feat, ctx, k, F);
    if (st != LBMS_OK) return ufail(u, st, "%s", u->feat.err.c_str());
    lbms::CaseView v;
    lbms::case_view(ctx, k, &v);
    const Levels lv = levels_of(1, (v.nx + 3) / 4 * 4, (v.ny + 3) / 4 * 4, (v.nz + 3) / 4 * 4);
    const Geo& g0 = lv.g[0];
    if (g0.V > u->vcap || !levels_fit(lv))
        return ufail(u, LBMS_EINVAL, "case %d needs %lld voxels, the network was made for %lld", k, (long long)g0.V,
                     (long long)u->vcap);
    UST(ensure_buffers(u, lv));
    cell_row_kernel<<<(v.nf + 255) / 256, 256>>>(F.cell, v.nf, v.nx, v.ny, g0, F.row);
    UCK(cudaGetLastError(), "cells");
    UCK(cudaMemsetAsync(u->x0, 0, (size_t)g0.Rp * kUInC * sizeof(bf16), 0), "inputs");
    unet_inputs_kernel<<<grid_for((int64_t)v.nf * kUInC), 256>>>(F.rows, F.row, v.nf, u->x0);
    UCK(cudaGetLastError(), "inputs");
    UST(unet_forward(u, lv, false, 0.0f));
    unet_post_kernel<<<(v.nf + 255) / 256, 256>>>(u->Y, F.row, v.nf, g0.Xp, F.xtab, F.pred);
    UCK(cudaGetLastError(), "prediction");
    UST(unet_check_gemm(u));
    st = take_prediction(&u->feat, ctx, k, F, Xout);
    return st == LBMS_OK ? st : ufail(u, st, "%s", u->feat.err.c_str());
}

}  // extern "C"

namespace {

// Uploads a host batch FP32 [B][17][Z][Y][X] (and targets [B][3][Z][Y][X])
// into x0 and T in the layout of `lv`; nfluid receives the mask's sum.
lbms_status upload_batch(lbms_unet* u, const float* x, const float* t, int B, int X, int Y, int Z, Levels* lv,
                         double* nfluid) {
    if (!x || B < 1 || X < 4 || Y < 4 || Z < 4 || X % 4 || Y % 4 || Z % 4)
        return ufail(u, LBMS_EINVAL, "need B >= 1 volumes with extents multiples of 4");
    *lv = levels_of(B, X, Y, Z);
    const Geo& g0 = lv->g[0];
    if (g0.V > u->vcap || !levels_fit(*lv))
        return ufail(u, LBMS_EINVAL, "the batch holds %lld voxels, the network was made for %lld", (long long)g0.V,
                     (long long)u->vcap);
    UST(ensure_buffers(u, *lv));
    const int64_t S = (int64_t)X * Y * Z, V = g0.V;
    double nf = 0.0;
    for (int b = 0; b < B; ++b)
        for (int64_t s = 0; s < S; ++s) nf += x[((int64_t)b * kUInReal + kUInReal - 1) * S + s];
    if (nfluid) *nfluid = nf;
    float* dev = nullptr;
    const size_t nin = (size_t)V * kUInReal, ntg = t ? (size_t)V * 3 : 0;
    UCK(lbms::dev_malloc(&dev, (nin + ntg) * sizeof(float)), "batch upload");
    lbms_status st = LBMS_OK;
    cudaError_t e = cudaMemcpy(dev, x, nin * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && t) e = cudaMemcpy(dev + nin, t, ntg * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(u->x0, 0, (size_t)g0.Rp * kUInC * sizeof(bf16));
    if (e == cudaSuccess) e = cudaMemset(u->T, 0, (size_t)g0.Rp * 4 * sizeof(float));
    if (e == cudaSuccess) {
        vol_in_kernel<<<warp_grid(V), 256>>>(dev, g0, u->x0, u->T);
        if (t) vol_target_kernel<<<grid_for(V), 256>>>(dev + nin, g0, u->T);
        e = cudaDeviceSynchronize();
    }
    if (e != cudaSuccess) st = ufail(u, LBMS_ECUDA, "batch upload: %s", cudaGetErrorString(e));
    cudaFree(dev);
    return st;
}

}  // namespace

extern "C" {

lbms_status lbms_unet_forward(lbms_unet* u, const float* x, int B, int X, int Y, int Z, float* y) {
    if (!u || !y) return LBMS_EINVAL;
    Levels lv;
    UST(upload_batch(u, x, nullptr, B, X, Y, Z, &lv, nullptr));
    UST(unet_forward(u, lv, false, 0.0f));
    const Geo& g0 = lv.g[0];
    std::vector<float> h((size_t)g0.R * 4);
    UCK(cudaMemcpy(h.data(), u->Y, h.size() * sizeof(float), cudaMemcpyDeviceToHost), "read output");
    UST(unet_check_gemm(u));
    const int64_t S = (int64_t)X * Y * Z;
    for (int b = 0; b < B; ++b)
        for (int z = 0; z < Z; ++z)
            for (int yy = 0; yy < Y; ++yy)
                for (int xx = 0; xx < X; ++xx) {
                    const int64_t r = (((int64_t)b * g0.Zp + z + 1) * g0.Yp + yy + 1) * g0.Xp + xx + 1;
                    const int64_t s = ((int64_t)z * Y + yy) * X + xx;
                    for (int c = 0; c < 3; ++c) y[((int64_t)b * 3 + c) * S + s] = h[(size_t)r * 4 + c];
                }
    return LBMS_OK;
}

lbms_status lbms_unet_train_batch(lbms_unet* u, const float* x, const float* t, int B, int X, int Y, int Z, double lr,
                                  double* loss) {
    if (!u || !t || !(lr >= 0.0)) return LBMS_EINVAL;
    double nf = 0.0;
    Levels lv;
    UST(upload_batch(u, x, t, B, X, Y, Z, &lv, &nf));
    UST(unet_forward(u, lv, true, (float)(1.0 / (3.0 * std::max(nf, 1.0)))));
    UST(unet_backward(u, lv));
    if (lr > 0.0) UST(unet_adam(u, lr));
    if (loss) UCK(cudaMemcpy(loss, u->loss, sizeof(double), cudaMemcpyDeviceToHost), "read loss");
    UCK(cudaDeviceSynchronize(), "train batch");
    return unet_check_gemm(u);
}

lbms_status lbms_unet_get(const lbms_unet* cu, int what, float* buf, int64_t count) {
    lbms_unet* u = const_cast<lbms_unet*>(cu);
    if (!u || !buf || (what != 0 && what != 1)) return LBMS_EINVAL;
    if (count < unet_params(u))
        return ufail(u, LBMS_EINVAL, "buffer holds %lld floats, need %lld", (long long)count, (long long)unet_params(u));
    const std::lock_guard<std::mutex> hold(u->flat_use);
    int64_t off = 0;
    for (const auto& l : u->L) {
        const int64_t n = layer_weights(l);
        layer_flat_kernel<<<grid_for(n + l.co), 256>>>(l, what ? l.g : l.W, what ? l.gb : l.b, n, u->flat + off, false);
        off += n + l.co;
    }
    UCK(cudaGetLastError(), "get");
    UCK(cudaMemcpy(buf, u->flat, (size_t)off * sizeof(float), cudaMemcpyDeviceToHost), "get");
    return LBMS_OK;
}

lbms_status lbms_unet_set(lbms_unet* u, const float* buf, int64_t count) {
    if (!u || !buf) return LBMS_EINVAL;
    if (count < unet_params(u))
        return ufail(u, LBMS_EINVAL, "buffer holds %lld floats, need %lld", (long long)count, (long long)unet_params(u));
    const std::lock_guard<std::mutex> hold(u->flat_use);
    UCK(cudaMemcpy(u->flat, buf, (size_t)unet_params(u) * sizeof(float), cudaMemcpyHostToDevice), "set");
    int64_t off = 0;
    for (const auto& l : u->L) {
        const int64_t n = layer_weights(l);
        UCK(cudaMemsetAsync(l.W, 0, (size_t)l.rows * l.K * sizeof(float), 0), "set");
        UCK(cudaMemsetAsync(l.b, 0, l.co_s * sizeof(float), 0), "set");
        layer_flat_kernel<<<grid_for(n + l.co), 256>>>(l, l.W, l.b, n, u->flat + off, true);
        UCK(cudaGetLastError(), "set");
        off += n + l.co;
        UST(cast_layer(u, l));
    }
    UCK(cudaDeviceSynchronize(), "set");
    return LBMS_OK;
}

}  // extern "C"
