// The products of the two networks on the tcgen05 tensor cores: convolutions
// (the 3-D U-Net), plain products (the pointwise network), input gradients and
// weight gradients, with what follows each product done on its accumulators.
//
// Activations are stored in a layout with a zero halo of one voxel between
// rows, planes and volumes, so the neighbour of every interior voxel at tap t = (dz, dy, dx) lies a
// fixed number of rows off(t) away and a convolution is an implicit GEMM: the
// A tile of tap t is the activation matrix [rows][C] read at shifted rows
// (TMA zero-fills rows outside it).  The three taps of a (dz, dy) row differ
// in dx only, so one window of 130 rows serves all three: the swizzle is a
// function of the shared-memory address, and an MMA may start any whole
// number of rows into the window.
//
// What bounds these products: an operand A of 128 rows is 4 KB of shared
// memory per MMA whatever N is, so at N = 32 (the full resolution) an MMA
// takes about 50 cycles where its arithmetic takes 8; storing 32 channels
// instead of 64 there quartered the MMAs.  The kernels of a training step on 4
// volumes of 96^3 take 6.5 ms, on 8 of 64x32x32 1.5 ms (calls that read the
// gradients 6.95 and 1.92; 48.5 and 13.2 with 64 channels stored, FP32 products
// in memory, transposed copies for the weight gradients and row-wise kernels
// between the products).  Of the 6.5 ms the 32-channel convolutions take 0.28 ms
// each (52 cycles an MMA, shared memory at 74 %) and the one that copies into a
// concatenation 0.5 (its stores), their input gradients 0.28, their weight
// gradients 0.22.  Reading the timer on every barrier wait and issuing from a
// single lane's branch cost twice that.
#include <cuda_bf16.h>

#include <algorithm>

#include "lbms_internal.h"
#include "lbms_umma.cuh"

namespace lbms {
namespace {

using bf16 = __nv_bfloat16;

constexpr int kSmemMax = 227 * 1024;
constexpr int kConvThreads = 64 + 2 * 128;
constexpr int align1k(int b) { return (b + 1023) / 1024 * 1024; }

// Interior coordinates of row r; false for halo and padding rows.
__device__ __forceinline__ bool voxel_of(const RowLayout& g, long long r, int& x, int& y, int& z, int& b) {
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
__device__ __forceinline__ long long row_of(const RowLayout& g, int b, int x, int y, int z) {
    return (((long long)b * g.Zp + z + 1) * g.Yp + y + 1) * g.Xp + x + 1;
}

__device__ __forceinline__ uint32_t pack2(float a, float b) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&p);
}

// Sum of v[c] over the warp's lanes, for column c = lane.
__device__ __forceinline__ float column_sum(float (&v)[32], int lane) {
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < o; ++i) {
            const float keep = up ? v[i + o] : v[i];
            const float send = up ? v[i] : v[i + o];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    return v[0];
}

// After a wait that ran out, once no warp of the CTA issues any more: the
// copies into the last stages land (or are waited for as long as any) before
// the CTA gives its shared memory back.  `issued` stages of the ring of ST in
// all; `once`: a barrier of copies issued once, or null.
__device__ __noinline__ void drain_copies(uint64_t* full, int ST, int issued, uint64_t* once) {
    for (int i = max(0, issued - ST); i < issued; ++i) mbar_wait(&full[i % ST], (uint32_t)(i / ST) & 1u);
    if (once) mbar_wait(once, 0);
}

// ---------------------------------------------------------------------------
// Convolution and plain product.  RB: bytes of an operand row in shared
// memory (64: 32 channels, 128: 64 channels; nblk such blocks make up C).
// N: output columns of a tile.  NT: taps per window (3, or 1 for a plain
// product).
//
// A persistent CTA per SM takes 128-row tiles in turn: warp 0 issues the TMA
// loads of a ring of stages, warp 1 the MMAs into one of two TMEM
// accumulators, warps 2-5 the epilogues of the tiles in the first, warps 6-9 of
// those in the second; what an epilogue reads from memory it loads before the
// wait for its accumulator.  Plain products are bound by their epilogues: the
// head of 4 volumes of 96^3 takes 0.144 ms and its input gradient 0.156, with
// one set of epilogue warps 0.197 and 0.235.  The weights stay in
// shared memory for the whole launch where they fit (27 N RB <= 108 KB, the
// layers at full resolution), else each stage brings its three taps'.
template <int RB, int N, int NT, int KIND>
struct ConvShape {
    static constexpr int kGroups = NT == 3 ? 9 : 1;
    static constexpr bool kResident = NT == 3 && RB * N <= 4096;
    static constexpr int kARows = NT == 3 ? 130 : 128;
    static constexpr int kABytes = align1k(kARows * RB);
    static constexpr int kBTile = N * RB;
    static constexpr int kGps = NT == 3 && RB == 64 && KIND != kOutSplit ? 3 : 1;   // windows (dz, dy rows) of a stage
    static constexpr int kStage = kGps * kABytes + (kResident ? 0 : NT * kBTile);
    static_assert(kGps == 1 || kResident, "a stage holds the weights of one window");
    static constexpr int kResBytes = kResident ? align1k(27 * kBTile) : 0;
    static constexpr int kStageFloats = KIND == kOutSplit ? 8 * 32 * 65 : 0;   // split: rows of each epilogue warp
    static constexpr int kFixed = 1024 + kResBytes + kStageFloats * 4 + N * 4 + 512;
    static constexpr int kFit = (kSmemMax - kFixed) / kStage;
    static constexpr int kStages = kFit < 8 ? kFit : 8;
    static constexpr int kSmem = kFixed + kStages * kStage;
    static constexpr int kCols = 2 * N < 32 ? 32 : 2 * N;
    static_assert(kStages >= 2, "shared memory");
};

template <int RB, int N, int NT, int KIND>
__global__ void __launch_bounds__(kConvThreads, 1) conv_kernel(const __grid_constant__ CUtensorMap mapA,
                                                      const __grid_constant__ CUtensorMap mapB, int rows, int nblk,
                                                      int ntn, unsigned int* __restrict__ err,
                                                      const __grid_constant__ ConvJob job) {
    using Sh = ConvShape<RB, N, NT, KIND>;
    constexpr int ST = Sh::kStages;
    constexpr int KS = RB / 32;
    constexpr int GPS = Sh::kGps;
    constexpr uint32_t idesc = umma_idesc(128, N, false);
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* resB = base;
    uint8_t* stages = base + Sh::kResBytes;
    float* split = reinterpret_cast<float*>(stages + ST * Sh::kStage);
    float* cs = split + Sh::kStageFloats;
    uint64_t* full = reinterpret_cast<uint64_t*>(cs + N);
    uint64_t* empty = full + ST;
    uint64_t* acc_full = empty + ST;
    uint64_t* acc_empty = acc_full + 2;
    uint64_t* res_full = acc_empty + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(res_full + 1);
    volatile uint32_t* failed = tmem_slot + 1;
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int tiles = (rows + 127) / 128 * ntn;
    const int per_tile = Sh::kGroups / GPS * nblk;   // stages of a tile: (dz, dy) rows x channel blocks

    if (threadIdx.x == 0) {
        for (int s = 0; s < ST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 4);
        }
        mbar_init(res_full, 1);
        *failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int c = threadIdx.x; c < N; c += kConvThreads) cs[c] = 0.0f;
    if (warp == 0) tmem_alloc(tmem_slot, Sh::kCols);
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;

    // A window starts at the lowest of its three offsets; tap d lies d rows
    // into it, or 2 - d where the offsets run backwards (input gradients).
    // Both issuing warps run their loops with all lanes and elect one for the
    // instruction itself, so that descriptors and addresses stay in uniform
    // registers: issued from a single lane's branch an MMA took 150 cycles.
    const bool back = NT == 3 && job.off[2] < job.off[0];
    int it = 0;      // stages whose loads are issued (warp 0)
    if (warp == 0) {
        const bool leader = elect_one();
        if (Sh::kResident && leader) {
            mbar_expect_tx(res_full, 27 * Sh::kBTile);
            for (int t = 0; t < 27; ++t) tma_load_2d(resB + t * Sh::kBTile, &mapB, t * (RB / 2), 0, res_full);
        }
        int s = 0;
        uint32_t ph = 1u;
        bool ok = true;
        for (int tile = blockIdx.x; ok && tile < tiles; tile += gridDim.x) {
            const int m0 = tile / ntn * 128, n0 = tile % ntn * N;
            for (int g = 0; ok && g < Sh::kGroups; g += GPS) {
                for (int c = 0; c < nblk; ++c) {
                    if (!mbar_wait(&empty[s], ph)) {   // the first pass through the ring finds it free
                        ok = false;
                        break;
                    }
                    if (leader) {
                        uint8_t* sa = stages + s * Sh::kStage;
                        mbar_expect_tx(&full[s], GPS * Sh::kARows * RB + (Sh::kResident ? 0 : NT * Sh::kBTile));
#pragma unroll
                        for (int i = 0; i < GPS; ++i)
                            tma_load_2d(sa + i * Sh::kABytes, &mapA, c * (RB / 2),
                                        NT == 1 ? m0 : m0 + job.off[3 * (g + i) + (back ? 2 : 0)], &full[s]);
                        if (!Sh::kResident)
                            for (int d = 0; d < NT; ++d)
                                tma_load_2d(sa + Sh::kABytes + d * Sh::kBTile, &mapB,
                                            ((NT * g + d) * nblk + c) * (RB / 2), n0, &full[s]);
                    }
                    ++it;
                    if (++s == ST) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
            }
        }
        if (!ok && lane == 0) {
            *failed = 1;
            atomicOr(err, 1u);
        }
    } else if (warp == 1) {
        const bool leader = elect_one();
        bool ok = !Sh::kResident || mbar_wait(res_full, 0);
        int nt = 0, s = 0;
        uint32_t ph = 0u;
        const uint64_t a0 = kmajor_desc(smem_u32(stages), RB);
        const uint64_t b0 = kmajor_desc(Sh::kResident ? smem_u32(resB) : smem_u32(stages) + Sh::kABytes, RB);
        for (int tile = blockIdx.x; ok && tile < tiles; tile += gridDim.x, ++nt) {
            const int b = nt & 1;
            if (nt >= 2 && !mbar_wait(&acc_empty[b], ((uint32_t)(nt >> 1) & 1u) ^ 1u)) {
                ok = false;
                break;
            }
            fence_after();
            const uint32_t d0 = tmem + b * N;
            for (int q = 0; q < per_tile; ++q) {
                if (!mbar_wait(&full[s], ph)) {
                    ok = false;
                    break;
                }
                fence_after();
                const uint64_t as = a0 + (uint32_t)((s * Sh::kStage) >> 4);
                const uint64_t bs = b0 + (uint32_t)((Sh::kResident ? q * GPS * 3 * Sh::kBTile : s * Sh::kStage) >> 4);
                if (leader) {
#pragma unroll
                    for (int i = 0; i < GPS; ++i)
#pragma unroll
                        for (int d = 0; d < NT; ++d) {
                            const uint64_t ad =
                                as + (uint32_t)((i * Sh::kABytes + (back ? 2 - d : d) * RB * (NT == 3)) >> 4);
#pragma unroll
                            for (int j = 0; j < KS; ++j)
                                umma_f16(d0, ad + 2 * j, bs + (((i * NT + d) * Sh::kBTile) >> 4) + 2 * j, idesc,
                                         (q | i | d | j) != 0);
                        }
                    umma_commit(&empty[s]);
                }
                __syncwarp();
                if (++s == ST) {
                    s = 0;
                    ph ^= 1u;
                }
            }
            if (!ok) break;
            if (leader) umma_commit(&acc_full[b]);
            __syncwarp();
        }
        if (!ok && lane == 0) {
            *failed = 1;
            atomicOr(err, 2u);
        }
    } else if (warp >= 2) {
        const ConvEpilogue& ep = job.ep;
        const int quarter = warp & 3;               // TMEM lanes this warp may read
        const int b = (warp - 2) >> 2;              // its accumulator
        int nt = b;
        double loss = 0.0;
        float hs[3] = {0.0f, 0.0f, 0.0f};
        for (int tile = blockIdx.x + b * gridDim.x; tile < tiles; tile += 2 * gridDim.x, nt += 2) {
            const int m0 = tile / ntn * 128, n0 = tile % ntn * N;
            const long long row = m0 + 32 * quarter + lane;
            const bool valid = row < rows;
            int x = 0, y = 0, z = 0, vb = 0;
            const bool in = KIND == kOutRelu && NT == 1 ? valid   // a plain layer: every row
                            : KIND != kOutReluBack && KIND != kOutStore && KIND != kOutHead &&
                                  voxel_of(ep.g, row, x, y, z, vb);
            uint4 acts[KIND == kOutReluBack ? N / 8 : 1];
            float4 target = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if constexpr (KIND == kOutReluBack) {
                const uint4* act = reinterpret_cast<const uint4*>(static_cast<const bf16*>(ep.act) + row * job.N + n0);
#pragma unroll
                for (int q = 0; q < N / 8; ++q) acts[q] = valid ? __ldg(act + q) : make_uint4(0u, 0u, 0u, 0u);
            }
            if (KIND == kOutHead && ep.T && valid) target = __ldg(reinterpret_cast<const float4*>(ep.T) + row);
            if (!mbar_wait(&acc_full[b], (uint32_t)(nt >> 1) & 1u)) {
                if (lane == 0) atomicOr(err, 4u);
                break;
            }
            fence_after();
            const uint32_t taddr = tmem + b * N + ((uint32_t)(32 * quarter) << 16);
            constexpr int kChunks = KIND == kOutHead ? 1 : N / 32;
#pragma unroll
            for (int ch = 0; ch < kChunks; ++ch) {
                uint32_t u[32];
                tmem_ld32(taddr + 32 * ch, u);
                tmem_wait_ld();
                if (ch == kChunks - 1) {   // the accumulator is free for the tile after next
                    fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&acc_empty[b]);
                }
                const int c0 = 32 * ch;
                if constexpr (KIND == kOutRelu) {
                    uint32_t wv[16];
#pragma unroll
                    for (int c = 0; c < 32; c += 2) {
                        const float a0 = in ? fmaxf(__uint_as_float(u[c]) + __ldg(ep.bias + n0 + c0 + c), 0.0f) : 0.0f;
                        const float a1 = in ? fmaxf(__uint_as_float(u[c + 1]) + __ldg(ep.bias + n0 + c0 + c + 1), 0.0f) : 0.0f;
                        wv[c / 2] = pack2(a0, a1);
                    }
                    if (valid) {
                        uint4* dst = reinterpret_cast<uint4*>(static_cast<bf16*>(ep.out) + row * job.N + n0 + c0);
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            dst[q] = make_uint4(wv[4 * q], wv[4 * q + 1], wv[4 * q + 2], wv[4 * q + 3]);
                        if (ep.cat) {
                            bf16* cat = static_cast<bf16*>(ep.cat) + row * ep.cat_ld;
                            if (!in) {
                                if (ch == 0)
                                    for (int q = 0; q < ep.cat_ld / 8; ++q)
                                        reinterpret_cast<uint4*>(cat)[q] = make_uint4(0u, 0u, 0u, 0u);
                            } else if (((ep.w | ep.cat_off | ep.cat_ld) & 1) == 0) {
                                uint32_t* dc = reinterpret_cast<uint32_t*>(cat + ep.cat_off + c0);
#pragma unroll
                                for (int c = 0; c < 32; c += 2)
                                    if (c0 + c < ep.w) dc[c / 2] = wv[c / 2];
                            } else {
                                uint16_t* dc = reinterpret_cast<uint16_t*>(cat + ep.cat_off + c0);
#pragma unroll
                                for (int c = 0; c < 32; ++c)
                                    if (c0 + c < ep.w) dc[c] = (uint16_t)(wv[c / 2] >> (16 * (c & 1)));
                            }
                        }
                    }
                } else if constexpr (KIND == kOutReluBack) {
                    float v[32];
                    uint4* dst = reinterpret_cast<uint4*>(static_cast<bf16*>(ep.out) + row * job.N + n0 + c0);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const uint4 av = acts[4 * ch + q];
                        const uint32_t aw[4] = {av.x, av.y, av.z, av.w};
                        uint32_t o[4];
#pragma unroll
                        for (int h = 0; h < 4; ++h) {
                            const int c = 8 * q + 2 * h;
                            // activations are relu outputs: positive unless both halves' bits are 0 (or -0)
                            v[c] = (aw[h] & 0x7FFFu) ? __uint_as_float(u[c]) : 0.0f;
                            v[c + 1] = (aw[h] & 0x7FFF0000u) ? __uint_as_float(u[c + 1]) : 0.0f;
                            o[h] = pack2(v[c], v[c + 1]);
                        }
                        if (valid) dst[q] = make_uint4(o[0], o[1], o[2], o[3]);
                    }
                    const float sum = column_sum(v, lane);
                    atomicAdd(ntn == 1 ? &cs[c0 + lane] : &ep.gb[n0 + c0 + lane], sum);
                } else if constexpr (KIND == kOutStore) {
                    if (valid) {
                        float4* dst = reinterpret_cast<float4*>(ep.P + row * N + c0);
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            dst[q] = make_float4(__uint_as_float(u[4 * q]), __uint_as_float(u[4 * q + 1]),
                                                 __uint_as_float(u[4 * q + 2]), __uint_as_float(u[4 * q + 3]));
                    }
                } else if constexpr (KIND == kOutSplit) {
                    // through shared memory (rows 65 words apart), 64 columns at a time, so that a
                    // warp writes one row's columns at a time
                    float* sw = split + (warp - 2) * 32 * 65;
#pragma unroll
                    for (int c = 0; c < 32; ++c) sw[lane * 65 + (ch & 1) * 32 + c] = __uint_as_float(u[c]);
                    if (ch & 1) {
                        __syncwarp();
                        const int par =
                            in ? (int)row_of(ep.other, vb, x >> 1, y >> 1, z >> 1) * 8 + (z & 1) * 4 + (y & 1) * 2 + (x & 1)
                               : -1;
                        const int cl = 64 * (ch >> 1) + lane;    // this lane's columns: cl and cl + 32
                        float sum[2] = {0.0f, 0.0f};
                        bf16* Gc = static_cast<bf16*>(ep.G) + cl;
                        float* Pc = ep.P + (long long)(m0 + 32 * quarter) * ep.Cg + cl - ep.w;
                        const int left = rows - (m0 + 32 * quarter);
                        const bool up0 = cl < ep.w, up1 = cl + 32 < ep.w;
                        const bool sk0 = !up0 && cl < 2 * ep.w, sk1 = !up1 && cl + 32 < 2 * ep.w;
#pragma unroll 8
                        for (int r = 0; r < 32; ++r) {
                            const int p = __shfl_sync(0xffffffffu, par, r);
                            const float v0 = p >= 0 ? sw[r * 65 + lane] : 0.0f;
                            const float v1 = p >= 0 ? sw[r * 65 + 32 + lane] : 0.0f;
                            sum[0] += v0;
                            sum[1] += v1;
                            if (up0 && p >= 0) Gc[(long long)p * ep.Cg] = __float2bfloat16_rn(v0);
                            if (up1 && p >= 0) Gc[(long long)p * ep.Cg + 32] = __float2bfloat16_rn(v1);
                            if (sk0 && r < left) Pc[(long long)r * ep.Cg] = v0;
                            if (sk1 && r < left) Pc[(long long)r * ep.Cg + 32] = v1;
                        }
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int c = 64 * (ch >> 1) + 32 * h + lane;
                            if (c < ep.w) atomicAdd(&cs[c], sum[h]);
                        }
                        __syncwarp();
                    }
                } else if constexpr (KIND == kOutUp) {
                    if (in) {
                        const int t = (n0 + c0) / ep.Cg, cb = (n0 + c0) % ep.Cg;
                        const long long child =
                            row_of(ep.other, vb, 2 * x + (t & 1), 2 * y + ((t >> 1) & 1), 2 * z + (t >> 2));
                        bf16* dst = static_cast<bf16*>(ep.cat) + child * ep.cat_ld + cb;
                        if (((ep.w | ep.cat_ld) & 3) == 0) {
#pragma unroll
                            for (int c = 0; c < 32; c += 4)
                                if (cb + c < ep.w)
                                    *reinterpret_cast<uint2*>(dst + c) =
                                        make_uint2(pack2(__uint_as_float(u[c]) + __ldg(ep.bias + cb + c),
                                                         __uint_as_float(u[c + 1]) + __ldg(ep.bias + cb + c + 1)),
                                                   pack2(__uint_as_float(u[c + 2]) + __ldg(ep.bias + cb + c + 2),
                                                         __uint_as_float(u[c + 3]) + __ldg(ep.bias + cb + c + 3)));
                        } else {
#pragma unroll
                            for (int c = 0; c < 32; ++c)
                                if (cb + c < ep.w)
                                    dst[c] = __float2bfloat16_rn(__uint_as_float(u[c]) + __ldg(ep.bias + cb + c));
                        }
                    }
                } else {   // kOutHead
                    if (valid) {
                        float yv[3], gv[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
                        for (int c = 0; c < 3; ++c) yv[c] = __uint_as_float(u[c]) + __ldg(ep.bias + c);
                        if (ep.Y) {
#pragma unroll
                            for (int c = 0; c < 3; ++c) ep.Y[row * 4 + c] = yv[c];
                        }
                        if (ep.T) {
                            const float tv[3] = {target.x, target.y, target.z};
#pragma unroll
                            for (int c = 0; c < 3; ++c) {
                                const float d = (yv[c] - tv[c]) * target.w;
                                loss += (double)d * d;
                                gv[c] = ep.grad_scale * d;
                                hs[c] += gv[c];
                            }
                            uint4* dst = reinterpret_cast<uint4*>(static_cast<bf16*>(ep.out) + row * N);
                            dst[0] = make_uint4(pack2(gv[0], gv[1]), pack2(gv[2], 0.0f), 0u, 0u);
#pragma unroll
                            for (int q = 1; q < N / 8; ++q) dst[q] = make_uint4(0u, 0u, 0u, 0u);
                        }
                    }
                }
            }
        }
        if constexpr (KIND == kOutReluBack || KIND == kOutSplit) {
            asm volatile("bar.sync 1, 256;" ::: "memory");   // the epilogue warps
            const int e = (int)threadIdx.x - 64;
            if (e < N && (KIND == kOutReluBack ? ntn == 1 : e < ep.w)) atomicAdd(&ep.gb[e], cs[e]);
        }
        if constexpr (KIND == kOutHead) {
            if (ep.T) {
                double sum[4] = {loss * ep.loss_scale, hs[0], hs[1], hs[2]};
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                    for (int c = 0; c < 4; ++c) sum[c] += __shfl_down_sync(0xffffffffu, sum[c], o);
                if (lane == 0) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) atomicAdd(&ep.loss[c], sum[c]);
                    __threadfence();
                    if (atomicAdd(ep.done, 1u) + 1u == 8u * gridDim.x) {   // the last epilogue warp
                        __threadfence();
#pragma unroll
                        for (int c = 0; c < 3; ++c) ep.gb[c] = (float)__ldcg(&ep.loss[1 + c]);
                    }
                }
            }
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 0) {
        if (*failed) drain_copies(full, ST, it, Sh::kResident ? res_full : nullptr);
        tmem_dealloc(tmem, Sh::kCols);
    }
}

// ---------------------------------------------------------------------------
// Weight gradient.  Both operands are read as they lie in memory, rows of
// channels, i.e. MN-major with K running over the rows: no transposed copies.
// RBA, NBA: row bytes and number of the A blocks of a window (32 channels: 64,
// 1; 64: 128, 1; 128: 128, 2); RBB, NBB the same of dz.  An MMA's 128 rows are
// the channels of 2 or 1 consecutive dx taps: the next block of M starts one
// row further into the same window (the leading offset of the descriptor), and
// the block past the third tap is not stored.
//
// A CTA reduces one chunk of rows for one of the nine (dz, dy) rows of taps
// (plain product: one of its 128-channel tiles) in the order of the rows.
constexpr int kWL = 64;                  // rows per stage
constexpr int kWRows = kWL + 3;          // window rows (taps up to 3 rows on)

template <int RBA, int NBA, int RBB, int NBB, int NT>
struct WgradShape {
    static constexpr int kTpm = NT == 1 ? 1 : (NBA == 2 ? 1 : 2);   // taps per MMA
    static constexpr int kMpg = NT == 1 ? 1 : (3 + kTpm - 1) / kTpm;    // MMAs per K slice
    static constexpr int kN = RBB / 2 * NBB;
    static constexpr int kABlock = align1k(kWRows * RBA);
    static constexpr int kBBlock = kWL * RBB;
    static constexpr uint32_t kCols = kMpg * kN <= 32 ? 32 : (kMpg * kN <= 128 ? 128 : (kMpg * kN <= 256 ? 256 : 512));
    static constexpr int kStage = NBA * kABlock + NBB * kBBlock;
    static constexpr int kStages = std::min(8, (kSmemMax - 2048) / kStage);
};

template <int RBA, int NBA, int RBB, int NBB, int NT>
__global__ void __launch_bounds__(192, 1) wgrad_kernel(const __grid_constant__ CUtensorMap mapA,
                                                       const __grid_constant__ CUtensorMap mapB, int chunk, int ST,
                                                       unsigned int* __restrict__ err,
                                                       const __grid_constant__ WgradJob job) {
    using Sh = WgradShape<RBA, NBA, RBB, NBB, NT>;
    constexpr uint32_t idesc = umma_idesc(128, Sh::kN, true);
    constexpr int CA = RBA / 2 * NBA;        // channels of a window
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    constexpr int stage = Sh::kStage;
    uint64_t* full = reinterpret_cast<uint64_t*>(base + ST * stage);
    uint64_t* empty = full + ST;
    uint64_t* done = empty + ST;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    volatile uint32_t* failed = tmem_slot + 1;
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int g = blockIdx.x;
    const int n0 = blockIdx.z * Sh::kN;
    const int r0 = blockIdx.y * chunk;
    const int nk = chunk / kWL;

    if (threadIdx.x == 0) {
        for (int s = 0; s < ST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        *failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(tmem_slot, Sh::kCols);
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;

    int it = 0;      // stages whose loads are issued (warp 0)
    if (warp == 0) {
        const bool leader = elect_one();
        int s = 0;
        uint32_t ph = 1u;
        bool ok = true;
        for (; it < nk; ++it) {
            if (!mbar_wait(&empty[s], ph)) {
                ok = false;
                break;
            }
            if (leader) {
                uint8_t* sa = base + s * stage;
                const int r = r0 + it * kWL;
                mbar_expect_tx(&full[s], NBA * kWRows * RBA + NBB * Sh::kBBlock);
                for (int c = 0; c < NBA; ++c)
                    tma_load_2d(sa + c * Sh::kABlock, &mapA, (NT == 1 ? g * CA : 0) + c * (RBA / 2),
                                NT == 1 ? r : r + job.off[3 * g], &full[s]);
                for (int c = 0; c < NBB; ++c)
                    tma_load_2d(sa + NBA * Sh::kABlock + c * Sh::kBBlock, &mapB, n0 + c * (RBB / 2), r, &full[s]);
            }
            if (++s == ST) {
                s = 0;
                ph ^= 1u;
            }
        }
        if (!ok && lane == 0) {
            *failed = 1;
            atomicOr(err, 8u);
        }
    } else if (warp == 1) {
        const bool leader = elect_one();
        int s = 0;
        uint32_t ph = 0u;
        const uint64_t a0 = mnmajor_desc(smem_u32(base), NBA == 2 ? Sh::kABlock : RBA, RBA);
        const uint64_t b0 = mnmajor_desc(smem_u32(base) + NBA * Sh::kABlock, Sh::kBBlock, RBB);
        for (int it = 0; it < nk; ++it) {
            if (!mbar_wait(&full[s], ph)) {
                if (lane == 0) {
                    *failed = 1;
                    atomicOr(err, 16u);
                }
                break;
            }
            fence_after();
            const uint64_t as = a0 + (uint32_t)((s * stage) >> 4);
            const uint64_t bs = b0 + (uint32_t)((s * stage) >> 4);
            if (leader) {
#pragma unroll
                for (int m = 0; m < Sh::kMpg; ++m)
#pragma unroll
                    for (int j = 0; j < kWL / 16; ++j)
                        umma_f16(tmem + m * Sh::kN, as + (m * Sh::kTpm + 16 * j) * (RBA / 16), bs + 16 * j * (RBB / 16),
                                 idesc, (it | j) != 0);
                umma_commit(&empty[s]);
            }
            __syncwarp();
            if (++s == ST) {
                s = 0;
                ph ^= 1u;
            }
        }
        if (leader) umma_commit(done);
        __syncwarp();
    } else if (warp >= 2) {
        if (!mbar_wait(done, 0)) {
            if (lane == 0) atomicOr(err, 32u);
        } else {
            fence_after();
            const int quarter = warp & 3;
            const int l = 32 * quarter + lane;
            const int tb = l / CA, c = l % CA;       // tap within the MMA, channel
            const int K = NT == 1 ? job.C : 27 * job.C;
            for (int m = 0; m < Sh::kMpg; ++m) {
                const int d = m * Sh::kTpm + tb;
                const bool keep = NT == 1 ? g * CA + l < job.C && tb == 0 : d < 3;
                const long long prow = NT == 1 ? (long long)g * CA + c : (long long)(3 * g + d) * job.C + c;
                float4* dst = reinterpret_cast<float4*>(job.P + ((long long)blockIdx.y * K + prow) * job.N + n0);
                const uint32_t taddr = tmem + m * Sh::kN + ((uint32_t)(32 * quarter) << 16);
#pragma unroll
                for (int n = 0; n < Sh::kN; n += 32) {
                    uint32_t u[32];
                    tmem_ld32(taddr + n, u);
                    tmem_wait_ld();
                    if (keep && n0 + n < job.N) {
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            dst[n / 4 + q] = make_float4(__uint_as_float(u[4 * q]), __uint_as_float(u[4 * q + 1]),
                                                         __uint_as_float(u[4 * q + 2]), __uint_as_float(u[4 * q + 3]));
                    }
                }
            }
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 0) {
        if (*failed) drain_copies(full, ST, it, nullptr);
        tmem_dealloc(tmem, Sh::kCols);
    }
}

// The weight gradient of a 3x3x3 convolution with at most 64 channels on
// either side, with the operands' roles turned round: the MMA's 128 rows are
// the channels of dz at consecutive rows (4 or 2 blocks of them, each one row
// further into the same window), its columns the channels of x in the three
// windows of a dz.  With x at row p and dz at row p - 2 + j the product belongs
// to tap dx = 2 - j.  An MMA reads its 128-row operand from shared memory at 32
// cycles whatever its columns are, so 96 or 192 columns instead of 32 or 64
// take a third of the MMAs: 4 volumes of 96^3, 32 by 32 channels 0.43 -> 0.22 ms.
// W windows a CTA: 3, or 1 where three would leave half the SMs without work.
template <int RBA, int RBB, int W>
struct Wgrad3Shape {
    static constexpr int CA = RBA / 2, CB = RBB / 2;     // channels of x and dz
    static constexpr int kTpm = 128 / CB;                // rows of dz (taps) of an MMA
    static constexpr int kMpg = CB == 32 ? 1 : 2;        // MMAs that cover three taps
    static constexpr int kN = W * CA;
    static constexpr int kRows = 128;                    // rows per stage
    static constexpr int kABytes = align1k((kRows + 3) * RBB);
    static constexpr int kBBlock = kRows * RBA;
    static constexpr int kStage = kABytes + W * kBBlock;
    static constexpr int kTwo = (113 * 1024 - 1536) / kStage;     // stages that leave room for a second CTA on the SM
    static constexpr int kStages = kTwo >= 2 ? std::min(4, kTwo) : std::min(4, (kSmemMax - 1536) / kStage);
    static constexpr int kSmem = 1024 + kStages * kStage + 512;
    static constexpr uint32_t kCols = kMpg * kN <= 128 ? 128 : (kMpg * kN <= 256 ? 256 : 512);
    static_assert(kStages >= 2, "shared memory");
};

template <int RBA, int RBB, int W>
__global__ void __launch_bounds__(192, 1) wgrad3_kernel(const __grid_constant__ CUtensorMap mapA,
                                                        const __grid_constant__ CUtensorMap mapB, int chunk,
                                                        unsigned int* __restrict__ err,
                                                        const __grid_constant__ WgradJob job) {
    using Sh = Wgrad3Shape<RBA, RBB, W>;
    constexpr int ST = Sh::kStages, WL = Sh::kRows;
    constexpr uint32_t idesc = umma_idesc(128, Sh::kN, true);
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* full = reinterpret_cast<uint64_t*>(base + ST * Sh::kStage);
    uint64_t* empty = full + ST;
    uint64_t* done = empty + ST;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    volatile uint32_t* failed = tmem_slot + 1;
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int g0 = blockIdx.x * W;
    const int r0 = blockIdx.y * chunk;
    const int nk = (chunk + WL - 1) / WL;      // the last stage may be half used (chunk: a multiple of 64)

    if (threadIdx.x == 0) {
        for (int s = 0; s < ST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        *failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(tmem_slot, Sh::kCols);
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;

    int it = 0;      // stages whose loads are issued (warp 0)
    if (warp == 0) {
        const bool leader = elect_one();
        int s = 0;
        uint32_t ph = 1u;
        bool ok = true;
        for (; it < nk; ++it) {
            if (!mbar_wait(&empty[s], ph)) {
                ok = false;
                break;
            }
            if (leader) {
                uint8_t* sa = base + s * Sh::kStage;
                const int r = r0 + it * WL;
                mbar_expect_tx(&full[s], (WL + 3) * RBB + W * Sh::kBBlock);
                tma_load_2d(sa, &mapA, 0, r - 2, &full[s]);
                for (int g = 0; g < W; ++g)
                    tma_load_2d(sa + Sh::kABytes + g * Sh::kBBlock, &mapB, 0, r + job.off[3 * (g0 + g)], &full[s]);
            }
            if (++s == ST) {
                s = 0;
                ph ^= 1u;
            }
        }
        if (!ok && lane == 0) {
            *failed = 1;
            atomicOr(err, 8u);
        }
    } else if (warp == 1) {
        const bool leader = elect_one();
        int s = 0;
        uint32_t ph = 0u;
        const uint64_t a0 = mnmajor_desc(smem_u32(base), RBB, RBB);
        const uint64_t b0 = mnmajor_desc(smem_u32(base) + Sh::kABytes, Sh::kBBlock, RBA);
        for (int it = 0; it < nk; ++it) {
            if (!mbar_wait(&full[s], ph)) {
                if (lane == 0) {
                    *failed = 1;
                    atomicOr(err, 16u);
                }
                break;
            }
            fence_after();
            const uint64_t as = a0 + (uint32_t)((s * Sh::kStage) >> 4);
            const uint64_t bs = b0 + (uint32_t)((s * Sh::kStage) >> 4);
            const int slices = min(WL, chunk - it * WL) / 16;
            if (leader) {
#pragma unroll
                for (int j = 0; j < WL / 16; ++j)
                    if (j < slices)
#pragma unroll
                        for (int m = 0; m < Sh::kMpg; ++m)
                            umma_f16(tmem + m * Sh::kN, as + (m * Sh::kTpm + 16 * j) * (RBB / 16),
                                     bs + 16 * j * (RBA / 16), idesc, (it | j) != 0);
                umma_commit(&empty[s]);
            }
            __syncwarp();
            if (++s == ST) {
                s = 0;
                ph ^= 1u;
            }
        }
        if (leader) umma_commit(done);
        __syncwarp();
    } else if (warp >= 2) {
        if (!mbar_wait(done, 0)) {
            if (lane == 0) atomicOr(err, 32u);
        } else {
            fence_after();
            const int quarter = warp & 3;
            const int l = 32 * quarter + lane;
            const int co = l % Sh::CB;
            for (int m = 0; m < Sh::kMpg; ++m) {
                const int d = 2 - (m * Sh::kTpm + l / Sh::CB);     // the same for all lanes of the warp
                if (d < 0) continue;
                const uint32_t taddr = tmem + m * Sh::kN + ((uint32_t)(32 * quarter) << 16);
                for (int n = 0; n < Sh::kN; n += 32) {
                    uint32_t u[32];
                    tmem_ld32(taddr + n, u);
                    tmem_wait_ld();
                    float* dst = job.P + ((long long)blockIdx.y * 27 * Sh::CA +
                                          (long long)(3 * (g0 + n / Sh::CA) + d) * Sh::CA + n % Sh::CA) * Sh::CB + co;
#pragma unroll
                    for (int q = 0; q < 32; ++q) dst[q * Sh::CB] = __uint_as_float(u[q]);
                }
            }
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 0) {
        if (*failed) drain_copies(full, ST, it, nullptr);
        tmem_dealloc(tmem, Sh::kCols);
    }
}

// ------------------------------------------------------------------ launch
int g_sms = 0;

template <int RB, int N, int NT, int KIND>
struct ConvK {
    using Sh = ConvShape<RB, N, NT, KIND>;
    static cudaError_t init() {
        return cudaFuncSetAttribute(conv_kernel<RB, N, NT, KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, Sh::kSmem);
    }
    static cudaError_t launch(const ConvJob& j, unsigned int* err, cudaStream_t st) {
        const int nblk = j.C / (RB / 2), ntn = j.N / N;
        CUtensorMap ma, mb;
        if (!make_map(&ma, j.x, j.C, j.rows, j.C, RB, Sh::kARows) ||
            !make_map(&mb, j.W, j.taps * j.C, j.N, j.taps * j.C, RB, N))
            return cudaErrorInvalidValue;
        const int tiles = (j.rows + 127) / 128 * ntn;
        conv_kernel<RB, N, NT, KIND><<<std::min(tiles, g_sms), kConvThreads, Sh::kSmem, st>>>(ma, mb, j.rows, nblk, ntn, err, j);
        return cudaGetLastError();
    }
};

template <int RBA, int NBA, int RBB, int NBB, int NT>
struct WgradK {
    using Sh = WgradShape<RBA, NBA, RBB, NBB, NT>;
    static cudaError_t init() {
        return cudaFuncSetAttribute(wgrad_kernel<RBA, NBA, RBB, NBB, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    kSmemMax);
    }
    static cudaError_t launch(const WgradJob& j, unsigned int* err, cudaStream_t st) {
        constexpr int CA = RBA / 2 * NBA;
        const int groups = NT == 1 ? (j.C + CA - 1) / CA : 9;
        CUtensorMap ma, mb;
        if (!make_map(&ma, j.x, j.C, j.rows, j.C, RBA, kWRows) || !make_map(&mb, j.dz, j.N, j.rows, j.N, RBB, kWL))
            return cudaErrorInvalidValue;
        // two CTAs an SM for the plain products of the pointwise network, whose chunks are a few stages long
        const int nk = j.rows / j.S / kWL;
        const int st_n = NT == 1 && nk <= 16 ? std::min(3, Sh::kStages) : Sh::kStages;
        wgrad_kernel<RBA, NBA, RBB, NBB, NT>
            <<<dim3(groups, j.S, (j.N + Sh::kN - 1) / Sh::kN), 192, 1024 + st_n * Sh::kStage + 512, st>>>(
                ma, mb, j.rows / j.S, st_n, err, j);
        return cudaGetLastError();
    }
};

template <int RBA, int RBB>
struct Wgrad3K {
    template <int W>
    static cudaError_t init_w() {
        return cudaFuncSetAttribute(wgrad3_kernel<RBA, RBB, W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    Wgrad3Shape<RBA, RBB, W>::kSmem);
    }
    static cudaError_t init() {
        const cudaError_t e = init_w<1>();
        return e == cudaSuccess ? init_w<3>() : e;
    }
    template <int W>
    static cudaError_t launch_w(const WgradJob& j, unsigned int* err, cudaStream_t st) {
        using Sh = Wgrad3Shape<RBA, RBB, W>;
        CUtensorMap ma, mb;
        if (!make_map(&ma, j.dz, j.N, j.rows, j.N, RBB, Sh::kRows + 3) ||
            !make_map(&mb, j.x, j.C, j.rows, j.C, RBA, Sh::kRows))
            return cudaErrorInvalidValue;
        wgrad3_kernel<RBA, RBB, W><<<dim3(9 / W, j.S), 192, Sh::kSmem, st>>>(ma, mb, j.rows / j.S, err, j);
        return cudaGetLastError();
    }
    static cudaError_t launch(const WgradJob& j, unsigned int* err, cudaStream_t st) {
        return 6 * j.S < g_sms ? launch_w<1>(j, err, st) : launch_w<3>(j, err, st);
    }
};

// Every shape the network uses (C, N stored channels).
#define LBMS_CONV_SHAPES(F)                                                                              \
    F(64, 32, 3, kOutRelu) F(64, 64, 3, kOutRelu) F(128, 64, 3, kOutRelu) F(128, 128, 3, kOutRelu)        \
    F(128, 32, 3, kOutRelu) F(64, 32, 3, kOutReluBack) F(64, 64, 3, kOutSplit) F(128, 64, 3, kOutReluBack) \
    F(128, 128, 3, kOutSplit) F(128, 128, 3, kOutReluBack) F(128, 64, 3, kOutStore)                       \
    F(128, 32, 3, kOutStore) F(128, 128, 1, kOutUp) F(128, 128, 1, kOutReluBack)                          \
    F(128, 64, 1, kOutReluBack) F(64, 32, 1, kOutHead) F(64, 32, 1, kOutReluBack)                         \
    F(128, 64, 1, kOutRelu) F(128, 64, 1, kOutHead)
#define LBMS_WGRAD_SHAPES(F)                                                                        \
    F(128, 1, 128, 2, 3)                                                                              \
    F(128, 2, 128, 1, 3) F(128, 2, 128, 2, 3) F(64, 1, 64, 1, 1) F(128, 2, 128, 1, 1) F(128, 2, 128, 2, 1)

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace

cudaError_t conv_init() {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
#define LBMS_INIT(RB, N, NT, KIND) \
    if (e == cudaSuccess) e = ConvK<RB, N, NT, KIND>::init();
    LBMS_CONV_SHAPES(LBMS_INIT)
#undef LBMS_INIT
    if (e == cudaSuccess) e = Wgrad3K<64, 64>::init();
    if (e == cudaSuccess) e = Wgrad3K<64, 128>::init();
    if (e == cudaSuccess) e = Wgrad3K<128, 64>::init();
    if (e == cudaSuccess) e = Wgrad3K<128, 128>::init();
#define LBMS_INIT(A, NA, B, NB, NT) \
    if (e == cudaSuccess) e = WgradK<A, NA, B, NB, NT>::init();
    LBMS_WGRAD_SHAPES(LBMS_INIT)
#undef LBMS_INIT
    return e;
}

cudaError_t umma_conv(const ConvJob& j, unsigned int* err, cudaStream_t st) {
    cudaError_t e = umma_init();
    if (e != cudaSuccess) return e;
    if (j.rows < 1 || (j.C != 32 && (j.C < 64 || j.C % 64)) || !aligned16(j.x) || !aligned16(j.W) ||
        !aligned16(j.ep.out) || !aligned16(j.ep.act) || !aligned16(j.ep.cat) || !aligned16(j.ep.P) ||
        (j.taps != 27 && j.taps != 1))
        return cudaErrorInvalidValue;
    const int dir = j.off[1] - j.off[0];
    for (int g = 0; g < 9 && j.taps == 27; ++g)   // the three taps of a row lie in one window
        if ((dir != 1 && dir != -1) || j.off[3 * g + 1] != j.off[3 * g] + dir ||
            j.off[3 * g + 2] != j.off[3 * g] + 2 * dir)
            return cudaErrorInvalidValue;
    const int rb = j.C == 32 ? 64 : 128, nt = j.taps == 27 ? 3 : 1;
    // columns of a tile: all of them, or 64 (128 for the transposed convolutions) where N is larger
    const int n = j.kind == kOutUp ? 128 : (j.N == 32 || (j.N == 128 && j.kind != kOutRelu) || nt == 3 ? j.N : 64);
    if (j.N % n || (nt == 3 && rb * n <= 4096 && j.C > 64)) return cudaErrorInvalidValue;
#define LBMS_TRY(RB, N, NT, KIND) \
    if (rb == RB && n == N && nt == NT && j.kind == KIND) return ConvK<RB, N, NT, KIND>::launch(j, err, st);
    LBMS_CONV_SHAPES(LBMS_TRY)
#undef LBMS_TRY
    return cudaErrorInvalidValue;
}

cudaError_t umma_wgrad(const WgradJob& j, unsigned int* err, cudaStream_t st) {
    cudaError_t e = umma_init();
    if (e != cudaSuccess) return e;
    if (j.rows < kWL || j.S < 1 || j.S > 65535 || j.rows % j.S || (j.rows / j.S) % kWL || !aligned16(j.x) ||
        !aligned16(j.dz) || !aligned16(j.P) || (j.taps != 27 && j.taps != 1))
        return cudaErrorInvalidValue;
    for (int g = 0; g < 9 && j.taps == 27; ++g)
        if (j.off[3 * g + 1] != j.off[3 * g] + 1 || j.off[3 * g + 2] != j.off[3 * g] + 2) return cudaErrorInvalidValue;
    const int nt = j.taps == 27 ? 3 : 1;
    // a plain product takes any multiple of 64 channels in tiles of 128 (those past C or N read as zero)
    const int rba = j.C == 32 ? 64 : 128, nba = j.C == 32 || (j.C == 64 && nt == 3) ? 1 : 2;
    const int rbb = j.N == 32 ? 64 : 128, nbb = j.N > 64 ? 2 : 1;
    if ((j.C != 32 && j.C % 64) || (j.N != 32 && j.N % 64) || j.C < 32 || j.N < 32 ||
        (nt == 3 && (j.C > 128 || j.N > 128 || j.C % (rba / 2 * nba) || j.N % (rbb / 2 * nbb))))
        return cudaErrorInvalidValue;
    if (nt == 3 && j.C <= 64 && j.N <= 64) {
        if (j.C == 32) return j.N == 32 ? Wgrad3K<64, 64>::launch(j, err, st) : Wgrad3K<64, 128>::launch(j, err, st);
        return j.N == 32 ? Wgrad3K<128, 64>::launch(j, err, st) : Wgrad3K<128, 128>::launch(j, err, st);
    }
#define LBMS_TRY(A, NA, B, NB, NT) \
    if (rba == A && nba == NA && rbb == B && nbb == NB && nt == NT) return WgradK<A, NA, B, NB, NT>::launch(j, err, st);
    LBMS_WGRAD_SHAPES(LBMS_TRY)
#undef LBMS_TRY
    return cudaErrorInvalidValue;
}

}  // namespace lbms
