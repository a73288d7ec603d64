// Instantiations and launches of the steps of handles that do not fill the
// GPU (lbms_step_small.cuh).
#include "lbms_step_launch.cuh"
#include "lbms_step_small.cuh"

namespace lbms {
namespace {

// How the launches of step_small_kernel overlap.  Blocks of the next step are
// placed wherever there is room, so where there is room beside some blocks of
// this step and not beside others they pile up on few SMs.
//  Two steps fit side by side (twice the blocks are resident): the next one is
// let in as soon as the wait of this one is over, not before, when a third and a
// fourth would come too.  us per step, let in after the gathers / after the
// wait / from the start: 2-D FP32 8.3 k cells 2.42 / 1.92 / 2.03, 18 k 2.65 / 2.2 /
// 2.8, 27 k 2.75 / 2.50 / 2.93; beyond, 30 k, 2.81 / 3.33 / 3.33; 3-D FP32 9.7 k 2.89 /
// 2.50 / 2.85, 19 k 3.37 / 2.94 / 3.36, 23.5 k (beyond) 3.63 / 3.91 / 3.91.
//  Else after the gathers, but in FP64, whose step is the pipe of the fullest
// SM, only where next to nothing of the next step finds room: with 3 to 5 blocks
// an SM in 2-D (6 resident) and 2.5 to 4 in 3-D (5 resident) overlapped launches
// took 24.2 us (16.8 k cells) and 33.2 us (13.4 k), ordinary ones 18.4 and 24.0;
// with more they gain 0.9 us.
struct Overlap {
    bool on, side;
};
Overlap small_overlap(const Launch& L) {
    const int64_t blocks = L.ncells / kSmallCells[kSmall], sms = L.sm_count;
    // by the registers of the kernels: 96 / 126 (FP64), 56 / 80
    const int resident = L.precision == 0 ? (L.dim == 2 ? 6 : 5) : (L.dim == 2 ? 12 : 8);
    const bool side = 2 * blocks <= resident * sms;
    return {L.precision != 0 || side || blocks > (resident - 1) * sms, side};
}

template <class Lat, typename XS, typename P>
SmallParams<XS, P> params(const Launch& L, int n) {
    SmallParams<XS, P> p;
    for (int k = 0; k < 2; ++k) {
        p.h[k] = static_cast<P*>(L.b.f[k]);
        p.x[k] = static_cast<XS*>(L.b.X[k]);
    }
    p.cur = L.cur;
    p.n = n;
    p.nbr32 = L.b.nbr;
    p.cell_code = L.b.cell_code;
    p.rowtab = reinterpret_cast<const uint2*>(L.b.rowtab);
    p.cases = static_cast<const CaseBC<XS>*>(L.b.cases);
    p.blk_case = L.b.blk_case[0];
    p.S = L.S;
    p.c = launch_detail::make_const<typename Xv<XS>::T>(L);
    return p;
}

template <class Lat, typename XS, typename P, int W>
cudaError_t block_w(const Launch& L, int n, cudaStream_t st) {
    using T = typename Xv<XS>::T;
    constexpr int smem = W * (3 * sizeof(T) + 3 * Lat::DIM * sizeof(T) + 3 * sizeof(XS) + 3 * Lat::Q * sizeof(P));
    cudaError_t e = cudaSuccess;
    if (smem > 48 * 1024)
        e = cudaFuncSetAttribute(block_steps_kernel<Lat, XS, P, W>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    block_steps_kernel<Lat, XS, P, W><<<L.n_cases, 3 * W, smem, st>>>(params<Lat, XS, P>(L, n));
    return cudaGetLastError();
}

template <class Lat, typename XS, typename P>
cudaError_t small_t(const Launch& L, cudaStream_t st) {
    constexpr int W = kSmallCells[kSmall];
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(L.ncells / W));
    cfg.blockDim = dim3(3 * W);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    const Overlap over = small_overlap(L);
    cfg.numAttrs = over.on ? 1 : 0;
    return cudaLaunchKernelEx(
        &cfg, over.side ? step_small_kernel<Lat, XS, P, W, true> : step_small_kernel<Lat, XS, P, W, false>,
        params<Lat, XS, P>(L, 1));
}

template <class Lat, typename XS, typename P>
cudaError_t block_t(const Launch& L, int n, cudaStream_t st) {
    switch (L.small) {
        case kBlock64: return block_w<Lat, XS, P, kSmallCells[kBlock64]>(L, n, st);
        case kBlock128: return block_w<Lat, XS, P, kSmallCells[kBlock128]>(L, n, st);
        case kBlock320:
            if constexpr (sizeof(XS) == 8) return cudaErrorInvalidValue;   // not chosen
            else return block_w<Lat, XS, P, kSmallCells[kBlock320]>(L, n, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

namespace {

// Whether a block per case is the faster step of small cases.  FP32 and FP16:
// a step is latency, so it is, but for 3-D cases of more than 128 cells while
// they leave most SMs idle (us per step of 1 / 15 / 30 / 45 / 60 cases of 300
// cells, block 3.0 at any, launches 2.2 / 2.4 / 2.8 / 3.1 / 3.3; FP16 3.2
// and 2.1 / 2.4 / 2.8 / 3.0 / 3.3).  FP64: the pipe of the fullest SM is the step,
// and a block puts a whole case on one (2-D, 1 case of 64, 120, 300 cells: 8.5,
// 16.7, 41.5 us, launches 6.7 at any), so it must not give that SM more warps
// than the launches would (80 cases of 64: 8.5, launches 9.9; 152 of 120: 16.7
// and 22); with 320 cells its registers spill and it was ahead nowhere.
bool block_pays(const Launch& L, int block) {
    if (L.precision != 0) return block != kBlock320 || L.dim == 2 || 8 * L.n_cases >= 3 * L.sm_count;
    if (block == kBlock320) return false;
    const int warps = 3 * kSmallCells[block] / 32, resident = block == kBlock64 ? 2 : 1;
    const int64_t a = L.sm_count, n = L.n_cases;
    const int64_t of_blocks = n <= a ? warps : (n + resident * a - 1) / (resident * a) * resident * warps;
    return of_blocks <= 3 * ((L.ncells / kSmallCells[kSmall] + a - 1) / a);
}

// Whether a launch of blocks of 32 cells and three threads a cell is the faster
// step, against the tiled one; `per` cells make one block of a tile on each SM.
// us per step, this / tiled: FP32 3-D 36 k cells 4.0 / 5.1, 42 k 5.4 / 5.1, 2-D 37 k
// 3.0 / 3.4, 44 k 3.2 / 3.1.  FP64, bound by the pipe of the fullest SM, gains from the
// finer blocks while there are few: 2-D 40 k cells 38 / 43, 57 k 50 / 50, 67 k 62 / 60, and
// once more where the tiled step starts a second wave of 8 blocks an SM: 81 k 71 /
// 80, 92 k 82 / 80; 3-D 41 k 60 / 70, 49 k 73 / 80, 52 k 73 / 80, 54 k 80 / 80.
bool small_pays(const Launch& L) {
    const int64_t n = L.ncells, per = (int64_t)kTile * L.sm_count;
    if (L.precision != 0) return n <= 4 * per;
    if (L.dim == 2) return n <= 6 * per || (n > 8 * per && n <= 9 * per);
    return 2 * n <= 11 * per;
}

}  // namespace

int choose_small(const Launch& L, int max_nf) {
    for (int block : {kBlock64, kBlock128, kBlock320})
        if (max_nf <= kSmallCells[block]) {
            if (block_pays(L, block)) return block;
            break;
        }
    return small_pays(L) ? kSmall : kNotSmall;
}

cudaError_t launch_steps_block(const Launch& L, int n, cudaStream_t st) {
    if (L.dim == 2) {
        if (L.precision == 0) return block_t<D2Q9, double, double>(L, n, st);
        if (L.precision == 1) return block_t<D2Q9, float, float>(L, n, st);
        return block_t<D2Q9, float, __half>(L, n, st);
    }
    if (L.precision == 0) return block_t<D3Q19, double, double>(L, n, st);
    if (L.precision == 1) return block_t<D3Q19, float, float>(L, n, st);
    return block_t<D3Q19, float, __half>(L, n, st);
}

cudaError_t launch_step_small(const Launch& L, cudaStream_t st) {
    if (L.dim == 2) {
        if (L.precision == 0) return small_t<D2Q9, double, double>(L, st);
        if (L.precision == 1) return small_t<D2Q9, float, float>(L, st);
        return small_t<D2Q9, float, __half>(L, st);
    }
    if (L.precision == 0) return small_t<D3Q19, double, double>(L, st);
    if (L.precision == 1) return small_t<D3Q19, float, float>(L, st);
    return small_t<D3Q19, float, __half>(L, st);
}

}  // namespace lbms
