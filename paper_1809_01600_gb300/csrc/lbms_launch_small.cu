// Instantiations and launches of the steps of handles that do not fill the
// GPU (lbms_step_small.cuh).
#include "lbms_step_launch.cuh"
#include "lbms_step_small.cuh"

namespace lbms {
namespace {

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
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, step_small_kernel<Lat, XS, P, W>, params<Lat, XS, P>(L, 1));
}

template <class Lat, typename XS, typename P>
cudaError_t block_t(const Launch& L, int n, cudaStream_t st) {
    switch (L.small) {
        case kBlock64: return block_w<Lat, XS, P, kSmallCells[kBlock64]>(L, n, st);
        case kBlock128: return block_w<Lat, XS, P, kSmallCells[kBlock128]>(L, n, st);
        case kBlock320: return block_w<Lat, XS, P, kSmallCells[kBlock320]>(L, n, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

int choose_small(const Launch& L, int max_nf) {
    if (max_nf <= 64) return kBlock64;
    if (max_nf <= 128) return kBlock128;
    if (max_nf <= 320) return kBlock320;
    return L.ncells < kTileMinCells ? kSmall : kNotSmall;
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
    if (L.small != kSmall) return launch_steps_block(L, 1, st);
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
