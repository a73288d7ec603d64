// Instantiations and launches of the default time step (lbms_step_tile.cuh).
#include "lbms_step_launch.cuh"
#include "lbms_step_tile.cuh"

namespace lbms {
namespace {

template <class Lat, typename XS, typename P, typename NBT>
cudaError_t tile_w(const Launch& L, cudaStream_t st) {
    using T = typename Xv<XS>::T;
    constexpr int MB = tile_min_blocks(Lat::DIM, sizeof(XS) == 8 ? 0 : (sizeof(P) == 4 ? 1 : 2));
    TileParams<XS, P> p;
    p.hin = static_cast<const P*>(L.b.f[L.cur]);
    p.hout = static_cast<P*>(L.b.f[L.cur ^ 1]);
    p.xin = static_cast<const XS*>(L.b.X[L.cur]);
    p.xout = static_cast<XS*>(L.b.X[L.cur ^ 1]);
    p.nbr32 = L.b.nbr;
    p.cell_code = L.b.cell_code;
    p.rowtab = reinterpret_cast<const uint2*>(L.b.rowtab);
    p.cases = static_cast<const CaseBC<XS>*>(L.b.cases);
    p.blk_case = L.b.blk_case[kTileBlkCase];
    p.S = L.S;
    p.pf_dist = L.sm_count * kTilePrefetch / kTile * kTile;
    p.c = launch_detail::make_const<T>(L);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(L.ncells / kTile));
    cfg.blockDim = dim3(kTile);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, step_tile_kernel<Lat, XS, P, NBT, kTile, MB>, p);
}

template <class Lat, typename XS, typename P>
cudaError_t tile_t(const Launch& L, cudaStream_t st) {
    return L.b.rowtab ? tile_w<Lat, XS, P, RowMaskNb>(L, st) : tile_w<Lat, XS, P, int>(L, st);
}

}  // namespace

size_t tile_cell_bytes(int dim, int precision) {
    if (precision == 2) return 4 * (dim == 2 ? TileLay<D2Q9, __half>::kRows : TileLay<D3Q19, __half>::kRows);
    return 3 * (dim == 2 ? D2Q9::Q : D3Q19::Q) * pop_size(precision);
}

cudaError_t launch_step_tile(const Launch& L, cudaStream_t st) {
    if (L.dim == 2) {
        if (L.precision == 0) return tile_t<D2Q9, double, double>(L, st);
        if (L.precision == 1) return tile_t<D2Q9, float, float>(L, st);
        return tile_t<D2Q9, float, __half>(L, st);
    }
    if (L.precision == 0) return tile_t<D3Q19, double, double>(L, st);
    if (L.precision == 1) return tile_t<D3Q19, float, float>(L, st);
    return tile_t<D3Q19, float, __half>(L, st);
}

}  // namespace lbms
