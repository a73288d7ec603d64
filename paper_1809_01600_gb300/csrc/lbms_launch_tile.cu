// Instantiations and launches of the default time step (lbms_step_tile.cuh).
#include "lbms_step_launch.cuh"
#include "lbms_step_tile.cuh"

#include <algorithm>

namespace lbms {
namespace {

// Whether consecutive launches overlap (programmatic dependent launch).  Blocks
// of the next step are placed wherever there is room; while this step leaves
// room on some SMs and not on others, they pile up there and the next step runs
// unevenly.  us per step without and with: 3-D FP32 41 k cells 5.5 and 6.9, 67 k
// 6.5 and 7.5, 79 k 7.52 and 7.53, 91 k 7.9 and 7.5; FP16 67 k 5.9 and 6.6, 79 k
// 7.0 and 6.6; 2-D FP32 60 k 4.0 and 4.4, 90 k 4.6 and 4.6, FP64 43 k 42.9 and 63.8,
// 67 k 60.0 and 65.3; 3-D FP64 (5 blocks an SM resident) 41 k 69.6 and 79.5, 49 k
// 80.0 and 79.8.  So from 8 blocks an SM on, or as many as are resident.
bool tile_overlaps(const Launch& L) {
    return L.ncells >= (int64_t)std::min(8, tile_min_blocks(L.dim, L.precision)) * kTile * L.sm_count;
}

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
    cfg.numAttrs = tile_overlaps(L) ? 1 : 0;
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
