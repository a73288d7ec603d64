// Instantiations and launches of the default time step (lbms_step_tile.cuh).
#include "lbms_step_launch.cuh"
#include "lbms_step_tile.cuh"

#include <algorithm>

namespace lbms {
namespace {

// Whether consecutive launches overlap (programmatic dependent launch).  Blocks
// of the next step are placed wherever there is room; while this step leaves
// room on some SMs and not on others, they pile up there and the next step runs
// unevenly.  us per step without and with: 3-D FP32 67 k cells 6.5 and 7.5, 79 k
// 7.52 and 7.53, 91 k 7.9 and 7.5; FP16 67 k 5.9 and 6.6, 79 k 7.0 and 6.6; 2-D FP32
// 60 k 4.0 and 4.4, 90 k 4.6 and 4.6, FP64 67 k 60.0 and 65.3.  So from 8 blocks an
// SM on, or as many as are resident; and where two steps are resident side by
// side, the next one let in after the wait (not a third from the start): 3-D
// FP32 42 k cells 5.57 and 5.06, FP16 5.05 and 4.45, 2-D FP32 44 k 3.66 and 3.13.
struct Overlap {
    bool on, side;
};
Overlap tile_overlap(const Launch& L) {
    const int64_t per = (int64_t)kTile * L.sm_count;
    const int resident = tile_resident(L.dim, L.precision);
    const bool side = 2 * (int64_t)L.ncells <= resident * per;
    return {!L.fine && (side || L.ncells >= std::min(8, resident) * per), side};
}

template <class Lat, typename XS, typename P, typename NBT, int W, int MB>
cudaError_t tile_w(const Launch& L, cudaStream_t st) {
    using T = typename Xv<XS>::T;
    const Overlap over = tile_overlap(L);
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
    p.side = over.side;
    p.pf_dist = L.sm_count * kTilePrefetch / kTile * kTile;
    p.c = launch_detail::make_const<T>(L);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(L.ncells / W));
    cfg.blockDim = dim3(W);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = over.on ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, step_tile_kernel<Lat, XS, P, NBT, W, MB>, p);
}

template <class Lat, typename XS, typename P, int W, int MB>
cudaError_t tile_nb(const Launch& L, cudaStream_t st) {
    return L.b.rowtab ? tile_w<Lat, XS, P, RowMaskNb, W, MB>(L, st) : tile_w<Lat, XS, P, int, W, MB>(L, st);
}

template <class Lat, typename XS, typename P>
cudaError_t tile_t(const Launch& L, cudaStream_t st) {
    constexpr int prec = sizeof(XS) == 8 ? 0 : (sizeof(P) == 4 ? 1 : 2);
    if constexpr (prec == 0 && Lat::DIM == 3)
        if (L.fine) return tile_nb<Lat, XS, P, kFineCells, kFineMinBlocks>(L, st);
    return tile_nb<Lat, XS, P, kTile, tile_min_blocks(Lat::DIM, prec)>(L, st);
}

}  // namespace

size_t tile_cell_bytes(int dim, int precision) {
    if (precision == 2) return 4 * (dim == 2 ? TileLay<D2Q9, __half>::kRows : TileLay<D3Q19, __half>::kRows);
    return 3 * (dim == 2 ? D2Q9::Q : D3Q19::Q) * pop_size(precision);
}

bool tile_fine(const Launch& L) {
    const int64_t n = L.ncells, per = (int64_t)kTile * L.sm_count, wave = tile_resident(L.dim, L.precision) * per;
    return L.dim == 3 && L.precision == 0 && n > wave && 4 * n <= 5 * wave;
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
