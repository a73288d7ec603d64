// The time steps of handles that do not fill the GPU.  There a step's work
// takes a microsecond or two and the launch between two steps about as much
// again.  One thread per (species, cell), as in step_kernel.
//  * block_steps_kernel: every case fits a block, which keeps the case's whole
//    state in shared memory over many steps; a step costs two block barriers.
//    15 strips of 64 nodes in FP32: 0.61 us per step, 1.79 with a launch each.
//  * step_small_kernel: one step per launch, launches overlapped (programmatic
//    dependent launch).  The three threads of a cell split its source rows
//    (row windows: 9 rows of D3Q19 as 3 + 2 + 4, 6 links each) or its row of
//    the 32-bit table and leave the links in shared memory, before the wait for
//    the preceding step: no step writes those tables.  When the next step may
//    be placed, and where launches overlap at all: small_overlap
//    (lbms_launch_small.cu).
// Keeping all blocks resident with a grid-wide barrier, or with flags between
// the blocks that exchange, was no faster than overlapped launches where FP32
// is the arithmetic: 26 k cells took 4.3 and 5.0 us per step, launches 3.9.
#pragma once

#include "lbms_internal.h"
#include "lbms_kernels.cuh"
#include "lbms_step_tile.cuh"

namespace lbms {

// The state's pointers carry no __restrict__, so that its loads stay ordinary
// (coherent) loads behind grid_wait.
template <typename XS, typename P>
struct SmallParams {
    P* h[2];
    XS* x[2];
    int cur;                            // lattice holding the state
    int n;                              // steps (block_steps_kernel)
    const int* nbr32;
    const uint32_t* cell_code;
    const uint2* rowtab;                // windows of the tiled step, or null: nbr32
    const CaseBC<XS>* cases;
    const int* blk_case;                // case of each run of 32 cells
    int64_t S;
    MsConst<typename Xv<XS>::T> c;
};

enum : int { kInletCell = 1, kOutletCell = 2 };

// After streaming: boundary rules, the moment and the lagged gradient of one
// species (d in storage units, h * kStore; dx the X differences of the links).
// (xb: the species' inlet mole fraction; qs: its outlet flux over the weight
// of the links along x, in storage units)
template <class L, typename XS, typename P>
__device__ __forceinline__ void close_stream(const Xv<XS>& xb, typename Xv<XS>::T qs, int flags, const Xv<XS>& xo,
                                             typename Xv<XS>::T (&d)[L::Q],
                                             const typename Xv<XS>::T (&dx)[L::Q], typename Xv<XS>::T& dX,
                                             typename Xv<XS>::T (&g)[L::DIM]) {
    using T = typename Xv<XS>::T;
    constexpr T sc = T(Pop<T, P>::kStore);
    if (flags & kOutletCell) {   // Eq. 39: every link from beyond x = nx - 1
#pragma unroll
        for (int k = 1; k < L::Q; ++k)
            if (L::e(k, 0) == -1) d[k] -= T(weight<L>(opp<L>(k))) * qs;
    }
    if (flags & kInletCell) {    // Eq. 36: f_k = (w_k + w_opp) X_in - f_opp
        const T din = xb.minus(xo) * sc;
#pragma unroll
        for (int k = 1; k < L::Q; ++k)
            if (L::e(k, 0) == 1) d[k] = T(weight<L>(k) + weight<L>(opp<L>(k))) * din - d[opp<L>(k)];
    }
    // in two chains: the latency of the sum is on the step's critical path
    T odd = d[1];
    dX = d[0];
#pragma unroll
    for (int k = 3; k < L::Q; k += 2) odd += d[k];
#pragma unroll
    for (int k = 2; k < L::Q; k += 2) dX += d[k];
    dX += odd;
    // central, one-sided along x at the inlet and outlet (whose missing
    // neighbour has difference 0)
#pragma unroll
    for (int a = 0; a < L::DIM; ++a) g[a] = (a == 0 && flags ? T(1) : T(0.5)) * (dx[2 + 2 * a] - dx[1 + 2 * a]);
}

// The coupling and the collision of one species: the stored populations q.
template <class L, typename XS, typename P>
__device__ __forceinline__ void collide(const MsConst<typename Xv<XS>::T>& c, int s,
                                        const typename Xv<XS>::T (&X)[3],
                                        const typename Xv<XS>::T (&g)[3][L::DIM],
                                        const typename Xv<XS>::T (&gs)[L::DIM], typename Xv<XS>::T dX,
                                        const typename Xv<XS>::T (&d)[L::Q], P (&q)[L::Q]) {
    using T = typename Xv<XS>::T;
    constexpr T sc = T(Pop<T, P>::kStore);
    T it, v[L::DIM];
    ms_couple(X, g, gs, c, s, it, v);
    const T Xs = s == 0 ? X[0] : (s == 1 ? X[1] : X[2]);
    const T keep = T(1) - it;
    const T A = T(3) * sc * Xs * it;
#pragma unroll
    for (int a = 0; a < L::DIM; ++a) v[a] *= A;
    T rest = T(0), rest1 = T(0);
#pragma unroll
    for (int k = 1; k < L::Q; k += 2) {
        T ev = T(0);
#pragma unroll
        for (int a = 0; a < L::DIM; ++a) {
            if (L::e(k, a) == 1) ev += v[a];
            if (L::e(k, a) == -1) ev -= v[a];
        }
        const T w = T(weight<L>(k));
        const T m = w * ev;
        q[k] = Pop<T, P>::quant_raw((d[k] - w * dX) * keep + m);
        q[k + 1] = Pop<T, P>::quant_raw((d[k + 1] - w * dX) * keep - m);
        rest -= Pop<T, P>::dequant_raw(q[k]);
        rest1 -= Pop<T, P>::dequant_raw(q[k + 1]);
    }
    q[0] = Pop<T, P>::quant_raw(rest + rest1);   // closes the sum on the stored values
}

// One block of 3 W threads per case of at most W cells; the state in shared
// memory as [3][Q][W] populations and [3][W] mole fractions (the words the
// neighbours exchange).
template <class L, typename XS, typename P, int W>
__global__ void __launch_bounds__(3 * W) block_steps_kernel(const SmallParams<XS, P> p) {
    using T = typename Xv<XS>::T;
    using XV = Xv<XS>;
    constexpr int Q = L::Q;
    constexpr int DIM = L::DIM;
    extern __shared__ __align__(16) unsigned char smem[];
    T (*sXv)[W] = reinterpret_cast<T (*)[W]>(smem);                    // [3] X of the step
    T (*sG)[DIM][W] = reinterpret_cast<T (*)[DIM][W]>(sXv + 3);        // [3] its gradients
    XS (*sX)[W] = reinterpret_cast<XS (*)[W]>(sG + 3);                 // [3] X the neighbours read
    P (*sH)[Q * W] = reinterpret_cast<P (*)[Q * W]>(sX + 3);           // [3] populations

    const int s = threadIdx.x / W;
    const int c = threadIdx.x - s * W;
    const CaseBC<XS>& cb = p.cases[blockIdx.x];
    const bool mine = c < cb.nf;
    const int i = cb.base + (mine ? c : 0);
    const int64_t S = p.S;
    uint32_t link[Q];    // element of sH[s] to pull | cell whose X to exchange with << 16
    int flags = 0;
    XV xo{}, xprev{};
    {
        const P* hs = p.h[p.cur] + (int64_t)s * Q * S;
        const XS* xs = p.x[p.cur];
        int nb[Q];
        load_neighbours<L>(p.nbr32, i, nb);
        flags = (nb[1] == NB_INLET ? kInletCell : 0) | (nb[2] == NB_OUTLET ? kOutletCell : 0);
#pragma unroll
        for (int k = 1; k < Q; ++k) {
            const int j = nb[k] >= 0 ? nb[k] - cb.base : c;
            link[k] = (uint32_t)((nb[k] >= 0 ? k : opp<L>(k)) * W + j) | ((uint32_t)j << 16);
        }
        if (mine) {
            xo = XV::own(xs, S, s, i);
#pragma unroll
            for (int k = 0; k < Q; ++k) sH[s][k * W + c] = hs[k * S + i];
            sX[s][c] = xo.exch_base();
        }
    }
    __syncthreads();
    constexpr T sc = T(Pop<T, P>::kStore);
    const XV xb = cb.xbc[s];
    const T qs = cb.qout[s] * sc / T(weight_xplus<L>());
    for (int t = 0; t < p.n; ++t) {
        T d[Q], dx[Q], dX = T(0), g[DIM];
        if (mine) {
            d[0] = Pop<T, P>::raw(&sH[s][c]);
#pragma unroll
            for (int k = 1; k < Q; ++k) {
                d[k] = Pop<T, P>::raw(&sH[s][link[k] & 0xFFFFu]);
                dx[k] = xo.exch(sX[s][link[k] >> 16]);
                d[k] += T(weight<L>(k) * sc) * dx[k];
            }
            close_stream<L, XS, P>(xb, qs, flags, xo, d, dx, dX, g);
            xprev = xo;
            xo = xo.plus(dX * T(1.0 / sc));
            sXv[s][c] = xo.value();
#pragma unroll
            for (int a = 0; a < DIM; ++a) sG[s][a][c] = g[a];
        }
        __syncthreads();
        if (mine) {
            T X[3], gall[3][DIM];
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                X[r] = sXv[r][c];
#pragma unroll
                for (int a = 0; a < DIM; ++a) gall[r][a] = sG[r][a][c];
            }
            P q[Q];
            collide<L, XS, P>(p.c, s, X, gall, g, dX, d, q);
#pragma unroll
            for (int k = 0; k < Q; ++k) sH[s][k * W + c] = q[k];
            sX[s][c] = xo.exch_base();
        }
        __syncthreads();
    }
    if (mine) {   // the state, and the mole fractions of the step before in the other lattice
        const int fin = p.cur ^ (p.n & 1);
        P* hs = p.h[fin] + (int64_t)s * Q * S;
#pragma unroll
        for (int k = 0; k < Q; ++k) hs[k * S + i] = sH[s][k * W + c];
        xo.store(p.x[fin], S, s, i);
        xprev.store(p.x[fin ^ 1], S, s, i);
    }
}

// Which of a cell's three threads looks up source row (dy, dz).
template <class L>
__host__ __device__ constexpr int row_owner(int dy, int dz) {
    if (L::DIM == 2) return dy == 0 ? 0 : (dy < 0 ? 1 : 2);
    if (dz == 0) return dy <= 0 ? 0 : 1;
    if (dy == 0) return dz < 0 ? 1 : 2;
    return dy < 0 && dz < 0 ? 0 : 2;
}

// Links of cell i (slot c of the block) from the rows that thread PART looks
// up (windows as in row_sources): the population to pull (element of the
// species, rows of stride S; bounce-back folded in) and the cell to exchange
// X with.
template <class L, int PART, int W>
__device__ __forceinline__ void share_rows(uint32_t code, const uint2* __restrict__ tab, int nx, int ny, int nz,
                                           int wpr, int i, int S, int c, int2 (*sN)[W], int* sF) {
    const bool pad = code == 0xFFFFFFFFu;   // padding cell between cases: walls all round
    if (pad) code = 0u;
    const int x = (int)(code & 2047u);
    const int y = (int)((code >> 11) & 1023u);
    const int z = (int)(code >> 21);
    const int b = (x & 15) + 8;
    const uint32_t below = (1u << b) - 1u;
    if (PART == 0) sF[c] = pad ? 0 : (x == 0 ? kInletCell : 0) | (x == nx - 1 ? kOutletCell : 0);
#pragma unroll
    for (int dz = -1; dz <= 1; ++dz) {
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy) {
            if (!row_used<L>(dy, dz) || row_owner<L>(dy, dz) != PART) continue;
            const int ys = dy == 0 ? y : (dy < 0 ? (y == 0 ? ny - 1 : y - 1) : (y == ny - 1 ? 0 : y + 1));
            const int zs = dz == 0 ? z : (dz < 0 ? (z == 0 ? nz - 1 : z - 1) : (z == nz - 1 ? 0 : z + 1));
            const uint2 e = __ldg(tab + (zs * ny + ys) * wpr + (x >> 4));
            const int at = (int)e.y - kTile + __popc(e.x & below);   // index x has (or would have)
            const uint32_t bits = pad ? 0u : e.x >> (b - 1);         // fluid flags of x - 1, x, x + 1
#pragma unroll
            for (int k = 1; k < L::Q; ++k) {
                if (-L::e(k, 1) != dy || -L::e(k, 2) != dz) continue;
                const int dx = -L::e(k, 0);
                const bool fluid = bits & (dx < 0 ? 1u : (dx == 0 ? 2u : 4u));
                const int j = dx < 0 ? at - 1 : (dx == 0 ? at : at + (int)((bits >> 1) & 1u));
                sN[k - 1][c] = make_int2(fluid ? k * S + j : opp<L>(k) * S + i, fluid ? j : i);
            }
        }
    }
}

// The same from the cell's row of the 32-bit table, a third of the links.
template <class L, int PART, int W>
__device__ __forceinline__ void share_table(const int* __restrict__ nbr, int i, int S, int c, int2 (*sN)[W], int* sF) {
    constexpr int N = (L::Q - 1 + 2) / 3;
    const int* row = nbr + (int64_t)i * nb_width<L>();
    int flags = 0;
#pragma unroll
    for (int k = 1 + PART * N; k < 1 + (PART + 1) * N && k < L::Q; ++k) {
        const int j = __ldg(row + (k - 1));
        sN[k - 1][c] = make_int2(j >= 0 ? k * S + j : opp<L>(k) * S + i, j >= 0 ? j : i);
        if (k <= 2) flags |= j == NB_INLET ? kInletCell : (j == NB_OUTLET ? kOutletCell : 0);
    }
    if (PART == 0) sF[c] = flags;   // links 1 and 2 (from x - 1 and x + 1) are part 0's
}

// One step of blocks of W = 32 cells (blocks of 16 and 64 were slower on one or
// another of 2-D and 3-D handles of 2 to 37 k cells in FP64, FP32 and FP16).
// us per step, with step_kernel / now: 2-D 2.2 k cells FP64 8.3 / 6.8, 2.4 k FP32
// 2.1 / 1.7; 9 k FP64 12.0 / 9.9; 3-D 5.2 k FP32 2.6 / 2.2, 26 k FP32 4.1 / 3.7, FP64 47 /
// 41, 36 k FP32 4.6 / 4.0.
// SIDE: the next step fits beside this one (small_overlap).
template <class L, typename XS, typename P, int W, bool SIDE>
__global__ void __launch_bounds__(3 * W, kSmallMinBlocks[kSmall]) step_small_kernel(const SmallParams<XS, P> p) {
    using T = typename Xv<XS>::T;
    using XV = Xv<XS>;
    constexpr int Q = L::Q;
    constexpr int DIM = L::DIM;
    __shared__ int2 sN[Q - 1][W];
    __shared__ int sF[W];
    __shared__ T sXv[3][W];
    __shared__ T sG[3][DIM][W];
    const int s = threadIdx.x / W;
    const int c = threadIdx.x - s * W;
    const int i = blockIdx.x * W + c;    // the cells of all cases are a multiple of 64
    const CaseBC<XS>& cb = p.cases[__ldg(p.blk_case + i / 32)];
    const int64_t S = p.S;
    const int S32 = (int)S;              // Q S < 2^31 (checked at create)
    if (p.rowtab) {
        const uint32_t code = __ldg(p.cell_code + i);
        const uint2* tab = p.rowtab + cb.tab;
        if (s == 0)
            share_rows<L, 0, W>(code, tab, cb.nx, cb.ny, cb.nz, cb.wpr, i, S32, c, sN, sF);
        else if (s == 1)
            share_rows<L, 1, W>(code, tab, cb.nx, cb.ny, cb.nz, cb.wpr, i, S32, c, sN, sF);
        else
            share_rows<L, 2, W>(code, tab, cb.nx, cb.ny, cb.nz, cb.wpr, i, S32, c, sN, sF);
    } else {
        if (s == 0)
            share_table<L, 0, W>(p.nbr32, i, S32, c, sN, sF);
        else if (s == 1)
            share_table<L, 1, W>(p.nbr32, i, S32, c, sN, sF);
        else
            share_table<L, 2, W>(p.nbr32, i, S32, c, sN, sF);
    }
    grid_wait();
    if constexpr (SIDE) grid_launch_next();
    const P* hs = p.h[p.cur] + (int64_t)s * Q * S;
    const XS* xh = p.x[p.cur] + s * S;
    XV xo = XV::own_rows(xh, p.x[p.cur] + (3 + s) * S, i);
    constexpr T sc = T(Pop<T, P>::kStore);
    T d[Q], dx[Q], dX, g[DIM];
    d[0] = Pop<T, P>::raw(hs + i);
    __syncthreads();
#pragma unroll
    for (int k = 1; k < Q; ++k) {
        const int2 n = sN[k - 1][c];
        d[k] = Pop<T, P>::raw(hs + n.x);
        dx[k] = xh[n.y];
    }
#pragma unroll
    for (int k = 1; k < Q; ++k) {
        dx[k] = xo.exch(dx[k]);
        d[k] += T(weight<L>(k) * sc) * dx[k];
    }
    const int flags = sF[c];
    close_stream<L, XS, P>(cb.xbc[s], cb.qout[s] * T(Pop<T, P>::kStore / weight_xplus<L>()), flags, xo, d, dx, dX, g);
    xo = xo.plus(dX * T(1.0 / sc));
    sXv[s][c] = xo.value();
#pragma unroll
    for (int a = 0; a < DIM; ++a) sG[s][a][c] = g[a];
    __syncthreads();
    T X[3], gall[3][DIM];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        X[r] = sXv[r][c];
#pragma unroll
        for (int a = 0; a < DIM; ++a) gall[r][a] = sG[r][a][c];
    }
    // Not earlier: blocks of the next step placed while these have just begun
    // crowd onto the SMs they find.
    if constexpr (!SIDE) grid_launch_next();
    P q[Q];
    collide<L, XS, P>(p.c, s, X, gall, g, dX, d, q);
    P* ho = p.h[p.cur ^ 1] + (int64_t)s * Q * S;
#pragma unroll
    for (int k = 0; k < Q; ++k) ho[k * S32 + i] = q[k];
    xo.store(p.x[p.cur ^ 1], S, s, i);
}

}  // namespace lbms
