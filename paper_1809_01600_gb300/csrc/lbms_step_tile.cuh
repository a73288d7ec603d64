// The default time step: one thread per fluid cell with the populations of
// all three species in registers, and the populations in tiles in memory.
//
// Tiled layout (TileLay): population (s, k) of cell j at unit
// (j / 64) R 64 + row(s, k) 64 + j % 64 of R rows a tile, so that all populations
// of a cell lie at compile-time distances from one address.  A link then costs one
// address for its three species and the stores of a cell one address in all,
// where rows of stride S need one per population; and a tile is one
// contiguous piece of memory (14.6 KB in FP32), which a single instruction
// prefetches into L2.  X keeps its rows of stride S.
//
// What bounds it (256x128x128 anode, 1,689,574 fluid cells, D3Q19): FP32
// moves 826 MB a step and takes 140 to 149 us on one GB300 or another, 5.6 to
// 5.9 TB/s of the 6.8 a copy reaches;
// with the neighbour decode, the address arithmetic and the boundary rules
// spread over the links the step before issued 108 M warp instructions and
// took 181 us, this one issues 66 M.  FP16 moves 449 MB in 101 us (151
// before): the latency of the gathers and their issue, so populations share
// 32-bit units (112 us with a 16-bit access for each, 57 loads and 57 stores a
// cell instead of 38 and 29).  FP64 takes 2231 us (2548): the FP64 pipe.
// The same with one thread per (cell, species) and the lookup shared through
// shared memory took 161 us (FP32) and 137 us (FP16): the L1 data stage, at
// 72-76 %, from the two-word link records read three times a cell.
//
// The lookup of the sources reads only tables that no time step writes, so it
// runs before the wait for the preceding launch (programmatic dependent
// launch).
#pragma once

#include "lbms_internal.h"
#include "lbms_kernels.cuh"

namespace lbms {

static_assert(kTile == kCaseAlign, "a case starts at a tile");

// Waits for the preceding launch of the stream and its memory operations;
// nothing to wait for when launched without the programmatic attribute.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Brings `bytes` (a multiple of 16) at the 16-byte aligned address a into L2.
__device__ __forceinline__ void prefetch_bulk(const void* a, unsigned bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(__cvta_generic_to_global(a)), "r"(bytes)
                 : "memory");
}

// As StepParams, for overlapped launches: the state's pointers carry no
// __restrict__, so that its loads stay ordinary (coherent) loads behind
// grid_wait; the tables and the boundary data are never written by a kernel.
template <typename XS, typename P>
struct TileParams {
    const P* hin;
    P* hout;
    const XS* xin;
    XS* xout;
    const int* nbr32;
    const uint32_t* cell_code;
    const uint2* rowtab;
    const CaseBC<XS>* cases;
    const int* blk_case;
    int64_t S;
    bool side;                          // the next step fits beside this one: let in after the wait
    int pf_dist;                        // cells ahead to prefetch into L2
    MsConst<typename Xv<XS>::T> c;
};

// Two values handled as one: the populations of a link and its opposite.
// FP32 pairs use the packed FP32 instructions (each half rounds as the scalar
// instruction does), which halves the arithmetic instructions of the step.
template <typename T>
struct Pk {
    T lo, hi;
    __device__ __forceinline__ static Pk make(T a, T b) { return Pk{a, b}; }
    __device__ __forceinline__ T low() const { return lo; }
    __device__ __forceinline__ T high() const { return hi; }
    __device__ __forceinline__ friend Pk operator+(Pk a, Pk b) { return Pk{a.lo + b.lo, a.hi + b.hi}; }
    __device__ __forceinline__ friend Pk operator*(Pk a, Pk b) { return Pk{a.lo * b.lo, a.hi * b.hi}; }
    __device__ __forceinline__ static Pk fma(Pk a, Pk b, Pk c) {
        return Pk{a.lo * b.lo + c.lo, a.hi * b.hi + c.hi};
    }
};
template <>
struct Pk<float> {
    unsigned long long v;
    __device__ __forceinline__ static Pk make(float a, float b) {
        Pk r;
        asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
        return r;
    }
    __device__ __forceinline__ float low() const {
        float a, b;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
        return a;
    }
    __device__ __forceinline__ float high() const {
        float a, b;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
        return b;
    }
    __device__ __forceinline__ friend Pk operator+(Pk a, Pk b) {
        Pk r;
        asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
        return r;
    }
    __device__ __forceinline__ friend Pk operator*(Pk a, Pk b) {
        Pk r;
        asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
        return r;
    }
    __device__ __forceinline__ static Pk fma(Pk a, Pk b, Pk c) {
        Pk r;
        asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
        return r;
    }
};

// Unit of row 0 of cell j in the tiled layout.
// Sources are counted from one tile before the first cell (index j + kTile,
// pointers one tile back), so that the step to the opposite link at a wall
// stays non-negative; 3 Q (S + kTile) < 2^32 (checked at create).
template <class L, typename P>
__device__ __forceinline__ uint32_t tile_off(int j) {
    return (uint32_t)j + (uint32_t)(j & ~(kTile - 1)) * (TileLay<L, P>::kRows - 1);
}

// A link's source, counted from one tile before the first cell: the cell
// whose X it exchanges with (the cell itself at a wall) and the unit to pull
// from less row(s, k) kTile (bounce-back folded in: the opposite link of the
// cell itself, one row on or back).
struct Source {
    uint32_t h;
    int x;
};

// Sources of a fluid cell from the 32-voxel windows of the rows (kNbRowMask
// of the tiled step).  code as in decode_neighbours; window (row, w) of a
// case: .x = fluid flags of voxels 16 w - 8 .. 16 w + 23 of the row (zero
// outside the grid), .y = kTile + the fluid index that the first fluid voxel
// at or after 16 w - 8 has (or would have).
template <class L, typename P>
__device__ __forceinline__ void row_sources(uint32_t code, const uint2* __restrict__ tab, int nx, int ny, int nz,
                                            int wpr, int i, Source (&src)[L::Q], bool& at_in, bool& at_out) {
    const bool pad = code == 0xFFFFFFFFu;   // padding cell between cases: walls all round
    if (pad) code = 0u;
    const int x = (int)(code & 2047u);
    const int y = (int)((code >> 11) & 1023u);
    const int z = (int)(code >> 21);
    const int b = (x & 15) + 8;
    const uint32_t below = (1u << b) - 1u;
    const int wx = x >> 4;
    const int ry[3] = {(y == 0 ? ny - 1 : y - 1) * wpr + wx, y * wpr + wx, (y == ny - 1 ? 0 : y + 1) * wpr + wx};
    const int plane = ny * wpr;
    const int rz[3] = {(z == 0 ? nz - 1 : z - 1) * plane, z * plane, (z == nz - 1 ? 0 : z + 1) * plane};
    i += kTile;
    const uint32_t own = tile_off<L, P>(i);
    at_in = x == 0 && !pad;
    at_out = x == nx - 1 && !pad;
#pragma unroll
    for (int dz = -1; dz <= 1; ++dz) {
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy) {
            if (!row_used<L>(dy, dz)) continue;
            const uint2 e = __ldg(tab + (L::DIM == 2 ? ry[dy + 1] : rz[dz + 1] + ry[dy + 1]));
            const int at = (int)e.y + __popc(e.x & below);     // index x has (or would have)
            const uint32_t bits = pad ? 0u : e.x >> (b - 1);   // fluid flags of x - 1, x, x + 1
#pragma unroll
            for (int k = 1; k < L::Q; ++k) {
                if (-L::e(k, 1) != dy || -L::e(k, 2) != dz) continue;
                const int dx = -L::e(k, 0);
                const bool fluid = bits & (dx < 0 ? 1u : (dx == 0 ? 2u : 4u));
                const int j = dx < 0 ? at - 1 : (dx == 0 ? at : at + (int)((bits >> 1) & 1u));
                src[k].h = fluid ? tile_off<L, P>(j) : own + (opp<L>(k) - k) * kTile;
                src[k].x = fluid ? j : i;
            }
        }
    }
}

// The same from the cell's row of the 32-bit table.
template <class L, typename P>
__device__ __forceinline__ void table_sources(const int* __restrict__ nbr, int i, Source (&src)[L::Q], bool& at_in,
                                              bool& at_out) {
    int nb[L::Q];
    load_neighbours<L>(nbr, i, nb);
    i += kTile;
    const uint32_t own = tile_off<L, P>(i);
    at_in = nb[1] == NB_INLET;      // links 1 and 2 pull from x - 1 and x + 1
    at_out = nb[2] == NB_OUTLET;
#pragma unroll
    for (int k = 1; k < L::Q; ++k) {
        const bool fluid = nb[k] >= 0;
        src[k].h = fluid ? tile_off<L, P>(nb[k] + kTile) : own + (opp<L>(k) - k) * kTile;
        src[k].x = fluid ? nb[k] + kTile : i;
    }
}

// The populations of link k of the three species from unit a (a source, rows
// from 0), as stored values.
template <class L, typename T, typename P>
__device__ __forceinline__ void load_link(const typename TileLay<L, P>::U* a, int k, T (&v)[3]) {
    using Lay = TileLay<L, P>;
    if constexpr (std::is_same<P, __half>::value) {
        const uint32_t w = a[Lay::row(0, k) * kTile];
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w));
        v[0] = f.x;
        v[1] = f.y;
        v[2] = Pop<T, P>::raw(reinterpret_cast<const __half*>(a + Lay::row(2, k) * kTile) + Lay::half(2, k));
    } else {
#pragma unroll
        for (int s = 0; s < 3; ++s) v[s] = Pop<T, P>::raw(a + Lay::row(s, k) * kTile);
    }
}

__device__ __forceinline__ uint32_t half_bits(__half2 h) { return *reinterpret_cast<const uint32_t*>(&h); }

template <class L, typename XS, typename P, typename NBT, int W, int MB>
__global__ void __launch_bounds__(W, MB) step_tile_kernel(const TileParams<XS, P> p) {
    using T = typename Xv<XS>::T;
    using XV = Xv<XS>;
    using PT = Pk<T>;
    static_assert(kTile % W == 0, "a block lies in a tile");
    using Lay = TileLay<L, P>;
    using U = typename Lay::U;
    constexpr bool kHalf = std::is_same<P, __half>::value;
    constexpr int Q = L::Q;
    constexpr int DIM = L::DIM;
    constexpr int NP = (Q - 1) / 2;          // link pairs (k, k + 1), opposite to each other
    constexpr T sc = T(Pop<T, P>::kStore);   // d, dX and the collision work in storage units (h * kStore)

    if (!p.side) grid_launch_next();
    const int i = blockIdx.x * W + threadIdx.x;
    const CaseBC<XS>& cb = p.cases[__ldg(p.blk_case + blockIdx.x / (kTile / W))];
    Source src[Q];
    bool at_in, at_out;
    if constexpr (std::is_same<NBT, RowMaskNb>::value)
        row_sources<L, P>(__ldg(p.cell_code + i), p.rowtab + cb.tab, cb.nx, cb.ny, cb.nz,
                       cb.wpr, i, src, at_in, at_out);
    else
        table_sources<L, P>(p.nbr32, i, src, at_in, at_out);
    grid_wait();
    if (p.side) grid_launch_next();

    const int64_t S = p.S;
    if (threadIdx.x < 4 && blockIdx.x % (kTile / W) == 0) {
        // the tile and the X rows that blocks a third of a wave later start from
        const int64_t j = (int64_t)blockIdx.x * W + p.pf_dist;   // a multiple of the tile
        if (j + kTile <= S) {
            if (threadIdx.x == 0)
                prefetch_bulk(reinterpret_cast<const U*>(p.hin) + j * Lay::kRows, Lay::kRows * kTile * sizeof(U));
            else
                prefetch_bulk(p.xin + (threadIdx.x - 1) * S + j, kTile * sizeof(XS));
        }
    }
    const XS* xh[3] = {p.xin, p.xin + S, p.xin + 2 * S};
    const uint32_t own = tile_off<L, P>(i);
    const U* hin = reinterpret_cast<const U*>(p.hin) - Lay::kRows * kTile;
    XV xo[3];
    T d0[3], g[3][DIM];
    PT d[3][NP];     // f_k(x) - w_k X_old(x) after streaming
#pragma unroll
    for (int s = 0; s < 3; ++s) xo[s] = XV::own_rows(xh[s], p.xin + (int64_t)(3 + s) * S, i);
    load_link<L, T, P>(reinterpret_cast<const U*>(p.hin) + own, 0, d0);
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        const int k = 1 + 2 * q;
        T ha[3], hb[3];
        load_link<L, T, P>(hin + src[k].h, k, ha);
        load_link<L, T, P>(hin + src[k + 1].h, k + 1, hb);
        const T w = T(weight<L>(k) * sc);
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const PT h = PT::make(ha[s], hb[s]);
            const T nx = -xo[s].exch_base();
            const PT dx = PT::make(xh[s][src[k].x - kTile], xh[s][src[k + 1].x - kTile]) + PT::make(nx, nx);
            d[s][q] = PT::fma(PT::make(w, w), dx, h);
            if (q < DIM) g[s][q] = dx.high() - dx.low();
        }
    }
    if (at_out) {   // Eq. 39: every link from beyond x = nx - 1 (the even link of a pair along x)
        constexpr T wx = T(weight_xplus<L>());
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const T qs = cb.qout[s] * sc;
#pragma unroll
            for (int q = 0; q < NP; ++q)
                if (L::e(1 + 2 * q, 0) == 1)
                    d[s][q] = PT::make(d[s][q].low(), d[s][q].high() - T(weight<L>(1 + 2 * q)) / wx * qs);
        }
    }
    if (at_in) {    // Eq. 36: f_k = (w_k + w_opp) X_in - f_opp (the odd link of a pair along x)
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const T din = cb.xbc[s].minus(xo[s]) * sc;
#pragma unroll
            for (int q = 0; q < NP; ++q)
                if (L::e(1 + 2 * q, 0) == 1)
                    d[s][q] = PT::make(T(2 * weight<L>(1 + 2 * q)) * din - d[s][q].high(), d[s][q].high());
        }
    }
    T X[3], dX[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        PT a = d[s][0];
#pragma unroll
        for (int q = 1; q < NP; ++q) a = a + d[s][q];
        dX[s] = d0[s] + (a.low() + a.high());
        // lagged gradient: central, one-sided along x at the inlet and outlet
        // (whose missing neighbour has difference 0)
#pragma unroll
        for (int b = 0; b < DIM; ++b) g[s][b] *= (b == 0 && (at_in || at_out)) ? T(1) : T(0.5);
        const XV xn = xo[s].plus(dX[s] * T(1.0 / sc));
        X[s] = xn.value();
        xn.store_rows(p.xout + s * S, p.xout + (3 + s) * S, i);
    }
    U* ho = reinterpret_cast<U*>(p.hout) + own;
    __half2 held[kHalf ? NP : 1];    // species 0, then pairs of species 2, until their units are complete
    __half held0;
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        T J[DIM], v[DIM], tau, xinv;
        ms_flux<T, DIM>(X, g, p.c, s, J);
        ms_relax<T, DIM>(X, g[s], J, p.c, s, tau, v, xinv);
        const T it = Arith<T>::div(T(1), tau);
        const T keep = T(1) - it;
        const T A = T(3) * sc * X[s] * it;
        // h* = keep (d - w dX) + w A (e . v); the rest population closes the
        // sum on the stored values
        PT vp[DIM];      // A v_a of a pair's links along +e_a and -e_a
#pragma unroll
        for (int b = 0; b < DIM; ++b) vp[b] = PT::make(A * v[b], -(A * v[b]));
        const PT keep2 = PT::make(keep, keep), ndX = PT::make(-dX[s], -dX[s]);
        PT rest = PT::make(T(0), T(0));
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            const int k = 1 + 2 * q;
            const PT w = PT::make(T(weight<L>(k)), T(weight<L>(k)));
            PT ev = PT::make(T(0), T(0));
            bool first = true;
#pragma unroll
            for (int b = 0; b < DIM; ++b) {
                if (L::e(k, b) == 0) continue;
                const PT t = L::e(k, b) == 1 ? vp[b] : PT::make(vp[b].high(), vp[b].low());
                ev = first ? t : ev + t;
                first = false;
            }
            const PT hk = PT::fma(PT::fma(w, ndX, d[s][q]), keep2, w * ev);
            if constexpr (kHalf) {
                const __half2 h2 = __floats2half2_rn(hk.low(), hk.high());
                const float2 r = __half22float2(h2);
                rest = rest + PT::make(r.x, r.y);
                if (s == 1) {
                    step_store(ho + Lay::row(0, k) * kTile, half_bits(__lows2half2(held[q], h2)));
                    step_store(ho + Lay::row(0, k + 1) * kTile, half_bits(__highs2half2(held[q], h2)));
                } else if (s == 2 && q % 2) {
                    step_store(ho + Lay::row(2, k) * kTile, half_bits(__lows2half2(held[q - 1], h2)));
                    step_store(ho + Lay::row(2, k + 1) * kTile, half_bits(__highs2half2(held[q - 1], h2)));
                } else {
                    held[q] = h2;
                }
            } else {
                const P q0 = Pop<T, P>::quant_raw(hk.low());
                const P q1 = Pop<T, P>::quant_raw(hk.high());
                rest = rest + PT::make(Pop<T, P>::dequant_raw(q0), Pop<T, P>::dequant_raw(q1));
                step_store(ho + Lay::row(s, k) * kTile, q0);
                step_store(ho + Lay::row(s, k + 1) * kTile, q1);
            }
        }
        const P q0 = Pop<T, P>::quant_raw(-(rest.low() + rest.high()));
        if constexpr (kHalf) {
            if (s == 0) {
                held0 = q0;
            } else if (s == 1) {
                step_store(ho + Lay::kRest * kTile, half_bits(__halves2half2(held0, q0)));
            } else if (NP % 2) {     // with the last pair of species 2
                step_store(ho + Lay::row(2, 0) * kTile, half_bits(__halves2half2(__low2half(held[NP - 1]), q0)));
                step_store(ho + (Lay::row(2, 0) + 1) * kTile, half_bits(__highs2half2(held[NP - 1], held[NP - 1])));
            } else {
                step_store(ho + Lay::row(2, 0) * kTile, half_bits(__halves2half2(q0, q0)));
            }
        } else {
            step_store(ho + Lay::row(s, 0) * kTile, q0);
        }
    }
}

}  // namespace lbms
