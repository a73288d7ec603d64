// Internal interface between the C ABI (lbms_capi.cu) and the kernel
// launchers (lbms_launch.cu).
#pragma once

#include <cstddef>
#include <cstdint>
#include <vector>
#include <cuda_runtime.h>

struct lbms_ctx;

namespace lbms {

constexpr int kCaseOutSlots = 16;      // doubles per case: residual sums (10) | boundary sums (6)

// Step-kernel variants the autotuner chooses from: (cells per block, minimum
// resident blocks per SM for the register budget, how neighbours are found,
// one thread per cell for all species instead of one per (cell, species)).
// Neighbours: kNbIndex32 reads a row of 32-bit fluid indices per cell,
// kNbOffset16 a row of 16-bit offsets, kNbRowMask decodes them from per-row
// fluid bitmasks and a 4-byte coordinate per cell (no per-link table).
enum { kNbIndex32 = 0, kNbOffset16 = 1, kNbRowMask = 2 };
constexpr int kStepVariants = 10;
constexpr int kVariantCells[kStepVariants] = {32, 32, 64, 32, 32, 64, 64, 32, 64, 32};
constexpr int kVariantMinBlocks[kStepVariants] = {8, 6, 4, 8, 6, 4, 8, 16, 8, 16};
constexpr int kVariantNb[kStepVariants] = {kNbIndex32,  kNbIndex32, kNbIndex32, kNbOffset16, kNbOffset16,
                                           kNbOffset16, kNbIndex32, kNbIndex32, kNbRowMask,  kNbRowMask};
constexpr int kVariantPerCell[kStepVariants] = {0, 0, 0, 0, 0, 0, 1, 1, 1, 1};

// The default step (lbms_step_tile.cuh): cells per tile of its population
// layout and per block, the variant whose block -> case table it shares, how
// many cells per SM ahead of a block it prefetches, and the blocks per SM its
// registers are budgeted for.  Measured on the 256x128x128 anode (1.69 M fluid
// cells, us per step), blocks per SM 5 / 6 / 8 / 9 / 10 / 12: FP32 151 / 151 /
// 143 / 153 / 140 / 191, FP64 2231 / 2253 / 2297 / 2306 / 2306 / 2308, FP16 at
// 8 / 9 / 10 / 12: 105 / 104 / 101 / 125; 2-D FP32 (1.22 M cells) 59 up to 10,
// 56.5 at 12, FP16 44.8 at any.  Prefetch none / 16 / 24 / 48 thousand cells
// ahead: FP32 155 / 144 / 143 / 145, FP16 (a 16-bit row per population) 122 /
// 113 / 112 / 113.
constexpr int kTile = 64;
constexpr int kTileBlkCase = 2;
constexpr int kTilePrefetch = 160;      // 24,320 cells on 152 SMs
constexpr int tile_min_blocks(int dim, int precision) {
    return dim == 2 ? (precision == 1 ? 12 : 8) : (precision == 0 ? 5 : 10);
}
// Blocks of a tile that its registers let an SM hold (FP64 in 3-D: 6 of 168
// registers a thread, though 5 are asked for).
constexpr int tile_resident(int dim, int precision) {
    return dim == 2 ? (precision == 0 ? 8 : 12) : (precision == 0 ? 6 : 10);
}
// FP64 in 3-D where a second wave of such blocks would be less than half full
// takes blocks of half a tile instead, 20 an SM with 96 registers a thread, all
// of them at once: 60 k cells 107 -> 95 us, 67 k 107 -> 99, but 55 k (one wave) 80
// -> 83, 74 k 107 -> 110 and 1.7 M 2230 -> 2300 us (16 an SM), from its spills.
constexpr int kFineCells = kTile / 2, kFineMinBlocks = 20;

// Steps of handles that do not fill the GPU (lbms_step_small.cuh): many steps
// of a block per case of at most 64, 128 or 320 cells, or a launch a step.  The
// rules stand in lbms_launch_small.cu.
enum { kNotSmall = 0, kBlock64, kBlock128, kBlock320, kSmall };
constexpr int kSmallCells[] = {0, 64, 128, 320, 32};        // cells per block of each
constexpr int kSmallMinBlocks[] = {0, 1, 1, 1, 4};          // and blocks per SM its registers are budgeted for
constexpr int kBlockSteps = 65536;   // steps of one launch at most

// Limits of the per-cell coordinate word of kNbRowMask (x | y << 11 | z << 21).
constexpr int kRowMaskMaxNx = 2048, kRowMaskMaxNy = 1024, kRowMaskMaxNz = 2048;

struct DevBuffers {
    void* f[2] = {nullptr, nullptr};   // non-equilibrium populations h = f* - w X, [3][Q][S]
    void* X[2] = {nullptr, nullptr};   // mole fractions (double or double-float blocks)
    double* snap = nullptr;            // residual snapshot, [3][S]
    int* nbr = nullptr;                // [S][nb_width]
    int16_t* nbr16 = nullptr;          // [S][nb16_width] offsets, when they all fit (else null)
    uint32_t* cell_code = nullptr;     // [S] x | y << 11 | z << 21 of each fluid cell (kNbRowMask; else null)
    uint4* rowtab = nullptr;           // per case [rows][words]: 64-bit fluid window + index (kNbRowMask); with
                                       // Launch::windows16 uint2 windows of 32 voxels (lbms_step_tile.cuh)
    int* rows = nullptr;               // [3][total rows]: x = 0, x = 1, x = nx-1 cell of each row (-1 if solid)
    int2* case_rows = nullptr;         // [cases]: first row, row count
    void* cases = nullptr;             // [cases] CaseBC<XS> (inlet values, outlet flux, range)
    int* blk_case[kStepVariants] = {};  // step-kernel block -> case
    int2* segs = nullptr;              // [segments]: first cell, cell count (reduction segments)
    int2* case_segs = nullptr;         // [cases]: first segment, segment count
    int* seg_case = nullptr;           // [segments]: case of each segment
    double* partials = nullptr;        // [segments][10]
    double* extrap = nullptr;          // [3][S] X of the last extrapolation check (lazy)
    double* coef = nullptr;            // [cases] extrapolation factors
    double* rre_ring = nullptr;        // [order + 1][3][S] X snapshots of a reduced-rank extrapolation cycle (lazy)
    double* rre_partials = nullptr;    // [segments][order (order + 1) / 2] Gram partials (lazy)
    double* rre_out = nullptr;         // [cases][order (order + 1) / 2] Gram matrices (lazy)
    double* rre_coef = nullptr;        // [cases][order] coefficients of the differences (lazy)
    double* case_out = nullptr;        // [cases][10] residual sums, then [cases][6] boundary sums
    double* case_out_host = nullptr;   // pinned: the residual sums again, written by the kernel
    unsigned int* seg_done = nullptr;  // [cases] finished segments of the running reduction, 0 between reductions
    void* fields = nullptr;            // [3 + 3 dim][S] of tau and u (lazy), FP64 or FP32
    double* dense = nullptr;           // X on the dense grid of the largest case (lazy)
};

struct Launch {
    int dim = 2;
    int precision = 1;                 // 0 = FP64, 1 = FP32, 2 = FP16 populations / FP32 compute
    int64_t S = 0;                     // padded row stride (elements), >= ncells
    int ncells = 0;                    // end of the last case's range (index space of the kernels)
    int n_cases = 1;
    int total_rows = 0;
    int n_segs = 0;
    int nblk[kStepVariants] = {};
    int variant = 0;                   // chosen step-kernel tile shape
    bool tiled = false;                // the step of lbms_step_tile.cuh and its population layout, instead of a variant
    int small = kNotSmall;             // which of the small handles' steps, instead of a variant
    bool fine = false;                 // the tiled step's blocks are half tiles
    bool windows16() const { return tiled || small != kNotSmall; }   // the row table's form (no 16-bit table then)
    int cur = 0;                       // lattice holding the latest post-collision state
    DevBuffers b;
    double D12 = 1, D13 = 1, D23 = 1;  // lattice binary diffusivities
    double stoich[3] = {-1, 1, 0};     // nu_i of the electrode reaction (Eq. 38)
    double tau_min = 1.0, tau_max = 5.0;
    int drift = 1;
    int grad_forward = 0;              // Eq. 35 forward difference along x only
    int outlet_extrap = 0;             // extrapolated wet-node outlet (per-cell step kernel only)
    int sm_count = 152;
};

// Host image of one case's boundary data; the launcher converts it to the
// device CaseBC layout of the precision in use.
struct CaseHostBC {
    double xin[3];
    double q[3];
    int base;
    int nf;
    int nx, ny, nz;     // grid of the case
    int wpr;            // row-table entries per (y, z) row: ceil(nx / 32)
    int tab;            // first row-table entry of the case
};

// cudaMalloc that leaves no error behind: a refused allocation is the caller's
// to report or to do without, and must not come back from the
// cudaGetLastError of a later launch.  *p is null then.
template <typename T>
inline cudaError_t dev_malloc(T** p, size_t bytes) {
    const cudaError_t e = cudaMalloc(reinterpret_cast<void**>(p), bytes);
    if (e != cudaSuccess) {
        *p = nullptr;
        (void)cudaGetLastError();
    }
    return e;
}

// First touch of freshly mapped host memory by the CPU: a device copy into
// untouched 64 KB pages takes a fault of some 25 us for each.
inline void touch_pages(double* p, int64_t n) {
    volatile double* v = p;
    for (int64_t i = 0; i < n; i += 512) v[i] = 0.0;
    if (n > 0) v[n - 1] = 0.0;
}

size_t pop_size(int precision);    // bytes per stored population
size_t x_size(int precision);      // bytes per stored mole fraction
size_t field_size(int precision);  // bytes per tau / u value of the fields kernel
size_t case_bc_size(int precision);
void pack_case_bc(int precision, const CaseHostBC& h, void* dst);  // host-side CaseBC image

cudaError_t launch_step(const Launch& L, cudaStream_t st);
cudaError_t launch_step_variant(const Launch& L, int variant, cudaStream_t st);
// the same with the grad_forward / outlet_extrap options compiled in
cudaError_t launch_step_variant_literal(const Launch& L, int variant, cudaStream_t st);
// the default step (lbms_step_tile.cuh); needs L.tiled; bytes of a cell's populations in its layout
size_t tile_cell_bytes(int dim, int precision);
bool tile_fine(const Launch& L);   // whether it takes kFineCells a block; L.ncells and sm_count are set
cudaError_t launch_step_tile(const Launch& L, cudaStream_t st);
// the step for a handle whose largest case has max_nf cells, or kNotSmall;
// L.ncells, n_cases and sm_count are set
int choose_small(const Launch& L, int max_nf);
cudaError_t launch_step_small(const Launch& L, cudaStream_t st);   // kSmall
// n <= kBlockSteps steps of a kBlock* handle; cur turns n & 1 times
cudaError_t launch_steps_block(const Launch& L, int n, cudaStream_t st);
cudaError_t launch_init(const Launch& L, int first, int count, cudaStream_t st);
cudaError_t launch_fields(const Launch& L, cudaStream_t st);
// X of species s, s + 1, ... (`count` of them) of a case's cells [base, base + nf)
// on its dense grid of N cells, dense[species - s][N] (coordinates from
// cell_code; solid voxels are not written), and back
cudaError_t launch_to_dense(const Launch& L, int base, int nf, int nx, int ny, int64_t N, int s, int count,
                            double* dense, cudaStream_t st);
cudaError_t launch_from_dense(const Launch& L, int base, int nf, int nx, int ny, int64_t N, int s, int count,
                              const double* dense, cudaStream_t st);
// X of a case's cells from [3][nf] values
cudaError_t launch_put_x(const Launch& L, int base, int nf, const double* values, cudaStream_t st);
cudaError_t launch_case_residuals(const Launch& L, int update, cudaStream_t st);
cudaError_t launch_case_boundary(const Launch& L, cudaStream_t st);
// per-case sums of (X - E)^2 etc. into case_out[c * 10 + v], E unchanged
cudaError_t launch_case_extrap_norms(const Launch& L, cudaStream_t st);
cudaError_t launch_extrapolate(const Launch& L, cudaStream_t st);
// reduced-rank extrapolation of order M (2..6): snapshot into slot, Gram
// matrices of the M differences into rre_out, and the update from rre_coef
cudaError_t launch_rre_snapshot(const Launch& L, int slot, cudaStream_t st);
cudaError_t launch_rre_gram(const Launch& L, int order, cudaStream_t st);
cudaError_t launch_rre_apply(const Launch& L, int order, cudaStream_t st);
constexpr int kRreMaxOrder = 6;

// Neighbour tables of one case built on the device from its dense
// fluid-index map (index_of[cell] = index in the case or -1) and its fluid
// cell list; nbr16 may be null.  counts[0..1] accumulate the fluid links and
// the links that do not fit the 16-bit table.
cudaError_t launch_build_neighbours(int dim, const int64_t* fluid_cell, const int* index_of, int nf, int base, int nx,
                                    int ny, int nz, int periodic_x, int* nbr, int16_t* nbr16,
                                    unsigned long long* counts, cudaStream_t st);
cudaError_t launch_fill16(int16_t* p, int64_t n, int16_t v, cudaStream_t st);

// Readies the tcgen05 kernels (lbms_umma.cu); the error if the device or driver lacks what they need.
cudaError_t umma_init();

// Products of the two networks (lbms_conv.cu).  The U-Net's activations are BF16
// rows [row][C] of a zero-halo layout: volumes of X x Y x Z voxels in Xp x Yp x Zp
// rows each, R rows in all.
struct RowLayout {
    int X = 0, Y = 0, Z = 0, Xp = 1, Yp = 1, Zp = 1;
    long long R = 0;
};

// What becomes of the product's FP32 accumulators acc[r][n] (kept in TMEM):
enum ConvOut {
    kOutRelu,       // out[r][n] = BF16(relu(acc + bias[n])) on interior rows (taps = 1: all rows), 0 elsewhere;
                    //   with cat, the first w columns also to cat[r][cat_off + n], and 0 to all of cat[r] elsewhere
    kOutReluBack,   // out[r][n] = BF16(act[r][n] > 0 ? acc : 0), gb[n] += the column sums (before rounding)
    kOutStore,      // P[r][n] = acc
    kOutSplit,      // gradient of a concatenation of two w-wide halves, interior rows: columns [0, w) as BF16 to
                    //   G[parent][t Cg + n] of the coarser layout (t = 4 dz + 2 dy + dx) and their sums to gb[n];
                    //   columns [w, 2 w) to P[r][n - w] (stride Cg), which is 0 on other rows
    kOutUp,         // transposed 2x2x2 convolution: column t Cg + n of an interior row, plus bias[n], to the row's
                    //   child t of the finer layout, cat[child][n] (n < w)
    kOutHead        // Y = acc + bias (3 columns): Y[r][4] if given; against T [r][4] = (targets, mask), if given,
                    //   out[r][n] = BF16(grad_scale (Y - T) mask) (0 for n >= 3), its column sums (FP32 over a
                    //   thread's rows, FP64 over the threads) to gb and loss_scale sum((Y - T)^2 mask^2) into loss
};
struct ConvEpilogue {
    const float* bias = nullptr;
    void* out = nullptr;          // BF16 [rows][N]
    const void* act = nullptr;    // BF16 [rows][N]
    void* cat = nullptr;          // BF16 [rows][cat_ld]
    int cat_ld = 0, cat_off = 0, w = 0;
    void* G = nullptr;            // BF16 [coarse rows][8 Cg]
    int Cg = 0;
    float* P = nullptr;
    float* gb = nullptr;
    const float* T = nullptr;
    float* Y = nullptr;
    double* loss = nullptr;       // kOutHead: loss and the three column sums, 0 before
    unsigned int* done = nullptr; // kOutHead: 0 before
    float grad_scale = 0.0f;
    double loss_scale = 0.0;
    RowLayout g;                  // the product's rows
    RowLayout other;              // kOutSplit: the coarser layout; kOutUp: the finer one
};

// acc[r][n] = sum_t sum_c x[r + off[t]][c] W[n][t C + c] over x [rows][C]
// (zeros outside) and W [N][taps C]: a 3x3x3 convolution or its input
// gradient (taps = 27; the three offsets of a (dz, dy) row consecutive) or a
// plain product (taps = 1, off[0] = 0).  *err is raised if a wait in the
// kernel timed out.  cudaErrorInvalidValue for shapes that are not built; plain
// products into kOutRelu, kOutReluBack and kOutHead take every C and N that are
// multiples of 64 (kOutHead: N = 64).
struct ConvJob {
    const void* x = nullptr;
    const void* W = nullptr;
    int rows = 0, C = 0, N = 0, taps = 27;
    int off[27] = {};
    ConvOut kind = kOutRelu;
    ConvEpilogue ep;
};
cudaError_t conv_init();
cudaError_t umma_conv(const ConvJob& j, unsigned int* err, cudaStream_t st);

// P[z][t C + c][n] = sum over the rows r of chunk z of x[r + off[t]][c]
// dz[r][n] (taps = 27, off[3 g + d] = off[3 g] + d), or P[z][c][n] with
// taps = 1; x [rows][C], dz [rows][N], S chunks of rows / S (a multiple of 64)
// rows each.  With taps = 27 the last two rows of dz are zero, and at most 64
// channels on either side a chunk takes the products whose x row off[3 g] on
// from dz lies in it.
struct WgradJob {
    const void* x = nullptr;
    const void* dz = nullptr;
    int rows = 0, C = 0, N = 0, S = 1, taps = 27;
    int off[27] = {};
    float* P = nullptr;
};
cudaError_t umma_wgrad(const WgradJob& j, unsigned int* err, cudaStream_t st);

// Read-only view of one case of a handle (for the warm-start network).
struct CaseView {
    int nx, ny, nz;
    int64_t N;                    // cells of the dense grid
    int nf;                       // fluid cells
    const int64_t* fluid_cell;    // dense index of each fluid cell (host)
    const uint32_t* cell_code;    // their coordinates x | y << 11 | z << 21 (device), or null
    double x_in[3];
    double current;               // A/cm2
    bool periodic_x;
    bool has_bc;
};
// False if k is out of range.
bool case_view(const lbms_ctx* c, int k, CaseView* v);
// The initial profile of Section 4.1 for case k at its current boundary
// data, prof[s * nx + x]; false if it goes negative (or the box is periodic
// in x).
bool case_profile_1d(const lbms_ctx* c, int k, std::vector<double>& prof);

// Restarts case k from X [3][nf] in device memory (f = w X), as
// lbms_batch_set_fields does from a host field; the values must be complete.
int case_restart_device(lbms_ctx* c, int k, const double* X);

}  // namespace lbms
