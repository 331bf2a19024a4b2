// lbm_internal.h -- launchers shared between the host API and the kernel units.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <utility>

#include "lbm_dd.cuh"
#include "lbm_device.cuh"

namespace lbm {

// Tile of the fused step kernel: TX x TY cells, one thread per cell.
constexpr int kTX = 32;
constexpr int kTY = 8;
// Fixed grid of the first totals pass (the result is deterministic for a given size).
constexpr int kTotalsBlocks = 1024;   // partials buffer: at least one wave of totals blocks
constexpr int kTotalsThreads = 256;

// All launchers enqueue on `st` and return the launch status.
// `prec` is the storage precision (0 = float64 f, 1 = float32 deviation g).
// Initialisation of interior rows row0 .. row0+rows-1 from fields [rows][nx] (device or mapped host
// addresses of the first of those rows); a bad cell sets *bad.
cudaError_t launch_init(const Params &P, int prec, void *f, const double *rho, const double *u, const double *v,
                        const double *T, int row0, int rows, int *bad, cudaStream_t st);
// Whether the plain step with tiles of 32 x ty cells takes 16 lanes per cell (small float64 grids).
bool lane_step(const Params &P, int prec, int ty);
// Ghost cells of the edges in `edges` (bit e: x-lo, x-hi, y-lo, y-hi); lanes: float64 walls with 16
// lanes per cell.  chain: as in launch_kernel (k_wall is always chained).
constexpr int kAllEdges = 15;
cudaError_t launch_ghost(const Params &P, int prec, void *f, cudaStream_t st, int edges = kAllEdges, bool lanes = false,
                         bool chain = true);

// Launch of a kernel that calls grid_dependency_wait before it touches memory.  chain: its CTAs may start
// (barrier initialisation, parameter fetches) while the stream's previous launch drains; else once
// everything before it in the stream is complete.
template <typename... KArgs, typename... Args>
cudaError_t launch_kernel(bool chain, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                          Args &&...args)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = chain ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}
template <typename... KArgs, typename... Args>
cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args &&...args)
{
    return launch_kernel(true, kernel, grid, block, smem, st, std::forward<Args>(args)...);
}
// Plain fused step with tiles of 32 x ty cells (ty = 4, 8 or 16).
cudaError_t launch_step(const Params &P, int prec, const void *fin, void *fout, cudaStream_t st, int ty = kTY,
                        bool chain = true);
// log2 of the plain kernels' tile width for a grid nx columns wide (5 for nx >= 32, else the
// smallest power of two >= nx); the tile has (kTX * kTY) >> log rows.
int plain_log_tx(int nx);
// threads (= cells) per CTA and tile of the batched step kernel: float32 groups, float64 groups
constexpr int kBatchThreads = kTX * kTY;
constexpr int kBatchThreadsFp64 = 64;

// One grid of a batch: its two population buffers, which one holds the current step, and the
// flag its TMA-fed kernels raise when a copy wait runs out.
struct BatchGrid {
    void *buf[2];
    int *err;
    int cur;
    int pad;
};
// Batched ghost fill (grid index = blockIdx.y) and batched fused step over a tile list
// (int4 {grid, x0, y0, 0}); `phase` = 0 reads buf[cur], 1 reads buf[cur ^ 1].
cudaError_t launch_ghost_batch(const Params *Pall, const BatchGrid *G, int ngrids, int max_ghost, int prec,
                               int phase, bool chain, cudaStream_t st);
cudaError_t launch_step_batch(const Params *Pall, const BatchGrid *G, const int4 *tiles, int ntiles, int prec,
                              int limiter, int nt, int ctas, int phase, bool chain, cudaStream_t st);
cudaError_t launch_moments(const Params &P, int prec, const void *f, int row0, int rows,
                           double *rho, double *u, double *v, double *T, double *delta,
                           double *dstar, int *flag, cudaStream_t st);
cudaError_t launch_totals(const Params &P, int prec, const void *f, double *partial, double *out,
                          double scale, cudaStream_t st);
cudaError_t launch_pack(const Params &P, int prec, const void *f, int row0, int rows, double *out,
                        cudaStream_t st);
cudaError_t launch_unpack(const Params &P, int prec, void *f, int row0, int rows, const double *in,
                          cudaStream_t st);

// TMA-staged step kernel: tiles of kTmaTX columns by TmaShape<R>::TR rows,
// kTmaTX x TT threads, each thread owns KR consecutive rows of one column.
// float32: 4 warps and 32 x 16 tiles (four CTAs per SM, so four tile copies in
// flight); the staged flow velocity is (u_x, u_y) pairs and 1/rho is recomputed
// from the cell's own density.  float64: 8 warps and 32 x 32 tiles, u_x, u_y and
// 1/rho staged.
constexpr int kTmaTX = 32;
constexpr int kTmaTT = 8;
template <typename R>
struct TmaShape {
    static constexpr int TT = sizeof(R) == sizeof(float) ? 4 : 8;   // warps per CTA
    static constexpr int CTAS = sizeof(R) == sizeof(float) ? (TT == 4 ? 4 : (TT == 3 ? 5 : 7)) : 1;   // per SM
    static constexpr int KR = 4;                       // rows per thread
    static constexpr int TR = TT * KR;                 // tile rows
    static constexpr int HX = 2;                       // x halo (8-byte elements: 16-byte TMA origin)
    static constexpr int SW = kTmaTX + 2 * HX;         // staged row
    static constexpr int SH = TR + 4;                  // staged rows: y halo of 2
    static constexpr int PL = SW * SH;                 // staged plane (float32: plane of pairs, in pairs)
    static constexpr int UW = kTmaTX + 2, UH = TR + 2; // flow-velocity tile with its ring
    static constexpr size_t tile_bytes = sizeof(R) * NQ * PL;
    static constexpr size_t smem_bytes = tile_bytes + sizeof(R) * (sizeof(R) == sizeof(float) ? 2 : 3) * UW * UH;
};
constexpr int kMaxGridY = 65535;        // a launch's limit on gridDim.y and z
bool tma_supported(const Params &P, int prec);
// Tiles of the double-float float64 kernels: 32 columns by TR rows, TT warps, KR rows per thread,
// CTAS CTAs per SM.  ROLES: two warps per row, one for the collision and one for the convection.
template <int TT_, int KR_, int CTAS_, bool ROLES_ = false>
struct DdShape {
    static constexpr int TT = TT_, KR = KR_, CTAS = CTAS_;
    static constexpr bool ROLES = ROLES_;
    static constexpr int TR = ROLES ? TT / 2 : TT * KR;
    static constexpr int HX = 2;                       // x halo (8-byte elements: 16-byte TMA origin)
    static constexpr int SW = kTmaTX + 2 * HX;
    static constexpr int SH = TR + 4;
    static constexpr int PL = SW * SH;
    static constexpr int UW = kTmaTX + 2, UH = TR + 2;
    static constexpr size_t tile_bytes = sizeof(double) * NQ * PL;
    // shared memory: the staged tile, (u_x, u_y) on the tile plus its ring, and the x edge values
    // of its rows
    static constexpr size_t uv_off = tile_bytes;
    static constexpr size_t edge_off = uv_off + 16 * UW * UH;
    static constexpr size_t acc_off = edge_off + 2 * 16 * 6 * TR;            // ROLES: the collision terms
    static constexpr size_t smem_bytes = acc_off + (ROLES ? 16 * 8 * kTmaTX * TR : 0);
};
using DdWideShape = DdShape<8, 2, 2>;            // 32 x 16: the fewest instructions per cell
using DdMidShape = DdShape<8, 1, 2>;             // 32 x 8
using DdNarrowShape = DdShape<8, 1, 2, true>;    // 32 x 4: the shortest step of a tile
enum { kDdWide = 0, kDdMid = 1, kDdNarrow = 2, kDdShapes = 3 };
constexpr int kDdRows[kDdShapes] = {DdWideShape::TR, DdMidShape::TR, DdNarrowShape::TR};
// Whether a grid's staged boxes of a shape fit its buffers.
bool dd_shape_supported(const Params &P, int shape);
// Estimated duration (us) of a step of `tiles` tiles of a shape on sms SMs, for choosing between shapes: a
// fixed part, whole waves of two CTAs per SM, then the remainder at one or two per SM (which overlaps the
// whole waves' tail).  Fitted to periodic grids on 152 SMs (MC, Pr != 1; graph runs), measured us per step on
// 32 x 16 / 32 x 8 / 32 x 4 tiles: 161 x 97 18.9 / 11.1 / 8.1, 608 x 64 16.8 / 10.4 / 10.5, 256^2 16.8 / 15.5 /
// 19.0, 320^2 26.4 / 21.5 / 27.0, 380^2 29.4 / 28.3 / 37.1, 400^2 38.7 / 33.9 / 43.2, 608 x 256 27.3 / 27.7 /
// 36.5, 608 x 448 47.3 / 45.9 / 62.2, 608 x 512 50.1 / 52.1 / 71.7, 1023 x 517 82.8 / 86.9 / 121, 608 x 1280
// 117 / 124 / 172.  The choice is the fastest on each of the 27 grids measured.
double dd_shape_time(int shape, long long tiles, int sms);
static_assert(DdWideShape::CTAS * (DdWideShape::smem_bytes + 2048) <= 228 * 1024, "wide tiles per SM");
// Coefficients of the double-float kernels in the order of the population pairs (lane e of pair
// p belongs to shell 2p + e); the column of row 13 in pEy is negated, as the kernel forms that
// row negated.
struct CoefDD {
    dd2 hh[2], hhy[2], cr[2], cry[2];
    dd2 pA[2][2], pEx[2][3], pEy[2][3], pB1[2], pB2[2];
    dd2 q89, g4;
    dd b, inv_b, two_b2, six_b, b4, four_inv_b, ry, pad_;
};
static_assert(sizeof(CoefDD) % 16 == 0, "CoefDD is copied in 16-byte words");
// Batched TMA-staged steps over the tiles of up to kTmaBatchGrids grids of a batch group, one
// CTA per tile of kTmaTX x TmaShape<R>::TR cells: grid k owns the launch's tiles first[k] ..
// first[k+1] - 1, row by row from row y0[k], ntx[k] to a row.  A CTA finds its grid and tile from blockIdx
// and this parameter block alone, so that its tile copy is issued before any load from global
// memory; the host resolves each grid's input map, output buffer and error flag for the
// launch's buffer parity.  float32 (the tile kernel) and float64 in double-float arithmetic.
constexpr int kTmaBatchGrids = 128;
struct TmaBatchArgs {
    CUtensorMap map[kTmaBatchGrids];   // grid k's input buffer (box of TmaShape<R>)
    const void *in[kTmaBatchGrids];     // grid k's input buffer
    void *out[kTmaBatchGrids];          // grid k's output buffer
    int *err[kTmaBatchGrids];           // grid k's copy-wait flag
    int first[kTmaBatchGrids + 1];      // first[n] = tiles of the launch
    int ntx[kTmaBatchGrids];            // tiles per row of grid k
    int y0[kTmaBatchGrids];             // first row of grid k's tiles in this launch
    int n;                              // grids of the launch
};
// Per-grid block of a batched launch (global memory, one per grid in launch order): the
// geometry and the coefficients that the tile kernels read (C = Coef<float> or CoefDD); each
// CTA copies its grid's block to shared memory while its tile copy is in flight.
template <typename C>
struct TileGrid {
    int nx, ny, pitch, has_c9;
    long long plane;
    long long member;           // the grid's index in the group's Params table (its edges)
    C cf;
};
cudaError_t launch_step_tma_batch(const TmaBatchArgs &A, const TileGrid<Coef<float>> *tg, const Params *Pall, int limiter,
                                  bool chain, cudaStream_t st);
// shape: kDdWide, kDdMid or kDdNarrow (the grids' maps have its box); walls: some grid has one.
cudaError_t launch_step_dd_batch(const TmaBatchArgs &A, const TileGrid<CoefDD> *tg, const Params *Pall, int limiter, int shape, bool walls,
                                 bool chain, cudaStream_t st);
// Failure-path check of the bounded mbarrier waits (lbm_wait_selftest): *flag = 1 when the
// wait on a phase that nothing completes gave up at its limit; *ms = the kernel's duration.
cudaError_t wait_selftest(int *flag, float *ms);
// Opt the kernels that a context (a batch's groups of a limiter) launches in to their dynamic shared
// memory.
cudaError_t tma_prepare(int prec, int limiter);
cudaError_t tma_batch_prepare(int limiter);
// `tmap` points to the CUtensorMap of the input buffer fin (3-D: pitch x (ny+4) x 16).  The tiles fill
// the ghost cells of every edge but walls themselves, from the interior of fin.
cudaError_t launch_step_tma(const Params &P, int prec, const void *tmap, const void *fin, void *fout, int *err,
                            cudaStream_t st, bool chain = true);

// Persistent double-buffered TMA-staged kernel (float32): CTAs walk tiles of kTmaTX columns
// by TR rows round-robin with two tile buffers, so that the copy of the next tile overlaps
// the work on the current one; each thread owns KR rows of one column.
struct TmaPipeShape {
    static constexpr int KR = 2;
    static constexpr int TR = kTmaTT * KR;
    static constexpr int HX = 2;
    static constexpr int SW = kTmaTX + 2 * HX;
    static constexpr int SH = TR + 4;
    static constexpr int PL = SW * SH;                 // staged plane of pairs, in pairs
    static constexpr int UW = kTmaTX + 2, UH = TR + 2;
    static constexpr size_t buf_bytes = sizeof(float) * NQ * PL;
    static constexpr size_t smem_bytes = 2 * buf_bytes + sizeof(float) * 3 * UW * UH;
};
bool tma_pipe_supported(const Params &P);
cudaError_t tma_pipe_prepare();
// `tmap`: CUtensorMap of the input buffer with box SW x SH x 8 pair planes.
cudaError_t launch_step_tma_pipe(const Params &P, const void *tmap, void *fout, int *err, cudaStream_t st);

// Streaming step kernel: a CTA of WARPS warps owns a strip of W columns and walks down a
// share of its rows through a ring of SLOTS row slots; a slot holds all planes of one row
// as two copies of BW columns (half strip + 4 halo columns on each side).  Sizes in
// elements of R (float32: 8 planes of pairs = 16 floats per column).
template <typename R>
struct StreamShape {
    static constexpr int WARPS = 8;
    static constexpr int W = 32 * WARPS;               // strip width
    static constexpr int BW = W / 2 + 8;               // columns per copy
    static constexpr int HALF = NQ * BW;               // elements per copy
    static constexpr int ROW = 2 * HALF;               // elements per slot
    static constexpr int SLOTS = 6;
    static constexpr unsigned copy_bytes = HALF * sizeof(R);
    static constexpr size_t smem_bytes = sizeof(R) * (size_t)SLOTS * ROW;
};
bool stream_supported(const Params &P);
cudaError_t stream_prepare();
// `tmap` points to the CUtensorMap of the input buffer with box BW x 1 x 16.
cudaError_t launch_step_stream(const Params &P, int prec, const void *tmap, void *fout, int *err, cudaStream_t st);

// Float64-mode step in double-float arithmetic on the float32 pipe (step_kernel 8, 9), on tiles of
// `shape`, `tmap` with its box; `coef` is the CoefDD of the context (coef_dd).  Ghost cells as in
// launch_step_tma.  chain: as in launch_kernel; rows: the first rows only (0: all), a multiple of the
// shape's.
void coef_dd(const Params &P, CoefDD *out);
// The kernels of one shape (lbm_step_dd.cuh).
template <typename S>
struct DdOps {
    static cudaError_t launch(const Params &P, const CoefDD &C, const CUtensorMap &tm, const double *a, double *b, int *err,
                              bool chain, int rows, cudaStream_t st);
    static cudaError_t launch_batch(const TmaBatchArgs &A, const TileGrid<CoefDD> *tg, const Params *Pall, int limiter,
                                    bool walls, bool chain, cudaStream_t st);
    static cudaError_t prepare(const Params &P);
    static cudaError_t prepare_batch(int limiter, bool walls);
};
extern template struct DdOps<DdWideShape>;
extern template struct DdOps<DdMidShape>;
extern template struct DdOps<DdNarrowShape>;
cudaError_t dd_prepare(const Params &P);
cudaError_t dd_batch_prepare(int limiter, bool walls);
cudaError_t launch_step_dd(const Params &P, const void *coef, const void *tmap, const void *fin, void *fout,
                           int *err, cudaStream_t st, int shape, bool chain = true, int rows = 0);

// Sustained float64 FMA rate of the current device in FLOP/s (FMA = 2).
cudaError_t measure_fp64_fma(double *flops);

}  // namespace lbm
