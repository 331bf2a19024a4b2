// lbm_tma_util.cuh -- device helpers shared by the shared-memory-staged step
// kernels: stencil orientation of each population, the bounded mbarrier wait,
// and the limited flux difference in scalar and packed float32-pair form.
#pragma once

#include "lbm_internal.h"

namespace lbm {
namespace {

__device__ __forceinline__ constexpr int tsgn_x(int q)
{
    return q < 8 ? ((q & 3) == 0 ? 1 : ((q & 3) == 2 ? -1 : 0)) : (((q & 3) == 0 || (q & 3) == 3) ? 1 : -1);
}
__device__ __forceinline__ constexpr int tsgn_y(int q)
{
    return q < 8 ? ((q & 3) == 1 ? 1 : ((q & 3) == 3 ? -1 : 0)) : (((q & 3) <= 1) ? 1 : -1);
}

// Waits on an mbarrier phase.  try_wait carries a suspend-time hint, so a waiting warp
// sleeps until the phase completes (or the hint runs out) instead of spinning on issue
// slots that the other warps need; the wait as a whole is bounded by the global timer.
constexpr unsigned kWaitHintNs = 20000;
constexpr unsigned long long kWaitLimitNs = 2000000000ull;   // 2 s

__device__ __forceinline__ bool mbar_try_wait(unsigned bar, unsigned phase)
{
    unsigned done;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done) : "r"(bar), "r"(phase), "r"(kWaitHintNs) : "memory");
    return done != 0;
}

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Bounded wait on phase `phase` of an mbarrier (true when the phase completed).
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned phase)
{
    if (mbar_try_wait(bar, phase)) return true;
    const unsigned long long t0 = global_ns();
    while (global_ns() - t0 < kWaitLimitNs)
        if (mbar_try_wait(bar, phase)) return true;
    return false;
}

// As mbar_wait, but gives up early once another warp of the CTA has raised `abort`.
__device__ __forceinline__ bool mbar_wait_or_abort(unsigned bar, unsigned phase, const volatile int *abort)
{
    if (mbar_try_wait(bar, phase)) return true;
    const unsigned long long t0 = global_ns();
    while (global_ns() - t0 < kWaitLimitNs) {
        if (mbar_try_wait(bar, phase)) return true;
        if (*abort) return false;
    }
    return false;
}

template <typename R, int Lim>
__device__ __forceinline__ R slope2(R a, R b)
{
    return Lim == 0 ? mc2(a, b) : (Lim == 1 ? R(2.0) * b : R(0.0));
}

// Programmatic dependent launch: a step kernel's CTAs may start while the previous launch of the
// stream drains, and wait here before they touch its results.  Every kernel of a chained launch waits,
// also one that reads nothing of the launch before it: the wait is what makes the results of all earlier
// launches visible to it, and its completion then stands for theirs.  A kernel that is launched so does not
// take its populations as __restrict__: until the wait is over the launch before it still writes them,
// and the qualifier would let the compiler read them through the non-coherent path, or above the wait.
// Functions called after the wait may (until the kernel ends nothing else writes what they read).
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Coordinate a read at v goes to along an axis of n cells: the wrapped cell past a periodic edge
// (kind 0), the edge cell past a zero-gradient one (1), else v itself.
__device__ __forceinline__ int ghost_source(int v, int n, int kind_lo, int kind_hi)
{
    if (v >= 0 && v < n) return v;
    const int kind = v < 0 ? kind_lo : kind_hi;
    if (kind == 1) return v < 0 ? 0 : n - 1;
    return kind == 0 ? ((v % n) + n) % n : v;
}

// Ghost cells of the tiles at an edge of the grid: periodic and zero-gradient edges are filled in
// the staged tile, with the values the ghost launch would have written; those of a
// fixed-equilibrium edge never change (lbm_create_ex fills them).  So no ghost launch precedes the
// step, but for walls in the float32 kernel and the float64 one of step_kernel 2 (the double-float
// kernels form them in the tile too: wall_fill).  One thread per ghost cell of the cross: the tile's
// columns in up to four ghost rows, its rows in up to four ghost columns.  The sources are interior
// cells, read from global memory while the tile copy is in flight; they replace the tile's ghost
// cells once it has landed.
// Measured per step, with the launches chained (launch_chained): 200 x 4 float64 20.5 -> 9.3 us,
// 256^2 float32 10.3 -> 6.2 us, 8192^2 float32 1.382 ms with its ghost launch -> 1.353 ms.
template <typename R>
struct TileElem { using T = double; static constexpr int N = NQ; };            // planes of a staged tile
template <>
struct TileElem<float> { using T = float2; static constexpr int N = NQ / 2; };

// Ghost cell k of a tile's cross: k < 128 in the ghost rows of the tile's columns, then in the ghost
// columns of its rows.
template <typename S>
struct GhostSlot {
    static constexpr int kSlots = 4 * kTmaTX + 4 * S::TR;
    bool row, in;              // in a ghost row (else column); within the staged tile and the grid
    int layer, edge;           // 0, 1: -1, -2; 2, 3: n, n + 1; x-lo, x-hi, y-lo, y-hi
    int along, g, at, fix;     // coordinate along the edge, across it; staged row or column; the other one
    template <typename PP>
    __device__ __forceinline__ GhostSlot(const PP &P, int k, int x0, int y0)
    {
        row = k < 4 * kTmaTX;
        const int j = row ? k : k - 4 * kTmaTX;
        layer = row ? j / kTmaTX : j / S::TR;
        along = row ? x0 + j % kTmaTX : y0 + j % S::TR;
        const int size = row ? P.ny : P.nx, first = row ? y0 : x0;
        g = layer < 2 ? -1 - layer : size + layer - 2;
        at = g - first + 2;
        fix = row ? along - x0 + S::HX : along - y0 + 2;
        edge = (row ? 2 : 0) + (layer >> 1);
        in = k < kSlots && at >= 0 && at < (row ? S::SH : S::SW) && along < (row ? P.nx : P.ny);
    }
    // offset in a staged plane of the cell at staged row (column) v across the edge
    __device__ __forceinline__ int offset(int v) const { return row ? v * S::SW + fix : fix * S::SW + v; }
};

template <typename R, typename S>
struct GhostFill {
    using E = typename TileElem<R>::T;
    static constexpr int N = TileElem<R>::N;
    static constexpr int kThreads = kTmaTX * S::TT;
    static constexpr int kRounds = (GhostSlot<S>::kSlots + kThreads - 1) / kThreads;
    E v[kRounds][N];
    int c[kRounds];            // cell of the staged tile, or -1

    // A tile whose staged cross reaches past an edge of the grid (uniform per CTA).
    template <typename PP>
    static __device__ __forceinline__ bool edge_tile(const PP &P, int x0, int y0)
    {
        return x0 == 0 || y0 == 0 || x0 + kTmaTX + S::HX > P.nx || y0 + S::TR + 2 > P.ny;
    }

    template <typename PP>
    __device__ __forceinline__ void load(const PP &P, const EdgeDev *edges, const R *fin, int x0, int y0, int tid)
    {
#pragma unroll
        for (int n = 0; n < kRounds; n++) {
            const GhostSlot<S> slot(P, tid + n * kThreads, x0, y0);
            c[n] = -1;
            if (!slot.in) continue;
            const EdgeDev &D = edges[slot.edge];
            if (D.kind > 1) continue;
            c[n] = slot.offset(slot.at);
            const int s = ghost_source(slot.g, slot.row ? P.ny : P.nx, D.kind, D.kind);
            const long long cell =
                (long long)((slot.row ? s : slot.along) + OY) * P.pitch + ((slot.row ? slot.along : s) + OX);
            const E *src = reinterpret_cast<const E *>(fin) + cell;
#pragma unroll
            for (int q = 0; q < N; q++) v[n][q] = src[q * P.plane];
        }
    }

    __device__ __forceinline__ void store(R *tile) const
    {
        E *t = reinterpret_cast<E *>(tile);
#pragma unroll
        for (int n = 0; n < kRounds; n++)
            if (c[n] >= 0) {
#pragma unroll
                for (int q = 0; q < N; q++) t[q * S::PL + c[n]] = v[n][q];
            }
    }
};

// ---- packed float32 pairs (Blackwell f32x2 arithmetic) -------------------
// Populations q and q + 4 (q = 0..3 axis shells 1 and 2, q = 8..11 diagonal shells 3 and 4)
// move in the same direction: their stencils have the same offsets and only the per-shell
// constants differ, so their convection runs as one float2 per pair.

// Batched launches: the grid of tile b (the largest k with first[k] <= b, a binary search on
// the parameter block, uniform across the CTA) and the tile's origin (grid k's tiles start at
// row y0[k]).
__device__ __forceinline__ int batch_tile(const TmaBatchArgs &A, int b, int tr, int &x0, int &y0)
{
    int lo = 0, hi = A.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (A.first[mid] <= b) lo = mid;
        else hi = mid - 1;
    }
    const int local = b - A.first[lo], nt = A.ntx[lo];
    const int ty = local / nt;
    x0 = (local - ty * nt) * kTmaTX;
    y0 = A.y0[lo] + ty * tr;
    return lo;
}

// Prologue of a batched tile CTA (thread 0): initialise the tile barrier, issue the copy of
// grid g's tile at (x0, y0) (tiles of TR rows; the x origin HX columns left of the tile's first
// interior column), and with ctas > 0 (resident CTAs per SM) prefetch into L2 the tile half a
// resident wave further down the launch.
template <int TR, int HX>
__device__ __forceinline__ void batch_issue(const TmaBatchArgs &A, int g, int x0, int y0, unsigned dst,
                                            unsigned bar_a, unsigned bytes, int ctas)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar_a) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar_a), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
                 " [%0], [%1, {%2, %3, %4}], [%5];"
                 ::"r"(dst), "l"(reinterpret_cast<unsigned long long>(&A.map[g])), "r"(x0 + OX - HX), "r"(y0),
                 "r"(0), "r"(bar_a) : "memory");
    if (ctas <= 0) return;
    unsigned nsm;
    asm("mov.u32 %0, %%nsmid;" : "=r"(nsm));
    const long long bn = (long long)blockIdx.x + (long long)ctas * nsm / 2;
    if (bn < A.first[A.n]) {
        int xn, yn;
        const int gn = batch_tile(A, (int)bn, TR, xn, yn);
        asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];"
                     ::"l"(reinterpret_cast<unsigned long long>(&A.map[gn])), "r"(xn + OX - HX), "r"(yn), "r"(0)
                     : "memory");
    }
}

template <int Lim>
__device__ __forceinline__ float2 slope2x2(float2 a, float2 b)
{
    if (Lim == 2) return f2(0.f, 0.f);
    if (Lim == 1) return mul2(b, f2(2.f, 2.f));
    // as mc2(float), per lane: t = +-min(|a|, |b|), positive when a and b agree in sign;
    // the result carries the sign of a + b and the magnitude min(4 max(t, 0), |a + b|)
    const float2 s = add2(a, b);
    float tx, ty;
    asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(tx) : "f"(a.x), "f"(b.x));
    asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(ty) : "f"(a.y), "f"(b.y));
    const float2 t4 = mul2(f2(tx, ty), f2(4.f, 4.f));
    const float mx = fmaxf(t4.x, 0.f), my = fmaxf(t4.y, 0.f);
    float rx, ry;
    asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(rx) : "f"(mx), "f"(s.x));
    asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(ry) : "f"(my), "f"(s.y));
    return f2(rx, ry);
}

// (F_out - F_in) of a pair in upwind order (f_{J-2s}, f_{J-s}, f_J, f_{J+s}); hh = h/2 per member.
template <int Lim>
__device__ __forceinline__ float2 flux_diff2(float2 fmm, float2 fm, float2 f0, float2 fp, float2 hh)
{
    const float2 d1 = sub2(f0, fm);
    if (Lim == 2) return d1;
    const float2 d2 = sub2(fp, f0);
    const float2 d0 = sub2(fm, fmm);
    return __ffma2_rn(hh, sub2(slope2x2<Lim>(d1, d2), slope2x2<Lim>(d0, d1)), d1);
}


}  // namespace
}  // namespace lbm
