// lbm_step_dd.cuh -- float64-mode fused step in double-float arithmetic (sm_103a).
//
// The populations are float64 in HBM, as in the other float64 kernels; the arithmetic of the
// step runs on the float32 pipe in double-float form (lbm_dd.cuh), which GB300 executes far
// faster than float64.  Layout and staging follow the TMA-staged tile kernel: one CTA owns a
// tile of 32 columns x TR rows and one elected thread brings all 16 float64 planes of the
// tile plus its stencil halo into shared memory with one tensor copy (bounded mbarrier wait);
// then
//   split    every staged value becomes hi + lo in place (8 bytes either way), the hi parts of the
//            population pair (q, q + 4) together in plane q, the lo parts in plane q + 4;
//   phase 1  per thread the residuals f_hat - f_hat^eq of its cells (Eq. 3 in the shell basis:
//            all of the collision but the energy-flux correction, which needs grad u) and their
//            flow velocity; the velocity of the ring; the face differences and slopes one column
//            outside the tile;
//   phase 2  the correction and the relaxation of the residuals, then pair by pair the limited x
//            and y convection
//            (Sec. III; each x face difference and slope is formed once, by the lane of its column,
//            and passed to the neighbour lane by a shuffle; y slopes from a window sliding down the
//            thread's column), the forward-Euler update, and one float64 store per population (the
//            double-float result rounded to float64).
// The formulas are those of the float64 kernels, operation for operation; each rounds at
// about 2^-47 instead of 2^-53, so results agree with the float64 kernels and the oracle to a
// few parts in 1e14 per step.
//
// What bounds it: the float32 pipe, about 3540 lane operations a cell (28 cycles of an SM at 128
// lanes), then the fixed latency of the double-float chains and the float64 pipe that rounds the
// results (48 operations a cell, 24 cycles).  Measured on 2048 x 2048 (MC, Pr != 1; the step
// kernel, CUDA events), starting from scalar operations with one 8-warp CTA per SM on 32 x 32
// tiles (245 registers a thread, issue slots 57% busy, most stalls on fixed latencies):
//   0.981 ms  start
//   0.940     the same operations on population pairs with f32x2 instructions (5263 -> 3600 thread
//             instructions a cell; the latencies of two warps per scheduler remain)
//   0.720     collision first, then convection pair by pair, so that 128 registers a thread do and
//             two 8-warp CTAs on 32 x 16 tiles run per SM (their phases overlap)
//   0.681     the tile of the CTA half a resident wave later prefetched into L2; the populations
//             read again after the collision instead of kept
//   0.643     the split in half the integer operations, Fast2Sum where the order is known
//   0.587     the residuals formed in phase 1 and kept in registers, so that no cell's shells are
//             formed twice and the ring is left out where s8 = s5 (3501 -> 3188
//             thread instructions a cell)
//   0.557     the pairs that move along both axes first; results stored evict-first
//   0.562     the slope set to zero where differences disagree in sign (mc2n)
// Other shapes (warps x rows per thread, CTAs per SM), same code: 16 x 2, one CTA 0.807 ms; 12 x 2,
// one CTA 0.843; 5 x 3, two CTAs 1.09; 4 x 4, two CTAs 1.31 (the unrolled rows spill), against 0.643;
// 6 x 2, two CTAs 0.677; 7 x 2, two CTAs 0.665; 10 x 2, one CTA 0.885, against 0.587.
// At their 128 registers the MC kernels on 32 x 16 tiles spill 8 to 24 bytes a thread, the batched ones on
// those tiles (coefficients in shared memory) 88 to 190.  The results are bit for bit those of scalar operations.
#pragma once

#include <cuda.h>

#include "lbm_dd.cuh"
#include "lbm_internal.h"
#include "lbm_tma_util.cuh"

namespace lbm {

namespace {

// ---- constants in double-float ------------------------------------------------------------
// Velocity-set constants that float32 does not hold exactly (Sec. II, Appendix A), split at
// compile time.
__host__ __device__ constexpr float hi_of(double x) { return (float)x; }
__host__ __device__ constexpr float lo_of(double x) { return (float)(x - (double)(float)x); }
__device__ __forceinline__ dd2 both(double x) { return dd2{f2(hi_of(x), hi_of(x)), f2(lo_of(x), lo_of(x))}; }

// ---- shells on population pairs (as shells2_of of the float32 path) ------------------------
struct ShellsDD { dd2 S[2], X[2], Y[2], Q[2]; };   // [0]: shells 1, 2; [1]: shells 3, 4

__device__ __forceinline__ ShellsDD shells_dd(const dd2 *fp)
{
    ShellsDD s;
    {
        const dd2 a = fp[0] + fp[2], b = fp[1] + fp[3];
        s.S[0] = a + b;
        s.Q[0] = a - b;
        s.X[0] = fp[0] - fp[2];
        s.Y[0] = fp[1] - fp[3];
    }
    {
        const dd2 a = fp[4] + fp[6], b = fp[5] + fp[7];
        const dd2 c = fp[4] - fp[6], d = fp[5] - fp[7];
        s.S[1] = a + b;
        s.Q[1] = a - b;
        s.X[1] = c - d;
        s.Y[1] = c + d;
    }
    return s;
}

__device__ __forceinline__ void unbutterfly_dd_axis(dd2 S, dd2 X, dd2 Y, dd2 Q, dd2 *p)
{
    const dd2 a = S + Q, b = S - Q;
    p[0] = a + X;
    p[2] = a - X;
    p[1] = b + Y;
    p[3] = b - Y;
}

__device__ __forceinline__ void unbutterfly_dd_diag(dd2 S, dd2 X, dd2 Y, dd2 Q, dd2 *p)
{
    const dd2 a = S + Q, b = S - Q, c = X + Y, d = X - Y;
    p[0] = a + c;
    p[2] = a - c;
    p[1] = b - d;
    p[3] = b + d;
}

// The staged tile after the split: population pair pr of the cell at offset c is
// (hi of q, hi of q + 4) in plane q = pair_q(pr) and (lo of q, lo of q + 4) in plane q + 4, so
// every access is 8 bytes wide and free of bank conflicts.
template <typename S>
__device__ __forceinline__ dd2 tile_pair(const float2 *t, int pr, int c)
{
    return dd2{t[pair_q(pr) * S::PL + c], t[(pair_q(pr) + 4) * S::PL + c]};
}

__device__ __forceinline__ float4 quad(dd2 a) { return make_float4(a.hi.x, a.hi.y, a.lo.x, a.lo.y); }
__device__ __forceinline__ dd2 unquad(float4 v) { return dd2{f2(v.x, v.y), f2(v.z, v.w)}; }

// (j_x, j_y) over the shells 1 .. 4.
__device__ __forceinline__ dd2 flux_dd(dd2 X0, dd2 X1, dd2 Y0, dd2 Y1)
{
    return ((firsts(X0, Y0) + seconds(X0, Y0) * f2(6.0f, 6.0f)) + both(kD3) * firsts(X1, Y1)) +
           both(kD4) * seconds(X1, Y1);
}

// (u_x, u_y) of the staged cell at offset c.
template <typename S>
__device__ __forceinline__ dd2 velocity_dd(const float2 *t, int c)
{
    dd2 fp[8];
#pragma unroll
    for (int pr = 0; pr < 8; pr++) fp[pr] = tile_pair<S>(t, pr, c);
    const dd2 S0 = (fp[0] + fp[2]) + (fp[1] + fp[3]), S1 = (fp[4] + fp[6]) + (fp[5] + fp[7]);
    const dd2 cc = fp[4] - fp[6], dm = fp[5] - fp[7];
    const dd rho = sum_lanes(S0) + sum_lanes(S1);
    return flux_dd(fp[0] - fp[2], cc - dm, fp[1] - fp[3], cc + dm) * bcast(recip(rho));
}

// f_hat - f_hat^eq of a cell (rows 5..16, in the pairs the inverse blocks take), its velocity and
// pressure: all of the collision that needs the cell's own populations only.
struct ResidualDD {
    dd2 d413, d78, d910, d1112, d515, d614, u;
    dd P;
};

// Float64 mode (zero reference state): the formulas of collide<double, false> on shell pairs, with
// the x and y rows as pairs.
__device__ __forceinline__ ResidualDD residual_dd(const CoefDD &C, const dd2 *fp)
{
    const ShellsDD s = shells_dd(fp);
    ResidualDD r;
    const dd ir = recip(sum_lanes(s.S[0]) + sum_lanes(s.S[1]));
    const dd2 j = flux_dd(s.X[0], s.X[1], s.Y[0], s.Y[1]);
    const dd2 u = j * bcast(ir);
    r.u = u;
    const dd2 e0 = s.S[0] * f2(7.25f, 36.0f), e1 = s.S[1] * f2(4.0f, 9.0f);
    const dd de = (sum_lanes(e0) + first(e1)) + second(e1);
    // rows 5..16 of Appendix A
    const dd2 XY0 = firsts(s.X[0], s.Y[0]), XY1 = seconds(s.X[0], s.Y[0]);
    const dd2 m78 = ((XY0 * f2(7.25f, 7.25f) + XY1 * f2(216.0f, 216.0f)) +
                     both(4.0 * kSqrt2) * firsts(s.X[1], s.Y[1])) + both(27.0 / kSqrt2) * seconds(s.X[1], s.Y[1]);
    const dd2 t13 = s.S[1] * f2(16.0f, 81.0f);
    const dd m13 = (sum_lanes(s.S[0] * f2(7.25f, 1296.0f)) + first(t13)) + second(t13);
    const dd2 m910 = m78 - XY0 * f2(6.25f, 6.25f);
    const dd2 m1112 = XY0 + XY1 * f2(216.0f, 216.0f);       // row 13 negated, as its column of cEy
    const dd2 m515 = bcast(first(s.Q[0])) * f2(1.0f, 7.25f) + bcast(second(s.Q[0])) * f2(36.0f, 1296.0f);
    const dd2 m614 = bcast(first(s.Q[1])) * f2(2.0f, 8.0f) + bcast(second(s.Q[1])) * f2(4.5f, 40.5f);
    // equilibria (Appendix A closed forms), as feq_hat_dev<R, false>
    const dd2 jj = j * u;
    const dd J2 = sum_lanes(jj), dxy = first(jj) - second(jj);
    const dd dP = (de - J2) * C.inv_b;
    r.P = dP;
    const dd P2 = scale2(dP, 2.0f);
    const dd q6 = first(j) * second(u);
    const dd q13 = ir * (dP * fma_dd(C.two_b2, dP, C.six_b * J2) + J2 * J2);
    const dd k = fma_dd(C.b4, dP, J2);
    const dd e2p = fma_dd(C.b, dP, J2) + P2;
    const dd2 q1415 = bcast(k) * pack(first(u), dxy) * pack(second(u), ir);   // rows 15, 16
    r.d413 = pack((de - first(s.S[0]) * 6.25f) - (P2 + J2), m13 - q13);
    r.d78 = m78 - bcast(e2p) * u;
    r.d910 = m910 - bcast(scale2(dP, 4.0f) + J2) * u;
    r.d1112 = m1112 - pack(P2 + dxy, P2 - dxy) * u;
    r.d515 = m515 - pack(dxy, second(q1415));
    r.d614 = m614 - pack(q6, first(q1415));
    return r;
}

// The energy-flux correction (Sec. II) of rows 8, 9; gx, gy: the differences of (u_x, u_y) along x
// and y, y differences weighted by ry = dx/dy (q89 carries 1/(2 dx)).
__device__ __forceinline__ void correct_dd(const CoefDD &C, ResidualDD &r, dd2 gx, dd2 gy)
{
    const dd div = first(gx) + C.ry * second(gy), shr = second(gx) + C.ry * first(gy);
    const dd2 g = C.g4 * pack(first(gx), second(gy)) - bcast(C.four_inv_b * div);
    const dd2 h = r.u * g + scale2(pack(second(r.u), first(r.u)) * bcast(shr), 2.0f);
    r.d78 = r.d78 + C.q89 * bcast(r.P) * h;
}

// dt M^-1 S of the residual, per population pair (Eq. 3).
__device__ __forceinline__ void relax_dd(const CoefDD &C, const ResidualDD &r, dd2 *out)
{
    const dd2 d4 = bcast(first(r.d413)), d13 = bcast(second(r.d413));
    const dd2 d7 = bcast(first(r.d78)), d9 = bcast(first(r.d910)), d11 = bcast(first(r.d1112));
    const dd2 d8 = bcast(second(r.d78)), d10 = bcast(second(r.d910)), d12 = bcast(second(r.d1112));
    const dd2 d5 = bcast(first(r.d515)), d15 = bcast(second(r.d515));
    const dd2 d6 = bcast(first(r.d614)), d14 = bcast(second(r.d614));
    unbutterfly_dd_axis(C.pA[0][0] * d4 + C.pA[0][1] * d13,
                        (C.pEx[0][0] * d7 + C.pEx[0][1] * d9) + C.pEx[0][2] * d11,
                        (C.pEy[0][0] * d8 + C.pEy[0][1] * d10) + C.pEy[0][2] * d12,
                        C.pB1[0] * d5 + C.pB1[1] * d15, out);
    unbutterfly_dd_diag(C.pA[1][0] * d4 + C.pA[1][1] * d13,
                        (C.pEx[1][0] * d7 + C.pEx[1][1] * d9) + C.pEx[1][2] * d11,
                        (C.pEy[1][0] * d8 + C.pEy[1][1] * d10) + C.pEy[1][2] * d12,
                        C.pB2[0] * d6 + C.pB2[1] * d14, out + 4);
}

__device__ __forceinline__ float2 shfl_down2(float2 v)
{
    return f2(__shfl_down_sync(0xffffffffu, v.x, 1), __shfl_down_sync(0xffffffffu, v.y, 1));
}
__device__ __forceinline__ float2 shfl_up2(float2 v)
{
    return f2(__shfl_up_sync(0xffffffffu, v.x, 1), __shfl_up_sync(0xffffffffu, v.y, 1));
}
__device__ __forceinline__ dd2 shfl_down_dd(dd2 v) { return dd2{shfl_down2(v.hi), shfl_down2(v.lo)}; }
__device__ __forceinline__ dd2 shfl_up_dd(dd2 v) { return dd2{shfl_up2(v.hi), shfl_up2(v.lo)}; }

// v, or the pair at shared address a where `own` holds (a predicated 16-byte load: no selects).
__device__ __forceinline__ void take_edge(dd2 &v, unsigned a, bool own)
{
    asm("{\n\t.reg .pred p;\n\t"
        "setp.ne.s32 p, %5, 0;\n\t"
        "@p ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n\t}"
        : "+f"(v.hi.x), "+f"(v.hi.y), "+f"(v.lo.x), "+f"(v.lo.y)
        : "r"(a), "r"((int)own));
}

// Face differences enter the MC slope normalised (norm_lim, once per difference: each feeds two
// slopes); the other limiters use them as they are.
template <int Lim>
__device__ __forceinline__ dd2 norm_lim(dd2 a)
{
    return Lim == 0 ? norm(a) : a;
}

template <int Lim>
__device__ __forceinline__ dd2 slope_dd(dd2 a, dd2 b)
{
    if (Lim == 0) return mc2n(a, b);
    if (Lim == 1) return scale2(b, 2.0f);
    return dd2{f2(0.0f, 0.0f), f2(0.0f, 0.0f)};
}

// x-moving pair e (0 .. 5) of the six, and its index among them
__device__ __forceinline__ constexpr int xpair(int e) { return e < 2 ? 2 * e : e + 2; }
__device__ __forceinline__ constexpr int xpair_index(int pr) { return pr < 4 ? pr >> 1 : pr - 2; }

// Limited flux differences (F_out - F_in) of pair pr along y, for KR cells of a column (the first at
// smem offset c, values f): emit(k, t).  The slopes come from a window sliding along the motion: last
// value, face difference, slope; downward pairs carry differences and slopes, and t, negated.
template <int Lim, typename S, typename F>
__device__ __forceinline__ void y_flux_dd(const CoefDD &C, const float2 *tile, int pr, int c, const dd2 *f, F &&emit)
{
    const int sy = tsgn_y(pair_q(pr)), sp = pr >> 2;
    const int first_row = sy > 0 ? -2 : -1;
    dd2 w = tile_pair<S>(tile, pr, c + first_row * S::SW);
    dd2 d = dd2{f2(0.0f, 0.0f), f2(0.0f, 0.0f)}, m = d;
#pragma unroll
    for (int i = 1; i < S::KR + 3; i++) {
        const int row = first_row + i;
        const dd2 wn = row >= 0 && row < S::KR ? f[row] : tile_pair<S>(tile, pr, c + row * S::SW);
        const dd2 dn = norm_lim<Lim>(wn - w);
        if (i >= 2) {
            const dd2 mn = sy > 0 ? slope_dd<Lim>(d, dn) : slope_dd<Lim>(dn, d);
            if (i >= 3) {
                const dd2 dm = sy > 0 ? mn - m : m - mn;
                // Lim 0: both slopes have the sign of d and at most 4 |d|, and hhy <= 1/4
                emit(i - 3, Lim == 2 ? d : Lim == 0 ? add_smaller(d, C.hhy[sp] * dm) : d + C.hhy[sp] * dm);
            }
            m = mn;
        }
        w = wn;
        d = dn;
    }
}

// The same along x for the cell of value f at smem offset c: the lane's face difference
// D(x) = f(x) - f(x-1) and slope S(x) = mc2(D(x), D(x+1)); the neighbours' values by shuffles, those
// one column outside the tile from the edge table at ea.  Negated for pairs moving left.
template <int Lim, typename S>
__device__ __forceinline__ dd2 x_flux_dd(const CoefDD &C, const float2 *tile, int pr, int c, dd2 f, unsigned ea,
                                         int lane)
{
    const int sx = tsgn_x(pair_q(pr)), sp = pr >> 2;
    const dd2 D = norm_lim<Lim>(f - tile_pair<S>(tile, pr, c - 1));
    dd2 Dr = shfl_down_dd(D);
    take_edge(Dr, ea, lane == kTmaTX - 1);
    const dd2 t = sx > 0 ? D : Dr;
    if (Lim == 2) return t;
    if (Lim == 1) return t + scale2(C.hh[sp], 2.0f) * (sx > 0 ? Dr - D : D - Dr);
    const dd2 Sx = mc2n(D, Dr);
    // upwind slope: S(x - 1) for pairs moving right; moving left, d1 = -D(x+1) with slopes -S(x) and
    // -S(x+1) (mc2n is odd and symmetric, up to the choice between candidates within 2^-47 of each
    // other)
    dd2 Su = sx > 0 ? shfl_up_dd(Sx) : shfl_down_dd(Sx);
    take_edge(Su, ea + 16u, lane == (sx > 0 ? 0 : kTmaTX - 1));
    return add_smaller(t, C.hh[sp] * (Sx - Su));   // as along y
}

// Flow velocity of the tile's ring (for grad u, where c9), and the values one column outside the tile
// for the x stencils: per row and x-moving pair D(x0 + 32) for lane 31, and the slope beyond the
// upwind end, S(x0 - 1) = mc2(D(x0 - 1), D(x0)) for pairs moving right, S(x0 + 32) =
// mc2(D(x0 + 32), D(x0 + 33)) for those moving left.  Shared by threads tid of `threads`.
template <int Lim, typename S>
__device__ __forceinline__ void ring_and_edges(const float2 *tile, float4 *suv, float4 *sedge, int tid, int threads,
                                               bool c9)
{
    constexpr int kRing = 2 * (kTmaTX + S::TR), kEdges = 6 * S::TR;
    for (int k = tid; k < kRing + kEdges; k += threads) {
        if (k < kRing) {
            if (!c9) continue;
            int i, j;                                                 // column, row in the tile + ring
            if (k < 2 * kTmaTX) {
                i = (k & (kTmaTX - 1)) + 1;
                j = k < kTmaTX ? 0 : S::TR + 1;
            } else {
                i = k < 2 * kTmaTX + S::TR ? 0 : kTmaTX + 1;
                j = (k - 2 * kTmaTX) % S::TR + 1;
            }
            suv[j * S::UW + i] = quad(velocity_dd<S>(tile, (j + 1) * S::SW + (i + S::HX - 1)));
        } else {
            const int n = k - kRing, r = n / 6, e = n - 6 * r, pr = xpair(e);
            const int row = (r + 2) * S::SW + S::HX;                  // smem offset of x0
            const float2 *hi = tile + pair_q(pr) * S::PL + row, *lo = hi + 4 * S::PL;
            auto at = [&](int x) { return dd2{hi[x], lo[x]}; };
            sedge[2 * n] = quad(norm_lim<Lim>(at(kTmaTX) - at(kTmaTX - 1)));
            if (Lim == 0) {
                const int c = tsgn_x(pair_q(pr)) > 0 ? -2 : kTmaTX - 1;
                sedge[2 * n + 1] = quad(mc2n(norm(at(c + 1) - at(c)), norm(at(c + 2) - at(c + 1))));
            }
        }
    }
}

// One ghost cell of a wall in the staged tile (before its split) from its mirror cell, in float64 as the
// ghost launch of the other kernels forms it: the two warps of a tile's wall cells take some 210 float64
// instructions each while the other warps wait (161 x 97 channel 14.8 us a step, 18.8 with a launch before
// the step, 512 x 512 52 and 53, 1023 x 517 94 and 114).  In double-float it was 10.3 us on 161 x 97, with
// three to four times the error of a step at the wall cells.  A function of its own: every tile shape,
// alone and in a batch, runs the same code and has the same bits.
__device__ __noinline__ void wall_cell64(const Coef<double> &C, const EdgeDev &E, const double *mirror, double *ghost,
                                         int plane)
{
    double g[NQ], fd[NQ];
#pragma unroll
    for (int q = 0; q < NQ; q++) g[q] = mirror[q * plane];
    wall_change<double, false>(C, E, g, fd);
#pragma unroll
    for (int q = 0; q < NQ; q++) ghost[q * plane] = g[q] + fd[q];
}

// Ghost cells of the walls at an edge tile, one thread per cell.  G: the grid's extents; P: its
// coefficients and edges.
template <typename S, typename PP>
__device__ __forceinline__ void wall_fill(const PP &G, const Params &P, double *tile, int x0, int y0, int tid)
{
    for (int k = tid; k < GhostSlot<S>::kSlots; k += kTmaTX * S::TT) {
        const GhostSlot<S> g(G, k, x0, y0);
        if (!g.in || P.edge[g.edge].kind != 3) continue;
        const int n = g.row ? G.ny : G.nx, depth = g.layer & 1;
        const int m = min(max(g.layer < 2 ? depth : n - 1 - depth, 0), n - 1);
        wall_cell64(P.cd, P.edge[g.edge], tile + g.offset(g.row ? m - y0 + 2 : m - x0 + S::HX), tile + g.offset(g.at),
                    S::PL);
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// The tile body shared by the single-grid and the batched kernel: the staged float64 tile in
// shared memory (smraw) is split, then phases 1 and 2 produce the tile's new float64 values.
// ---------------------------------------------------------------------------
// P: the context's Params, or the TileGrid block of a batched launch (nx, ny, pitch, plane).
// S: the tile shape.
// C9: whether the energy-flux correction runs (0, 1), or 2 to ask P.has_c9.
template <int Lim, int C9, typename S, typename PP>
__device__ __forceinline__ void dd_tile(const PP &P, const CoefDD &C, unsigned char *smraw,
                                        double *__restrict__ fout, int x0, int y0)
{
    double *tile64 = reinterpret_cast<double *>(smraw);
    float2 *tile = reinterpret_cast<float2 *>(smraw);
    float4 *suv = reinterpret_cast<float4 *>(smraw + S::uv_off);        // (u_x, u_y), tile + ring
    float4 *sedge = reinterpret_cast<float4 *>(smraw + S::edge_off);    // x edge values per row and pair
    const bool c9 = C9 == 2 ? P.has_c9 != 0 : C9 != 0;
    const int lane = threadIdx.x, ty = threadIdx.y, tid = ty * kTmaTX + lane;
    constexpr int kThreads = kTmaTX * S::TT;
    const int nx = P.nx, ny = P.ny;
    // ---- split: float64 -> hi + lo in place, population pairs (q, q + 4)
#pragma unroll 4
    for (int k = tid; k < 8 * S::PL; k += kThreads) {
        const int a = k < 4 * S::PL ? k : k + 4 * S::PL, b = a + 4 * S::PL;
        const dd2 v = dd_split2(tile64[a], tile64[b]);
        tile[a] = v.hi;
        tile[b] = v.lo;
    }
    __syncthreads();

    const unsigned edge_a = (unsigned)__cvta_generic_to_shared(sedge);
    const int gx = x0 + lane;
    if constexpr (S::ROLES) {
        // ---- warps 0 .. TR-1: residual and relaxation of their row; warps TR .. 2 TR-1: ring, edge
        // values and convection of theirs.  A small grid has one CTA of these per SM: a warp's chain
        // of instructions is what its step lasts, and each half is about half of it.
        float4 *sacc = reinterpret_cast<float4 *>(smraw + S::acc_off);
        const bool convect = ty >= S::TR;
        const int r = convect ? ty - S::TR : ty;
        const int c0 = (r + 2) * S::SW + lane + S::HX;
        sacc += r * 8 * kTmaTX + lane;
        dd2 py[8], px[8];                                   // c_y and c_x times the flux differences
        ResidualDD res;
        if (convect) {
            ring_and_edges<Lim, S>(tile, suv, sedge, tid - S::TR * kTmaTX, S::TR * kTmaTX, c9);
#pragma unroll
            for (int pr = 0; pr < 8; pr++) {
                if (tsgn_y(pair_q(pr)) == 0) continue;
                const dd2 f = tile_pair<S>(tile, pr, c0);
                y_flux_dd<Lim, S>(C, tile, pr, c0, &f, [&](int, dd2 t) { py[pr] = C.cry[pr >> 2] * t; });
            }
        } else {
            dd2 fp[8];
#pragma unroll
            for (int pr = 0; pr < 8; pr++) fp[pr] = tile_pair<S>(tile, pr, c0);
            res = residual_dd(C, fp);
            if (c9) suv[(r + 1) * S::UW + (lane + 1)] = quad(res.u);
        }
        __syncthreads();
        if (convect) {
#pragma unroll
            for (int pr = 0; pr < 8; pr++) {
                if (tsgn_x(pair_q(pr)) == 0) continue;
                px[pr] = C.cr[pr >> 2] * x_flux_dd<Lim, S>(C, tile, pr, c0, tile_pair<S>(tile, pr, c0),
                                                         edge_a + 32u * (unsigned)(6 * r + xpair_index(pr)), lane);
            }
        } else {
            if (c9) {
                const int ui = (r + 1) * S::UW + (lane + 1);
                correct_dd(C, res, unquad(suv[ui + 1]) - unquad(suv[ui - 1]),
                           unquad(suv[ui + S::UW]) - unquad(suv[ui - S::UW]));
            }
            dd2 acc[8];
            relax_dd(C, res, acc);
#pragma unroll
            for (int pr = 0; pr < 8; pr++) sacc[pr * kTmaTX] = quad(acc[pr]);
        }
        __syncthreads();
        if (!convect) return;
        const int gy = y0 + r;
        if (gx >= nx || gy >= ny) return;
        double *o = fout + (long long)(gy + OY) * P.pitch + (gx + OX);
#pragma unroll
        for (int pr = 0; pr < 8; pr++) {
            const int qa = pair_q(pr), sx = tsgn_x(qa), sy = tsgn_y(qa);
            // f - C - c_x (F_out - F_in)_x - c_y (F_out - F_in)_y
            dd2 out = tile_pair<S>(tile, pr, c0) - unquad(sacc[pr * kTmaTX]);
            if (sy != 0) out = sy > 0 ? out - py[pr] : out + py[pr];
            if (sx != 0) out = sx > 0 ? out - px[pr] : out + px[pr];
            o[qa * P.plane] = dd_to_double(first(out));
            o[(qa + 4) * P.plane] = dd_to_double(second(out));
        }
        return;
    } else {
    // ---- phase 1: the ring, the edge values, and the residuals of rows ty*KR .. ty*KR+KR-1 of the
    // tile, column `lane`
    ring_and_edges<Lim, S>(tile, suv, sedge, tid, kThreads, c9);
    const int r0 = ty * S::KR;
    const int c0 = (r0 + 2) * S::SW + lane + S::HX;
    ResidualDD res[S::KR];
#pragma unroll
    for (int k = 0; k < S::KR; k++) {
        dd2 fp[8];
#pragma unroll
        for (int pr = 0; pr < 8; pr++) fp[pr] = tile_pair<S>(tile, pr, c0 + k * S::SW);
        res[k] = residual_dd(C, fp);
        if (c9) suv[(r0 + k + 1) * S::UW + (lane + 1)] = quad(res[k].u);
    }
    __syncthreads();

    // ---- phase 2: the collision terms C of the thread's cells, then pair by pair their
    // convection and update (a pair's windows are dead before the next one's are formed)
    dd2 acc[S::KR][8];
#pragma unroll
    for (int k = 0; k < S::KR; k++) {
        if (c9) {
            const int ui = (r0 + k + 1) * S::UW + (lane + 1);
            correct_dd(C, res[k], unquad(suv[ui + 1]) - unquad(suv[ui - 1]),
                       unquad(suv[ui + S::UW]) - unquad(suv[ui - S::UW]));
        }
        relax_dd(C, res[k], acc[k]);
    }
    // the cells' populations are read again below: kept in registers from the collision (which the
    // compiler does for loads from equal addresses) they would be spilled
    int c1 = c0;
    asm volatile("" : "+r"(c1));
    // f - C - c_x (F_out - F_in)_x - c_y (F_out - F_in)_y
#pragma unroll
    for (int n = 0; n < 8; n++) {
        const int pr = n ^ 4;                               // the diagonal pairs first
        const int qa = pair_q(pr);
        const int sx = tsgn_x(qa), sy = tsgn_y(qa);
        const int sp = pr >> 2;                             // shell pair
        dd2 f[S::KR], out[S::KR];
#pragma unroll
        for (int k = 0; k < S::KR; k++) {
            f[k] = tile_pair<S>(tile, pr, c1 + k * S::SW);
            out[k] = f[k] - acc[k][pr];
        }
        if (sy != 0)
            y_flux_dd<Lim, S>(C, tile, pr, c1, f, [&](int k, dd2 t) {
                out[k] = sy > 0 ? out[k] - C.cry[sp] * t : out[k] + C.cry[sp] * t;
            });
#pragma unroll
        for (int k = 0; k < S::KR; k++) {
            if (sx != 0) {
                const dd2 t = x_flux_dd<Lim, S>(C, tile, pr, c1 + k * S::SW, f[k],
                                                edge_a + 32u * (unsigned)(6 * (r0 + k) + xpair_index(pr)), lane);
                out[k] = sx > 0 ? out[k] - C.cr[sp] * t : out[k] + C.cr[sp] * t;
            }
            const int gy = y0 + r0 + k;
            if (gx < nx && gy < ny) {
                double *o = fout + (long long)(gy + OY) * P.pitch + (gx + OX);
                __stcs(o + qa * P.plane, dd_to_double(first(out[k])));
                __stcs(o + (qa + 4) * P.plane, dd_to_double(second(out[k])));
            }
        }
    }
    }
}

// ---------------------------------------------------------------------------
// The single-grid kernel.  Walls: a grid with walls (an instantiation of its own: with the call of
// wall_fill the step of grids without any takes 1.5% longer).
// ---------------------------------------------------------------------------
template <int Lim, bool C9, bool Walls, typename S>
__global__ void __launch_bounds__(kTmaTX * S::TT, S::CTAS)
k_step_dd(const __grid_constant__ Params P, const __grid_constant__ CoefDD C, const __grid_constant__ CUtensorMap tm,
          const double *fin, double *fout, int *err)
{
    extern __shared__ __align__(128) unsigned char smraw[];
    double *tile64 = reinterpret_cast<double *>(smraw);
    __shared__ __align__(8) unsigned long long bar;

    const int tid = threadIdx.y * kTmaTX + threadIdx.x;
    // tile rows past 65535, the grid dimension's limit, go on along z (DdOps::launch)
    const int x0 = blockIdx.x * kTmaTX, row = blockIdx.z * gridDim.y + blockIdx.y, y0 = row * S::TR;
    if (y0 >= P.ny) return;
    const unsigned bar_a = (unsigned)__cvta_generic_to_shared(&bar);
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar_a) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    grid_dependency_wait();
    grid_launch_dependents();
    if (tid == 0) {
        // box origin: interior column x0 - HX = padded column x0 + OX - HX; interior row y0 - 2 =
        // padded row y0
        const unsigned dst = (unsigned)__cvta_generic_to_shared(tile64);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar_a),
                     "r"((unsigned)S::tile_bytes) : "memory");
        asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
                     " [%0], [%1, {%2, %3, %4}], [%5];"
                     ::"r"(dst), "l"(reinterpret_cast<unsigned long long>(&tm)), "r"(x0 + OX - S::HX), "r"(y0),
                     "r"(0), "r"(bar_a) : "memory");
        // bring the tile of the CTA half a resident wave later into L2
        unsigned nsm;
        asm("mov.u32 %0, %%nsmid;" : "=r"(nsm));
        const long long bn = (long long)row * gridDim.x + blockIdx.x + (long long)S::CTAS * nsm / 2;
        const int xn = (int)(bn % gridDim.x) * kTmaTX + OX - S::HX, yn = (int)(bn / gridDim.x) * S::TR;
        if (yn < P.ny) {
            asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];"
                         ::"l"(reinterpret_cast<unsigned long long>(&tm)), "r"(xn), "r"(yn), "r"(0) : "memory");
        }
    }
    GhostFill<double, S> ghost;
    const bool edge = GhostFill<double, S>::edge_tile(P, x0, y0);
    if (edge) ghost.load(P, P.edge, fin, x0, y0, tid);
    const bool ok = mbar_wait(bar_a, 0);
    if (!__syncthreads_and(ok)) {
        if (tid == 0) {
            atomicExch(err, 1);
            mbar_wait(bar_a, 0);               // let a late copy land before the CTA exits (bounded)
        }
    } else {
        if (edge) {
            ghost.store(tile64);
            if (Walls) wall_fill<S>(P, P, tile64, x0, y0, tid);
            __syncthreads();
        }
        dd_tile<Lim, C9, S>(P, C, smraw, fout, x0, y0);
    }
}

// ---------------------------------------------------------------------------
// Batched form: one CTA per tile of the launch's grids (TmaBatchArgs).  Thread 0 issues the
// tile copy with the grid's tensor map from the parameter block, then the CTA copies the grid's
// TileGrid block (geometry and double-float coefficients) into shared memory while the copy is
// in flight.  The energy-flux
// correction runs where the grid has one.
// ---------------------------------------------------------------------------
template <int Lim, bool Walls, typename S>
__global__ void __launch_bounds__(kTmaTX * S::TT, S::CTAS)
k_step_dd_batch(const __grid_constant__ TmaBatchArgs A, const TileGrid<CoefDD> *__restrict__ TG,
                const Params *__restrict__ Pall)
{
    using T = TileGrid<CoefDD>;
    static_assert(sizeof(T) % 16 == 0, "TileGrid copy");
    extern __shared__ __align__(128) unsigned char smraw[];
    __shared__ __align__(16) T Ts;
    __shared__ __align__(8) unsigned long long bar;
    const int tid = threadIdx.y * kTmaTX + threadIdx.x;
    constexpr int kThreads = kTmaTX * S::TT;
    int x0, y0;
    const int g = batch_tile(A, blockIdx.x, S::TR, x0, y0);
    const unsigned bar_a = (unsigned)__cvta_generic_to_shared(&bar);
    grid_dependency_wait();
    grid_launch_dependents();
    if (tid == 0)
        batch_issue<S::TR, S::HX>(A, g, x0, y0, (unsigned)__cvta_generic_to_shared(smraw), bar_a,
                                  (unsigned)S::tile_bytes, S::CTAS);
    // the grid's block, while the tile copy is in flight
    {
        const int4 *src = reinterpret_cast<const int4 *>(TG + g);
        int4 *dst = reinterpret_cast<int4 *>(&Ts);
        for (int k = tid; k < (int)(sizeof(T) / sizeof(int4)); k += kThreads) dst[k] = src[k];
    }
    __syncthreads();                            // the barrier is initialised
    GhostFill<double, S> ghost;
    const bool edge = GhostFill<double, S>::edge_tile(Ts, x0, y0);
    if (edge) ghost.load(Ts, Pall[Ts.member].edge, static_cast<const double *>(A.in[g]), x0, y0, tid);
    const bool ok = mbar_wait(bar_a, 0);
    if (!__syncthreads_and(ok)) {
        if (tid == 0) {
            atomicExch(A.err[g], 1);
            mbar_wait(bar_a, 0);               // let a late copy land before the CTA exits (bounded)
        }
    } else {
        if (edge) {
            ghost.store(reinterpret_cast<double *>(smraw));
            if (Walls) wall_fill<S>(Ts, Pall[Ts.member], reinterpret_cast<double *>(smraw), x0, y0, tid);
            __syncthreads();
        }
        dd_tile<Lim, 2, S>(Ts, Ts.cf, smraw, static_cast<double *>(A.out[g]), x0, y0);
    }
}

static bool has_walls(const Params &P)
{
    return P.edge[0].kind == 3 || P.edge[1].kind == 3 || P.edge[2].kind == 3 || P.edge[3].kind == 3;
}

template <bool Walls, typename S>
static auto dd_kernel_of(const Params &P)
{
    return P.limiter == 0   ? (P.has_c9 ? k_step_dd<0, true, Walls, S> : k_step_dd<0, false, Walls, S>)
           : P.limiter == 1 ? (P.has_c9 ? k_step_dd<1, true, Walls, S> : k_step_dd<1, false, Walls, S>)
                            : (P.has_c9 ? k_step_dd<2, true, Walls, S> : k_step_dd<2, false, Walls, S>);
}

template <typename S>
static auto dd_kernel(const Params &P)
{
    return has_walls(P) ? dd_kernel_of<true, S>(P) : dd_kernel_of<false, S>(P);
}

template <typename S>
static auto dd_batch_kernel(int limiter, bool walls)
{
    if (walls)
        return limiter == 0   ? k_step_dd_batch<0, true, S>
               : limiter == 1 ? k_step_dd_batch<1, true, S>
                              : k_step_dd_batch<2, true, S>;
    return limiter == 0   ? k_step_dd_batch<0, false, S>
           : limiter == 1 ? k_step_dd_batch<1, false, S>
                          : k_step_dd_batch<2, false, S>;
}

template <typename S, typename K>
static cudaError_t dd_allow(K *kernel)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::smem_bytes);
}

template <typename S>
cudaError_t DdOps<S>::launch(const Params &P, const CoefDD &C, const CUtensorMap &tm, const double *a, double *b, int *err,
                             bool chain, int rows, cudaStream_t st)
{
    const dim3 block(kTmaTX, S::TT);
    // tile rows in y, and in z by as few as y holds
    const int trows = (rows + S::TR - 1) / S::TR, z = (trows + kMaxGridY - 1) / kMaxGridY;
    const dim3 grid((P.nx + kTmaTX - 1) / kTmaTX, (trows + z - 1) / z, z);
    return launch_kernel(chain, dd_kernel<S>(P), grid, block, S::smem_bytes, st, P, C, tm, a, b, err);
}

template <typename S>
cudaError_t DdOps<S>::launch_batch(const TmaBatchArgs &A, const TileGrid<CoefDD> *tg, const Params *Pall, int limiter,
                                   bool walls, bool chain, cudaStream_t st)
{
    return launch_kernel(chain, dd_batch_kernel<S>(limiter, walls), dim3(A.first[A.n]), dim3(kTmaTX, S::TT), S::smem_bytes,
                         st, A, tg, Pall);
}

template <typename S>
cudaError_t DdOps<S>::prepare(const Params &P)
{
    return dd_allow<S>(dd_kernel<S>(P));
}

template <typename S>
cudaError_t DdOps<S>::prepare_batch(int limiter, bool walls)
{
    return dd_allow<S>(dd_batch_kernel<S>(limiter, walls));
}

}  // namespace lbm
