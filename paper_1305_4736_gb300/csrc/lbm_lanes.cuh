// lbm_lanes.cuh -- float64 cell arithmetic with one lane per population.
//
// GB300's float64 unit takes 0.4 lanes per cycle in each of an SM's four partitions: a warp
// instruction costs its partition about 78 cycles whether its 32 lanes hold 32 cells or one cell's
// populations.  Where a launch has few cells (walls; grids of a few thousand cells) the number of
// float64 instructions in one warp is what it lasts, so here 16 lanes share a cell: the butterflies
// of the shells take one instruction a stage, a block of the transformation four, an equilibrium
// row six, 79 instead of 398 for a whole step (47 without the energy-flux correction; 40 against 12 per
// cell: the price where cells abound).  Everything stays in float64.
//
// Lane q of a cell holds population q = 4 shell + i, and in the shell basis the coefficient
// `i` of its shell: 0 S, 1 Q, 2 X, 3 Y.  A moment row r of a component's block sits in the lane of
// shell r: S: m1, m4, m5, m14; X: m2, m8, m10, m12; Y: m3, m9, m11, m13; Q: m6, m16, m7, m15.
#pragma once

#include "lbm_device.cuh"

namespace lbm {
namespace {

constexpr int kCellLanes = 16;

__device__ __forceinline__ double shfl16(double v, int src) { return __shfl_sync(0xffffffffu, v, src, kCellLanes); }
__device__ __forceinline__ double xor16(double v, int m) { return __shfl_xor_sync(0xffffffffu, v, m, kCellLanes); }
// v or -v: the sign bit on the integer pipe (a float64 negation would cost a float64 instruction)
__device__ __forceinline__ double flip(double v, bool minus)
{
    return __hiloint2double(__double2hiint(v) ^ (minus ? (int)0x80000000 : 0), __double2loint(v));
}

// Blocks of the transformation matrix in the shell basis (Appendix A), row by lane.
__device__ const double kLaneRows[16][4] = {
    {1.0, 1.0, 1.0, 1.0}, {1.0, 36.0, 0.0, 0.0}, {1.0, 6.0, kD3, kD4}, {1.0, 6.0, kD3, kD4},
    {kW1, 36.0, 4.0, 9.0}, {kW1, 1296.0, 0.0, 0.0},
    {kW1, 216.0, 4.0 * kSqrt2, 27.0 / kSqrt2}, {kW1, 216.0, 4.0 * kSqrt2, 27.0 / kSqrt2},
    {1.0, 36.0, 4.0, 9.0}, {0.0, 0.0, 2.0, 4.5},
    {1.0, 216.0, 4.0 * kSqrt2, 27.0 / kSqrt2}, {1.0, 216.0, 4.0 * kSqrt2, 27.0 / kSqrt2},
    {kW1, 1296.0, 16.0, 81.0}, {0.0, 0.0, 8.0, 40.5}, {1.0, 216.0, 0.0, 0.0}, {-1.0, -216.0, 0.0, 0.0}};

struct Lane {
    int q, shell, comp;
    double row[4];             // this lane's row of the forward block
    double ca, cb, c6;         // equilibrium row: ((ca P + cb Z) F1 + c6 J2^2) F2
    int z, f1, f2;             // Z: 0 J2, 1 dxy, 2 rho;  F1: 0 one, 1 ux, 2 uy, 3 P, 4 dxy;  F2: 0 one, 1 uy, 2 1/rho
};

__device__ __forceinline__ Lane lane_of(const Coef<double> &C, int q)
{
    Lane L;
    L.q = q;
    L.shell = q >> 2;
    L.comp = q & 3;
#pragma unroll
    for (int k = 0; k < 4; k++) L.row[k] = kLaneRows[q][k];
    L.ca = 0.0;
    L.cb = 1.0;
    L.c6 = 0.0;
    L.z = L.f1 = L.f2 = 0;
    switch (q) {
    case 0: L.z = 2; break;                                              // m1: rho
    case 4: L.ca = C.b; break;                                           // m4: b P + J2
    case 8: L.ca = 2.0; break;                                           // m5: 2 P + J2
    case 12: L.ca = C.two_b2; L.cb = C.six_b; L.f1 = 3; L.f2 = 2; L.c6 = 1.0; break;   // m14
    case 2: case 3: L.z = 2; L.f1 = L.comp - 1; break;                   // m2, m3: rho u
    case 6: case 7: L.ca = C.b + 2.0; L.f1 = L.comp - 1; break;          // m8, m9: (e + 2 P) u
    case 10: case 11: L.ca = 4.0; L.f1 = L.comp - 1; break;              // m10, m11: (4 P + J2) u
    case 14: L.ca = 2.0; L.z = 1; L.f1 = 1; break;                       // m12: (2 P + dxy) ux
    case 15: L.ca = -2.0; L.z = 1; L.f1 = 2; break;                      // m13: (dxy - 2 P) uy
    case 1: L.z = 1; break;                                              // m6: dxy
    case 9: L.z = 2; L.f1 = 1; L.f2 = 1; break;                          // m7: rho ux uy
    case 13: L.ca = C.b4; L.f1 = 1; L.f2 = 1; break;                     // m15: ((b + 4) P + J2) ux uy
    default: L.ca = C.b4; L.f1 = 4; L.f2 = 2; break;                     // m16 (lane 5): (...) dxy / rho
    }
    return L;
}

// Rows of the collision's inverse blocks (dt s_k folded in; conserved columns zero) and of the full
// inverse, for this lane's coefficient.
__device__ __forceinline__ void lane_collision(const Coef<double> &C, const Lane &L, double *k)
{
    k[0] = k[1] = k[2] = k[3] = 0.0;
    if (L.comp == 0) {
        k[2] = C.cA[L.shell][0];
        k[3] = C.cA[L.shell][1];
    } else if (L.comp == 1) {
        if (L.shell < 2) {
            k[0] = C.cB1[L.shell][0];
            k[1] = C.cB1[L.shell][1];
        } else {
            k[2] = C.cB2[L.shell - 2][0];
            k[3] = C.cB2[L.shell - 2][1];
        }
    } else {
        const double *e = L.comp == 2 ? C.cEx[L.shell] : C.cEy[L.shell];
        for (int j = 0; j < 3; j++) k[j + 1] = e[j];
    }
}

__device__ __forceinline__ void lane_inverse(const Coef<double> &C, const Lane &L, double *k)
{
    k[0] = k[1] = k[2] = k[3] = 0.0;
    if (L.comp == 1) {
        for (int j = 0; j < 2; j++) {
            if (L.shell < 2) k[j] = C.iB1[L.shell][j];
            else k[2 + j] = C.iB2[L.shell - 2][j];
        }
    } else {
        const double *e = L.comp == 0 ? C.iA[L.shell] : (L.comp == 2 ? C.iEx[L.shell] : C.iEy[L.shell]);
        for (int j = 0; j < 4; j++) k[j] = e[j];
    }
}

// Shell coefficient of this lane from the populations.
__device__ __forceinline__ double lane_butterfly(const Lane &L, double p)
{
    const bool hi = L.comp & 2, diag = L.shell >= 2;
    const double t = xor16(p, 2) + flip(p, hi);                    // p0 + p2, p1 + p3, p0 - p2, p1 - p3
    const double w = xor16(t, 1);
    const double r = flip(t, L.comp == 1) + flip(w, L.comp == 2);  // a + b, a - b, c - d, c + d
    return hi && !diag ? t : r;
}

// Population of this lane from the (normalised) shell coefficients.
__device__ __forceinline__ double lane_unbutterfly(const Lane &L, double v)
{
    const bool hi = L.comp & 2, diag = L.shell >= 2;
    const double w = xor16(v, 1);
    const double r = w + flip(v, L.comp & 1);                      // S + Q, S - Q, X + Y, X - Y
    const double t = hi && !diag ? v : r;
    const double o = xor16(t, 2);
    // axis: a + X, b + Y, a - X, b - Y; diagonal: a + c, b - d, a - c, b + d
    const bool neg_o = diag && L.comp == 1, neg_t = hi && !(diag && L.comp == 3);
    return flip(t, neg_t) + flip(o, neg_o);
}

// A block of four by four, row by lane, applied to the component's values of the four shells.
__device__ __forceinline__ double lane_block(const Lane &L, const double *k, double v)
{
    double s = k[0] * shfl16(v, L.comp);
#pragma unroll
    for (int j = 1; j < 4; j++) s = fma(k[j], shfl16(v, 4 * j + L.comp), s);
    return s;
}

// Conserved moments' state, equal in the 16 lanes of a cell.
struct LaneState { double rho, ir, ux, uy, J2, dxy, P; };

__device__ __forceinline__ void lane_kinetic(LaneState &s, double jx, double jy)
{
    s.ux = jx * s.ir;
    s.uy = jy * s.ir;
    const double jx2 = jx * s.ux, jy2 = jy * s.uy;
    s.J2 = jx2 + jy2;
    s.dxy = jx2 - jy2;
}

// State of the cell whose moment rows are in m (jx, jy in lanes 2, 3; rho in 0, e in 4).
__device__ __forceinline__ LaneState lane_state(const Coef<double> &C, double m, double &jx, double &jy)
{
    LaneState s;
    s.rho = shfl16(m, 0);
    jx = shfl16(m, 2);
    jy = shfl16(m, 3);
    const double e = shfl16(m, 4);
    s.ir = recip(s.rho);
    lane_kinetic(s, jx, jy);
    s.P = (e - s.J2) * C.inv_b;
    return s;
}

// This lane's row of f_hat^eq.
__device__ __forceinline__ double lane_feq(const Lane &L, const LaneState &s)
{
    const double Z = L.z == 0 ? s.J2 : (L.z == 1 ? s.dxy : s.rho);
    const double F1 = L.f1 == 0 ? 1.0 : (L.f1 == 1 ? s.ux : (L.f1 == 2 ? s.uy : (L.f1 == 3 ? s.P : s.dxy)));
    const double F2 = L.f2 == 0 ? 1.0 : (L.f2 == 1 ? s.uy : s.ir);
    const double t = fma(L.ca, s.P, L.cb * Z);
    return fma(t, F1, L.c6 * (s.J2 * s.J2)) * F2;
}

}  // namespace
}  // namespace lbm
