// lbm_step_dd.cu -- host side of the double-float float64 kernels (lbm_step_dd.cuh, instantiated per tile
// shape in lbm_step_dd_wide.cu, _mid.cu and _narrow.cu, which compile in parallel): their coefficients, the
// choice between tile shapes, and the launches.
#include "lbm_internal.h"

namespace lbm {

// Coefficients in double-float from the float64 tables (host).
void coef_dd(const Params &P, CoefDD *out)
{
    const Coef<double> &C = P.cd;
    auto pair = [](double x, double y) {
        const dd a = dd_host(x), b = dd_host(y);
        return dd2{make_float2(a.hi, b.hi), make_float2(a.lo, b.lo)};
    };
    for (int p = 0; p < 2; p++) {
        out->hh[p] = pair(C.hh[2 * p], C.hh[2 * p + 1]);
        out->hhy[p] = pair(C.hhy[2 * p], C.hhy[2 * p + 1]);
        out->cr[p] = pair(C.cr[2 * p], C.cr[2 * p + 1]);
        out->cry[p] = pair(C.cry[2 * p], C.cry[2 * p + 1]);
        for (int j = 0; j < 2; j++) out->pA[p][j] = pair(C.cA[2 * p][j], C.cA[2 * p + 1][j]);
        for (int j = 0; j < 3; j++) {
            const double sg = j == 2 ? -1.0 : 1.0;          // row 13 enters negated
            out->pEx[p][j] = pair(C.cEx[2 * p][j], C.cEx[2 * p + 1][j]);
            out->pEy[p][j] = pair(sg * C.cEy[2 * p][j], sg * C.cEy[2 * p + 1][j]);
        }
        out->pB1[p] = pair(C.cB1[0][p], C.cB1[1][p]);
        out->pB2[p] = pair(C.cB2[0][p], C.cB2[1][p]);
    }
    out->q89 = pair(C.q8, C.q9);
    out->g4 = pair(C.g4[0], C.g4[1]);
    out->b = dd_host(C.b);
    out->inv_b = dd_host(C.inv_b);
    out->two_b2 = dd_host(C.two_b2);
    out->six_b = dd_host(C.six_b);
    out->b4 = dd_host(C.b4);
    out->four_inv_b = dd_host(C.four_inv_b);
    out->ry = dd_host(C.ry);
    out->pad_ = dd{0.0f, 0.0f};
}

bool dd_shape_supported(const Params &P, int shape)
{
    return P.pitch >= DdWideShape::SW && P.nx >= kTmaTX && P.ny >= kDdRows[shape];
}

double dd_shape_time(int shape, long long tiles, int sms)
{
    constexpr double fixed[kDdShapes] = {4.9, 3.1, 2.0}, whole[kDdShapes] = {22.4, 12.3, 8.6},
                     one[kDdShapes] = {11.5, 6.7, 5.2}, two[kDdShapes] = {22.0, 11.0, 9.0};
    const long long slots = 2LL * sms, rest = tiles % slots;
    return fixed[shape] + (double)(tiles / slots) * whole[shape] +
           (rest == 0 ? 0.0 : (rest <= sms ? one[shape] : two[shape]));
}

cudaError_t launch_step_dd(const Params &P, const void *coef, const void *tmap, const void *fin, void *fout,
                           int *err, cudaStream_t st, int shape, bool chain, int rows)
{
    const CUtensorMap &tm = *reinterpret_cast<const CUtensorMap *>(tmap);
    const CoefDD &C = *reinterpret_cast<const CoefDD *>(coef);
    const double *a = (const double *)fin;
    double *b = (double *)fout;
    if (rows == 0) rows = P.ny;
    return shape == kDdNarrow ? DdOps<DdNarrowShape>::launch(P, C, tm, a, b, err, chain, rows, st)
           : shape == kDdMid  ? DdOps<DdMidShape>::launch(P, C, tm, a, b, err, chain, rows, st)
                              : DdOps<DdWideShape>::launch(P, C, tm, a, b, err, chain, rows, st);
}

cudaError_t launch_step_dd_batch(const TmaBatchArgs &A, const TileGrid<CoefDD> *tg, const Params *Pall, int limiter,
                                 int shape, bool walls, bool chain, cudaStream_t st)
{
    if (A.first[A.n] <= 0) return cudaSuccess;
    return shape == kDdNarrow ? DdOps<DdNarrowShape>::launch_batch(A, tg, Pall, limiter, walls, chain, st)
           : shape == kDdMid  ? DdOps<DdMidShape>::launch_batch(A, tg, Pall, limiter, walls, chain, st)
                              : DdOps<DdWideShape>::launch_batch(A, tg, Pall, limiter, walls, chain, st);
}

cudaError_t dd_prepare(const Params &P)
{
    cudaError_t e = DdOps<DdWideShape>::prepare(P);
    if (e == cudaSuccess) e = DdOps<DdMidShape>::prepare(P);
    if (e == cudaSuccess) e = DdOps<DdNarrowShape>::prepare(P);
    return e;
}

cudaError_t dd_batch_prepare(int limiter, bool walls)
{
    cudaError_t e = DdOps<DdWideShape>::prepare_batch(limiter, walls);
    if (e == cudaSuccess) e = DdOps<DdMidShape>::prepare_batch(limiter, walls);
    if (e == cudaSuccess) e = DdOps<DdNarrowShape>::prepare_batch(limiter, walls);
    return e;
}

}  // namespace lbm
