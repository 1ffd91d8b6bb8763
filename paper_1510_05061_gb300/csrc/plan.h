// plan.h -- the launch shape (tile variant and z partition) a 3D solve takes
// unless the caller or the autotuner chooses another.
#pragma once

#include <algorithm>

#include "../../include/hydro.h"
#include "launchers.h"

namespace hydro {

struct LaunchPlan {
    int variant;   // TILE3D_SHAPES index
    int zchunk;    // planes per CTA, or -1: the balanced grid over whole columns (PieceIter)
};

// Every candidate runs on the balanced grid (min(resident CTAs, plane-tiles)
// CTAs with equal shares of the plane-tiles): against the z-chunks of 8 to 64
// planes taken before, it has no partial last wave and repeats fewer planes
// (a chunk predicts two planes and stages four beyond its own): measured on
// GB300, us per MUSCL-Hancock step, z-chunks -> balanced, same tile: FP64 16^3
// 288 -> 74, 101x75x130 1251 -> 1001, 128^3 1999 -> 1751; FP32 32^3 40 -> 19,
// 128^3 147 -> 114.
//
// The tile is the one with the least modelled time
//   max(alone, k unit) (ceil(W / (SMs k)) + fixed),   k = min(ctas, ceil(W / SMs)),
// W = plane-tiles (tiles x nz), `unit` the time of a plane of one CTA divided
// by the CTAs sharing an SM, `alone` a plane's latency on an SM of its own,
// `fixed` the planes' worth of work a CTA repeats; the constants are fitted to
// the same sweep (16^3 .. 320^3, 200x40x100, 300x40x200) and reproduce its
// times within 10 %.
struct TileCost {
    int variant, ctas;
    double alone, unit, fixed;   // us
};

inline LaunchPlan default_plan(const hydro_problem &p)
{
    constexpr int SMS = 152;
    const bool fp32 = p.precision == HYDRO_FP32;
    // FP64: 16 x 16 tiles, 32 x 8 where they fit the grid better (200x40x100:
    // 838 against 875 us), 32 x 4 for grids of few tiles (16^3: 61 against 74 us)
    static const TileCost f64[] = {{6, 1, 31.0, 31.0, 2.45}, {4, 1, 33.2, 33.2, 2.3}, {5, 1, 25.6, 25.6, 1.4}};
    // FP32: 32 x 8 tiles, three CTAs per SM; 32 x 16, one CTA; 16 x 16, two;
    // 32 x 4 for the smallest grids
    static const TileCost f32[] = {{0, 3, 3.5, 1.86, 2.3}, {3, 1, 3.76, 3.76, 2.3}, {2, 2, 3.5, 2.1, 2.3},
                                   {5, 4, 3.0, 1.2, 2.3}};
    // piecewise parabolic stages hold two more planes and a deeper halo: the
    // 512-thread tile is the fastest by a quarter (128^3: 327 against 422 us)
    static const TileCost f32_ppm[] = {{3, 1, 3.76, 3.76, 3.5}};
    const TileCost *c = fp32 ? (p.recon == HYDRO_RECON_PPM ? f32_ppm : f32) : f64;
    const int nc = fp32 ? (p.recon == HYDRO_RECON_PPM ? 1 : 4) : 3;
    LaunchPlan best{c[0].variant, -1};
    double tbest = 0.0;
    for (int i = 0; i < nc; ++i) {
        const TileShape s = TILE3D_SHAPES[c[i].variant];
        const long long W = (long long)((p.n[0] + s.tx - 1) / s.tx) * ((p.n[1] + s.ty - 1) / s.ty) * p.n[2];
        const long long k = std::min<long long>(c[i].ctas, (W + SMS - 1) / SMS);
        const long long planes = (W + SMS * k - 1) / (SMS * k);
        const double t = std::max(c[i].alone, k * c[i].unit) * (planes + c[i].fixed);
        if (i == 0 || t < tbest) {
            tbest = t;
            best.variant = c[i].variant;
        }
    }
    // an FP32 state well beyond the 129 MB L2: 32 x 8 tiles on z-chunks of 32
    // planes, whose many waves march neighbouring tiles at the same heights, so
    // that they find each other's halo rows in L2 (320^3: 1393 us, balanced
    // 1526, the 32 x 16 tile balanced 1539; 100x300x320: 545 against 556 and
    // 560; at 192^3, 141 MB, the balanced grid still wins, 343 against 351)
    const double bytes = (double)p.n[0] * p.n[1] * p.n[2] * 5 * 4;
    if (fp32 && p.recon != HYDRO_RECON_PPM && bytes > 160e6 && p.n[2] >= 32) best = LaunchPlan{0, 32};
    return best;
}

// Launch shape of the 2D step: march = threads of a marched strip, or 0 and
// the tile (tx x ty).
struct Plan2D {
    int march, tx, ty;
};

// Tiles (measured, us per MUSCL-Hancock step): FP64 16 x 16 cells (512^2 152
// against 160 with 32 x 8; 517x331 111 against 117), 16 x 8 while those fit one
// per SM (128^2: 26 against 33); FP32 32 x 16 (384^2 12.6 against 14.5), 16 x 16
// for the parabolic stages (1448^2 179 against 187).  A strip (linear states)
// is taken where its modelled time, row time x (rows per CTA + 2.2), is below
// the tiles' time per padded cell; the row times at full residency and the
// tiles' cell times are fitted at 512^2 to 2048^2.  The crossing lies near 700^2
// (FP64: 266 against 293) and 1024^2 (FP32: 38.3 against 37.9).
inline Plan2D plan2d(int nx, int ny, bool fp32, bool ppm)
{
    constexpr int SMS = 152;
    const auto along = [](long long n, int t) { return (n + t - 1) / t; };
    Plan2D best{0, fp32 && !ppm ? 32 : 16, 16};
    if (!fp32 && along(nx, 16) * along(ny, 8) <= SMS) best.ty = 8;
    if (ppm) return best;
    const double cells = (double)along(nx, best.tx) * best.tx * along(ny, best.ty) * best.ty;
    double tbest = fp32 ? 4.0 + 31.5e-6 * cells : 10.0 + 525e-6 * cells;
    struct Strip { int nt, ctas; double row; };
    static const Strip f64[] = {{128, 3, 22.9}};
    static const Strip f32[] = {{128, 6, 2.5}, {256, 3, 2.5}};
    const Strip *c = fp32 ? f32 : f64;
    for (int i = 0; i < (fp32 ? 2 : 1); ++i) {
        const double t = c[i].row * (along(along(nx, c[i].nt - 4) * ny, SMS * c[i].ctas) + 2.2);
        if (t < tbest) {
            tbest = t;
            best.march = c[i].nt;
        }
    }
    return best;
}

}  // namespace hydro
