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

// The balanced grid (min(resident CTAs, plane-tiles) CTAs with equal shares of
// the plane-tiles) has no partial last wave and repeats fewer planes than the
// z-chunks of 8 to 64 planes taken before (a piece predicts two planes and
// stages four beyond its own): measured on GB300, us per MUSCL-Hancock step, same
// tile and kernels, FP64 16^3 288 -> 74, 101x75x130 1251 -> 1001, 128^3 1999 ->
// 1751; FP32 32^3 40 -> 19, 128^3 147 -> 114.  Where one wave of CTAs holds every
// tile, z-chunks of one piece per CTA can beat it, because its CTAs march parts
// of two columns: FP64 64^3 232 against 248, 80^3 374 against 412.
//
// Tile and partition are those with the least modelled time, with
//   time = max(alone, k unit) (planes + pieces fixed),   k = min(ctas, ceil(W / SMs)),
// planes and pieces of the longest CTA, W = plane-tiles (tiles x nz), `unit` the
// time of a plane of one CTA divided by the CTAs sharing an SM, `alone` a
// plane's latency on an SM of its own, `fixed` the planes' worth of work a piece
// repeats.  The constants are fitted to sweeps from 16^3 to 320^3, 200x40x100 and
// 300x40x200 and reproduce their times within 10 %.
struct TileCost {
    int variant, ctas;
    double alone, unit, fixed;   // us
};

inline LaunchPlan default_plan(const hydro_problem &p)
{
    constexpr int SMS = 152;
    const bool fp32 = p.precision == HYDRO_FP32;
    // FP64: 16 x 16 tiles (128^3: 1356 us, 32 x 8 1593, 32 x 4 2141), 32 x 8 where
    // those waste more of the grid, 32 x 4 for grids of few tiles (16^3: 50
    // against 70 us)
    static const TileCost f64[] = {{2, 1, 24.0, 24.0, 1.2}, {0, 1, 28.2, 28.2, 1.2}, {1, 1, 19.5, 19.5, 1.2}};
    // FP32: 32 x 8 tiles, three CTAs per SM; 32 x 16, one CTA; 16 x 16, two;
    // 32 x 4 for the smallest grids
    static const TileCost f32[] = {{0, 3, 3.5, 1.86, 1.2}, {3, 1, 3.76, 3.76, 1.2}, {2, 2, 3.5, 2.1, 1.2},
                                   {5, 4, 3.0, 1.2, 1.2}};
    // piecewise parabolic stages hold two more planes and a deeper halo: the
    // 512-thread tile is the fastest by a quarter (128^3: 327 against 422 us)
    static const TileCost f32_ppm[] = {{3, 1, 3.76, 3.76, 1.8}};
    const TileCost *c = fp32 ? (p.recon == HYDRO_RECON_PPM ? f32_ppm : f32) : f64;
    const int nc = fp32 ? (p.recon == HYDRO_RECON_PPM ? 1 : 4) : 3;
    LaunchPlan best{c[0].variant, -1};
    double tbest = 0.0;
    for (int i = 0; i < nc; ++i) {
        const TileShape s = TILE3D_SHAPES[c[i].variant];
        const long long W = (long long)((p.n[0] + s.tx - 1) / s.tx) * ((p.n[1] + s.ty - 1) / s.ty) * p.n[2];
        const long long k = std::min<long long>(c[i].ctas, (W + SMS - 1) / SMS);
        const long long planes = (W + SMS * k - 1) / (SMS * k);
        const long long tiles = W / p.n[2], G = SMS * k;
        const double tp = std::max(c[i].alone, k * c[i].unit);
        // the balanced grid's longest CTA, which marches parts of two columns
        // unless the shares divide the columns; or, where one wave holds every
        // tile, z-chunks of one piece each
        const bool split = planes > 1 && !(G % tiles == 0 && p.n[2] % (G / tiles) == 0);
        double t = tp * (planes + (split ? 2 : 1) * c[i].fixed);
        int z = -1;
        if (tiles <= G) {
            const int zc = (int)((p.n[2] + G / tiles - 1) / (G / tiles));
            if (tp * (zc + c[i].fixed) < t) {
                t = tp * (zc + c[i].fixed);
                z = zc;
            }
        }
        if (i == 0 || t < tbest) {
            tbest = t;
            best = LaunchPlan{c[i].variant, z};
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

// z partition of the tile of variant v chosen by the caller: planes per CTA,
// -1 for the balanced grid, or 0 for chunks in several waves (the caller's).
// One piece per CTA where a single wave of the kernel's resident CTAs holds every
// tile and the balanced grid would split columns, else the balanced grid, as in
// default_plan.  Measured on 24^3 to 320^3, us, several-wave chunks -> this:
// FP32 24^3 25 to 38 -> 13 to 16, 96^3 56 to 79 -> 54 to 66, 128^3 122 to 179 -> 112 to
// 142, FP64 64^3 234 to 344 -> 234 to 324.  The FP32 32 x 8 tile keeps those chunks
// where the state's buffers pass 110 MB, the 16 x 16 tile where they pass 250 MB:
// their neighbouring tiles march at the same heights and find each other's halo
// rows in L2 (32 x 8, 192^3: 337 against 355, Runge-Kutta 660 against 864).
inline int tile_zchunk(const hydro_problem &p, int v)
{
    constexpr int SMS = 152;
    const TileShape s = TILE3D_SHAPES[v];
    const bool fp32 = p.precision == HYDRO_FP32, rk = p.scheme != HYDRO_SCHEME_HANCOCK, ppm = p.recon == HYDRO_RECON_PPM;
    const bool async = v >= 4 && !rk;
    const int shape = v % 4;
    // resident CTAs that share an SM without loss
    const int k = !fp32 || shape == 3 ? 1 : (shape == 0 && !async && !ppm ? 3 : (shape == 2 && ppm ? 1 : 2));
    const double buffers = (rk ? 3.0 : 2.0) * 5 * (fp32 ? 4 : 8) * p.n[0] * p.n[1] * p.n[2];
    if (fp32 && !async && !ppm && ((shape == 0 && buffers > 110e6) || (shape == 2 && buffers > 250e6))) return 0;
    const long long T = (long long)((p.n[0] + s.tx - 1) / s.tx) * ((p.n[1] + s.ty - 1) / s.ty), G = (long long)SMS * k;
    const long long planes = (T * p.n[2] + G - 1) / G;
    if (T > G) return -1;
    const double fixed = ppm ? 1.8 : 1.2;
    const bool split = planes > 1 && !(G % T == 0 && p.n[2] % (G / T) == 0);
    const int zc = (int)((p.n[2] + G / T - 1) / (G / T));
    return zc + fixed < planes + (split ? 2 : 1) * fixed ? zc : -1;
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
// is taken where its modelled time, base + row x rows per CTA, is below the
// tiles', a constant and a time per padded cell.  FP64: fitted at 512^2 to 2048^2;
// the crossing lies near 700^2 (266 against 293).  FP32: fitted to 46 shapes from
// 61^2 to 2048^2, 40 x 30000 and 2600 x 48 within 6 %, the tiles' time taken 3 %
// short so that the Runge-Kutta stages, whose strips cost a little more, gain too;
// us, strip and tile: 600^2 19.7 and 18.3, 2600 x 100 18.6 and 15.9, 800 x 700 25.5
// and 23.7, 250 x 2600 24.6 and 27.6, 1024^2 36.1 and 37.4, 2048^2 101 and 129.
inline Plan2D plan2d(int nx, int ny, bool fp32, bool ppm)
{
    constexpr int SMS = 152;
    const auto along = [](long long n, int t) { return (n + t - 1) / t; };
    Plan2D best{0, fp32 && !ppm ? 32 : 16, 16};
    if (!fp32 && along(nx, 16) * along(ny, 8) <= SMS) best.ty = 8;
    if (ppm) return best;
    const double cells = (double)along(nx, best.tx) * best.tx * along(ny, best.ty) * best.ty;
    double tbest = fp32 ? 7.8 + 28.9e-6 * cells : 10.0 + 525e-6 * cells;
    struct Strip { int nt, ctas; double base, row; };
    static const Strip f64[] = {{128, 3, 50.4, 22.9}};
    static const Strip f32[] = {{128, 6, 13.0, 2.1}, {256, 3, 11.5, 2.15}};
    const Strip *c = fp32 ? f32 : f64;
    for (int i = 0; i < (fp32 ? 2 : 1); ++i) {
        const double t = c[i].base + c[i].row * along(along(nx, c[i].nt - 4) * ny, SMS * c[i].ctas);
        if (t < tbest) {
            tbest = t;
            best.march = c[i].nt;
        }
    }
    return best;
}

}  // namespace hydro
