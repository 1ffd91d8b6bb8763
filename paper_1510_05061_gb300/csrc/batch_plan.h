// batch_plan.h -- how a batch's 3D columns are shared out among the CTAs of the
// persistent step unless the caller or the autotuner chooses a tile and chunks.
#pragma once

#include <algorithm>
#include <vector>

#include "hydro_internal.h"
#include "plan.h"

namespace hydro {

// Tile and cut of a batch's 3D columns: all columns end to end, cut into
// `shares` shares of `budget` planes, each piece of a column costing `fixed`
// planes beside its own.
struct BatchPlan {
    int variant, shares;
    double budget, fixed;
};

// The cut a batch of fixed membership takes by default: the tile (only: that
// variant) and number of shares with the least modelled time,
//   time = max(alone, k unit) budget,   budget = (planes + fixed pieces) / shares,
// alone and unit as in default_plan, k shares per SM.  The chunks of at most 64
// planes that the CTAs claimed before, largest first, left most of the chip idle
// on small batches and a last round on the others; the costs are fitted to
// sweeps of those chunks, 8 to 256 planes long, whose times a simulated claim
// order reproduces within 6 % rms.  us per step, chunks -> shares, FP32: 3 boxes
// of 16^3 to 40^3 with a 2D box 162 -> 40, 6 of 24^3 to 90^3 with two 247 -> 89,
// 11 of 32^3 to 128^3 with three 394 -> 362; FP64 6 boxes of 24^3 to 90^3 1647 ->
// 894, 11 of 32^3 to 128^3 5038 -> 4560.
//
// FP32 states whose two buffers pass the 129 MB L2 take the 32 x 16 tile, which
// re-reads the least halo (8 boxes of 36^3 to 128^3, 101 MB: 298 against 330 with
// 16 x 16), and those well beyond it keep the chunks (shares = 0): their CTAs
// march neighbouring tiles at the same heights and find each other's halo rows
// in L2 (default_plan's line; 126 MB: 362 shared, 394 in chunks; 344 MB 1310 and
// 1136; 1.3 GB 4200 and 3641).
constexpr TileCost BATCH_F64[3] = {{2, 1, 24.0, 24.0, 2.0}, {0, 1, 28.2, 28.2, 2.0}, {1, 1, 19.5, 19.5, 2.0}};
constexpr TileCost BATCH_F32[3] = {{2, 2, 3.5, 1.8, 3.0}, {7, 1, 3.5, 3.5, 3.0}, {1, 2, 2.5, 1.0, 3.0}};

inline BatchPlan batch_plan(const hydro_problem *const *p, int count, bool fp32, int only)
{
    constexpr int SMS = 152;
    BatchPlan best{};
    double tbest = 0.0, cells = 0.0;
    for (int j = 0; j < count; ++j) cells += (double)p[j]->n[0] * p[j]->n[1] * p[j]->n[2];
    if (fp32 && cells * 5 * 4 > 160e6) return best;
    const bool beyond_l2 = fp32 && 2 * cells * 5 * 4 > 129e6;
    for (int i = 0; i < 3; ++i) {
        const TileCost &c = fp32 ? BATCH_F32[i] : BATCH_F64[i];
        if (only >= 0 ? only % 4 != c.variant % 4 : beyond_l2 && i != 1) continue;
        const TileShape s = TILE3D_SHAPES[c.variant];
        long long cols = 0, W = 0;
        for (int j = 0; j < count; ++j) {
            const long long tiles = (long long)((p[j]->n[0] + s.tx - 1) / s.tx) * ((p[j]->n[1] + s.ty - 1) / s.ty);
            cols += tiles;
            W += tiles * p[j]->n[2];
        }
        for (int k = 1; k <= c.ctas; ++k) {
            const long long G = std::min<long long>(SMS * k, W);
            const double budget = (W + c.fixed * (cols + G)) / G, t = std::max(c.alone, k * c.unit) * budget;
            if (best.shares == 0 || t < tbest) {
                tbest = t;
                best = BatchPlan{only >= 0 ? only : c.variant, (int)G, budget, c.fixed};
            }
        }
    }
    return best;
}

// Longest z-chunk of an instance's column where the columns are claimed in
// chunks of nearly equal length: long chunks re-read few halo planes (4 per
// chunk), and the largest-first claim order keeps the SMs balanced even when
// whole columns are single items.
constexpr int BATCH_ZCHUNK_DEFAULT = 64;

inline int batch_chunk(int nz, int longest)
{
    const int nch = (nz + longest - 1) / longest;
    return (nz + nch - 1) / nch;
}

// Whether an FP32 batch takes the plan's shares rather than chunks with the
// tile of variant `otherwise`.  The shares cut the columns into more pieces,
// each costing `fixed` planes: a batch that has the chip to itself gains (the
// CTAs end together), but where several batches step on streams of their own,
// idle CTAs are filled by the others and only the work counts.  So the shares
// are taken where their modelled work is no more than the chunks', or where even
// three batches' chunks leave CTAs idle (busy, the part of one batch's CTAs that
// its chunks keep working, below a third; up to a half a ratio a little below 1
// is made up: at 0.42 0.945: 1.010, at 0.46 0.927: 0.936).  Three batches at once, shares
// against chunks, at a ratio of modelled works of 0.956 (5 boxes of 35^3 to
// 115^3): 0.952, 0.991 (38^3 to 134^3): 0.992, 1.008: 1.010, 1.03: 1.03; busy
// below a third 1.01 to 3.2.  Alone the shares' gain is 1.1 to 1.4 where they are given
// up, 1.07 to 4.9 where they stay.  The 16 x 16 tile's halo rows cost 3 to 5 %
// more where three batches' buffers are well beyond the L2 (from 100 MB each;
// 22^3 to 112^3, ratio 1.026: 0.977); from 190 MB the shares are about 1 %
// better than the ratio (32^3 to 128^3, 0.993: 1.004).
inline bool shares_pay(const BatchPlan &plan, const hydro_problem *const *p, int count, int otherwise)
{
    constexpr int SMS = 152;
    const TileCost *s = nullptr, *c = nullptr;
    for (const TileCost &t : BATCH_F32) {
        if (t.variant % 4 == plan.variant % 4) s = &t;
        if (t.variant % 4 == otherwise % 4) c = &t;
    }
    if (!s || !c) return s != nullptr;
    const TileShape ss = TILE3D_SHAPES[plan.variant], cs = TILE3D_SHAPES[otherwise];
    double bytes = 0.0, shares = plan.fixed * plan.shares, chunks = 0.0, longest = 0.0;
    for (int j = 0; j < count; ++j) {
        const int *n = p[j]->n, zc = batch_chunk(n[2], BATCH_ZCHUNK_DEFAULT);
        const auto tiles = [n](const TileShape &t) { return (double)((n[0] + t.tx - 1) / t.tx) * ((n[1] + t.ty - 1) / t.ty); };
        bytes += 2.0 * 5 * 4 * n[0] * n[1] * n[2];
        shares += tiles(ss) * (n[2] + plan.fixed);
        chunks += tiles(cs) * (n[2] + c->fixed * ((n[2] + zc - 1) / zc));
        longest = std::max(longest, zc + c->fixed);
    }
    const double spill = plan.variant % 4 == 2 && bytes > 100e6 ? 1.05 : (bytes > 190e6 ? 0.99 : 1.0);
    const double ratio = c->unit * chunks / (spill * s->unit * shares), busy = chunks / (SMS * c->ctas * longest);
    return busy < 1.0 / 3 || ratio >= (busy < 0.5 ? 0.92 + 0.39 * (busy - 1.0 / 3) : 1.0);
}

// The 3D columns of a batch cut into equal shares (batch_plan), one for each
// CTA: the columns end to end, instance by instance, a share's pieces
// linked by `next`.  While the list is built an item's `next` is its share.
struct CutState {
    int shares;      // shares begun
    double room;     // planes the last share still takes
};

inline void cut_columns(const BatchPlan &plan, int inst, int tiles, int nz, CutState &c, std::vector<BatchItem> &items,
                 int *local)
{
    for (int t = 0; t < tiles; ++t)
        for (int z = 0; z < nz;) {
            if (c.shares == 0 || (c.room < plan.fixed + 1.0 && c.shares < plan.shares)) {
                c.shares += 1;
                c.room += plan.budget;   // (and what the share before left of its own)
            }
            int n = std::max(1, (int)(c.room - plan.fixed));
            if (c.shares == plan.shares || n > nz - z) n = nz - z;
            items.push_back(BatchItem{inst, t, z, z + n, (*local)++, c.shares - 1});
            c.room -= n + plan.fixed;
            z += n;
        }
}

// The shares' first pieces, then the others, each linked to the share's next.
inline std::vector<BatchItem> claim_order(const std::vector<BatchItem> &items)
{
    std::vector<BatchItem> out;
    out.reserve(items.size());
    for (size_t k = 0; k < items.size(); ++k)
        if (k == 0 || items[k].next != items[k - 1].next) out.push_back(items[k]);
    int follow = (int)out.size(), first = -1;
    for (size_t k = 0; k < items.size(); ++k) {
        const bool more = k + 1 < items.size() && items[k + 1].next == items[k].next;
        int at;
        if (k == 0 || items[k].next != items[k - 1].next) {
            at = ++first;
        } else {
            at = (int)out.size();
            out.push_back(items[k]);
        }
        out[at].next = more ? follow++ : -1;
    }
    return out;
}

}  // namespace hydro
