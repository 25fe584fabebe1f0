// How work is dealt out to CTAs: the ranges of the GEMV and the GEMM, and the GEMM's choice of a split.  No CUDA in it but the mark that
// lets kernels use the ranges.
#pragma once
#include <stdint.h>

#include "layout.h"

namespace tf {

// How a sequence of units (tiles) is dealt out to CTAs as contiguous ranges.  A CTA finds its range without a division, which would
// sit between its start and its first copy: of the first on_time CTAs `more` get size + 1 units, the rest size, and the others, the late
// ones, likewise.  (GEMM 24x4096x14336 18.2 us with two divisions per CTA, 16.8 without, 40x8192x8192 20.5 and 18.8; GEMV 16 tokens
// 14336x4096 10.9 and 10.5, 4 tokens 9.0 and 8.8.)
// CTAs start in the order of their index as SMs come free; in a chain of kernels that take a whole SM each, the last ten or so start up
// to 3 us behind the others, and the call ends with them.  So they can be given shorter ranges.
struct Ranges {
    int on_time, size, more, bulk;             // the first on_time CTAs share the first bulk units
    int late_size, late_more;
    // `late` CTAs get about `less` units less than the others (less than 0: more).  ctas > late >= 0; with units >= ctas every range
    // has a unit: the owner of a cut tile waits for every CTA that holds a part of it.
    static Ranges make(int units, int ctas, int late = 0, int less = 0) {
        Ranges r;
        int late_units = 0;
        if (late > 0) {
            late_units = late * ((units + late * less) / ctas - less);
            if (late_units > units - (ctas - late)) late_units = units - (ctas - late);
            if (late_units < late) late_units = late;
        }
        r.on_time = ctas - late;
        r.bulk = units - late_units;
        r.size = r.bulk / r.on_time; r.more = r.bulk % r.on_time;
        r.late_size = late > 0 ? late_units / late : 0; r.late_more = late > 0 ? late_units % late : 0;
        return r;
    }
    TF_HD int start(int cta) const {
        const int c = cta - on_time;
        return c <= 0 ? cta * size + (cta < more ? cta : more) : bulk + c * late_size + (c < late_more ? c : late_more);
    }
    TF_HD int owner(int unit) const {
        const bool late = unit >= bulk;
        const int u = late ? unit - bulk : unit, q = late ? late_size : size, m = late ? late_more : more, head = m * (q + 1);
        return (late ? on_time : 0) + (int)(u < head ? (uint32_t)u / (uint32_t)(q + 1) : m + (uint32_t)(u - head) / (uint32_t)q);
    }
};

// How the work is spread over the CTAs.  Whole tiles only: nothing has to be put together, but the last wave of tiles may
// leave SMs idle.  Split of the (tile, k-tile) units over `grid` CTAs: the owner of a cut tile adds up the others' parts
// at the end of its range.  The candidates are one CTA per SM, in equal ranges, and, where there are fewer tiles than SMs, every whole
// number of CTAs per tile; the one with the smallest estimate is taken.  In ns: a k-tile 350 + 1.5 bt (dequantization up to
// about 128 tokens, MMAs above), a cut 3000 (parts stored, flagged and seen) and 550 for every trip to the L2 that brings the
// parts: two CTAs' at a time, 64 tokens at a time; 1000 less where a range is longer than two tiles, whose first part was
// stored long before.  (With 450 + 1.5 bt and 2000, the times of an earlier form: 33x1536x8960 8.22 us, now 7.08, 128x2048x11008 12.97 and
// 11.7, 100x4096x1024 10.8 and 10.1, 90x4096x2048 int8 10.6 and 10.1; others within 1 %.)
struct GemmSplit {
    int grid, rows;            // CTAs; rows of the grid: one, or one per tile
    bool whole_tiles;
    Ranges ranges;             // of whole tiles, or of units
};
inline GemmSplit split_gemm(int tiles, int ktiles, int bt, int sm_count) {
    const long long units = (long long)tiles * ktiles, t_unit = 350 + 3 * bt / 2;
    GemmSplit best;
    best.grid = tiles < sm_count ? tiles : sm_count;
    best.whole_tiles = true;
    long long best_cost = (long long)((tiles + best.grid - 1) / best.grid) * ktiles * t_unit;
    auto consider = [&](int grid, long long others) {        // others: CTAs besides the owner that hold a part of a tile
        const long long len = (units + grid - 1) / grid;
        const long long cost = len * t_unit + 3000 - (len >= 2 * ktiles ? 1000 : 0) + 550 * ((others + 1) / 2) * ((bt + 63) / 64);
        if (cost < best_cost) { best_cost = cost; best.grid = grid; best.whole_tiles = false; }
    };
    for (int per_tile = 2; per_tile * tiles <= sm_count && per_tile <= ktiles; ++per_tile) consider(per_tile * tiles, per_tile - 1);
    if (tiles % sm_count != 0 && units >= sm_count) consider(sm_count, (ktiles + units / sm_count - 1) / (units / sm_count));
    // Up to 128 tokens, one CTA per SM: the last ten CTAs get what they are late by, about 2 us, less (77x2944x11016 14.3 -> 14.1 us, 24x4096x14336
    // 16.8 -> 16.3, 40x8192x8192 18.8 -> 18.6, 128 tokens no difference).  Wider tiles are long calls, and fewer SMs than CTAs leave
    // nobody late.
    constexpr int kLate = 10, kLateNs = 1600;
    // Several CTAs per tile: the owner of the last k-tile takes as much more as its k-tiles last while the others' parts are on
    // their way (us with even shares / this: 128x4096x4096 12.5 / 12.3, 60x4096x1024 8.25 / 8.05, int8 300x4096x4096 17.7 / 17.2).
    constexpr int kOwnNs = 1500;
    const int mean = (int)(units / sm_count), late_less = (int)(kLateNs / t_unit);
    const bool some_late = best.grid == sm_count && bt <= 128 && sm_count >= 8 * kLate;
    best.rows = !best.whole_tiles && best.grid % tiles == 0 ? tiles : 1;
    if (best.whole_tiles) best.ranges = Ranges::make(tiles, best.grid);
    else if (best.rows > 1) best.ranges = Ranges::make(ktiles, best.grid / best.rows, 1, -(int)(kOwnNs / t_unit));
    else best.ranges = Ranges::make((int)units, best.grid, some_late ? kLate : 0, late_less < mean / 2 ? late_less : mean / 2);
    return best;
}

}  // namespace tf
