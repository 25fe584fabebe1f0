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
// number of CTAs per tile; the one with the smallest estimate is taken.  In ns, for a call in a chain: a k-tile 360 + 0.9 bt
// (dequantization up to about 128 tokens, MMAs above); the drain of the last tile 9 bt, of every other tile of a CTA 12 bt above 128 tokens
// (one accumulator: nothing runs under it) and 600 below; a cut 1000, storing and reading the parts 9 bt + 2.5 bt for each of the others, and 350 for
// every trip to the L2 that brings them (two CTAs' parts at a time, 64 tokens at a time); 1100 where more than half of the SMs are taken, as
// the start of the next call of a chain then no longer hides behind this one.  Fitted to 4700 timings (4-bit and int8, 20 to 3100 tokens,
// 0.5 to 59 M weights), for the differences between candidates: over 400 sizes the choice costs 0.8 % over the best one.  It is no time of a call:
// what every candidate pays is left out, and under the power limit the clock is lower than in the fit.  Of 76 sizes the estimate is 27 % below the time
// of a chained call up to 10 us, 19 % from 10 to 30, 21 to 22 % above (2 to 50 %; 2048x4096x14336 142 and 168 us, 1024x4096x8584 44 and 53 to 67).
struct GemmSplit {
    int grid, rows;            // CTAs; rows of the grid: one, or one per tile
    bool whole_tiles;
    long long cost;            // the estimate
    Ranges ranges;             // of whole tiles, or of units
};
inline GemmSplit split_gemm(int tiles, int ktiles, int bt, int sm_count) {
    const long long units = (long long)tiles * ktiles;
    const int t_unit = 360 + 9 * bt / 10;
    const auto range = [&](int grid, long long len) {        // a CTA's range of k-tiles, with the drains of all its tiles
        return len * t_unit + 9 * bt + (len - 1) / ktiles * (bt > 128 ? 12 * bt : 600) + (2 * grid > sm_count ? 1100 : 0);
    };
    GemmSplit best;
    best.grid = tiles < sm_count ? tiles : sm_count;
    best.whole_tiles = true;
    best.cost = range(best.grid, (long long)((tiles + best.grid - 1) / best.grid) * ktiles);
    auto consider = [&](int grid, long long others) {        // others: CTAs besides the owner that hold a part of a tile
        const long long cost = range(grid, (units + grid - 1) / grid) + 1000 + 350 * ((others + 1) / 2) * ((bt + 63) / 64) + 9 * bt + 5 * others * bt / 2;
        if (cost < best.cost) { best.cost = cost; best.grid = grid; best.whole_tiles = false; }
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
    const int mean = (int)(units / sm_count), late_less = kLateNs / t_unit;
    const bool some_late = best.grid == sm_count && bt <= 128 && sm_count >= 8 * kLate;
    best.rows = !best.whole_tiles && best.grid % tiles == 0 ? tiles : 1;
    if (best.whole_tiles) best.ranges = Ranges::make(tiles, best.grid);
    else if (best.rows > 1) best.ranges = Ranges::make(ktiles, best.grid / best.rows, 1, -(kOwnNs / t_unit));
    else best.ranges = Ranges::make((int)units, best.grid, some_late ? kLate : 0, late_less < mean / 2 ? late_less : mean / 2);
    return best;
}

// Token tiles of a GEMM call.  `width`: 32, 64, 128 or 256, what the kernel is built for; the tiles are equal: 297 tokens are two tiles of 160
// columns (149 and 148 of them real), not 256 + 41.  The widest that M fills unpacks each weight least often and is right where the SMs
// have enough to do.  Where there are few output tiles a narrower one, at twice the unpacking, has more tiles for the SMs and less to put
// together (us, 4-bit: 256x4096x4096 17.5 in one tile of 256 cut four ways, 14.1 in two of 128 cut two ways, x8192x2048 22.5 and 15.7,
// 200x1024x4096 8.2 and 6.2, 128x2048x2048 9.0 and 7.2 in tiles of 64); taken where the estimate is at least 3 % smaller.
struct GemmTiling {
    int width, m_tiles, bt;    // bt: token columns of a tile, a multiple of 16
    bool pair;                 // two CTAs per tile of 256 columns; the split then counts pairs, and bt is a multiple of 32
    GemmSplit split;
};
inline int gemm_widest_tile(int M) { return M > 128 ? 256 : M > 64 ? 128 : M > 32 ? 64 : 32; }
inline GemmTiling choose_gemm_tiling(int M, int n_tiles, int ktiles, int sm_count) {
    GemmTiling best;
    long long best_cost = 0;
    for (int width = gemm_widest_tile(M), widest = width; width >= 32; width /= 2) {
        GemmTiling t;
        t.width = width;
        t.pair = false;
        t.m_tiles = (M + width - 1) / width;
        t.bt = ((M + t.m_tiles - 1) / t.m_tiles + 15) / 16 * 16;
        t.split = split_gemm(n_tiles * t.m_tiles, ktiles, t.bt, sm_count);
        const long long cost = width == widest ? t.split.cost : t.split.cost * 103 / 100;
        if (width == widest || cost < best_cost) { best = t; best_cost = cost; }
    }
    // Pairs of CTAs, for the widest tile: 6 % less for the work (see gemm.cu), 1200 ns more for a call (a cluster starts later and overlaps
    // less with its neighbours), token columns in steps of 32 and weight columns in steps of 256.  With both sides measured over 133 sizes the estimate
    // takes the better one to within 0.2 % on average, 2.8 % at worst: us alone / in pairs 200x512x16384 7.3 / 8.6, 400x1536x8960 12.3 / 13.7, 700x8192x8192
    // 75.9 / 78.1 (tiles of 240 tokens become 256), 512x4096x8584 31.1 / 29.5, 1024x11008x4096 71.8 / 67.0, 2048x8192x8192 230 / 219.
    if (best.width == 256 && n_tiles > 1 && sm_count > 1) {
        GemmTiling t = best;
        t.pair = true;
        t.bt = ((M + t.m_tiles - 1) / t.m_tiles + 31) / 32 * 32;
        t.split = split_gemm((n_tiles + 1) / 2 * t.m_tiles, ktiles, t.bt, sm_count / 2);
        if (t.split.cost * 94 / 100 + 1200 < best_cost) best = t;
    }
    return best;
}

}  // namespace tf
