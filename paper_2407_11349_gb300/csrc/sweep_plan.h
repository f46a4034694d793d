// How the symmetric sweep of a problem, or of a batch, is cut into work items, on
// the host.  Plain C++ without allocations: the allocation-free entry point plans
// its sweep too, and the rule can be checked without a GPU.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

namespace hk {

// Work items of `chunk` column tiles, by the row-tile kernel of the selected
// variant (k_sweep) or by the column-split kernel (k_sweep_cs); with `band`, the
// row tiles leave out the columns of their own rows, which the column-split kernel
// takes.
struct SweepPlan {
    bool split;
    int chunk;
    bool band;
};

constexpr int PLAN_TC = 256;      // events per column tile
constexpr int PLAN_CHUNK = 16;    // longest item that a plan chooses by itself

// The row-tile variant (rows per tile, resident CTAs per SM) and the rows of the
// column-split kernel's items.
struct PlanKernels {
    int tile_rows, resident, split_rows;
};

// Column tiles of all row tiles of `tr` rows in the causal triangle of n events.
inline int64_t plan_units(int64_t n, int tr) {
    int64_t u = 0;
    for (int64_t r = 0; r < n; r += tr) u += (std::min<int64_t>(r + tr, n) + PLAN_TC - 1) / PLAN_TC;
    return u;
}

inline int pow2_floor(double v, int cap) {
    int p = 1;
    while (2 * p <= cap && 2 * p <= v) p *= 2;
    return p;
}

// The plan for `count` problems of sizes ns[] swept together.
//   chunk: most column tiles per item, up to PLAN_CHUNK (0: PLAN_CHUNK); above that
//   many, exactly that many.
//   band: the work list may have a diagonal band (SweepPlan).
//
// With a band.  A row tile's units that lie partly above the diagonal leave
// warps idle, and a persistent kernel ends on whole items of up to PLAN_CHUNK units
// (N = 100,000: 62 units per SM).  So the row tiles take only the columns
// below their own rows, and the column-split kernel takes the band between;
// it starts while the row tiles' last items run and fills the SMs they leave:
// N = 100,000 3.96 -> 3.75 ms, 50,000 1.047 -> 0.956, 30,000 0.402 -> 0.379.
// Items are as long as the rounds over the SMs come out shortest, in units of
// one row tile x one column tile (62 us of one SM); an item's row flush costs 0.07
// of one.
//
// Row tiles with the band, or the column-split kernel alone, by what each takes in
// these units, fitted to 50 sizes from 4,000 to 65,536 events at 152 SMs (within 4%
// up to 25,000):
//   - column split: 1.12 times the pairs' units per SM, and 0.2;
//   - row tiles: 0.93 for each unit of an item and 0.06 for the item, in every round,
//     and 0.3.  The band (1.1 times its pairs' units) runs beside them, on the SMs that
//     the last round leaves idle and beside a last row tile with at most half of its
//     warps' rows (0.58 of its time); what finds no room adds itself and 0.65.
// From 4.9 units of pairs per SM (27,700 events) the row tiles are always taken: they
// win by up to 11% there (43,000 events 0.722 ms for 0.801; 33,000, the one exception
// seen, 0.481 for 0.478).  Below, they win where they fill their rounds: 17,103 events
// 0.137 ms for 0.143, 24,550 0.248 for 0.275; but 10,250 0.064 for 0.075, 17,500
// 0.144 for 0.181 and 22,000 0.226 for 0.243 are column split.  Of the sizes timed the
// slower plan is taken at 27,000 (0.337 for 0.329) and where the two are within 2%.
//
// Without: column split where the row tiles cover more than 1.1 times its pairs
// (N below about 36,000); items for 16 per SM.
//
// Column-split items: from three items per SM up to 4 tiles (N = 17,103:
// 0.144 ms with 4, 0.163 with 1; N = 5,000: 0.023 with 1, 0.028 with 2), and 8
// where 64 items per SM are left.
inline SweepPlan sweep_plan(const int64_t* ns, size_t count, int sms, const PlanKernels& k, int chunk, bool band) {
    const int tr = k.tile_rows;
    double rows = 0.0, split = 0.0;  // units: tr x PLAN_TC, split_rows x PLAN_TC
    // units below the row tiles' own rows; those of them without rows (of a last row
    // tile that is partly filled); and the SM time that such a tile leaves
    double below = 0.0, dead = 0.0, thin = 0.0;
    for (size_t p = 0; p < count; ++p) {
        const int64_t n = ns[p];
        const double full = static_cast<double>((n - 1) / tr);  // row tiles with columns below them
        rows += static_cast<double>(plan_units(n, tr));
        split += static_cast<double>(plan_units(n, k.split_rows));
        below += full * (full + 1.0) / 2.0 * (tr / PLAN_TC);
        const double last = static_cast<double>(n - static_cast<int64_t>(full) * tr) / tr;
        dead += full * (tr / PLAN_TC) * (1.0 - last);
        thin += last <= 0.5 ? 0.42 * full * (tr / PLAN_TC) : 0.0;
    }
    SweepPlan pl{rows * tr > 1.1 * split * k.split_rows, chunk, false};
    int best = pow2_floor(rows / (16.0 * sms), PLAN_CHUNK);
    if (band) {
        const double slots = static_cast<double>(sms) * k.resident, all = split * k.split_rows / tr, flush = 0.07;
        double least = 1e300;
        for (int c = PLAN_CHUNK; c >= 1; c /= 2) {
            const double items = below / c;
            const double t = std::max(std::ceil(items / slots) * (c + flush), (all + flush * items) / slots);
            if (t < least) {
                least = t;
                best = c;
            }
        }
        const double rounds = std::ceil(below / best / slots);
        const double room = (slots * rounds - below / best) * (best + flush) + thin;
        const double left = 1.1 * (all - below + dead) - room;  // of the band, when the row tiles end
        const double tiles = rounds * (0.93 * best + 0.06) + 0.3 + (left > 0.0 ? left / slots + 0.65 : 0.0);
        pl.split = below == 0.0 || (all < 4.9 * slots && 1.12 * all / slots + 0.2 < tiles);
        pl.band = !pl.split;
    }
    if (pl.split) best = std::max(pow2_floor(split / (3.0 * sms), 4), pow2_floor(split / (64.0 * sms), 8));
    if (chunk <= PLAN_CHUNK) pl.chunk = chunk <= 0 ? best : std::min(best, chunk);
    return pl;
}

}  // namespace hk
