// xm_plan.cuh -- sizes of an index build's partition, from the numbers of rows
// and zones alone (host code without CUDA, so that it is tested by itself).
#pragma once

#include <stdint.h>

namespace xm {

// Units: consecutive cells whose first rows fall in the same window of
// 2^kUnitRowBits rows, of zones in the same kUnitZones, form one unit; a part
// of a zone, and a cell of more rows than a window, begins a unit (which ends
// with it: the next cell begins in a later window). So a unit of several
// cells holds fewer than two windows' rows, and only a unit of one cell can
// hold more than k_place_b stages.
constexpr int kUnitRowBits = 9, kUnitZoneBits = 6;
constexpr int kUnitZones = 1 << kUnitZoneBits;

// Digits of a split: the units of a small catalogue, or the bins of the first
// of two splits, or the units of a bin in the second. A bin covers zones with
// the same z >> kBinZoneBits (records carry the low bits of their zone).
constexpr int kMaxUnits = 2048, kMaxBins = 1024, kMaxDigits = 1536;
constexpr int kBinZoneBits = 11;
constexpr int kMaxZones = 648000;  // of at least 1 arcsec
static_assert((kMaxZones >> kBinZoneBits) + 2 <= kMaxBins, "bins of a few rows fit every zone count");

// The zone count's 16-bit counters: a block adds kCountThreads * kCountLoads
// sources a loop, a barrier every kFoldLoops loops. A counter is below 0x8000
// after a barrier; before the next it takes at most all that is added between
// them, stays below 2^16 (no carry into its neighbour) and reaches 0x8000 once.
constexpr int kCountThreads = 1024, kCountLoads = 4, kFoldLoops = 7;
static_assert(kCountThreads * kCountLoads * kFoldLoops < 0x8000, "16-bit counters of zones hold");

struct BuildPlan {
    bool two;            // two splits: into bins, and those into units
    int kb;              // a bin's window holds 2^kb rows
    int nbins;           // bins (0: one split, into units), at most kMaxBins
    int64_t cells_cap;   // cells and units at most
    int64_t units_cap;
};

// The bins of one split are the units; past kMaxUnits units (some 4e5 rows in
// zones of 20 arcsec, 5.2e5 in the widest) there are two splits: into bins of
// 2^kb rows, at least a unit's window, so that units do not straddle bins. The
// rows make 384 to 767 bins, and the zones one more per 2^kBinZoneBits (316 in
// zones of 1 arcsec); where the two together would pass kMaxBins the bins hold
// twice the rows.
inline BuildPlan build_plan(int64_t n, int32_t nz) {
    BuildPlan p;
    p.cells_cap = nz;
    p.units_cap = 2 * (n >> kUnitRowBits) + (nz >> kUnitZoneBits) + 1;
    p.two = p.units_cap > kMaxUnits;
    p.kb = kUnitRowBits;
    p.nbins = 0;
    if (!p.two) return p;
    const int64_t zone_bins = (nz >> kBinZoneBits) + 1;
    while ((n >> (p.kb + 1)) >= 384 || (n >> p.kb) + zone_bins > kMaxBins) p.kb++;
    p.nbins = (int)((n >> p.kb) + zone_bins);
    // parts of zones: of half of kPartRows rows or more, of zones past kPartMin
    p.cells_cap += n / 200 + 16;
    p.units_cap += n / 160 + 16;
    return p;
}

}  // namespace xm
