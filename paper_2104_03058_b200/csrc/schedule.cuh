// Launch schedule shared by the gather kernels: how a sweep over one column tile of one chunk is cut
// into block ranges (hub segments first, then the degree classes from high to low).
#pragma once

#include "common.cuh"

namespace gnnfd {

#ifndef GNNFD_GATHER_BLOCK
#define GNNFD_GATHER_BLOCK 256
#endif
constexpr int kBlock = GNNFD_GATHER_BLOCK;      // threads per block of the gather kernels
constexpr int kMaxRanges = kNumBins - 1 + kOctaves;     // hub segments, the octaves of the fourth class, three classes
constexpr int kMaxGridY = 65535;               // chunks one launch of a gather kernel covers (grid y)

struct Range {
    int32_t first_block;   // first block (within one column tile of one sweep) of this range
    int32_t item_first;    // rows: place of the first one to take in row_order
    int32_t item_step;     // rows: -1 from the longest row down, 1 from the shortest up
    int32_t item_count;
    int32_t ep_log2;       // log2 of the edge-parallel groups per row
    int32_t hub;           // 1: items are hub segments writing partial results
    int32_t warps_log2;    // log2 of the warps that share an item (more than one only where a row has all lanes of a warp)
};

inline int ilog2(int x) { int l = 0; while ((1 << l) < x) ++l; return l; }

// Edge-parallel groups per row for a degree class, at most (the lanes a row may use limit them further).  The gathers: rows of up to 32
// entries get one group, rows of up to 128 four: a short row is bound by its chain of dependent loads
// (row number -> row pointer -> indices -> features), so more rows in flight per block beat more lanes per
// row (config 2 at 64 columns 0.128 -> 0.115 ms, GAT on config 3 0.189 -> 0.167 ms, config 5 at 64 columns
// 1.81 -> 1.62 ms against 4 and 8 groups).
struct Groups { int want[kNumBins]; };

inline Groups gather_groups()
{
#ifndef GNNFD_EP_BIN1
#define GNNFD_EP_BIN1 1
#endif
#ifndef GNNFD_EP_BIN2
#define GNNFD_EP_BIN2 4
#endif
#ifndef GNNFD_EP_BIN3
#define GNNFD_EP_BIN3 32
#endif
    return Groups{{1, GNNFD_EP_BIN1, GNNFD_EP_BIN2, GNNFD_EP_BIN3, 32}};
}

// Warps of a block that share a row (or hub segment) of up to `entries` entries.  A warp walks its row in steps of
// `per_step` entries whose loads are in flight together, one step after the other, so on a graph that
// does not keep the chip busy for long the time of a launch is that of its longest walk, whatever the rest does.
// A walk is therefore split until it is no longer than `limit` steps.
inline int warps_log2_for(int entries, int per_step, int64_t limit)
{
    int w = 0;
    while ((1 << w) < kBlock / 32 && (entries >> w) > per_step * limit) ++w;
    return w;
}

// The longest walk to allow, in steps: twice what a warp slot of the chip has to do on average in the sweep over one chunk, and
// not under 16 (of the gathers' steps).  A chunk's column tiles run side by side and count; chunks run one after the other, so the
// longest rows end every one of their sweeps, and a column slab of whole chunks is cut like the full width, with the same
// bits.  In entries the limit is 2 * nnz * tiles / 3552: with one tile, rows are split on graphs of up to 3.6 M entries.  fp32 GCN
// against unsplit rows (one warp up to 2048 entries): 4,000 rows of 10 entries and 304 columns 76 -> 18 us, 20,000 of 50 and
// 128 columns 101 -> 40, 100,000 of 20 and 64 columns 75 -> 50.  With the average itself or four times it as the limit: 38 and
// 58 us for the second, 52 and 75 for the third.  `blocks_per_sm`: blocks of the kernel that an SM holds.  Kernels with four are slower per warp and have
// more slots: counted as three, SAGE of 72 / 96 fp32 columns on 20,000 rows of 50 took 32 us instead of 26.5, on 100,000 of 20 61 / 62 instead
// of 48 / 49, of 64 columns on 20,000 rows of 50 23 instead of 20.
inline int64_t walk_limit(const gnnfd_csr_t* csr, int per_step, int64_t tiles, int64_t at_least = 16, int blocks_per_sm = 3)
{
    const int64_t warp_slots = (int64_t)148 * blocks_per_sm * (kBlock / 32);
    const int64_t limit = 2 * (csr->nnz * tiles / (per_step * warp_slots));
    return limit > at_least ? limit : at_least;
}

// Fills ranges for `lpr` lanes per row; returns the blocks of one column tile of one sweep.  `per_step`: entries a whole warp
// has in flight; `limit`: steps of the longest walk.
inline int64_t plan_ranges(const gnnfd_csr_t* csr, const Groups& groups, int lpr, int per_step, int64_t limit, Range* range,
                           int32_t* n_ranges)
{
    auto ep_for_bin = [&](int bin) { return groups.want[bin] < 32 / lpr ? groups.want[bin] : 32 / lpr; };
    int nr = 0;
    int64_t blocks = 0;
    auto add = [&](int64_t begin, int64_t count, int ep, int entries, int hub, bool octave = false) {
        const int w = lpr * ep == 32 ? warps_log2_for(entries, per_step, limit) : 0;
        const int per_block = kBlock / (lpr * ep) >> w;
        if (octave && nr > 0 && !range[nr - 1].hub && range[nr - 1].warps_log2 == w) {
            // the octave before the last one in the order, cut in the same way: one range
            Range& r = range[nr - 1];
            r.item_count += (int32_t)count;
            blocks = r.first_block + (r.item_count + per_block - 1) / per_block;
            return;
        }
        range[nr++] = Range{(int32_t)blocks, (int32_t)(begin + count - 1), -1, (int32_t)count, ilog2(ep), hub, w};
        blocks += (count + per_block - 1) / per_block;
    };
    if (csr->n_segments > 0) add(0, csr->n_segments, ep_for_bin(4), kHubSegment, 1);
    int64_t end = csr->bin_start[3] + csr->bin_count[3];
    for (int o = kOctaves - 1; o >= 0; --o) {
        end -= csr->octave_count[o];
        if (csr->octave_count[o] > 0) add(end, csr->octave_count[o], ep_for_bin(3), kBinDeg2 << (o + 1), 0, true);
    }
    const int longest[3] = {kBinDeg0, kBinDeg1, kBinDeg2};
    for (int bin = 2; bin >= 0; --bin)
        if (csr->bin_count[bin] > 0) add(csr->bin_start[bin], csr->bin_count[bin], ep_for_bin(bin), longest[bin], 0);
    *n_ranges = nr;
    return blocks;
}

}  // namespace gnnfd
