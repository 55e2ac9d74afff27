// build_sizes.h -- the sizes a build chooses by itself: root batches, slices and
// what the autotuner tries (host code, no CUDA).
#pragma once

#include <algorithm>
#include <cstdint>

namespace pll {

// An entry of the frontier whose vertex has more than SLICE neighbours is
// expanded in slices of SLICE arcs, so that no warp of the expand sweep is
// left with a hub's list while the others are done (R-MAT-20's expand sweeps: 55.3,
// 57.0, 59.1, 64 ms with slices of 64, 128, 256, 512).
constexpr uint32_t SLICE = 64;
// Slices of one level that a build has room for (16 bytes each; a level with more
// expands its entries whole): one for every arc, which a first batch's 64 roots do
// not exceed, between 1 MiB and 1 GiB, and at most a sixteenth of the free memory.
constexpr uint64_t SLICE_CAP = 64ull << 20;
inline uint64_t slice_entries(uint64_t nnz, uint64_t free_b) {
    const uint64_t most = std::min<uint64_t>(SLICE_CAP, free_b / 16 / 16);
    return std::max<uint64_t>(std::min(nnz, most), 1ull << 16);
}

// Size of the next root batch, after `roots_done` roots and a batch that emitted
// `last_entries` entries. A batch costs its launches, about 0.35 ms (0.5 with its
// host round trip); roots in one batch do not prune with each other, so a larger
// one labels, expands and drops again more surplus entries, about 0.75 ns each.
// While batches are small (their launches are what they cost) the roots done
// quadruple with each, then double; a batch with more than a million entries
// fills the device, and its successors are held to two fifths of the roots done
// and to BATCH_FULL. Late batches emit little again and grow up to the largest
// size. Builds of R-MAT-20, the batch of 96 graphs, BA-10k and R-MAT-15 both ways:
//   doubling from 64 to 16384               115.2  147.1  4.19  12.5 ms
//   this rule                                91.0  143.0  3.44  12.2
//   with at most 16384 / 32768 roots        +9.4 / +2.5, +6.1 / +0.2 ms on the
//                                           first two (the late batches' launches)
//   shares of 0.25, 0.33, 0.5 for 0.4       R-MAT-20 90.6 90.9 93.4, batch 143.4 142.6 140.6
//   lines at 64K entries (for 256K)         BA-10k 3.7 to 4.0; at 512K R-MAT-15 15.2
//   the first batches five times the roots done   R-MAT-20 98.9
constexpr uint32_t BATCH_MAX = 1u << 16, BATCH_FULL = 16384;
inline uint32_t next_batch(uint64_t roots_done, uint64_t last_entries, uint32_t bmax) {
    uint64_t b = roots_done;
    if (last_entries < (256u << 10)) b = 3 * roots_done;
    else if (last_entries >= (1u << 20)) b = std::min<uint64_t>(roots_done * 2 / 5, BATCH_FULL);
    return (uint32_t)std::min<uint64_t>(std::max<uint64_t>(b, 64), bmax);
}

// The root batches that the autotuner tries: powers of two from 1024 to BATCH_FULL,
// and on to `dflt`, the largest batch that a build without options uses, as far as
// the graph's n vertices reach. Returns how many.
inline int autotune_batches(uint32_t n, uint32_t dflt, uint32_t (&sizes)[7]) {
    int count = 0;
    for (uint32_t b = 1024; b <= BATCH_MAX; b *= 2)
        if (b <= BATCH_FULL || (b <= dflt && b / 2 < n)) sizes[count++] = b;
    return count;
}

}  // namespace pll
