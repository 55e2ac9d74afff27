// bp_nibble.h -- arithmetic of the expand sweep's distance test on nibble rows
// (host and device).
//
// A nibble row holds min(d(r_i, v), 7) in four bits a root (7 for an
// unreachable root and for the padding), so the row of 64 roots is one 32-byte
// sector instead of two, and 32-bit arithmetic tests eight roots at once. Root
// i sits in word 4 (i / 32) + (i % 4) of its row, nibble (i % 32) / 4: four
// words of compare bits then interleave into a 32-bit root mask with shifts.
// With thr = level - d(v_k, r_i), clamped to [-1, 7], root i prunes w iff its
// nibble is <= thr; the nibble of (8 + thr) - q has its top bit set exactly
// then, and no borrow leaves a nibble (8 + thr >= 7 >= q).
//
// The test is exact for candidate levels L <= NIB_LEVEL (it is asked about
// sums of at most L, L + 1 and L + 2): a 7 stands for a distance >= 7 > L + 1,
// and only w = r_i (d = 0) could meet L + 2 = 7 with a larger one, which a BFS
// that reached r_i at level L rules out. d(v_k, r_i) >= 1, as bit-parallel
// roots run no pruned BFS.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define PLL_HD __host__ __device__ __forceinline__
#else
#define PLL_HD inline
#endif

namespace pll {

constexpr uint32_t NIB_LEVEL = 5;
constexpr uint32_t NIB_TOP = 0x88888888u;

// 8 + thr of the eight roots of word q of v_k's row, for sums of at most lv <= 7
PLL_HD uint32_t nib_thresholds(uint32_t q, uint32_t lv) {
    const uint32_t y = (8u + lv) * 0x11111111u - q;  // 8 + lv - q in every nibble
    const uint32_t m = y & NIB_TOP, full = m | (m - (m >> 3));
    return (y & full) | (0x77777777u & ~full);       // max(y, 7)
}

// top bits set where a nibble of w's word q is within its threshold
PLL_HD uint32_t nib_within(uint32_t thr, uint32_t q) { return (thr - q) & NIB_TOP; }

// the compare bits of a chunk's four words as a mask over its 32 roots
PLL_HD uint32_t nib_roots(uint32_t a, uint32_t b, uint32_t c, uint32_t d) { return a >> 3 | b >> 2 | c >> 1 | d; }

// word w (0..3) of a chunk of 32 roots from their distance bytes, four bytes a word
PLL_HD uint32_t nib_pack(const uint32_t (&bytes)[8], int w) {
    uint32_t q = 0;
    for (int j = 0; j < 8; ++j) {
        const uint32_t d = (bytes[j] >> (8 * w)) & 0xffu;
        q |= (d < 7 ? d : 7u) << (4 * j);
    }
    return q;
}

}  // namespace pll
