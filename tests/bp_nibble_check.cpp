// The nibble-row distance test (csrc/bp_nibble.h) against the plain sums, for
// every pair of distances (1..12 and unreachable at the BFS root's end, 0..12
// and unreachable at the candidate's) in every position of a 32-root chunk and
// every level the test is used at. A root itself (distance 0) reached at level
// L is at distance at most L from the BFS root, so pairs with d = 0 beyond that
// do not occur. Prints "ok <comparisons>" and exits 0, or prints the first
// difference and exits 1.
#include <cstdint>
#include <cstdio>

#include "bp_nibble.h"

static void pack(const uint8_t *d, uint32_t *row) {
    uint32_t bytes[8];
    for (int j = 0; j < 8; ++j)
        bytes[j] = d[4 * j] | d[4 * j + 1] << 8 | d[4 * j + 2] << 16 | (uint32_t)d[4 * j + 3] << 24;
    for (int w = 0; w < 4; ++w) row[w] = pll::nib_pack(bytes, w);
}

static uint32_t within(const uint32_t *k, const uint32_t *w, uint32_t lv) {
    uint32_t b[4];
    for (int x = 0; x < 4; ++x) b[x] = pll::nib_within(pll::nib_thresholds(k[x], lv), w[x]);
    return pll::nib_roots(b[0], b[1], b[2], b[3]);
}

int main() {
    const uint8_t far = 255;
    unsigned long long done = 0;
    uint32_t state = 1;
    auto rnd = [&](uint32_t n) { return (state = state * 1664525u + 1013904223u, (state >> 8) % n); };
    for (uint32_t L = 1; L <= pll::NIB_LEVEL; ++L)
        for (int trial = 0; trial < 200; ++trial)
            for (uint32_t a = 1; a <= 13; ++a)
                for (uint32_t b = 0; b <= 13; ++b) {
                    uint8_t dk[32], dw[32];
                    for (int i = 0; i < 32; ++i) {  // other pairs around the one at hand
                        dk[i] = (uint8_t)(1 + rnd(13));
                        dw[i] = (uint8_t)rnd(14);
                    }
                    const int at = (int)rnd(32);
                    dk[at] = (uint8_t)a;
                    dw[at] = (uint8_t)b;
                    for (int i = 0; i < 32; ++i) {
                        if (dk[i] == 13) dk[i] = far;
                        if (dw[i] == 13) dw[i] = far;
                        if (dw[i] == 0 && dk[i] > L) dk[i] = (uint8_t)L;
                    }
                    uint32_t rk[4], rw[4];
                    pack(dk, rk);
                    pack(dw, rw);
                    for (uint32_t lv = L; lv <= L + 2; ++lv) {
                        uint32_t want = 0;
                        for (int i = 0; i < 32; ++i)
                            if (dk[i] != far && dw[i] != far && dk[i] + dw[i] <= (int)lv) want |= 1u << i;
                        const uint32_t got = within(rk, rw, lv);
                        if (got != want) {
                            std::printf("level %u, sums <= %u: got %08x, want %08x\n", L, lv, got, want);
                            return 1;
                        }
                        done += 32;
                    }
                }
    std::printf("ok %llu\n", done);
    return 0;
}
