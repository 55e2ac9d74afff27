// k_pruned.cu -- pruned BFSs (Alg. 1) for a batch of roots [k0, k0 + B).
//
// Alg. 2 runs Alg. 1 for k = 1..n one after another: the BFS from v_k is
// pruned at u when Query(v_k, u, L'_{k-1}) <= P[u]. Here a whole batch of
// roots runs at once and each root is pruned only with the labels of hubs
// < k0 (finished batches) plus the bit-parallel labels (Sec. 5.4). That
// emits a superset of the entries Alg. 1 would add; the cleanup pass in
// k_labels.cu removes exactly the surplus (an entry (u, k, d) is surplus iff
// an in-batch hub h < k lies on a shortest k-u path, and then both (h, .) in
// L(v_k) and (h, .) in L(u) were emitted by this batch). The result is the
// label set of the sequential algorithm for any batch size.
//
// The BFSs of all roots of the batch advance level by level together, as
// bulk-synchronous sweeps over one flat frontier of (root slot, vertex)
// pairs, so the work of a level is spread over the whole GPU whatever the
// mix of large and small BFSs:
//
//   init    per root: the level-0 entry (v_k, k, 0) (the root is never
//           pruned: Query(v_k, v_k) >= 2 for v_k outside X), its visited bit,
//           a hash table of its label L(v_k) -- the root array T of Sec.
//           4.5.1 ("Querying"), so a prune test costs O(|L(u)|) probes.
//   expand  the arcs (u, w) of the entries (u, k, d) of the level, w of rank >=
//           k0 (lower ranks are always pruned). First the cheap part of the
//           prune test, which decides 19 of 20 on power-law graphs: the
//           bit-parallel distances -- with d~_i = d(v_k,r_i) + d(r_i,w), some
//           d~_i <= d + 1 prunes (Sec. 5.3: the distance through {r_i} U S_{r_i}
//           is at most d~_i) -- on rows of four bits a root (eight roots per
//           instruction; bytes past level NIB_LEVEL). A w that it leaves is
//           looked up in the root's visited row (a bitmap [B][ceil(n / 32)],
//           one row per root of the batch: the per-root visited set of Alg.
//           1). If unvisited: which roots could still reach the bound with
//           their masks (d~_i = d + 2 needs a reduction of 1, d~_i = d + 3
//           the S^{-1} intersection; neither can come from empty sets), then the
//           masks of the first QUICK roots: roots come in rank order, so these
//           are the largest hubs and they decide most mask tests. Survivors
//           are claimed with an atomicOr; freshly claimed (slot, w) pairs and
//           the remaining feasible roots are the next level's candidates. A
//           vertex the bit-parallel labels prune stays unmarked: the
//           bit-parallel bound of a pair does not depend on the level, so if
//           it prunes w at level d + 1 it prunes w again at any later level
//           where w is reached, and leaving the bit clear changes no label.
//   test    the rest of the test, 32 candidates per warp: the mask pairs of
//           their feasible bit-parallel roots compared, one a lane; then, root
//           by root, the near entries of the labels L(w) of the candidates that
//           are left, past the root's reach table to its hash table. Survivors
//           are appended as (w, k, d + 1).
//   clear   after the batch, the lazy reset of Sec. 4.5.1 ("Initialization"):
//           the only bits set are those of the roots and of the recorded
//           candidates, so their words are zeroed and nothing else is touched
//           (instead of clearing B * n / 8 bytes per batch).
//
// Level boundaries live in a device descriptor, advanced by the last block of
// each sweep of the graph loop (by a one-thread kernel where the host enqueues
// the levels, several ahead); sweeps over an empty range return at once.
#include "bp_nibble.h"
#include "pll_internal.cuh"

namespace pll {
namespace {

// threads an SM of the test sweep (64 registers each; at 1280 it spills: R-MAT-20's
// test sweeps 41.6 ms against 32.8, the batch's 74.2 against 69.0)
constexpr int TEST_TPS = 1024;

constexpr unsigned FULL = 0xffffffffu;
constexpr uint32_t HT_EMPTY = 0xffffffffu;

// Slot of hub rank h in a table of mask + 1 = 2^lg slots (lg >= 5): the top lg
// bits of a two-multiply mix of h. Hub ranks of one graph in a batch share
// their low bits (ranks interleave the graphs), so an unmixed product would
// crowd them into few slots.
__device__ __forceinline__ uint32_t ht_slot(uint32_t h, uint32_t mask) {
    uint32_t x = h * 0x9E3779B1u;
    x ^= x >> 15;
    x *= 0x2C1B3C6Du;
    x ^= x >> 12;
    const uint32_t lg = 31 - __clz(mask + 1);
    return x >> (32 - lg);
}

// warp-aggregated append: returns this lane's slot (valid where want is true)
__device__ __forceinline__ unsigned long long warp_append(unsigned long long *counter, bool want,
                                                          int lane) {
    const unsigned m = __ballot_sync(FULL, want);
    unsigned long long base = 0;
    const int leader = m ? __ffs(m) - 1 : 0;
    if (m && lane == leader) base = atomicAdd(counter, (unsigned long long)__popc(m));
    base = __shfl_sync(FULL, base, leader);
    return base + __popc(m & ((1u << lane) - 1u));
}

// A root's reach table: a byte per hash of a hub, four for every slot of its
// hash table (up to REACH_MAX bytes), in which bit r (r < 8) says that some
// hub with that hash is within r of the root (bit 7: at any distance). A
// candidate's entry (h, d) can prune at level L only if bit min(L - d, 7) of
// its hub's byte is set: one byte answers it for nearly every entry, and only
// the others go to the hash table, whose chains cost dependent loads.
__device__ __forceinline__ uint32_t reach_slot(uint32_t h, uint32_t lg) { return (h * 0x85EBCA6Bu) >> (32 - lg); }
__device__ __forceinline__ uint32_t reach_lg(uint32_t tmask) {  // of a hash table of tmask + 1 slots
    return min(34u - __clz(tmask), REACH_LG_MAX);
}

// Neighbours of rank < k0 need no test: they are pruned at whatever level they
// are reached. (A hub of a finished batch answers every distance to itself
// exactly, Thm 4.1, and so do the bit-parallel labels for a vertex of X:
// Query(v_k, w) = d(v_k, w) <= level.) Lists are ascending, so rstart cuts them
// off as a prefix, unread: on power-law graphs most arcs lead to hubs. Levels
// next to the deepest distance read the whole list, so that a vertex at depth
// 255 is found (and is an error) exactly where it would be without the cut: a
// vertex adjacent to one at depth 254 is at depth 253 at least.
constexpr uint32_t WHOLE_LEVEL = 250;
__device__ __forceinline__ uint32_t first_arc(const BatchArgs &a, uint32_t u, uint32_t nlevel) {
    return nlevel >= WHOLE_LEVEL ? a.roff[u] : a.rstart[u];
}

__global__ void k_row_starts(uint32_t n, uint32_t k0, const uint32_t *__restrict__ roff,
                             const uint32_t *__restrict__ rcol, uint32_t *rstart) {
    for (uint32_t u = blockIdx.x * blockDim.x + threadIdx.x; u < n; u += gridDim.x * blockDim.x) {
        uint32_t lo = k0 ? rstart[u] : roff[u];
        const uint32_t first = lo, end = roff[u + 1];
        if (lo < end && rcol[lo] < k0) {
            // gallop, then search the last step: batches move the cut a little
            uint32_t step = 1;
            while (step < end - lo && rcol[lo + step] < k0) {
                lo += step;
                step <<= 1;
            }
            uint32_t hi = end - lo < step ? end : lo + step;
            ++lo;
            while (lo < hi) {
                const uint32_t mid = lo + ((hi - lo) >> 1);
                if (rcol[mid] < k0) lo = mid + 1; else hi = mid;
            }
        }
        if (lo != first || k0 == 0) rstart[u] = lo;
    }
}

// New entries (w, k) of level `level` (the lanes with keep): those of more than
// SLICE arcs to expand leave the arcs past the first SLICE as slices.
__device__ __forceinline__ void append_slices(const BatchArgs &a, bool keep, int lane, uint32_t w, uint32_t k,
                                              uint32_t level) {
    uint32_t rb = 0, deg = 0;
    if (keep) {
        rb = first_arc(a, w, level + 1);
        deg = a.roff[w + 1] - rb;
    }
    for (unsigned m = __ballot_sync(FULL, deg > SLICE); m; m &= m - 1) {
        const int j = __ffs(m) - 1;
        const uint32_t b = __shfl_sync(FULL, rb, j), e = b + __shfl_sync(FULL, deg, j);
        const uint32_t kj = __shfl_sync(FULL, k, j), cnt = (e - b - 1) / SLICE;
        unsigned long long base = 0;
        if (lane == j) base = atomicAdd(&a.ctr->slice_n, (unsigned long long)cnt);
        base = __shfl_sync(FULL, base, j);
        for (uint32_t i = lane; i < cnt; i += 32) {
            const uint32_t x = b + (i + 1) * SLICE;
            if (base + i < a.slice_cap) a.slices[base + i] = make_uint4(kj, x, e - x < SLICE ? e : x + SLICE, 0);
        }
    }
}

__global__ void k_batch_init(BatchArgs a) {
    const int lane = threadIdx.x & 31;
    const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t slot = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; slot < a.B; slot += warps) {
        const uint32_t k = a.k0 + slot;
        if (a.inX[k]) continue;  // bit-parallel vertices get no pruned BFS
        if (lane == 0) {
            const unsigned long long pos = atomicAdd(&a.ctr->out_n, 1ull);
            if (pos < a.out_cap) a.out[pos] = pack_tuple(k, k, 0);
            else atomicOr(&a.ctr->err, ERR_BUF);
            atomicOr(&a.visited[(size_t)slot * a.NW + (k >> 5)], 1u << (k & 31));
        }
        append_slices(a, lane == 0, lane, k, k, 0);
        const uint32_t len = a.lab_len[k], slots = ht_size(len);
        // root array T as a hash table of 2 x |L(v_k)| slots (very long labels,
        // and tables past the pool's end, are binary-searched instead; the host
        // grows the pool for the next batches)
        unsigned long long tb = 0;
        if (slots && lane == 0) tb = atomicAdd(&a.ctr->ht_top, (unsigned long long)slots);
        tb = __shfl_sync(FULL, tb, 0);
        const bool fits = slots && tb + slots <= a.ht_cap;
        if (lane == 0) {
            a.tab[slot] = make_uint2((uint32_t)(tb / HT_MIN), fits ? slots - 1 : NONE);
            if (slots && !fits) atomicOr(&a.ctr->err, ERR_TABLE);
        }
        if (fits) {
            uint32_t *ht = a.ht + tb;
            const uint32_t mask = slots - 1;
            uint32_t *reach = a.reach + tb;
            const uint32_t lg = reach_lg(mask);
            const uint4 empty = make_uint4(HT_EMPTY, HT_EMPTY, HT_EMPTY, HT_EMPTY);
            for (uint32_t s = lane; s <= mask / 4; s += 32) reinterpret_cast<uint4 *>(ht)[s] = empty;
            for (uint32_t s = lane; s < 1u << (lg - 4); s += 32)
                reinterpret_cast<uint4 *>(reach)[s] = make_uint4(0, 0, 0, 0);
            __syncwarp();
            const uint32_t *lab = a.pool + a.lab_off[k];
            for (uint32_t j = lane; j < len; j += 32) {
                const uint32_t e = lab[j];
                const uint32_t rs = reach_slot(entry_hub(e), lg), within = (0xffu << min(entry_dist(e), 7u)) & 0xffu;
                atomicOr(&reach[rs >> 2], within << (8 * (rs & 3)));
                uint32_t s = ht_slot(entry_hub(e), mask);
                while (atomicCAS(&ht[s], HT_EMPTY, e) != HT_EMPTY) s = (s + 1) & mask;
            }
        }
    }
}

// Cheap part of the prune test, one thread: bit-parallel distances only. With
// d~_i = d(v_k, r_i) + d(r_i, w), some d~_i <= level prunes (Sec. 5.3: the
// distance through {r_i} U S_{r_i} is at most d~_i); roots with d~_i = level + 1
// or level + 2 may still prune through their masks. kr and wq are the rows of
// v_k and w (nq 16-byte chunks, four roots per 32-bit word); the byte sums
// saturate at 255, so this form needs level + 2 < 255.

// Phase 1: is some d~_i <= level? Two byte instructions per four roots, with
// an exit at the first word that prunes: roots come in rank order (Sec. 5.4),
// so the first words, the largest hubs, prune most vertices, and the exit saves
// a fifth of the sweep's time against testing all t roots first.
__device__ __forceinline__ bool bp_prunes(const uint4 *kr, const uint4 (&wq)[PLL_MAX_T / 16], uint32_t nq,
                                          uint32_t lv) {
#pragma unroll
    for (uint32_t c = 0; c < PLL_MAX_T / 16; ++c) {
        if (c < nq) {
            const uint4 r = kr[c], q = wq[c];
            if (__vcmpleu4(__vaddus4(q.x, r.x), lv)) return true;
            if (__vcmpleu4(__vaddus4(q.y, r.y), lv)) return true;
            if (__vcmpleu4(__vaddus4(q.z, r.z), lv)) return true;
            if (__vcmpleu4(__vaddus4(q.w, r.w), lv)) return true;
        }
    }
    return false;
}

// bytes 0x00 / 0xff of x -> bits 0..3 (the four 0/1 bits gathered by one multiply)
__device__ __forceinline__ uint32_t byte_lanes(uint32_t x) { return ((x & 0x01010101u) * 0x01020408u) >> 24; }

// Phase 2, after phase 1 found no prune: c1 = roots with d~_i = level + 1,
// c2 = roots with d~_i = level + 2.
__device__ __forceinline__ void bp_feasible(const uint4 *kr, const uint4 (&wq)[PLL_MAX_T / 16], uint32_t nq,
                                            uint32_t level, uint64_t &c1, uint64_t &c2) {
    const uint32_t l1 = (level + 1) * 0x01010101u, l2 = (level + 2) * 0x01010101u;
    c1 = c2 = 0;
#pragma unroll
    for (uint32_t c = 0; c < PLL_MAX_T / 16; ++c) {
        if (c < nq) {
            const uint4 r = kr[c], q = wq[c];
            const uint32_t sx = __vaddus4(q.x, r.x), sy = __vaddus4(q.y, r.y);
            const uint32_t sz = __vaddus4(q.z, r.z), sw = __vaddus4(q.w, r.w);
            const uint32_t a1 = byte_lanes(__vcmpeq4(sx, l1)) | byte_lanes(__vcmpeq4(sy, l1)) << 4 |
                                byte_lanes(__vcmpeq4(sz, l1)) << 8 | byte_lanes(__vcmpeq4(sw, l1)) << 12;
            const uint32_t a2 = byte_lanes(__vcmpeq4(sx, l2)) | byte_lanes(__vcmpeq4(sy, l2)) << 4 |
                                byte_lanes(__vcmpeq4(sz, l2)) << 8 | byte_lanes(__vcmpeq4(sw, l2)) << 12;
            c1 |= (uint64_t)a1 << (16 * c);
            c2 |= (uint64_t)a2 << (16 * c);
        }
    }
}

// The clamped rows: bp_c holds min(d(r_i, v), 63) for every byte of bp_d
// (unreachable, 255, also becomes 63). Two clamped bytes add up to at most
// 126 with no carry between bytes, so plain 32-bit arithmetic tests four roots
// at once (the byte-SIMD intrinsics above take several instructions each).
// For a candidate level L <= FAST_LEVEL the test is exact: a clamped byte
// stands for a distance >= 63 > L + 2, so its sum can neither reach L nor
// equal L + 1 or L + 2, clamped or not.
constexpr uint32_t CLAMP = 63;
constexpr uint32_t FAST_LEVEL = CLAMP - 3;

// Phase 1 on clamped rows: with lb = (0x80 + L) in every byte, the byte of
// lb - (q + r) keeps its top bit iff q + r <= L (no borrow crosses a byte:
// every byte of lb is above every byte sum).
__device__ __forceinline__ bool bp_prunes_c(const uint4 *kr, const uint4 (&wq)[PLL_MAX_T / 16], uint32_t nq,
                                            uint32_t lb) {
#pragma unroll
    for (uint32_t c = 0; c < PLL_MAX_T / 16; ++c) {
        if (c < nq) {
            const uint4 r = kr[c], q = wq[c];
            if ((lb - (q.x + r.x)) & 0x80808080u) return true;
            if ((lb - (q.y + r.y)) & 0x80808080u) return true;
            if ((lb - (q.z + r.z)) & 0x80808080u) return true;
            if ((lb - (q.w + r.w)) & 0x80808080u) return true;
        }
    }
    return false;
}

// bits 0..3: which bytes of s equal those of cb (every byte of s ^ cb is
// below 0x80, so (x | 0x80) - 1 keeps its top bit iff the byte x is not 0)
__device__ __forceinline__ uint32_t eq_lanes(uint32_t s, uint32_t cb) {
    const uint32_t x = s ^ cb;
    const uint32_t z = ~((x | 0x80808080u) - 0x01010101u) & 0x80808080u;
    return ((z >> 7) * 0x01020408u) >> 24;
}

// Phase 2 on clamped rows: c1 = roots with d~_i = L + 1, c2 = roots with L + 2.
__device__ __forceinline__ void bp_feasible_c(const uint4 *kr, const uint4 (&wq)[PLL_MAX_T / 16], uint32_t nq,
                                              uint32_t level, uint64_t &c1, uint64_t &c2) {
    const uint32_t l1 = (level + 1) * 0x01010101u, l2 = (level + 2) * 0x01010101u;
    c1 = c2 = 0;
#pragma unroll
    for (uint32_t c = 0; c < PLL_MAX_T / 16; ++c) {
        if (c < nq) {
            const uint4 r = kr[c], q = wq[c];
            const uint32_t sx = q.x + r.x, sy = q.y + r.y, sz = q.z + r.z, sw = q.w + r.w;
            const uint32_t a1 = eq_lanes(sx, l1) | eq_lanes(sy, l1) << 4 | eq_lanes(sz, l1) << 8 |
                                eq_lanes(sw, l1) << 12;
            const uint32_t a2 = eq_lanes(sx, l2) | eq_lanes(sy, l2) << 4 | eq_lanes(sz, l2) << 8 |
                                eq_lanes(sw, l2) << 12;
            c1 |= (uint64_t)a1 << (16 * c);
            c2 |= (uint64_t)a2 << (16 * c);
        }
    }
}

// The same test for depths near 255, where byte sums would overflow: a plain
// loop over the roots. Returns true if some d~_i <= level.
__device__ __noinline__ bool bp_test_plain(const BatchArgs &a, uint32_t k, uint32_t w, uint32_t level,
                                           uint64_t &c1, uint64_t &c2) {
    const uint8_t *dw = a.bp_d + (size_t)w * a.tp, *dk = a.bp_d + (size_t)k * a.tp;
    c1 = c2 = 0;
    for (uint32_t i = 0; i < a.t; ++i) {
        const uint32_t x = dw[i], y = dk[i];
        if (x == INF8 || y == INF8) continue;
        const uint32_t td = x + y;
        if (td <= level) return true;
        if (td == level + 1) c1 |= 1ull << i;
        if (td == level + 2) c2 |= 1ull << i;
    }
    return false;
}

// Masks of the first QUICK bit-parallel roots, one thread. The roots are
// chosen in rank order (Sec. 5.4), so the first ones are the largest hubs and
// settle most mask tests; checking them here keeps most candidates out of
// the test sweep and away from the rest of their 1 KiB mask rows. Clears
// those roots from c1 / c2.
constexpr uint32_t QUICK = 4;
__device__ __forceinline__ bool quick_masks(const BatchArgs &a, uint32_t k, uint32_t w, uint64_t &c1,
                                            uint64_t &c2) {
    const uint32_t q1 = (uint32_t)c1 & ((1u << QUICK) - 1u), q2 = (uint32_t)c2 & ((1u << QUICK) - 1u);
    c1 &= ~(uint64_t)((1u << QUICK) - 1u);
    c2 &= ~(uint64_t)((1u << QUICK) - 1u);
    if (!(q1 | q2)) return false;
    const ulonglong2 *wm = reinterpret_cast<const ulonglong2 *>(a.bp_m) + (size_t)w * a.t;
    const ulonglong2 *km = reinterpret_cast<const ulonglong2 *>(a.bp_m) + (size_t)k * a.t;
    bool p = false;
#pragma unroll
    for (uint32_t i = 0; i < QUICK; ++i) {
        if (((q1 | q2) >> i) & 1u) {
            const ulonglong2 m = wm[i], r = km[i];
            if (((q1 >> i) & 1u) && ((((r.x | r.y) & m.x) | (r.x & m.y)) != 0)) p = true;
            if (((q2 >> i) & 1u) && ((r.x & m.x) != 0)) p = true;
        }
    }
    return p;
}


// ---- nibble rows (bp_nibble.h): bp_q holds the distances clamped to 7, four
// bits a root, for levels up to NIB_LEVEL
__device__ __forceinline__ uint4 nib_thresholds4(uint4 q, uint32_t lv) {
    return make_uint4(nib_thresholds(q.x, lv), nib_thresholds(q.y, lv), nib_thresholds(q.z, lv),
                      nib_thresholds(q.w, lv));
}
__device__ __forceinline__ uint32_t nib_any(uint4 p, uint4 q) {
    return nib_within(p.x, q.x) | nib_within(p.y, q.y) | nib_within(p.z, q.z) | nib_within(p.w, q.w);
}
__device__ __forceinline__ uint32_t nib_mask(uint4 p, uint4 q) {
    return nib_roots(nib_within(p.x, q.x), nib_within(p.y, q.y), nib_within(p.z, q.z), nib_within(p.w, q.w));
}

// The nibble row of vertex v (qn = 1 or 2 chunks; the second chunk is zero
// without one): one 32-byte load a lane where the row has 32 bytes. The sweep
// is bound by the L1's rate of scattered accesses (81 % of its peak on the
// heaviest R-MAT-19 launch), and two 16-byte loads of one sector count twice
// there: R-MAT-20's sweeps take 51.4 ms with one load, 55.3 ms with two.
__device__ __forceinline__ void load_row(const BatchArgs &a, uint32_t v, uint4 &q0, uint4 &q1) {
    if (a.qn > 1) {
        const uint4 *row = a.bp_q + 2 * (size_t)v;
        asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
            : "=r"(q0.x), "=r"(q0.y), "=r"(q0.z), "=r"(q0.w), "=r"(q1.x), "=r"(q1.y), "=r"(q1.z), "=r"(q1.w)
            : "l"(row));
    } else {
        q0 = __ldg(a.bp_q + v);
        q1 = make_uint4(0, 0, 0, 0);
    }
}

// How a sweep tests the bit-parallel distances of candidates of one level.
enum BpMode : uint32_t {
    BP_NONE,    // t = 0, or a level past the last distance (every new vertex is an error)
    BP_NIBBLE,  // level <= NIB_LEVEL
    BP_CLAMP,   // level <= FAST_LEVEL: clamped bytes
    BP_BYTES,   // saturating bytes
    BP_PLAIN    // level + 2 would overflow a byte
};
__device__ __forceinline__ BpMode bp_mode(const BatchArgs &a, uint32_t nlevel) {
    if (a.t == 0 || nlevel >= INF8) return BP_NONE;
    if (nlevel <= NIB_LEVEL) return BP_NIBBLE;
    if (nlevel <= FAST_LEVEL) return BP_CLAMP;
    return nlevel + 2 < INF8 ? BP_BYTES : BP_PLAIN;
}

// Deeper levels (past NIB_LEVEL): does a bit-parallel distance prune w, and if
// not, which roots' masks may (c1, c2)? The byte rows, 16 roots a step.
__device__ __noinline__ bool bp_test_deep(const BatchArgs &a, BpMode mode, uint32_t k, uint32_t w,
                                          uint32_t nlevel, uint64_t &c1, uint64_t &c2) {
    if (mode == BP_PLAIN) return bp_test_plain(a, k, w, nlevel, c1, c2);
    const uint32_t nq = a.tp >> 4;
    const uint8_t *rows = mode == BP_CLAMP ? a.bp_c : a.bp_d;
    uint4 kr[PLL_MAX_T / 16], wq[PLL_MAX_T / 16];
#pragma unroll
    for (uint32_t c = 0; c < PLL_MAX_T / 16; ++c) {
        const bool in = c < nq;
        kr[c] = in ? __ldg(reinterpret_cast<const uint4 *>(rows + (size_t)k * a.tp) + c) : make_uint4(0, 0, 0, 0);
        wq[c] = in ? __ldg(reinterpret_cast<const uint4 *>(rows + (size_t)w * a.tp) + c) : make_uint4(0, 0, 0, 0);
    }
    c1 = c2 = 0;
    if (mode == BP_CLAMP) {
        if (bp_prunes_c(kr, wq, nq, (0x80u + nlevel) * 0x01010101u)) return true;
        bp_feasible_c(kr, wq, nq, nlevel, c1, c2);
    } else {
        if (bp_prunes(kr, wq, nq, nlevel * 0x01010101u)) return true;
        bp_feasible(kr, wq, nq, nlevel, c1, c2);
    }
    return false;
}

__device__ __forceinline__ void append_cand(const BatchArgs &a, bool keep, int lane, uint32_t slot, uint32_t w,
                                            uint64_t c1, uint64_t c2) {
    if (__any_sync(FULL, keep)) {
        const unsigned long long pos = warp_append(&a.ctr->cand_n, keep, lane);
        if (keep) {
            if (pos < a.cand_cap) {
                a.cand[pos] = ((uint64_t)slot << 32) | w;
                reinterpret_cast<ulonglong2 *>(a.candc)[pos] = make_ulonglong2(c1, c2);
            } else {
                atomicOr(&a.ctr->err, ERR_BUF);
            }
        }
    }
}

// What a warp of the expand sweep keeps in shared memory: for each entry of
// its chunk the nibble row of the root (q) and its prune thresholds (p), and
// the arcs that the distances did not prune.
struct ExpandWarp {
    uint4 p[32][2], q[32][2];
    uint32_t queue[64];  // w << 5 | entry of the chunk
};

// The second part of the expand sweep, for up to 32 arcs of the queue at once:
// look w up in the root's visited row; if unvisited, which roots' masks may
// still prune it, and the first masks; claim w if it survives.
__device__ __forceinline__ void expand_open(const BatchArgs &a, const ExpandWarp &sw, uint32_t at, uint32_t count,
                                            uint32_t k_lane, uint32_t nlevel, BpMode mode, uint32_t &nreach) {
    const int lane = threadIdx.x & 31;
    const bool act = (uint32_t)lane < count;
    const uint32_t item = act ? sw.queue[at + lane] : 0u;
    const uint32_t j = item & 31u, w = item >> 5;
    const uint32_t k = __shfl_sync(FULL, k_lane, j), slot = k - a.k0;
    bool keep = false;
    uint64_t c1 = 0, c2 = 0;
    if (act) {
        uint32_t *word = a.visited + (size_t)slot * a.NW + (w >> 5);
        const uint32_t wbit = 1u << (w & 31);
        if (!(*word & wbit)) {
            ++nreach;
            bool pruned = false;
            if (nlevel >= INF8) {
                atomicOr(&a.ctr->err, ERR_DEPTH);
                pruned = true;
            } else if (mode == BP_NIBBLE) {
                uint4 q[2];
                load_row(a, w, q[0], q[1]);
                uint32_t m1[2] = {0, 0}, m2[2] = {0, 0};
#pragma unroll
                for (uint32_t c = 0; c < 2; ++c) {
                    if (c < a.qn) {
                        const uint4 kq = sw.q[j][c];
                        m1[c] = nib_mask(nib_thresholds4(kq, nlevel + 1), q[c]);
                        m2[c] = nib_mask(nib_thresholds4(kq, nlevel + 2), q[c]) & ~m1[c];
                    }
                }
                c1 = (uint64_t)m1[1] << 32 | m1[0];
                c2 = (uint64_t)m2[1] << 32 | m2[0];
            } else if (mode != BP_NONE) {
                pruned = bp_test_deep(a, mode, k, w, nlevel, c1, c2);
            }
            if (c1 | c2) {
                // a reduction of 2 needs S^{-1} of both ends non-empty, one of 1
                // S^{-1} of one end and S^{-1} or S^0 of the other
                const ulonglong2 ew = __ldg(a.bp_e + w), ek = __ldg(a.bp_e + k);
                c1 &= (ek.x & ew.y) | (ek.y & ew.x);
                c2 &= ek.x & ew.x;
                pruned = quick_masks(a, k, w, c1, c2);
            }
            if (!pruned) keep = !(atomicOr(word, wbit) & wbit);
        }
    }
    append_cand(a, keep, lane, slot, w, c1, c2);
}

// Entries of at least this many arcs are taken 32 arcs at a time: with slices of as
// many, whole slices and full first ones (and the long lists of a level whose slices
// found no room), which leave no lane idle and need no owner search. A line at 32 to
// 1000 made no difference to the time. And threads an SM of the expand sweep (builds
// of R-MAT-20 and of the batch of 96 graphs: 144.9 and 176.4 ms at 1280, 138.5 and
// 170.6 at 1024)
constexpr uint32_t HEAVY_DEG = 64;
constexpr int EXPAND_TPS = 1024;

// The next chunk of G of a sweep's items for this warp: the first chunk of each
// warp is its own (small levels need no counter), the others are handed out as
// warps come free. Chunks differ much in their work; dealt out in turn, a third of
// the warps of a heavy expand launch were done early (22 of 32 active on average).
// R-MAT-20: expand 32.9 -> 30.7 ms, test 16.2 -> 15.4; the batch of 96 graphs:
// 40.0 -> 38.6, 62.2 -> 58.6. Chunks of at most 16: expand 32.3 and 39.8 ms, test
// 18.2 and 61.5; two or four chunks a warp in levels that have no more: BA-10k's
// sweeps 0.89 -> 1.1 ms.
__device__ __forceinline__ unsigned long long next_chunk(const BatchArgs &a, unsigned long long items,
                                                         unsigned long long nwarps, uint32_t G) {
    if (items <= nwarps * G) return items;
    unsigned long long c = 0;
    if ((threadIdx.x & 31) == 0) c = atomicAdd(&a.ctr->taken, (unsigned long long)G);
    return nwarps * G + __shfl_sync(FULL, c, 0);
}

// The expand sweep: entries [b, e) of level `level` and the slices of its long
// entries -> candidates of the next, by the warps of a grid. A warp takes a
// chunk of up to 32 of them (fewer when the level has fewer than that for
// every warp): lane j fetches entry j's key,
// row bounds and nibble row, so these dependent loads are in flight for the
// whole chunk, and then the arcs are tested: those of an entry of at least
// HEAVY_DEG neighbours 32 at a time, the others' laid end to end over the lanes.
//
// An arc (u, w) is first put to the bit-parallel distances, which need one
// 32-byte sector of w (an L2-resident table) and prune 19 of 20; only then is
// w looked up in the root's visited row, a scattered DRAM access. (Vertices
// that the distances prune are never marked, so the order of the two tests
// changes nothing.) The arcs that are left go through a queue in shared
// memory, so that the rest of the test runs with full warps.
//
// Bound by the L1's rate of scattered accesses (one row per arc). 1024 threads
// per SM (64 registers; the graph loop's form keeps 100 bytes of its chunk in local
// memory, the separate launch 12; at 1280 threads more: 52.9 against 51.4 ms). All of
// R-MAT-20's expand sweeps (t = 64; 3.15G arcs): 95.1 ms with a warp per
// entry, 64-byte rows and the visited word first; 71.9 ms with chunks, the
// queue and nibble rows; 55.3 ms with long lists in slices; 51.4 ms with one
// load a row; 39.2 ms with the lists cut at rank k0 (1.64G arcs left);
// 32.9 ms with the batch sizes of next_batch (1.3G).
__device__ __forceinline__ void expand_body(const BatchArgs &a, unsigned long long b, unsigned long long e,
                                            unsigned long long slice_n, uint32_t level, ExpandWarp &sw,
                                            uint32_t &nexp, uint32_t &nreach) {
    const int lane = threadIdx.x & 31;
    const unsigned long long nwarps = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
    const unsigned long long gw = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nlevel = level + 1;  // level of the candidates
    const BpMode mode = bp_mode(a, nlevel);
    // slices that did not all fit: every entry is expanded whole
    const uint32_t most = slice_n <= a.slice_cap ? SLICE : ~0u;
    const unsigned long long ne = e - b, items = ne + (slice_n <= a.slice_cap ? slice_n : 0);
    const unsigned long long per = (items + nwarps - 1) / nwarps;
    const uint32_t G = per < 1 ? 1u : per < 32 ? (uint32_t)per : 32u;
    for (unsigned long long c0 = gw * G; c0 < items; c0 = next_chunk(a, items, nwarps, G)) {
        // entries and candidates are written by other SMs between the phases of
        // one launch (k_batch_levels): read them from L2, never from a line the
        // L1 kept from an earlier level
        const uint32_t cnt = items - c0 < G ? (uint32_t)(items - c0) : G;
        uint32_t k = a.k0, eb = 0, deg = 0;
        __syncwarp();  // the previous chunk is done with sw
        if ((uint32_t)lane < cnt) {
            if (c0 + lane < ne) {
                const uint64_t key = __ldcg(a.out + b + c0 + lane);
                const uint32_t u = (uint32_t)(key >> 32);
                k = entry_hub((uint32_t)key);
                eb = first_arc(a, u, nlevel);
                deg = min(a.roff[u + 1] - eb, most);
            } else {
                const uint4 sl = __ldcg(a.slices + (c0 + lane - ne));
                k = sl.x;
                eb = sl.y;
                deg = sl.z - sl.y;
            }
            nexp += deg;
            if (mode == BP_NIBBLE) {
                uint4 q[2];
                load_row(a, k, q[0], q[1]);
#pragma unroll
                for (uint32_t c = 0; c < 2; ++c) {
                    sw.q[lane][c] = q[c];
                    sw.p[lane][c] = nib_thresholds4(q[c], nlevel);
                }
            }
        }
        __syncwarp();
        // entries with at least HEAVY_DEG neighbours one by one (arcs [x, xe) of
        // entry j are next), then the other entries' arcs end to end
        uint32_t heavy = __ballot_sync(FULL, deg >= HEAVY_DEG);
        const uint32_t len = deg < HEAVY_DEG ? deg : 0;
        uint32_t incl = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += y;
        }
        const uint32_t total = __shfl_sync(FULL, incl, 31);
        const uint32_t excl = incl - len;
        uint32_t x = 0, xe = 0, j = 0, x0 = 0, nqueue = 0;
        for (;;) {
            bool open;
            uint32_t arc;
            if (x >= xe && heavy) {
                j = __ffs(heavy) - 1;
                heavy &= heavy - 1;
                x = __shfl_sync(FULL, eb, j);
                xe = x + __shfl_sync(FULL, deg, j);
            }
            const bool more = x < xe || x0 < total;
            if (x < xe) {
                arc = x + lane;
                open = arc < xe;
                x += 32;
            } else {
                const uint32_t y = x0 + lane;
                j = 0;  // owner: the last entry whose first arc is <= y
#pragma unroll
                for (uint32_t step = 16; step > 0; step >>= 1)
                    if (__shfl_sync(FULL, excl, j + step) <= y) j += step;
                arc = __shfl_sync(FULL, eb - excl, j) + y;
                open = y < total;
                x0 += 32;
            }
            uint32_t w = 0;
            if (open) {
                w = a.rcol[arc];
                if (mode == BP_NIBBLE) {
                    uint4 q0, q1;
                    load_row(a, w, q0, q1);
                    uint32_t hit = nib_any(sw.p[j][0], q0);
                    if (a.qn > 1) hit |= nib_any(sw.p[j][1], q1);
                    open = hit == 0;
                    nreach += hit != 0;
                }
            }
            const unsigned m = __ballot_sync(FULL, open);
            if (open) sw.queue[nqueue + __popc(m & ((1u << lane) - 1u))] = w << 5 | j;
            nqueue += __popc(m);
            if (nqueue >= 32 || (!more && nqueue)) {
                __syncwarp();
                const uint32_t take = min(nqueue, 32u);
                nqueue -= take;
                expand_open(a, sw, nqueue, take, k, nlevel, mode, nreach);
                __syncwarp();
            }
            if (!more && nqueue == 0) break;
        }
    }
}

// warp sums of the work counters into ctr->work[w0], ctr->work[w0 + 1]
__device__ __forceinline__ void flush_work(const BatchArgs &a, int w0, uint32_t x, uint32_t y) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        x += __shfl_xor_sync(FULL, x, o);
        y += __shfl_xor_sync(FULL, y, o);
    }
    if ((threadIdx.x & 31) == 0 && x) atomicAdd(&a.ctr->work[w0], (unsigned long long)x);
    if ((threadIdx.x & 31) == 0 && y) atomicAdd(&a.ctr->work[w0 + 1], (unsigned long long)y);
}

__device__ __forceinline__ ExpandWarp &expand_warp(uint4 *dyn) {
    return reinterpret_cast<ExpandWarp *>(dyn)[threadIdx.x >> 5];
}

template <int BLOCK>
__global__ void __launch_bounds__(BLOCK, EXPAND_TPS / BLOCK) k_batch_expand(BatchArgs a) {
    extern __shared__ uint4 s_dyn[];
    uint32_t nexp = 0, nreach = 0;
    expand_body(a, a.desc->lvl_b, a.desc->lvl_e, a.desc->slice_n, a.desc->level, expand_warp(s_dyn), nexp, nreach);
    flush_work(a, 2, nexp, nreach);
}

template <int BLOCK>
constexpr size_t expand_smem() { return (size_t)(BLOCK / 32) * sizeof(ExpandWarp); }

// bp_c = min(bp_d, CLAMP) bytewise, 16 bytes per thread and step
__global__ void k_clamp_rows(const uint4 *bp_d, uint4 *bp_c, size_t n16) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += (size_t)gridDim.x * blockDim.x) {
        uint4 v = bp_d[i];
        uint32_t *x = reinterpret_cast<uint32_t *>(&v);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            // bytes >= 64 have one of their two top bits set: they become 63
            const uint32_t hi = x[j] & 0xC0C0C0C0u;
            const uint32_t big = ((hi >> 6) | (hi >> 7)) & 0x01010101u;
            x[j] = (x[j] & 0x3F3F3F3Fu) | (big * CLAMP);
        }
        bp_c[i] = v;
    }
}

// Nibble rows (see expand_body): thread g of vertex v turns the 32 bytes of
// roots 32 g .. 32 g + 31 (16 where the row ends) into four words.
__global__ void k_nibble_rows(const uint8_t *__restrict__ bp_d, uint32_t tp, uint32_t qn, uint4 *bp_q, size_t nrows) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nrows; i += (size_t)gridDim.x * blockDim.x) {
        const size_t v = i / qn;
        const uint32_t g = (uint32_t)(i - v * qn);
        const uint4 *row = reinterpret_cast<const uint4 *>(bp_d + v * tp) + 2 * g;
        uint32_t d[8];
        const uint4 lo = __ldg(row);
        const uint4 hi = 32 * g + 16 < tp ? __ldg(row + 1) : make_uint4(~0u, ~0u, ~0u, ~0u);
        d[0] = lo.x; d[1] = lo.y; d[2] = lo.z; d[3] = lo.w;
        d[4] = hi.x; d[5] = hi.y; d[6] = hi.z; d[7] = hi.w;
        bp_q[i] = make_uint4(nib_pack(d, 0), nib_pack(d, 1), nib_pack(d, 2), nib_pack(d, 3));
    }
}

// Lazy reset: zero the visited words of the batch's roots and candidates (the
// only bits the batch set; several candidates may share a word). A batch whose
// candidates overflowed their buffer did not record them all: its rows are
// zeroed whole (it runs again with a larger buffer).
__global__ void k_batch_clear(BatchArgs a) {
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    const unsigned long long i0 = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (a.ctr->err & ERR_BUF) {
        const unsigned long long words = (unsigned long long)a.B * a.NW;
        uint4 *v4 = reinterpret_cast<uint4 *>(a.visited);  // the bitmap is 256-byte aligned
        for (unsigned long long i = i0; i < words / 4; i += stride) v4[i] = make_uint4(0, 0, 0, 0);
        for (unsigned long long i = (words & ~3ull) + i0; i < words; i += stride) a.visited[i] = 0;
        return;
    }
    const unsigned long long cn = a.ctr->cand_n < a.cand_cap ? a.ctr->cand_n : a.cand_cap;
    for (unsigned long long i = i0; i < a.B; i += stride)
        a.visited[i * a.NW + ((a.k0 + (uint32_t)i) >> 5)] = 0;
    for (unsigned long long i = i0; i < cn; i += stride) {
        const uint64_t c = a.cand[i];
        a.visited[(c >> 32) * a.NW + ((uint32_t)c >> 5)] = 0;
    }
}

// The rest of the prune test for 32 candidates per warp (lane j holds
// candidate j), in two parts:
//   masks   the (candidate, feasible root) pairs of all 32 laid end to end over
//           the lanes, a mask pair compared by each (Sec. 5.3). A candidate has
//           four of them on R-MAT-20: one candidate at a time over the lanes
//           left 28 of 32 idle behind two dependent loads (its test sweeps: 32.8
//           -> 21.9 ms, the batch's 69.0 -> 64.4);
//   labels  of the candidates the masks did not prune, root by root (the sweeps
//           keep a root's candidates together: 4 to 6 of 32 share one on
//           average). The root's reach table is copied to shared memory, and
//           the labels L(w) are read past it, four entries a lane: a long one
//           (at least LONG_LABEL entries) by the whole warp; the others' quads
//           of entries laid end to end over the lanes (a quad's candidate found
//           by a binary search over a warp scan of the lengths). An entry at
//           distance d >= level can prune nothing (every hub is at least 1 from
//           the root): 95 of 100 entries on power-law graphs and more than half on
//           the high-diameter ones, most of which are not even read (the labels are
//           read from their near copy, k_labels.cu, up to distance level - 1,
//           and from the store past what the copy holds); an
//           entry that the table lets through is looked up in the root's hash
//           table T (or, without one, by a binary search of L(v_k)), and
//           d + T[h] <= level prunes the candidate. A candidate found pruned
//           takes no further entries.
//
// Bound by instruction issue (0.57 to 0.7 of the slots on the batch's heavy
// launches) and the latency of the labels. All test sweeps of the batch of 96
// uneven graphs (t = 16; 33G label entries, 15G of them nearer than the
// candidate): 325 ms with every entry probed in the hash table (gathers from
// L2), 124 ms with the reach tables and single entries on the lanes, 106.6 ms
// with quads. R-MAT-20 (t = 64; 7.8G entries, 0.4G nearer): 65.9, 47.0, 43.3
// ms; with the near copy, which leaves the near entries and those of the last
// batches (16G and 1.05G), 69.0 and 32.8 ms; with the masks end to end and the
// small groups together 60.1 and 18.9; with the batch sizes of next_batch 62.2 and
// 16.2 (170M and 106M candidates). Without effect or slower: two quads a lane in
// flight, a second hash of the reach table, the entries it lets through queued
// and looked up 32 at a time (64 to 67 ms on the batch, 15.8 on R-MAT-20).
// candidates whose labels have at least this many entries are scanned one by
// one by the whole warp (no owner search per entry, and an exit at the first
// step that prunes); shorter labels are laid end to end over the lanes (the
// line at 32: 2 ms more on R-MAT-20; at 64 to 256 no difference; none: 25 ms
// more on the batch)
constexpr uint32_t LONG_LABEL = 128;
// a root's table is staged for at least this many label entries of its
// candidates; the others' candidates are taken together, each lane reading its
// candidate's table where it lies (128, 256, 512: 60.3, 60.1, 63.1 ms of test
// sweeps on the batch, 19.1, 18.9, 19.1 on R-MAT-20; root by root without
// staging 64.4 and 21.9)
constexpr uint32_t STAGE_ENTRIES = 256;

// Where the label entries of a candidate lie that a test reads: the near copy's
// entries of distance < level, then those appended since its last rebuild (all
// of them without a near copy).
struct Spans {
    const uint32_t *near, *rest;
    uint32_t near_n, rest_n;  // entries
    uint32_t first, near_q;   // the candidate's first quad of those laid end to end; near_n in quads
};

// What a warp of the test sweep keeps in shared memory.
struct TestWarp {
    uint4 reach[REACH_MAX / 16];  // the staged table of the root at hand
    Spans spans[32];              // the candidates' labels
};

// The root whose candidates are at hand (the same on every lane).
struct TestRoot {
    unsigned long long tb;  // its tables in the table pools
    uint32_t k, klen;
    uint32_t tmask;         // hash-table slots - 1, NONE without a table
    uint32_t lg;            // log2 of the reach table's bytes
    bool staged;            // the reach table is in shared memory
};

// distance from the root to hub h, INF8 if h is not in its label
__device__ __forceinline__ uint32_t root_distance(const BatchArgs &a, const TestRoot &r, uint32_t h) {
    if (r.tmask != NONE) {
        const uint32_t *ht = a.ht + r.tb;
        for (uint32_t sl = ht_slot(h, r.tmask);; sl = (sl + 1) & r.tmask) {
            const uint32_t y = ht[sl];
            if (y == HT_EMPTY) return INF8;
            if (entry_hub(y) == h) return entry_dist(y);
        }
    }
    const uint32_t *rlab = a.pool + a.lab_off[r.k];
    uint32_t lo = 0, hi = r.klen;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (entry_hub(rlab[mid]) < h) lo = mid + 1; else hi = mid;
    }
    return lo < r.klen && entry_hub(rlab[lo]) == h ? entry_dist(rlab[lo]) : (uint32_t)INF8;
}

// Label entries arrive four to a lane (every label starts on 16 bytes and owns
// whole quads; those past its end read as distance 255, which prunes nothing).
// Does one of the quad's entries prune at `level` against root r? The reach
// bytes first, read as signed: shifted right by level - d (of at most 31) they
// give bit min(level - d, 7).
struct Quad {
    uint32_t e[4];
};
__device__ __forceinline__ Quad load_quad(const uint32_t *lab, uint32_t q, uint32_t len) {
    const uint4 v = *reinterpret_cast<const uint4 *>(lab + 4 * q);
    Quad r{{v.x, v.y, v.z, v.w}};
    if (4 * q + 4 > len) {
#pragma unroll
        for (uint32_t u = 1; u < 4; ++u)
            if (4 * q + u >= len) r.e[u] = INF8;
    }
    return r;
}
// quad q of a candidate's spans
__device__ __forceinline__ Quad span_quad(const Spans &sp, uint32_t q) {
    return q < sp.near_q ? load_quad(sp.near, q, sp.near_n) : load_quad(sp.rest, q - sp.near_q, sp.rest_n);
}
__device__ __forceinline__ bool quad_prunes(const BatchArgs &a, const TestWarp &tw, const TestRoot &r, const Quad &q,
                                            uint32_t level) {
    const int8_t *sh = reinterpret_cast<const int8_t *>(tw.reach);
    const int8_t *gl = reinterpret_cast<const int8_t *>(a.reach + r.tb);
    uint32_t open = 0;  // the entries that the table lets through
    if (r.staged) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int t = (int)level - (int)entry_dist(q.e[u]);
            const int near = sh[reach_slot(entry_hub(q.e[u]), r.lg)];
            if (t > 0) open |= (uint32_t)(near >> min(t, 31) & 1) << u;
        }
    } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int t = (int)level - (int)entry_dist(q.e[u]);
            if (t > 0) {
                const int near = r.tmask != NONE ? gl[reach_slot(entry_hub(q.e[u]), r.lg)] : -1;
                open |= (uint32_t)(near >> min(t, 31) & 1) << u;
            }
        }
    }
    for (; open; open &= open - 1) {
        const uint32_t lo = open & 1 ? q.e[0] : q.e[1], hi = open & 4 ? q.e[2] : q.e[3], e = open & 3 ? lo : hi;
        const uint32_t t = root_distance(a, r, entry_hub(e));
        if (t != INF8 && t + entry_dist(e) <= level) return true;
    }
    return false;
}

// The sweep over candidates [b, e) of level `level` by the warps of a grid.
// Adds the label entries it reads and the mask pairs it reads to n_scan /
// n_mask.
__device__ __forceinline__ void test_body(const BatchArgs &a, unsigned long long b, unsigned long long e,
                                          uint32_t level, TestWarp &tw, uint32_t &n_scan, uint32_t &n_mask) {
    const int lane = threadIdx.x & 31;
    // each warp takes up to 32 consecutive candidates, fewer when the level has
    // fewer than that for every warp (a warp tests them one root after another)
    const unsigned long long nwarps = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
    const unsigned long long gw = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const unsigned long long total_c = e - b, per = (total_c + nwarps - 1) / nwarps;
    const uint32_t G = per < 1 ? 1u : per < 32 ? (uint32_t)per : 32u;
    for (unsigned long long i0 = gw * G; i0 < total_c; i0 = next_chunk(a, total_c, nwarps, G)) {
        const uint32_t cnt = total_c - i0 < G ? (uint32_t)(total_c - i0) : G;
        const bool valid = (uint32_t)lane < cnt;
        ulonglong2 mc = make_ulonglong2(0, 0);
        uint32_t wlen = 0, klen = 0, slot = 0, w = 0, tb = 0, tmask = NONE, wquads = 0;
        __syncwarp();  // the previous candidates' spans have been read
        if (valid) {  // per-candidate metadata, loaded in parallel
            const uint64_t mine = __ldcg(a.cand + b + i0 + lane);
            mc = __ldcg(reinterpret_cast<const ulonglong2 *>(a.candc) + b + i0 + lane);
            w = (uint32_t)mine;
            slot = (uint32_t)(mine >> 32);
            Spans sp{nullptr, a.vis_pool + a.vis_off[w], 0, a.vis_len[w], 0, 0};
            if (a.near) {
                const NearLabel nl = a.near_lab[w];
                sp.near = a.near + nl.off;
                sp.near_n = level <= NEAR_CLASSES ? a.near_end[(size_t)(level - 1) * a.n + w] : nl.base;
                sp.near_q = (sp.near_n + 3) / 4;
                sp.rest += nl.base;
                sp.rest_n -= nl.base;
            }
            wlen = sp.near_n + sp.rest_n;
            wquads = sp.near_q + (sp.rest_n + 3) / 4;
            tw.spans[lane] = sp;
            klen = a.lab_len[a.k0 + slot];
            const uint2 t = a.tab[slot];
            tb = t.x;
            tmask = t.y;
        }
        // ---- masks: the (candidate, root) pairs laid end to end
        uint32_t pruned = 0;
        {
            uint64_t open = mc.x | mc.y;
            const uint32_t mine_n = __popcll(open);
            uint32_t incl = mine_n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(FULL, incl, o);
                if (lane >= o) incl += y;
            }
            const uint32_t total = __shfl_sync(FULL, incl, 31);
            // no table is staged yet: its place holds the list
            static_assert(32 * PLL_MAX_T * sizeof(uint16_t) <= REACH_MAX, "every root of every candidate fits");
            uint16_t *items = reinterpret_cast<uint16_t *>(tw.reach);
            for (uint32_t at = incl - mine_n; open; open &= open - 1) {
                const uint32_t i = __ffsll(open) - 1;
                items[at++] = (uint16_t)(lane | i << 5 | (uint32_t)(mc.x >> i & 1) << 11 |
                                         (uint32_t)(mc.y >> i & 1) << 12);
            }
            __syncwarp();
            for (uint32_t x0 = 0; x0 < total; x0 += 32) {
                const uint32_t it = x0 + lane < total ? items[x0 + lane] : 0, j = it & 31, i = it >> 5 & 63;
                const uint32_t wj = __shfl_sync(FULL, w, j), kj = a.k0 + __shfl_sync(FULL, slot, j);
                bool p = false;
                if (x0 + lane < total && !((pruned >> j) & 1)) {
                    ++n_mask;
                    const ulonglong2 mw = reinterpret_cast<const ulonglong2 *>(a.bp_m)[(size_t)wj * a.t + i];
                    const ulonglong2 r = reinterpret_cast<const ulonglong2 *>(a.bp_m)[(size_t)kj * a.t + i];
                    if ((it >> 11 & 1) && (((r.x | r.y) & mw.x) | (r.x & mw.y))) p = true;  // reduction >= 1
                    if ((it >> 12 & 1) && (r.x & mw.x)) p = true;                           // reduction 2
                }
                pruned |= __reduce_or_sync(FULL, p ? 1u << j : 0u);
            }
        }
        // ---- labels, root by root
        uint32_t todo = __ballot_sync(FULL, valid && !((pruned >> lane) & 1) && wlen && klen), loose = 0;
        while (todo) {
            const uint32_t j0 = __ffs(todo) - 1;
            const uint32_t s0 = __shfl_sync(FULL, slot, j0);
            const bool in = ((todo >> lane) & 1) && slot == s0;
            const uint32_t group = __ballot_sync(FULL, in);
            todo &= ~group;
            TestRoot r;
            r.k = a.k0 + s0;
            r.klen = __shfl_sync(FULL, klen, j0);
            r.tmask = __shfl_sync(FULL, tmask, j0);
            r.tb = (unsigned long long)__shfl_sync(FULL, tb, j0) * HT_MIN;
            r.lg = reach_lg(r.tmask);
            r.staged = __reduce_add_sync(FULL, in ? min(wlen, 0xffffu) : 0u) >= STAGE_ENTRIES;
            if (r.tmask != NONE && !r.staged) {
                loose |= group;
                continue;
            }
            r.staged = r.tmask != NONE;
            __syncwarp();  // the previous root's table has been read
            if (r.staged) {
                const uint4 *src = reinterpret_cast<const uint4 *>(a.reach + r.tb);
                for (uint32_t x = lane; x < 1u << (r.lg - 4); x += 32) tw.reach[x] = src[x];
            }
            __syncwarp();
            // long labels, 32 quads a step, leaving at the first step that prunes
            for (uint32_t m = __ballot_sync(FULL, in && wlen >= LONG_LABEL); m; m &= m - 1) {
                const uint32_t j = __ffs(m) - 1;
                const Spans sp = tw.spans[j];
                const uint32_t quads = __shfl_sync(FULL, wquads, j);
                for (uint32_t q0 = 0; q0 < quads; q0 += 32) {
                    const uint32_t q = q0 + lane;
                    if (__any_sync(FULL, q < quads && quad_prunes(a, tw, r, span_quad(sp, q), level))) {
                        pruned |= 1u << j;
                        break;
                    }
                }
                n_scan += lane == 0 ? sp.near_n + sp.rest_n : 0;
            }
            // short labels, their quads laid end to end
            const bool mine_short = in && wlen < LONG_LABEL;
            const uint32_t nq = mine_short ? wquads : 0;
            n_scan += mine_short ? wlen : 0;
            uint32_t incl = nq;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(FULL, incl, o);
                if (lane >= o) incl += y;
            }
            const uint32_t total = __shfl_sync(FULL, incl, 31);
            const uint32_t excl = incl - nq;
            tw.spans[lane].first = excl;
            __syncwarp();
            for (uint32_t x0 = 0; x0 < total; x0 += 32) {
                const uint32_t x = x0 + lane;
                uint32_t j = 0;  // owner: the last candidate whose first quad is <= x
#pragma unroll
                for (uint32_t step = 16; step > 0; step >>= 1)
                    if (__shfl_sync(FULL, excl, j + step) <= x) j += step;
                bool p = false;
                if (x < total) {
                    const Spans sp = tw.spans[j];
                    p = quad_prunes(a, tw, r, span_quad(sp, x - sp.first), level);
                }
                pruned |= __reduce_or_sync(FULL, p ? 1u << j : 0u);
            }
        }
        // the groups with few entries, together: each lane reads its candidate's table where it lies
        if (loose) {
            const uint32_t nq = (loose >> lane) & 1 ? wquads : 0;
            n_scan += nq ? wlen : 0;
            uint32_t incl = nq;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(FULL, incl, o);
                if (lane >= o) incl += y;
            }
            const uint32_t total = __shfl_sync(FULL, incl, 31);
            const uint32_t excl = incl - nq;
            __syncwarp();
            tw.spans[lane].first = excl;
            __syncwarp();
            for (uint32_t x0 = 0; x0 < total; x0 += 32) {
                const uint32_t x = x0 + lane;
                uint32_t j = 0;
#pragma unroll
                for (uint32_t step = 16; step > 0; step >>= 1)
                    if (__shfl_sync(FULL, excl, j + step) <= x) j += step;
                TestRoot r{};
                r.tmask = __shfl_sync(FULL, tmask, j);
                r.tb = (unsigned long long)__shfl_sync(FULL, tb, j) * HT_MIN;
                r.lg = reach_lg(r.tmask);
                r.staged = false;
                bool p = false;
                if (x < total) {
                    const Spans sp = tw.spans[j];
                    p = quad_prunes(a, tw, r, span_quad(sp, x - sp.first), level);
                }
                pruned |= __reduce_or_sync(FULL, p ? 1u << j : 0u);
            }
        }
        const bool keep = valid && !((pruned >> lane) & 1);
        if (__any_sync(FULL, keep)) {
            const unsigned long long pos = warp_append(&a.ctr->out_n, keep, lane);
            if (keep) {
                if (pos < a.out_cap) a.out[pos] = pack_tuple(w, a.k0 + slot, level);
                else atomicOr(&a.ctr->err, ERR_BUF);
            }
            append_slices(a, keep, lane, w, a.k0 + slot, level);
        }
    }
}

template <int BLOCK>
constexpr size_t test_smem() { return (size_t)(BLOCK / 32) * sizeof(TestWarp); }
// the cooperative loop's sweeps take turns with the same shared memory
template <int BLOCK>
constexpr size_t levels_smem() {
    return expand_smem<BLOCK>() > test_smem<BLOCK>() ? expand_smem<BLOCK>() : test_smem<BLOCK>();
}
__device__ __forceinline__ TestWarp &test_warp(uint4 *dyn) {
    return reinterpret_cast<TestWarp *>(dyn)[threadIdx.x >> 5];
}

template <int BLOCK>
__global__ void __launch_bounds__(BLOCK, TEST_TPS / BLOCK) k_batch_test(BatchArgs a) {
    extern __shared__ uint4 s_dyn[];
    uint32_t n_scan = 0, n_mask = 0;
    test_body(a, a.desc->cand_b, a.desc->cand_e, a.desc->level + 1, test_warp(s_dyn), n_scan, n_mask);
    flush_work(a, 0, n_scan, n_mask);
}

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// Grid-wide barrier of a cooperative launch (every CTA resident). The last
// CTA to arrive takes a snapshot of the counters (error word, candidate and
// entry counts) before it releases the others, so every CTA decides the next
// step from the same values. A wait longer than the state's timeout_ns sets
// ERR_TIMEOUT and returns false: the CTA leaves the level loop, and the
// others leave it at their next barrier, each wait bounded the same way.
__device__ __forceinline__ bool grid_barrier(const BatchArgs &a, LoopState *ls) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        __threadfence();
        const unsigned int gen = *(volatile unsigned int *)&ls->gen;
        if (atomicAdd(&ls->count, 1u) == gridDim.x - 1) {
            ls->count = 0;
            ls->err = atomicOr(&a.ctr->err, 0u);
            ls->cand_n = atomicAdd(&a.ctr->cand_n, 0ull);
            ls->out_n = atomicAdd(&a.ctr->out_n, 0ull);
            a.ctr->taken = 0;
            ls->slice_n = atomicExch(&a.ctr->slice_n, 0ull);  // the sweep before the barrier wrote or read them all
            __threadfence();
            atomicAdd(&ls->gen, 1u);
        } else {
            const unsigned long long t0 = global_ns(), lim = ls->timeout_ns;
            while (*(volatile unsigned int *)&ls->gen == gen) {
                if (global_ns() - t0 > lim) {
                    atomicOr(&a.ctr->err, ERR_TIMEOUT);
                    ok = 0;
                    break;
                }
                __nanosleep(64);
            }
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// Every level of a root batch in one cooperative launch: expand, barrier,
// test, barrier, until the frontier is empty (or a buffer overflows, a depth
// reaches 255, or a barrier times out). Level bounds live in registers, the
// same in every CTA (they come from the barrier's snapshots), so no level
// needs the host. Block 0 adds the phases' wall times to the loop state.
// At blocks of 128 and 256 the bound of 1280 threads an SM leaves 48 registers and
// spills (R-MAT-20's build 121 ms); at 512 and 1024 it comes to 1024 threads and 64
// registers (83 ms, the graph loop's 87).
template <int BLOCK>
__global__ void __launch_bounds__(BLOCK, 1280 / BLOCK) k_batch_levels(BatchArgs a) {
    extern __shared__ uint4 s_dyn[];
    LoopState *ls = a.loop;
    ExpandWarp &sw = expand_warp(s_dyn);
    TestWarp &tw = test_warp(s_dyn);
    const bool timer = blockIdx.x == 0 && threadIdx.x == 0;
    unsigned long long lvl_b = a.desc->lvl_b, lvl_e = a.desc->lvl_e, slice_n = a.desc->slice_n, cand_e = 0;
    uint32_t level = 0, nexp = 0, nreach = 0, n_scan = 0, n_mask = 0;
    unsigned long long ns_e = 0, ns_t = 0;
    constexpr uint32_t STOP = ERR_DEPTH | ERR_BUF | ERR_TIMEOUT;
    while (lvl_b < lvl_e) {
        const unsigned long long t0 = timer ? global_ns() : 0;
        expand_body(a, lvl_b, lvl_e, slice_n, level, sw, nexp, nreach);
        if (!grid_barrier(a, ls)) break;
        const unsigned long long t1 = timer ? global_ns() : 0;
        if (*(volatile uint32_t *)&ls->err & STOP) break;
        const unsigned long long cand_b = cand_e;
        const unsigned long long cn = *(volatile unsigned long long *)&ls->cand_n;
        cand_e = cn < a.cand_cap ? cn : a.cand_cap;
        test_body(a, cand_b, cand_e, level + 1, tw, n_scan, n_mask);
        if (!grid_barrier(a, ls)) break;
        if (timer) {
            const unsigned long long t2 = global_ns();
            ns_e += t1 - t0;
            ns_t += t2 - t1;
        }
        if (*(volatile uint32_t *)&ls->err & STOP) break;
        const unsigned long long on = *(volatile unsigned long long *)&ls->out_n;
        lvl_b = lvl_e;
        lvl_e = on < a.out_cap ? on : a.out_cap;
        slice_n = *(volatile unsigned long long *)&ls->slice_n;
        ++level;
    }
    flush_work(a, 2, nexp, nreach);
    flush_work(a, 0, n_scan, n_mask);
    if (timer) {
        ls->ns_expand += ns_e;
        ls->ns_test += ns_t;
        ls->levels += level;
    }
}

// descriptor steps between sweeps (one thread)
__device__ __forceinline__ void advance_desc(const BatchArgs &a, int phase) {
    LevelDesc *d = a.desc;
    const unsigned long long cn = *(volatile unsigned long long *)&a.ctr->cand_n;
    const unsigned long long on = *(volatile unsigned long long *)&a.ctr->out_n;
    const unsigned long long sn = *(volatile unsigned long long *)&a.ctr->slice_n;
    a.ctr->taken = 0;
    if (phase == 0) {          // after init: level 0 = the roots
        d->lvl_b = 0;
        d->lvl_e = on < a.out_cap ? on : a.out_cap;
        d->roots_n = d->lvl_e;
        d->level = 0;
        d->cand_b = 0;
        d->cand_e = 0;
        d->slice_n = sn;
        a.ctr->slice_n = 0;
        if (a.loop) a.loop->t_mark = global_ns();
    } else if (phase == 1) {   // after expand: candidates of level + 1
        d->cand_b = d->cand_e;
        d->cand_e = cn < a.cand_cap ? cn : a.cand_cap;
    } else {                   // after test: survivors become the level
        d->lvl_b = d->lvl_e;
        d->lvl_e = on < a.out_cap ? on : a.out_cap;
        d->level += 1;
        d->slice_n = sn;
        a.ctr->slice_n = 0;
    }
}

__global__ void k_batch_advance(BatchArgs a, int phase) { advance_desc(a, phase); }

// ---- the level loop as a CUDA graph: a while node whose body is expand, then
// test; the last block of each takes the step to the next phase, the second of
// which sets the loop condition. The kernels read the batch's arguments from
// device memory (the host writes them before each launch of the graph), so one
// instantiated graph serves every batch of a build.
// the batch's arguments, copied once per CTA from device memory into shared
// memory (read there as cheaply as kernel parameters)
__device__ __forceinline__ const BatchArgs &args_to_shared(const BatchArgs *ap, BatchArgs *sa) {
    static_assert(sizeof(BatchArgs) % 8 == 0, "BatchArgs is copied in 8-byte words");
    constexpr unsigned W = sizeof(BatchArgs) / 8;
    for (unsigned i = threadIdx.x; i < W; i += blockDim.x)
        reinterpret_cast<uint64_t *>(sa)[i] = reinterpret_cast<const uint64_t *>(ap)[i];
    __syncthreads();
    return *sa;
}

// The step after a sweep of the graph loop, by the block that finishes last (a
// kernel of its own costs a launch gap, 2.5 us a step): phase 1 / 2 of
// advance_desc, plus the phases' wall times; phase 2 sets the loop's condition:
// another level while the frontier is not empty and no buffer overflowed and no
// depth reached 255.
__device__ __forceinline__ void last_block_step(const BatchArgs &a, int phase, cudaGraphConditionalHandle h) {
    __syncthreads();
    if (threadIdx.x != 0) return;
    LoopState *ls = a.loop;
    __threadfence();
    if (atomicAdd(&ls->done, 1u) != gridDim.x - 1) return;
    __threadfence();  // every block's appends are behind its arrival
    ls->done = 0;
    advance_desc(a, phase);
    const unsigned long long now = global_ns();
    if (phase == 1) {
        ls->ns_expand += now - ls->t_mark;
    } else {
        ls->ns_test += now - ls->t_mark;
        ls->levels += 1;
        const bool more = a.desc->lvl_b < a.desc->lvl_e &&
                          !(*(volatile uint32_t *)&a.ctr->err & (ERR_DEPTH | ERR_BUF));
        cudaGraphSetConditional(h, more ? 1u : 0u);
    }
    ls->t_mark = now;
}

template <int BLOCK>
__global__ void __launch_bounds__(BLOCK, EXPAND_TPS / BLOCK) k_batch_expand_g(const BatchArgs *__restrict__ ap,
                                                                               cudaGraphConditionalHandle h) {
    extern __shared__ uint4 s_dyn[];
    __shared__ BatchArgs s_args;
    const BatchArgs &a = args_to_shared(ap, &s_args);
    uint32_t nexp = 0, nreach = 0;
    expand_body(a, a.desc->lvl_b, a.desc->lvl_e, a.desc->slice_n, a.desc->level, expand_warp(s_dyn), nexp, nreach);
    flush_work(a, 2, nexp, nreach);
    last_block_step(a, 1, h);
}

template <int BLOCK>
__global__ void __launch_bounds__(BLOCK, TEST_TPS / BLOCK) k_batch_test_g(const BatchArgs *__restrict__ ap,
                                                                           cudaGraphConditionalHandle h) {
    extern __shared__ uint4 s_dyn[];
    __shared__ BatchArgs s_args;
    const BatchArgs &a = args_to_shared(ap, &s_args);
    uint32_t n_scan = 0, n_mask = 0;
    test_body(a, a.desc->cand_b, a.desc->cand_e, a.desc->level + 1, test_warp(s_dyn), n_scan, n_mask);
    flush_work(a, 0, n_scan, n_mask);
    last_block_step(a, 2, h);
}

}  // namespace

template <int BLOCK>
static cudaError_t occupancy(int *pe, int *pt) {
    cudaError_t e = cudaFuncSetAttribute(k_batch_expand<BLOCK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)expand_smem<BLOCK>());
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(pe, k_batch_expand<BLOCK>, BLOCK, expand_smem<BLOCK>());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_batch_test<BLOCK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)test_smem<BLOCK>());
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(pt, k_batch_test<BLOCK>, BLOCK, test_smem<BLOCK>());
    return e;
}

// grid[0]: expand sweep, grid[1]: test sweep (resident CTAs of each)
int batch_grid(uint32_t block, int *grid) {
    int dev = 0, sms = 0, pe = 0, pt = 0;
    PLL_TRY(cudaGetDevice(&dev));
    PLL_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    cudaError_t e;
    switch (block) {
        case 128: e = occupancy<128>(&pe, &pt); break;
        case 512: e = occupancy<512>(&pe, &pt); break;
        case 1024: e = occupancy<1024>(&pe, &pt); break;
        default: e = occupancy<256>(&pe, &pt); break;
    }
    PLL_TRY(e);
    grid[0] = sms * (pe > 0 ? pe : 1);
    grid[1] = sms * (pt > 0 ? pt : 1);
    return PLL_OK;
}

int batch_init(const BatchArgs &a, cudaStream_t s) {
    const int g = (int)((a.B * 32ull + 255) / 256);
    k_batch_init<<<g > 0 ? g : 1, 256, 0, s>>>(a);
    k_batch_advance<<<1, 1, 0, s>>>(a, 0);
    PLL_TRY(cudaGetLastError());
    return PLL_OK;
}

template <int BLOCK>
static void level_sweeps(const BatchArgs &a, const int *grid, cudaStream_t s, cudaEvent_t *ev) {
    if (ev) cudaEventRecord(ev[0], s);
    k_batch_expand<BLOCK><<<grid[0], BLOCK, expand_smem<BLOCK>(), s>>>(a);
    if (ev) cudaEventRecord(ev[1], s);
    k_batch_advance<<<1, 1, 0, s>>>(a, 1);
    if (ev) cudaEventRecord(ev[2], s);
    k_batch_test<BLOCK><<<grid[1], BLOCK, test_smem<BLOCK>(), s>>>(a);
    if (ev) cudaEventRecord(ev[3], s);
    k_batch_advance<<<1, 1, 0, s>>>(a, 2);
}

int batch_clamp_rows(const uint8_t *bp_d, uint8_t *bp_c, size_t bytes, int grid, cudaStream_t s) {
    if (bytes == 0) return PLL_OK;
    k_clamp_rows<<<grid > 0 ? grid : 1, 256, 0, s>>>(reinterpret_cast<const uint4 *>(bp_d),
                                                     reinterpret_cast<uint4 *>(bp_c), bytes / 16);
    PLL_TRY(cudaGetLastError());
    return PLL_OK;
}

int batch_row_starts(uint32_t n, uint32_t k0, const uint32_t *roff, const uint32_t *rcol, uint32_t *rstart,
                     int grid, cudaStream_t s) {
    const int want = (int)((n + 255) / 256);
    k_row_starts<<<want < 4 * grid ? want : 4 * grid, 256, 0, s>>>(n, k0, roff, rcol, rstart);
    PLL_TRY(cudaGetLastError());
    return PLL_OK;
}

int batch_nibble_rows(const uint8_t *bp_d, uint32_t n, uint32_t tp, uint32_t qn, uint4 *bp_q, int grid,
                      cudaStream_t s) {
    if (n == 0 || qn == 0) return PLL_OK;
    k_nibble_rows<<<grid > 0 ? grid : 1, 256, 0, s>>>(bp_d, tp, qn, bp_q, (size_t)n * qn);
    PLL_TRY(cudaGetLastError());
    return PLL_OK;
}

int batch_clear(const BatchArgs &a, int grid, cudaStream_t s) {
    k_batch_clear<<<grid > 0 ? grid : 1, 256, 0, s>>>(a);
    PLL_TRY(cudaGetLastError());
    return PLL_OK;
}

template <int BLOCK>
static cudaError_t levels_grid(int *grid) {
    int dev = 0, sms = 0, coop = 0, per = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_batch_levels<BLOCK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)levels_smem<BLOCK>());
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_batch_levels<BLOCK>, BLOCK, levels_smem<BLOCK>());
    *grid = (e == cudaSuccess && coop && per > 0) ? sms * per : 0;
    return e;
}

int batch_levels_grid(uint32_t block, int *grid) {
    cudaError_t e;
    switch (block) {
        case 128: e = levels_grid<128>(grid); break;
        case 512: e = levels_grid<512>(grid); break;
        case 1024: e = levels_grid<1024>(grid); break;
        default: e = levels_grid<256>(grid); break;
    }
    PLL_TRY(e);
    return PLL_OK;
}

template <int BLOCK>
static cudaError_t launch_levels(const BatchArgs &a, int grid, cudaStream_t s) {
    BatchArgs arg = a;
    void *args[] = {&arg};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(k_batch_levels<BLOCK>), dim3(grid),
                                       dim3(BLOCK), args, levels_smem<BLOCK>(), s);
}

int batch_levels(const BatchArgs &a, uint32_t block, int grid, cudaStream_t s) {
    cudaError_t e;
    switch (block) {
        case 128: e = launch_levels<128>(a, grid, s); break;
        case 512: e = launch_levels<512>(a, grid, s); break;
        case 1024: e = launch_levels<1024>(a, grid, s); break;
        default: e = launch_levels<256>(a, grid, s); break;
    }
    PLL_TRY(e);
    return PLL_OK;
}

template <int BLOCK>
static int graph_build(const int *grid, const BatchArgs *d_args, cudaGraph_t *pg, cudaGraphExec_t *pexec) {
    cudaGraph_t g = nullptr;
    PLL_TRY(cudaGraphCreate(&g, 0));
    struct Guard {
        cudaGraph_t g;
        ~Guard() { if (g) cudaGraphDestroy(g); }
    } guard{g};
    PLL_TRY(cudaFuncSetAttribute(k_batch_expand_g<BLOCK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)expand_smem<BLOCK>()));
    PLL_TRY(cudaFuncSetAttribute(k_batch_test_g<BLOCK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)test_smem<BLOCK>()));
    cudaGraphConditionalHandle h;
    PLL_TRY(cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault));
    cudaGraphNodeParams cp{};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = h;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t cnode;
    PLL_TRY(cudaGraphAddNode(&cnode, g, nullptr, nullptr, 0, &cp));
    cudaGraph_t body = cp.conditional.phGraph_out[0];
    const BatchArgs *ap = d_args;
    void *args[] = {&ap, &h};
    cudaKernelNodeParams kp{};
    cudaGraphNode_t n[2];
    kp.func = reinterpret_cast<void *>(k_batch_expand_g<BLOCK>);
    kp.gridDim = dim3(grid[0]);
    kp.blockDim = dim3(BLOCK);
    kp.sharedMemBytes = (unsigned)expand_smem<BLOCK>();
    kp.kernelParams = args;
    PLL_TRY(cudaGraphAddKernelNode(&n[0], body, nullptr, 0, &kp));
    kp.func = reinterpret_cast<void *>(k_batch_test_g<BLOCK>);
    kp.gridDim = dim3(grid[1]);
    kp.sharedMemBytes = (unsigned)test_smem<BLOCK>();
    PLL_TRY(cudaGraphAddKernelNode(&n[1], body, &n[0], 1, &kp));
    PLL_TRY(cudaGraphInstantiate(pexec, g, 0));
    *pg = g;
    guard.g = nullptr;
    return PLL_OK;
}

int batch_graph_build(uint32_t block, const int *grid, const BatchArgs *d_args, cudaGraph_t *g,
                      cudaGraphExec_t *exec) {
    switch (block) {
        case 128: return graph_build<128>(grid, d_args, g, exec);
        case 512: return graph_build<512>(grid, d_args, g, exec);
        case 1024: return graph_build<1024>(grid, d_args, g, exec);
        default: return graph_build<256>(grid, d_args, g, exec);
    }
}

// ev: null, or four events recorded around the expand and test sweeps
int batch_level(const BatchArgs &a, const int *grid, uint32_t block, cudaStream_t s,
                cudaEvent_t *ev) {
    switch (block) {
        case 128: level_sweeps<128>(a, grid, s, ev); break;
        case 512: level_sweeps<512>(a, grid, s, ev); break;
        case 1024: level_sweeps<1024>(a, grid, s, ev); break;
        default: level_sweeps<256>(a, grid, s, ev); break;
    }
    PLL_TRY(cudaGetLastError());
    return PLL_OK;
}

}  // namespace pll
