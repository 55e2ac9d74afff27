// pair_device.cuh -- device code shared by the distance queries (k_query.cu) and
// the shortest-path queries (pll_paths.cu): one pair (s, t) of an index.
#pragma once

#include "pll_internal.cuh"

namespace pll {
namespace pairs {

constexpr unsigned FULL = 0xffffffffu;
constexpr uint32_t BIG = 1u << 20;
struct QueryArgs {
    uint32_t n, t, tp;
    const uint32_t *inv;
    const uint32_t *graph;  // graph of each rank (batch indices), or null
    const uint8_t *bp_d;
    const uint64_t *bp_m;
    const uint64_t *lab_off;
    const uint32_t *lab;
    const uint32_t *src, *dst;
    uint32_t stride;  // pair qi is (src[qi * stride], dst[qi * stride])
    uint64_t q;
    uint8_t *out;
    unsigned long long *err;  // [0] finite distance >= 255, [1] id >= n
};

inline QueryArgs query_args(const pll_index *ix, const uint32_t *src, const uint32_t *dst, uint32_t stride,
                            uint64_t q, uint8_t *out, unsigned long long *err) {
    return QueryArgs{ix->n, ix->t, ix->tp, ix->d_inv, ix->d_graph, ix->d_bp_d, ix->d_bp_m, ix->d_lab_off,
                     ix->d_lab, src, dst, stride, q, out, err};
}

__device__ __forceinline__ uint32_t warp_min(uint32_t v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(FULL, v, o));
    return v;
}

__device__ __forceinline__ uint32_t bp_reduce(uint32_t td, const uint64_t *__restrict__ ms,
                                              const uint64_t *__restrict__ mt) {
    ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(ms);
    ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(mt);
    if (a.x & b.x) return td - 2;
    if ((a.y & b.x) | (a.x & b.y)) return td - 1;
    return td;
}

// Resolves the cases that need no labels. Returns true with *ans set when
// the pair is decided (bad id, s == t, different graphs of a batch index).
__device__ __forceinline__ bool trivial_pair(const QueryArgs &a, uint32_t sid, uint32_t tid,
                                             uint32_t *s, uint32_t *t, uint32_t *ans, bool *bad) {
    *bad = false;
    if (sid >= a.n || tid >= a.n) { *ans = INF8; *bad = true; return true; }
    *s = a.inv[sid];
    *t = a.inv[tid];
    if (*s == *t) { *ans = 0; return true; }
    // graphs of a batch share slot numbers but not roots: no distance across
    if (a.graph && a.graph[*s] != a.graph[*t]) { *ans = INF8; return true; }
    return false;
}

// Bit-parallel distances d~ of the lane's roots (lane, lane + 32) and their
// warp-wide minimum d*.
__device__ __forceinline__ void bp_tilde(const QueryArgs &a, uint32_t s, uint32_t t, int lane,
                                         uint32_t *td0, uint32_t *td1, uint32_t *dstar) {
    *td0 = BIG;
    *td1 = BIG;
    const size_t ds = (size_t)s * a.tp, dt = (size_t)t * a.tp;
    if (lane < a.t) {
        uint32_t x = a.bp_d[ds + lane], y = a.bp_d[dt + lane];
        if (x != INF8 && y != INF8) *td0 = x + y;
    }
    if (lane + 32 < a.t) {
        uint32_t x = a.bp_d[ds + lane + 32], y = a.bp_d[dt + lane + 32];
        if (x != INF8 && y != INF8) *td1 = x + y;
    }
    *dstar = warp_min(min(*td0, *td1));
}

// min over common hubs of the two normal labels, over the entries
// first, first + step, ... of the shorter label taken by this lane's warp.
__device__ __forceinline__ uint32_t label_min(const QueryArgs &a, uint32_t s, uint32_t t, int lane,
                                              uint32_t first, uint32_t step) {
    const uint64_t os = a.lab_off[s], ot = a.lab_off[t];
    const uint32_t ls = (uint32_t)(a.lab_off[s + 1] - os), lt = (uint32_t)(a.lab_off[t + 1] - ot);
    const uint32_t *A = a.lab + (ls <= lt ? os : ot);
    const uint32_t *B = a.lab + (ls <= lt ? ot : os);
    const uint32_t la = ls <= lt ? ls : lt, lb = ls <= lt ? lt : ls;
    uint32_t best = BIG;
    for (uint32_t j = first; j < la; j += step) {
        if (j + lane < la) {
            const uint32_t e = A[j + lane], h = entry_hub(e);
            uint32_t lo = 0, hi = lb;
            while (lo < hi) {
                uint32_t mid = (lo + hi) >> 1;
                if (entry_hub(B[mid]) < h) lo = mid + 1; else hi = mid;
            }
            if (lo < lb && entry_hub(B[lo]) == h) best = min(best, entry_dist(e) + entry_dist(B[lo]));
        }
    }
    return warp_min(best);
}

#ifndef PLL_MERGE_RATIO
#define PLL_MERGE_RATIO 4
#endif

// min over common hubs of the two normal labels for one warp: a merge of the
// hub-sorted labels 32 entries at a time (the merge join of Sec. 3.3 done by
// a warp). Each lane holds one entry of the shorter label's window and finds
// its hub in the other window by a 5-step search over the lanes (shuffles);
// then the window whose last hub is smaller is passed whole and the other is
// advanced past the hubs not above it, which can meet nothing that is left.
// Labels read once, in coalesced 128-byte rows. When one label is more than
// PLL_MERGE_RATIO times longer, binary searches of its entries (label_min)
// touch less of it and are used instead. os / ls, ot / lt: the offsets and
// lengths of L(s) and L(t), already loaded by the caller.
__device__ __forceinline__ uint32_t label_min_merge_at(const QueryArgs &a, uint32_t s, uint32_t t,
                                                      uint64_t os, uint32_t ls, uint64_t ot, uint32_t lt,
                                                      int lane) {
    const uint32_t la = ls <= lt ? ls : lt, lb = ls <= lt ? lt : ls;
    if (la == 0) return BIG;
    if (lb > PLL_MERGE_RATIO * la) return label_min(a, s, t, lane, 0, 32);
    const uint32_t *A = a.lab + (ls <= lt ? os : ot);
    const uint32_t *B = a.lab + (ls <= lt ? ot : os);
    uint32_t best = BIG, ia = 0, ib = 0;
    while (ia < la && ib < lb) {
        const uint32_t na = min(32u, la - ia), nb = min(32u, lb - ib);
        const bool va = (uint32_t)lane < na, vb = (uint32_t)lane < nb;
        const uint32_t ea = va ? A[ia + lane] : NONE;  // padding sorts after every hub
        const uint32_t eb = vb ? B[ib + lane] : NONE;
        const uint32_t ha = entry_hub(ea), hb = entry_hub(eb);
        // lower bound of ha in the window of B held across the lanes
        uint32_t pos = 0;
#pragma unroll
        for (uint32_t stp = 16; stp > 0; stp >>= 1)
            if (entry_hub(__shfl_sync(FULL, eb, pos + stp - 1)) < ha) pos += stp;
        const uint32_t ep = __shfl_sync(FULL, eb, pos);
        if (va && pos < nb && entry_hub(ep) == ha) best = min(best, entry_dist(ea) + entry_dist(ep));
        const uint32_t lastA = entry_hub(__shfl_sync(FULL, ea, na - 1));
        const uint32_t lastB = entry_hub(__shfl_sync(FULL, eb, nb - 1));
        if (lastA <= lastB) {
            ia += na;
            ib += __popc(__ballot_sync(FULL, vb && hb <= lastA));
        } else {
            ib += nb;
            ia += __popc(__ballot_sync(FULL, va && ha <= lastB));
        }
    }
    return warp_min(best);
}

// The bit-parallel answer, fetching masks only where they can beat `best`
// (a label answer, or BIG).
__device__ __forceinline__ uint32_t finish_pair(const QueryArgs &a, uint32_t s, uint32_t t, int lane,
                                                uint32_t td0, uint32_t td1, uint32_t dstar,
                                                uint32_t best) {
    const size_t rs = (size_t)s * a.t, rt = (size_t)t * a.t;
    uint32_t bpb = BIG;
    if (dstar < BIG) {
        bpb = dstar;
        if (td0 <= dstar + 1 && td0 - 2 < best && td0 - 2 < bpb)
            bpb = min(bpb, bp_reduce(td0, a.bp_m + 2 * (rs + lane), a.bp_m + 2 * (rt + lane)));
        if (td1 <= dstar + 1 && td1 - 2 < best && td1 - 2 < bpb)
            bpb = min(bpb, bp_reduce(td1, a.bp_m + 2 * (rs + lane + 32), a.bp_m + 2 * (rt + lane + 32)));
        bpb = warp_min(bpb);
    }
    return min(best, bpb);
}

// the answer of a pair's minimum: its byte (255 for none or for a finite distance
// of 255 or more), and a bit above it for an error
constexpr uint32_t ANS_FAR = 1u << 8, ANS_BAD = 1u << 9;  // a finite distance >= 255, an id >= n
__device__ __forceinline__ uint32_t pair_answer(uint32_t best) {
    return best >= BIG ? INF8 : best >= INF8 ? INF8 | ANS_FAR : best;
}

// Adds the errors among a warp's answers to its block's counts (in shared memory).
__device__ __forceinline__ void count_errors(uint32_t *count, uint32_t ans, int lane) {
    if (!__any_sync(FULL, ans > INF8)) return;
    const unsigned far = __ballot_sync(FULL, ans & ANS_FAR), bad = __ballot_sync(FULL, ans & ANS_BAD);
    if (lane == 0) {
        atomicAdd(&count[0], __popc(far));
        atomicAdd(&count[1], __popc(bad));
    }
}

// An open pair: the ends' ranks, and where their labels are.
struct OpenPair {
    uint64_t os, ot;
    uint32_t s, t, ls, lt;
};

// v's bit-parallel row holds no distance (nothing reaches v from any root)
__device__ __forceinline__ bool row_empty(const QueryArgs &a, uint32_t v) {
    const uint4 *row = reinterpret_cast<const uint4 *>(a.bp_d + (size_t)v * a.tp);
    for (uint32_t c = 0; c < a.tp / 16; ++c) {
        const uint4 r = row[c];
        if ((r.x & r.y & r.z & r.w) != 0xffffffffu) return false;
    }
    return true;
}

// One thread: a pair with an end x that no bit-parallel root reaches and whose
// label has at most one entry (h, d), on power-law graphs mostly an isolated
// vertex, 4 of 10 on R-MAT-20 and so 6 of 10 uniform pairs. The pair's distance
// is d + d(h, y) if h is in the label of the other end y, none otherwise;
// a label's hubs are at most its vertex's own rank. *hub, *ds: that hub and its
// distance from s.
__device__ __forceinline__ bool lone_pair(const QueryArgs &a, uint32_t s, uint64_t os, uint32_t ls, uint32_t t,
                                          uint64_t ot, uint32_t lt, uint32_t *dist, uint32_t *hub, uint32_t *ds) {
    if (ls > 1 && lt > 1) return false;
    const bool at_s = ls <= 1 && row_empty(a, s);
    if (!at_s && !(lt <= 1 && row_empty(a, t))) return false;
    *dist = BIG;
    if ((at_s ? ls : lt) == 0) return true;
    const uint32_t e = a.lab[at_s ? os : ot], h = entry_hub(e), y = at_s ? t : s;
    if (h > y) return true;
    const uint32_t *B = a.lab + (at_s ? ot : os);
    const uint32_t lb = at_s ? lt : ls;
    uint32_t lo = 0, hi = lb;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (entry_hub(B[mid]) < h) lo = mid + 1; else hi = mid;
    }
    if (lo < lb && entry_hub(B[lo]) == h) {
        *dist = entry_dist(e) + entry_dist(B[lo]);
        *hub = h;
        *ds = entry_dist(at_s ? e : B[lo]);
    }
    return true;
}

// Entries of L(v) that can be part of a distance below ub through a hub that is
// neither end, compacted into `keep` (KEEP places): at most ub - 2 from v, as
// the other end is at least 1 from such a hub. *direct: the distance of v to
// `other`, if that is one of its hubs. AHEAD windows of 32 entries are loaded
// together. Returns how many are kept (over KEEP: too many, not all looked at). What
// other lanes wrote to or read from `keep` before (for the last pair, which may have
// ended early) is done first; the caller waits before it reads other lanes' places.
constexpr int AHEAD = 2;
template <uint32_t KEEP>
__device__ __forceinline__ uint32_t keep_near(const uint32_t *__restrict__ lab, uint32_t len, uint32_t v,
                                              uint32_t ub, uint32_t other, int lane, uint32_t *keep,
                                              uint32_t *direct) {
    uint32_t cnt = 0;
    __syncwarp();
    for (uint32_t x0 = 0; x0 < len && cnt <= KEEP; x0 += 32 * AHEAD) {
        uint32_t e[AHEAD];
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {
            const uint32_t x = x0 + 32 * u + lane;
            e[u] = x < len ? lab[x] : NONE;
        }
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {
            const uint32_t h = entry_hub(e[u]), d = entry_dist(e[u]);
            if (h == other) *direct = d;
            const bool in = e[u] != NONE && d + 2 <= ub && h != v;
            const unsigned m = __ballot_sync(FULL, in);
            const uint32_t pos = cnt + __popc(m & ((1u << lane) - 1u));
            if (in && pos < KEEP) keep[pos] = e[u];
            cnt += __popc(m);
        }
    }
    return cnt;
}

// The distance of an open pair, one warp, the labels first: the merge join, then the
// masks of the bit-parallel roots that can beat its answer.
__device__ __forceinline__ uint32_t pair_merged(const QueryArgs &a, const OpenPair &p, int lane) {
    uint32_t td0, td1, dstar;
    bp_tilde(a, p.s, p.t, lane, &td0, &td1, &dstar);
    const uint32_t best = label_min_merge_at(a, p.s, p.t, p.os, p.ls, p.ot, p.lt, lane);
    return finish_pair(a, p.s, p.t, lane, td0, td1, dstar, best);
}

// The same, reading as little of the labels as can be. The bit-parallel answer ub comes
// first: a common hub of the labels matters only below it. A label's hubs are
// at most its vertex's own rank, so of the two ends only the one of lower rank,
// h, can be a hub of the other, v: L(v) is read first, for h itself and for the
// near entries that can be on a path through a third hub (on power-law graphs,
// with ub 3 or 4, 1 entry in 20, often none), and L(h) only if there are some.
// The reads are one pass of independent loads; the merge join's windows wait
// for one another. (Bounded by the least d~ alone, with the masks after the
// labels, twice as many entries stay: 0.6 ms more on the 10M pairs of
// R-MAT-20; with both labels loaded along with the rows: 1 ms more.) With a bound
// past NEAR_MOST most entries are near, and the labels come first after all, as
// without a bound (t = 0, or ends that no root reaches); with too many near entries
// or where one label is long against the other, the merge join or its binary
// searches decide. 10M pairs with NEAR_MOST = 3, 4, 5 and none: R-MAT-20, t = 64, 3.50,
// 3.28, 3.30, 3.31 ms; BA of 50,000 vertices, t = 16, 8.43, 8.97, 9.59, 9.59 (8.26 with
// the labels first throughout).
constexpr uint32_t NEAR_MOST = 4;
constexpr uint32_t LONG_LABEL = 256;
constexpr uint32_t KEEP = 32;
__device__ __forceinline__ uint32_t pair_bounded(const QueryArgs &a, const OpenPair &p, int lane, uint32_t *keep) {
    uint32_t td0, td1, dstar;
    bp_tilde(a, p.s, p.t, lane, &td0, &td1, &dstar);
    if (dstar > NEAR_MOST) {
        const uint32_t best = label_min_merge_at(a, p.s, p.t, p.os, p.ls, p.ot, p.lt, lane);
        return finish_pair(a, p.s, p.t, lane, td0, td1, dstar, best);
    }
    uint32_t ub = finish_pair(a, p.s, p.t, lane, td0, td1, dstar, BIG);
    const bool low = p.s < p.t;  // h = s, v = t
    const uint32_t h = low ? p.s : p.t, v = low ? p.t : p.s, lh = low ? p.ls : p.lt, lv = low ? p.lt : p.ls;
    if (ub <= 1 || lv == 0) return ub;
    if (lv > LONG_LABEL && lv > PLL_MERGE_RATIO * lh) return min(ub, label_min(a, p.s, p.t, lane, 0, 32));
    uint32_t direct = BIG;
    const uint32_t cv = keep_near<KEEP>(a.lab + (low ? p.ot : p.os), lv, v, ub, h, lane, keep, &direct);
    if (cv > KEEP) return min(ub, label_min_merge_at(a, p.s, p.t, p.os, p.ls, p.ot, p.lt, lane));
    ub = min(ub, warp_min(direct));
    if (cv == 0 || ub <= 2) return ub;
    __syncwarp();
    const uint32_t *H = a.lab + (low ? p.os : p.ot);
    uint32_t best = ub;
    if (lh > LONG_LABEL) {  // a lane for each kept entry
        if ((uint32_t)lane < cv) {
            const uint32_t e = keep[lane];
            uint32_t lo = 0, hi = lh;
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                if (entry_hub(H[mid]) < entry_hub(e)) lo = mid + 1; else hi = mid;
            }
            if (lo < lh && entry_hub(H[lo]) == entry_hub(e)) best = min(best, entry_dist(e) + entry_dist(H[lo]));
        }
    } else {
        const uint32_t e = (uint32_t)lane < cv ? keep[lane] : NONE;
        const uint32_t ch = keep_near<KEEP>(H, lh, h, ub, NONE, lane, keep, &direct);
        if (ch > KEEP) return min(ub, label_min_merge_at(a, p.s, p.t, p.os, p.ls, p.ot, p.lt, lane));
        __syncwarp();
        for (uint32_t i = 0; i < ch; ++i) {
            const uint32_t f = keep[i];
            if (entry_hub(f) == entry_hub(e)) best = min(best, entry_dist(e) + entry_dist(f));
        }
    }
    return warp_min(best);
}

}  // namespace pairs
}  // namespace pll
