// pll_paths.cu -- shortest-path queries (Sec. 6, "Shortest-Path Queries").
//
// The paper keeps with each label entry (h, d) of L(v) the parent of v in the
// pruned BFS tree of h and restores an s-t path by climbing that tree from
// both ends. Here the parents are found once, after the build, from the
// finished labels: for (h, d) in L(v) with d > 0, the first neighbour w of v
// (in rank order) whose label holds (h, d - 1). Such a w is one hop nearer to
// h, and it holds h one hop lower in turn, so the climb reaches h in d steps.
// The BFS-tree parent itself is one such neighbour (the pruned BFS of h
// labels every vertex it expands); which one is kept does not change the
// path's length.
//
// When the bit-parallel label alone reaches d(s, t), the path runs through
// r_i or a member of S_{r_i}. The label gives that vertex's exact distance to
// every v: d(r_i, v) - 1, d(r_i, v) or d(r_i, v) + 1 as the member is in
// S^{-1}_{r_i}(v), S^0_{r_i}(v) or neither (Sec. 5.1). So each end walks to it
// one hop at a time, always to the first neighbour one hop nearer. The
// paper leaves paths through bit-parallel labels open; this is the reading
// taken here.
//
// Kernels: k_parents (a warp per vertex, lanes per label entry, each lane
// binary-searching the labels of the vertex's neighbours); path lengths come
// from the distance query; k_paths (a warp for up to 32 pairs: ranks, offsets and
// lone pairs on the lanes, the witnesses of the others one by one by the whole
// warp, then all climbs, a lane each, and all bit-parallel walks, eight lanes
// each, side by side).
#include <algorithm>
#include <new>
#include <vector>

#include <cub/device/device_scan.cuh>
#include <thrust/iterator/counting_iterator.h>
#include <thrust/iterator/transform_iterator.h>

#include "pair_device.cuh"

using namespace pll;
using namespace pll::pairs;

// Shortest-path support over a built index (borrowed: it must outlive this).
struct pll_paths {
    const pll_index *ix = nullptr;
    uint32_t *d_roff = nullptr;  // the graph in rank space, neighbours by rank
    uint32_t *d_rcol = nullptr;
    uint32_t *d_par = nullptr;   // parent (rank) of each label entry
};

namespace {

constexpr uint64_t NOPOS = ~0ull;
constexpr int PATH_BLOCKS = 8;  // of k_paths on an SM

// errors of the path kernels, a bit each of their error word
enum : uint32_t {
    PERR_ID,      // vertex id >= n
    PERR_SLOT,    // path_off not non-decreasing, past cap, or a slot too short
    PERR_RANGE,   // finite distance >= 255
    PERR_WALK,    // a climb or a walk found no next vertex (graph is not the index's)
    PERR_KINDS
};

// position of the packed entry `key` in the hub-sorted label lab[lo, hi)
// (hubs are unique in a label, so packed entries are sorted too)
__device__ __forceinline__ uint64_t find_entry(const uint32_t *__restrict__ lab, uint64_t lo,
                                               uint64_t hi, uint32_t key) {
    const uint64_t end = hi;
    while (lo < hi) {
        const uint64_t mid = (lo + hi) >> 1;
        if (lab[mid] < key) lo = mid + 1; else hi = mid;
    }
    return (lo < end && lab[lo] == key) ? lo : NOPOS;
}

struct ParentArgs {
    uint32_t n;
    const uint32_t *roff, *rcol;
    const uint64_t *lab_off;
    const uint32_t *lab;
    uint32_t *par;
    uint32_t *err;
};

// One warp per vertex v; each lane takes label entries of v and tries v's
// neighbours in rank order until one holds (h, d - 1).
__global__ void __launch_bounds__(256) k_parents(ParentArgs a) {
    const int lane = threadIdx.x & 31;
    const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t v = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < a.n; v += warps) {
        const uint64_t b = a.lab_off[v], e = a.lab_off[v + 1];
        const uint32_t nb = a.roff[v], ne = a.roff[v + 1];
        for (uint64_t j = b + lane; j < e; j += 32) {
            const uint32_t ent = a.lab[j], h = entry_hub(ent), d = entry_dist(ent);
            uint32_t p = NONE;
            if (d == 0) {
                if (h == (uint32_t)v) p = (uint32_t)v;
            } else {
                const uint32_t key = pack_entry(h, d - 1);
                for (uint32_t x = nb; x < ne; ++x) {
                    const uint32_t w = a.rcol[x];
                    if (find_entry(a.lab, a.lab_off[w], a.lab_off[w + 1], key) != NOPOS) { p = w; break; }
                }
            }
            if (p == NONE) atomicOr(a.err, 1u << PERR_WALK);
            a.par[j] = p;
        }
    }
}

struct PathArgs {
    QueryArgs x;               // the index and the pairs
    const uint32_t *order, *par;
    const uint32_t *roff, *rcol;
    const uint32_t *bp_root, *bp_S;  // [graphs][t], [graphs][t][64]
    uint32_t graphs;
    const uint64_t *path_off;  // slot of pair i is [path_off[i], path_off[i + 1])
    uint64_t cap;
    uint32_t *path;
    uint32_t *err;
};

__device__ __forceinline__ uint64_t warp_min64(uint64_t v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const uint64_t u = __shfl_xor_sync(FULL, v, o);
        v = u < v ? u : v;
    }
    return v;
}

// The common hub of L(s) and L(t) with the least distance sum (lowest rank
// among equals), as (sum << 32) | (hub << 8) | d(hub, s); NOPOS if none.
// Lanes take entries of the shorter label and binary-search the longer.
__device__ __forceinline__ uint64_t best_hub(const QueryArgs &a, const OpenPair &p, int lane) {
    const bool sa = p.ls <= p.lt;
    const uint32_t *A = a.lab + (sa ? p.os : p.ot), *B = a.lab + (sa ? p.ot : p.os);
    const uint32_t la = sa ? p.ls : p.lt, lb = sa ? p.lt : p.ls;
    uint64_t best = NOPOS;
    for (uint32_t j = lane; j < la; j += 32) {
        const uint32_t ea = A[j], h = entry_hub(ea);
        uint32_t lo = 0, hi = lb;
        while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if (entry_hub(B[mid]) < h) lo = mid + 1; else hi = mid;
        }
        if (lo < lb && entry_hub(B[lo]) == h) {
            const uint32_t da = entry_dist(ea), db = entry_dist(B[lo]);
            const uint64_t key = ((uint64_t)(da + db) << 32) | ((uint64_t)h << 8) | (sa ? da : db);
            best = key < best ? key : best;
        }
    }
    return warp_min64(best);
}

// The common hub with the least distance sum if that is at most ub (a key of
// best_hub's, or a larger one), from the near entries of both labels as in
// pair_bounded; hubs that only reach ub count here, so entries up to ub - 1 do.
constexpr uint32_t PATH_KEEP = 64;
__device__ __forceinline__ uint64_t near_hub(const QueryArgs &a, const OpenPair &p, uint32_t ub, int lane,
                                             uint32_t *keep) {
    const bool low = p.s < p.t;  // h = s, v = t
    const uint32_t h = low ? p.s : p.t, v = low ? p.t : p.s, lh = low ? p.ls : p.lt, lv = low ? p.lt : p.ls;
    if (max(lh, lv) > LONG_LABEL && max(lh, lv) > PLL_MERGE_RATIO * min(lh, lv)) return best_hub(a, p, lane);
    uint32_t direct = BIG;
    const uint32_t cv = keep_near<PATH_KEEP>(a.lab + (low ? p.ot : p.os), lv, v, ub + 1, h, lane, keep, &direct);
    if (cv > PATH_KEEP) return best_hub(a, p, lane);
    direct = warp_min(direct);
    uint64_t best = direct < BIG ? ((uint64_t)direct << 32) | ((uint64_t)h << 8) | (low ? 0u : direct) : NOPOS;
    if (cv == 0) return best;
    __syncwarp();
    const uint32_t e0 = (uint32_t)lane < cv ? keep[lane] : NONE, e1 = lane + 32u < cv ? keep[lane + 32] : NONE;
    const uint32_t ch = keep_near<PATH_KEEP>(a.lab + (low ? p.os : p.ot), lh, h, ub + 1, NONE, lane, keep, &direct);
    if (ch > PATH_KEEP) return best_hub(a, p, lane);
    __syncwarp();
    for (uint32_t i = 0; i < ch; ++i) {
        const uint32_t f = keep[i];
        if (entry_hub(f) == entry_hub(e0) || entry_hub(f) == entry_hub(e1)) {
            const uint32_t e = entry_hub(f) == entry_hub(e0) ? e0 : e1;
            const uint64_t key = ((uint64_t)(entry_dist(e) + entry_dist(f)) << 32) | ((uint64_t)entry_hub(f) << 8) |
                                 (low ? entry_dist(f) : entry_dist(e));
            best = key < best ? key : best;
        }
    }
    return warp_min64(best);
}

// The lowest bit-parallel slot that gives the bit-parallel distance ub, as
// (slot << 8) | (kind << 6) | bit: kind 0 meets in S^{-1} of both ends (d~ - 2),
// kind 1 in S^{-1} of one and S^0 of the other (d~ - 1), kind 2 at r_i (d~); bit
// = the lowest member where they meet. No slot gives less than ub, so a slot
// with d~ = ub meets at r_i, one with d~ = ub + 1 or ub + 2 reaches ub only by
// the matching reduction.
__device__ __forceinline__ uint32_t bp_slot(const QueryArgs &a, uint32_t s, uint32_t t, uint32_t ub, uint32_t td0,
                                            uint32_t td1, int lane) {
    uint32_t best = NONE;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t td = h ? td1 : td0, i = lane + 32 * h;
        if (td == ub) {
            best = min(best, i << 8 | 2u << 6);
        } else if (td == ub + 1 || td == ub + 2) {
            const ulonglong2 ms = reinterpret_cast<const ulonglong2 *>(a.bp_m)[(size_t)s * a.t + i];
            const ulonglong2 mt = reinterpret_cast<const ulonglong2 *>(a.bp_m)[(size_t)t * a.t + i];
            const uint64_t meet = td == ub + 2 ? ms.x & mt.x : (ms.x & mt.y) | (ms.y & mt.x);
            if (meet) best = min(best, i << 8 | (td == ub + 2 ? 0u : 1u << 6) | (uint32_t)(__ffsll((long long)meet) - 1));
        }
    }
    return warp_min(best);
}

// How a pair's path runs: through hub `at` (by >= 0: `by` from s), or through
// the bit-parallel vertex at = bp_slot's value (by < 0). d = BIG: there is none.
struct Witness {
    uint32_t d, at;
    int by;
};
__device__ __forceinline__ Witness pair_witness(const QueryArgs &a, const OpenPair &p, int lane, uint32_t *keep) {
    uint32_t td0 = BIG, td1 = BIG, dstar = BIG;
    if (a.t) bp_tilde(a, p.s, p.t, lane, &td0, &td1, &dstar);
    const uint32_t ub = finish_pair(a, p.s, p.t, lane, td0, td1, dstar, BIG);
    const uint64_t hk = ub < BIG ? near_hub(a, p, ub, lane, keep) : best_hub(a, p, lane);
    const uint32_t dn = hk == NOPOS ? BIG : (uint32_t)(hk >> 32);
    if (dn <= ub) return Witness{dn, (uint32_t)(hk >> 8) & 0xffffffu, (int)((uint32_t)hk & 0xffu)};
    return Witness{ub, bp_slot(a, p.s, p.t, ub, td0, td1, lane), -1};
}

// Distance from the bit-parallel vertex of slot i (r_i for kind 2, else member
// `bit` of S_{r_i}) to v; BIG if unreachable.
__device__ __forceinline__ uint32_t bp_dist_to(const PathArgs &a, uint32_t i, uint32_t kind,
                                               uint32_t bit, uint32_t v) {
    const uint32_t d = a.x.bp_d[(size_t)v * a.x.tp + i];
    if (d == INF8) return BIG;
    if (kind == 2) return d;
    const uint64_t *m = a.x.bp_m + 2 * ((size_t)v * a.x.t + i);
    const uint64_t b = 1ull << bit;
    if (m[0] & b) return d - 1;
    if (m[1] & b) return d;
    return d + 1;
}

// Walks from v (at distance dv) down to the bit-parallel vertex, writing the
// dv + 1 vertices at path[pos], path[pos + step], ...; by the WALK lanes of
// `group` (lane g of them), each step to the first neighbour one hop nearer.
// Every lane returns the same value: false if some vertex has no nearer neighbour.
// The last step is to the bit-parallel vertex itself, which a binary search finds in
// v's list (1M pairs of a complete graph of 1500 vertices, all of whose paths are
// such steps: 6.6 ms with a scan of the list by these lanes, 6.0 by 32, 0.57 so).
constexpr int WALK = 8;  // 4 or 16 lanes: 3 % slower
__device__ bool bp_walk(const PathArgs &a, uint32_t i, uint32_t kind, uint32_t bit, uint32_t v,
                        uint32_t dv, int64_t pos, int step, unsigned group, int g) {
    if (g == 0) a.path[pos] = a.order[v];
    while (dv > 0) {
        const uint32_t b = a.roff[v], e = a.roff[v + 1];
        uint32_t next = NONE;
        if (dv == 1) {
            const uint32_t gi = a.x.graph ? a.x.graph[v] : 0;
            if (gi >= a.graphs) return false;  // a file's graph ids are not checked
            const size_t slot = (size_t)gi * a.x.t + i;
            const uint32_t goal = kind == 2 ? a.bp_root[slot] : a.bp_S[slot * BPW + bit];
            uint32_t lo = b, hi = e;
            while (lo < hi) {
                const uint32_t mid = lo + ((hi - lo) >> 1);
                if (a.rcol[mid] < goal) lo = mid + 1; else hi = mid;
            }
            if (lo < e && a.rcol[lo] == goal) next = goal;
        } else {
            for (uint32_t x = b; x < e; x += WALK) {
                const uint32_t w = x + g < e ? a.rcol[x + g] : NONE;
                const unsigned m = __ballot_sync(group, w != NONE && bp_dist_to(a, i, kind, bit, w) == dv - 1) & group;
                if (m) { next = __shfl_sync(group, w, __ffs(m) - 1); break; }
            }
        }
        if (next == NONE) return false;
        v = next;
        --dv;
        pos += step;
        if (g == 0) a.path[pos] = a.order[v];
    }
    return true;
}

// Climbs the pruned BFS tree of hub h from v, which holds (h, d), writing the
// d + 1 vertices at path[pos], path[pos + step], ... (one thread).
__device__ bool climb(const PathArgs &a, uint32_t h, uint32_t v, uint32_t d, int64_t pos, int step) {
    for (uint32_t k = d;; --k) {
        a.path[pos] = a.order[v];
        if (k == 0) return v == h;
        const uint64_t j = find_entry(a.x.lab, a.x.lab_off[v], a.x.lab_off[v + 1], pack_entry(h, k));
        if (j == NOPOS) return false;
        v = a.par[j];
        if (v >= a.x.n) return false;
        pos += step;
    }
}

// Vertices on pair i's path, from its distance byte: d + 1, 0 if unreachable (and
// for a bad id or an out-of-range distance); 0 past the last pair.
struct PathLength {
    const uint8_t *dist;
    uint64_t q;
    __host__ __device__ uint64_t operator()(uint64_t i) const {
        return i < q && dist[i] != INF8 ? (uint64_t)dist[i] + 1 : 0;
    }
};

// One shortest path per pair into its slot; the rest of the slot (all of it
// for an unreachable pair) is filled with NONE. A warp takes up to G pairs:
// what each lane can settle about its own pair, then the witnesses of the open
// ones one by one, then the climbs and walks of all of them side by side (two
// ends each; a climb is a chain of dependent searches, and a walk's steps wait
// for one another too). Bound by the latency of those chains: eight blocks an SM
// (32 registers and 116 bytes of local memory; five blocks of 47 registers 10 %
// slower). 1M uniform pairs of R-MAT-20, t = 64, with the lengths: 2.90 ms with a warp
// per pair, binary searches for every witness and the climbs on two lanes; 1.70 ms
// so, of which (by leaving steps out) 0.6 ms was the witnesses, 0.5 the walks, 0.05
// the climbs; 1.45 ms with a search for a walk's last step and one copy each of the
// climb and the walk for both ends.
__global__ void __launch_bounds__(256, PATH_BLOCKS) k_paths(PathArgs a, uint32_t G) {
    __shared__ uint32_t s_keep[8][PATH_KEEP];
    __shared__ OpenPair s_pair[8][32];
    __shared__ Witness s_wit[8][32];
    __shared__ uint64_t s_slot[8][32];
    __shared__ uint8_t s_item[8][64];
    __shared__ uint8_t s_err[PERR_KINDS];  // what errors the block met
    if (threadIdx.x < PERR_KINDS) s_err[threadIdx.x] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    OpenPair *pair = s_pair[warp];
    Witness *wit = s_wit[warp];
    uint64_t *slot = s_slot[warp];
    uint8_t *item = s_item[warp];
    const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t q0 = (((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * G; q0 < a.x.q; q0 += warps * G) {
        const uint64_t qi = q0 + lane;
        uint64_t o0 = 0, o1 = 0, len = 0;
        bool open = false, routed = false;  // needs a witness; has one
        if ((uint32_t)lane < G && qi < a.x.q) {
            o0 = a.path_off[qi];
            o1 = a.path_off[qi + 1];
            if (o1 < o0 || o1 > a.cap) {
                s_err[PERR_SLOT] = 1;
                o1 = o0;  // nothing is written
            } else {
                OpenPair p;
                uint32_t ans = 0;
                bool bad = false;
                const uint32_t sid = a.x.src[qi];
                if (trivial_pair(a.x, sid, a.x.dst[qi], &p.s, &p.t, &ans, &bad)) {
                    if (bad) {
                        s_err[PERR_ID] = 1;
                    } else if (ans == 0) {  // s = t
                        if (o1 > o0) {
                            a.path[o0] = sid;
                            len = 1;
                        } else {
                            s_err[PERR_SLOT] = 1;
                        }
                    }
                } else {
                    p.os = a.x.lab_off[p.s];
                    p.ot = a.x.lab_off[p.t];
                    p.ls = (uint32_t)(a.x.lab_off[p.s + 1] - p.os);
                    p.lt = (uint32_t)(a.x.lab_off[p.t + 1] - p.ot);
                    pair[lane] = p;
                    uint32_t d, hub, ds;
                    if (lone_pair(a.x, p.s, p.os, p.ls, p.t, p.ot, p.lt, &d, &hub, &ds)) {
                        if (d < BIG) {
                            wit[lane] = Witness{d, hub, (int)ds};
                            routed = true;
                        }
                    } else {
                        open = true;
                    }
                }
            }
        }
        __syncwarp();
        for (unsigned m = __ballot_sync(FULL, open); m; m &= m - 1) {
            const int j = __ffs(m) - 1;
            const Witness w = pair_witness(a.x, pair[j], lane, s_keep[warp]);
            if (lane == j) {
                wit[j] = w;
                routed = w.d < BIG;
            }
        }
        bool climbs = false, walks = false;
        if (routed) {
            const Witness w = wit[lane];
            if (w.d >= INF8) {
                s_err[PERR_RANGE] = 1;
            } else if (o1 - o0 < (uint64_t)w.d + 1) {
                s_err[PERR_SLOT] = 1;
            } else {
                climbs = w.by >= 0;
                walks = !climbs;
                slot[lane] = o0;
            }
        }
        __syncwarp();
        // a common hub: climb its tree from both ends
        uint32_t failed = 0;
        unsigned m = __ballot_sync(FULL, climbs);
        if (climbs) {
            const int at = 2 * __popc(m & ((1u << lane) - 1u));
            item[at] = (uint8_t)lane;
            item[at + 1] = (uint8_t)(lane | 32);
        }
        __syncwarp();
        for (int x = lane; x < 2 * __popc(m); x += 32) {
            const int j = item[x] & 31;
            const Witness w = wit[j];
            const bool from_t = item[x] & 32;
            const bool ok = climb(a, w.at, from_t ? pair[j].t : pair[j].s, from_t ? w.d - w.by : w.by,
                                  (int64_t)(from_t ? slot[j] + w.d : slot[j]), from_t ? -1 : 1);
            if (!ok) failed |= 1u << j;
        }
        __syncwarp();
        // through r_i or a member of S_{r_i}: walk to it from both ends
        m = __ballot_sync(FULL, walks);
        if (walks) {
            const int at = 2 * __popc(m & ((1u << lane) - 1u));
            item[at] = (uint8_t)lane;
            item[at + 1] = (uint8_t)(lane | 32);
        }
        __syncwarp();
        const unsigned group = ((1u << WALK) - 1u) << (lane & ~(WALK - 1));
        for (int x = lane / WALK; x < 2 * __popc(m); x += 32 / WALK) {
            const int j = item[x] & 31;
            const Witness w = wit[j];
            const bool from_t = item[x] & 32;
            const uint32_t i = w.at >> 8, kind = (w.at >> 6) & 3u, bit = w.at & 63u;
            const uint32_t ds = bp_dist_to(a, i, kind, bit, pair[j].s), dt = bp_dist_to(a, i, kind, bit, pair[j].t);
            const bool ok = ds + dt == w.d &&
                            bp_walk(a, i, kind, bit, from_t ? pair[j].t : pair[j].s, from_t ? dt : ds,
                                    (int64_t)(from_t ? slot[j] + w.d : slot[j]), from_t ? -1 : 1, group, lane & (WALK - 1));
            if (!ok) failed |= 1u << j;
        }
        failed = __reduce_or_sync(FULL, failed);
        if (climbs || walks) {
            if ((failed >> lane) & 1) s_err[PERR_WALK] = 1;
            else len = (uint64_t)wit[lane].d + 1;
        }
        __syncwarp();  // the walks' writes come before the fill that may cover them
        for (m = __ballot_sync(FULL, o0 + len < o1); m; m &= m - 1) {
            const int j = __ffs(m) - 1;
            const uint64_t b = __shfl_sync(FULL, o0 + len, j), e = __shfl_sync(FULL, o1, j);
            for (uint64_t x = b + lane; x < e; x += 32) a.path[x] = NONE;
        }
        __syncwarp();  // the next group writes the shared arrays
    }
    __syncthreads();
    // written once: a.err may be host memory
    if (threadIdx.x < PERR_KINDS && s_err[threadIdx.x]) atomicOr_system(a.err, 1u << threadIdx.x);
}

int warp_grid(uint64_t items, int per_sm, int *blocks) {
    int dev = 0, sms = 0;
    PLL_TRY(cudaGetDevice(&dev));
    PLL_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const uint64_t want = (items + 7) / 8;  // 8 warps per block
    const uint64_t most = (uint64_t)(sms > 0 ? sms : 1) * per_sm;
    *blocks = (int)(want < most ? (want > 0 ? want : 1) : most);
    return PLL_OK;
}

// stream-ordered 4-byte error word, one per call
struct ErrWord {
    PoolMem m;
    uint32_t *p = nullptr;
    cudaStream_t s;
    explicit ErrWord(cudaStream_t st) : m(st), s(st) {}
    int alloc() {
        PLL_CHECK(m.alloc(4));
        p = m.as<uint32_t>();
        PLL_TRY(cudaMemsetAsync(p, 0, 4, s));
        return PLL_OK;
    }
    int read(uint32_t *h) {
        PLL_TRY(cudaMemcpyAsync(h, p, 4, cudaMemcpyDeviceToHost, s));
        PLL_TRY(cudaStreamSynchronize(s));
        return PLL_OK;
    }
};

int path_status(uint32_t e) {
    if (e & (1u << PERR_ID | 1u << PERR_SLOT | 1u << PERR_WALK)) return PLL_E_INVAL;
    if (e & (1u << PERR_RANGE)) return PLL_E_RANGE;
    return PLL_OK;
}

void paths_release(pll_paths *p) {
    if (!p) return;
    dev_free(p->d_roff);
    dev_free(p->d_rcol);
    dev_free(p->d_par);
    delete p;
}

}  // namespace

extern "C" {

PLL_API int pll_paths_create(const pll_index *idx, const uint32_t *offsets, const uint32_t *cols,
                             uint32_t n, uint64_t nnz, void *stream, pll_paths **out) {
    if (!out) return PLL_E_INVAL;
    *out = nullptr;
    if (!idx || n != idx->n || nnz != idx->nnz) return PLL_E_INVAL;
    if ((n > 0 && !offsets) || (nnz > 0 && !cols)) return PLL_E_INVAL;
    cudaStream_t s = (cudaStream_t)stream;
    pll_paths *p = new (std::nothrow) pll_paths();
    if (!p) return PLL_E_NOMEM;
    struct Guard {
        pll_paths *p;
        ~Guard() { paths_release(p); }
    } guard{p};
    p->ix = idx;
    ErrWord err(s);
    PLL_CHECK(err.alloc());
    uint32_t h = 0;
    Graph g;
    g.n = n; g.nnz = nnz; g.off = offsets; g.col = cols;
    PLL_CHECK(prep_validate_csr(g, err.p, s));
    PLL_CHECK(err.read(&h));
    if (h) return PLL_E_INVAL;
    PLL_TRY(dev_malloc(&p->d_roff, ((size_t)n + 1) * 4));
    PLL_TRY(dev_malloc(&p->d_rcol, std::max<uint64_t>(nnz, 1) * 4));
    PLL_TRY(dev_malloc(&p->d_par, std::max<uint64_t>(idx->entries, 1) * 4));
    {
        PoolMem inv(s);  // relabel writes an inverse order; the index keeps its own
        PLL_CHECK(inv.alloc(std::max<size_t>((size_t)n * 4, 4)));
        PLL_CHECK(prep_relabel(g, idx->d_order, inv.as<uint32_t>(), p->d_roff, p->d_rcol, nullptr, nullptr, s));
    }
    if (n > 0 && idx->entries > 0) {
        ParentArgs a{n, p->d_roff, p->d_rcol, idx->d_lab_off, idx->d_lab, p->d_par, err.p};
        int blocks = 0;
        PLL_CHECK(warp_grid(n, 8, &blocks));
        k_parents<<<blocks, 256, 0, s>>>(a);
        PLL_TRY(cudaGetLastError());
    }
    PLL_CHECK(err.read(&h));
    if (h) return PLL_E_INVAL;  // some entry has no parent: not the index's graph
    guard.p = nullptr;
    *out = p;
    return PLL_OK;
}

PLL_API int pll_paths_parents(const pll_paths *p, uint32_t *parents) {
    if (!p) return PLL_E_INVAL;
    const pll_index *ix = p->ix;
    if (ix->entries && !parents) return PLL_E_INVAL;
    const uint32_t n = ix->n;
    std::vector<uint64_t> off((size_t)n + 1);
    std::vector<uint32_t> par(ix->entries), inv(n), order(n);
    PLL_TRY(cudaMemcpy(off.data(), ix->d_lab_off, ((size_t)n + 1) * 8, cudaMemcpyDeviceToHost));
    if (ix->entries)
        PLL_TRY(cudaMemcpy(par.data(), p->d_par, ix->entries * 4, cudaMemcpyDeviceToHost));
    if (n) {
        PLL_TRY(cudaMemcpy(inv.data(), ix->d_inv, (size_t)n * 4, cudaMemcpyDeviceToHost));
        PLL_TRY(cudaMemcpy(order.data(), ix->d_order, (size_t)n * 4, cudaMemcpyDeviceToHost));
    }
    uint64_t k = 0;
    for (uint32_t v = 0; v < n; ++v) {
        const uint32_t r = inv[v];
        for (uint64_t j = off[r]; j < off[(size_t)r + 1]; ++j, ++k)
            parents[k] = par[j] < n ? order[par[j]] : NONE;
    }
    return PLL_OK;
}

PLL_API int pll_path_offsets(const pll_paths *p, const uint32_t *src, const uint32_t *dst, uint64_t q,
                             uint64_t *path_off, uint64_t *total, void *stream) {
    if (!p || !path_off || !total) return PLL_E_INVAL;
    if (q > 0 && (!src || !dst)) return PLL_E_INVAL;
    if (q >= 0x7fffffffull) return PLL_E_RANGE;
    cudaStream_t s = (cudaStream_t)stream;
    // the pairs' distances, then one scan of the lengths they stand for; the
    // total comes back behind the call's error counters
    CallErrors err(s, p->ix->ctx);
    PLL_CHECK(err.begin(nullptr));
    PoolMem dist(s), temp(s);
    PLL_CHECK(dist.alloc(q));
    PLL_CHECK(query_launch(p->ix, src, dst, q, dist.as<uint8_t>(), err.p, s));
    auto lengths = thrust::make_transform_iterator(thrust::counting_iterator<uint64_t>(0),
                                                   PathLength{dist.as<uint8_t>(), q});
    size_t tb = 0;
    PLL_TRY(cub::DeviceScan::ExclusiveSum(nullptr, tb, lengths, path_off, (int)(q + 1), s));
    PLL_CHECK(temp.alloc(tb));
    PLL_TRY(cub::DeviceScan::ExclusiveSum(temp.p, tb, lengths, path_off, (int)(q + 1), s));
    PLL_TRY(cudaMemcpyAsync(err.p + 2, path_off + q, 8, cudaMemcpyDefault, s));
    unsigned long long h[4];
    PLL_CHECK(err.finish(h));
    *total = h[2];
    return error_status(h);
}

PLL_API int pll_path_query(const pll_paths *p, const uint32_t *src, const uint32_t *dst, uint64_t q,
                           const uint64_t *path_off, uint64_t cap, uint32_t *path, void *stream) {
    if (!p) return PLL_E_INVAL;
    if (q == 0) return PLL_OK;
    if (!src || !dst || !path_off || (cap > 0 && !path)) return PLL_E_INVAL;
    cudaStream_t s = (cudaStream_t)stream;
    CallErrors err(s, p->ix->ctx);  // the first word takes the error bits
    PLL_CHECK(err.begin(nullptr));
    PathArgs a{};
    a.x = query_args(p->ix, src, dst, 1, q, nullptr, err.p);
    a.order = p->ix->d_order; a.par = p->d_par;
    a.roff = p->d_roff; a.rcol = p->d_rcol;
    a.bp_root = p->ix->d_bp_root; a.bp_S = p->ix->d_bp_S; a.graphs = p->ix->graphs;
    a.path_off = path_off;
    a.cap = cap;
    a.path = path;
    a.err = reinterpret_cast<uint32_t *>(err.p);
    int blocks = 0;
    PLL_CHECK(warp_grid(q, PATH_BLOCKS, &blocks));
    // pairs a warp takes at once: up to 32, fewer while warps would be left idle
    const uint64_t per = q / ((uint64_t)blocks * 8);
    k_paths<<<blocks, 256, 0, s>>>(a, per >= 32 ? 32u : per > 1 ? (uint32_t)per : 1u);
    PLL_TRY(cudaGetLastError());
    unsigned long long h[4];
    PLL_CHECK(err.finish(h));
    return path_status((uint32_t)h[0]);
}

PLL_API void pll_paths_free(pll_paths *p) { paths_release(p); }

}  // extern "C"
