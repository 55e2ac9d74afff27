// k_query.cu -- batched distance queries over a built index.
//
// d(s, t) = min( bit-parallel query (Sec. 5.3), Query(s, t, L) (Sec. 3.3) ).
//
// A persistent grid (a few CTAs per SM) walks the pairs; one warp answers one
// pair, the labels first (pair_merged) or, where the labels are larger than the L2,
// the bit-parallel part, which bounds what the labels can add (pair_bounded).
// Pairs with an end that nothing reaches are settled by one lane each (lone_pair).
// A launch too small to fill the GPU that way (up to 4 pairs per
// resident block) gives each pair 2, 4 or 8 warps instead, which split the
// label scan and meet in shared memory. Lanes own bit-parallel roots (lane, lane + 32): the t distance bytes
// of s and of t arrive in one coalesced load each, and d~_i = d(s,r_i) +
// d(r_i,t). Since the answer through {r_i} U S_{r_i} lies in [d~_i - 2, d~_i],
// only roots with d~_i <= min_i d~_i + 1 can decide the minimum, and only
// those whose d~_i - 2 beats the normal-label answer fetch their 16-byte mask
// pairs. The normal labels are hub-sorted (hub ranks, Sec. 4.5.1): a warp
// merges them 32 entries at a time (the merge join of Sec. 3.3, with the
// comparisons of a window done by shuffles), or, when one label is much
// longer, each lane takes entries of the shorter label and binary-searches the
// longer one; both find the same common hubs. No sentinel is needed
// (Sec. 4.5.2): bounds are explicit.
#include <atomic>

#include "pair_device.cuh"

namespace pll {
using namespace pairs;
namespace {

constexpr int QUERY_BLOCKS = 8;

// One warp per pair, PG pairs at a time: lane j < PG first fetches pair j's
// ids, ranks and label offsets (three dependent loads, in flight for PG pairs
// at once instead of one after another), and answers the trivial and the lone
// pairs; the warp then answers the others one by one, their ranks and offsets
// in shared memory. PG is 32 for launches that fill the GPU that way and smaller
// for launches that would otherwise leave warps idle. Bound by the traffic and
// the latency of scattered loads, so it wants resident warps: eight blocks an
// SM, 32 registers a thread, for which 28 or 56 bytes of a thread's state go to local
// memory (six blocks, without: 10 % slower). 10M uniform pairs of
// R-MAT-20, t = 64: 5.02 ms with the merge join for every pair, 3.28 ms so, of
// which (by leaving steps out) 0.3 ms for ranks, offsets and lone pairs, 0.3
// for the rows, 1.0 for the masks and 0.8 for each end's label.
//
// NEAR: near entries only (pair_bounded), for indices whose labels are larger than the
// L2, where what it leaves unread counts; otherwise the labels first (pair_merged):
// the near entries are a second reading of what the L2 holds, and the masks they
// are bounded by are most of the work. 10M uniform pairs, near entries against
// labels first: R-MAT-17, 18, 20, 21 at t = 64 (labels of 5, 21, 288 and 998 MB)
// 2.26 and 1.93, 2.51 and 2.24, 3.27 and 3.37, 4.02 and 4.59 ms; R-MAT-19 at t = 64,
// 48, 32, 16, 8, 4 (77, 98, 127, 168, 225 and 268 MB) 2.77 and 2.67, 2.87 and 2.83,
// 2.79 and 2.82, 3.12 and 3.27, 3.77 and 4.08, 4.22 and 4.60; BA of 10,000 and 50,000
// vertices at t = 16 (1 and 32 MB) 4.59 and 3.46, 9.57 and 8.26.
template <int PG, bool NEAR>
__global__ void __launch_bounds__(256, QUERY_BLOCKS) k_query(QueryArgs a) {
    __shared__ uint32_t s_keep[NEAR ? 8 : 1][KEEP];
    __shared__ OpenPair s_pair[8][PG];
    __shared__ uint32_t s_errors[2];
    if (threadIdx.x < 2) s_errors[threadIdx.x] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    uint32_t *keep = s_keep[NEAR ? threadIdx.x >> 5 : 0];
    OpenPair *pair = s_pair[threadIdx.x >> 5];
    const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t q0 = (((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * PG; q0 < a.q;
         q0 += warps * PG) {
        const uint64_t qi = q0 + lane;
        const bool mine = lane < PG && qi < a.q;
        uint32_t ans = 0;
        bool open = false;
        if (mine) {
            OpenPair p;
            bool bad = false;
            open = !trivial_pair(a, a.src[qi * a.stride], a.dst[qi * a.stride], &p.s, &p.t, &ans, &bad);
            if (open) {
                p.os = a.lab_off[p.s];
                p.ot = a.lab_off[p.t];
                p.ls = (uint32_t)(a.lab_off[p.s + 1] - p.os);
                p.lt = (uint32_t)(a.lab_off[p.t + 1] - p.ot);
                uint32_t d, hub, ds;
                if (lone_pair(a, p.s, p.os, p.ls, p.t, p.ot, p.lt, &d, &hub, &ds)) {
                    ans = pair_answer(d);
                    open = false;
                } else {
                    pair[lane] = p;
                }
            } else if (bad) {
                ans |= ANS_BAD;
            }
        }
        __syncwarp();
        for (uint32_t m = __ballot_sync(FULL, open); m; m &= m - 1) {
            const int j = __ffs(m) - 1;
            const OpenPair p = pair[j];
            const uint32_t best = NEAR ? pair_bounded(a, p, lane, keep) : pair_merged(a, p, lane);
            if (lane == j) ans = pair_answer(best);  // best is the same on every lane
        }
        // the group's answers in one coalesced store (the output may be host
        // memory that the GPU writes directly)
        if (mine) a.out[qi] = (uint8_t)ans;
        count_errors(s_errors, ans, lane);
        __syncwarp();  // the next group writes pair
    }
    // What errors the block has counted, by each warp as it ends (its own are among
    // them): the counters may be host memory, where an addition costs 12 ns (10M pairs,
    // every id out of range: 3.6 ms with one a group of pairs, 0.2 so). A barrier at the end
    // costs the server, whose runs overlap, 4 % on R-MAT-22.
    if (lane < 2 && s_errors[lane]) {
        const uint32_t count = atomicExch(&s_errors[lane], 0u);
        if (count) atomicAdd_system(a.err + lane, (unsigned long long)count);
    }
}

// G warps of a block per pair, for launches too small to fill the GPU with
// one warp per pair: the label scan is split G ways (warp g takes entries
// 32 g, 32 (g + G), ...), which shortens the chain of dependent loads each
// pair waits on; the partial minima meet in shared memory.
template <int G>
__global__ void __launch_bounds__(256) k_query_wide(QueryArgs a) {
    __shared__ uint32_t part[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int member = warp % G;
    const uint64_t qi = (uint64_t)blockIdx.x * (8 / G) + warp / G;
    uint32_t s = 0, t = 0, ans = 0, td0 = BIG, td1 = BIG, dstar = BIG;
    bool bad = false, decided = true;
    if (qi < a.q) decided = trivial_pair(a, a.src[qi * a.stride], a.dst[qi * a.stride], &s, &t, &ans, &bad);
    if (!decided) {
        if (member == 0) bp_tilde(a, s, t, lane, &td0, &td1, &dstar);
        const uint32_t m = label_min(a, s, t, lane, 32u * member, 32u * G);
        if (lane == 0) part[warp] = m;
    }
    __syncthreads();  // every warp of the block arrives: no early exit above
    if (member != 0 || qi >= a.q) return;
    if (decided) {
        if (lane == 0) {
            a.out[qi] = (uint8_t)ans;
            if (bad) atomicAdd_system(a.err + 1, 1ull);  // at most four times R in a launch
        }
        return;
    }
    uint32_t best = BIG;
#pragma unroll
    for (int g = 0; g < G; ++g) best = min(best, part[warp + g]);
    best = finish_pair(a, s, t, lane, td0, td1, dstar, best);
    if (lane == 0) {
        ans = pair_answer(best);
        a.out[qi] = (uint8_t)ans;
        if (ans & ANS_FAR) atomicAdd_system(a.err, 1ull);
    }
}

template <bool NEAR>
void launch_query(const QueryArgs &a, uint64_t per, unsigned blocks, cudaStream_t s) {
    if (per >= 32) k_query<32, NEAR><<<blocks, 256, 0, s>>>(a);
    else if (per >= 8) k_query<8, NEAR><<<blocks, 256, 0, s>>>(a);
    else if (per >= 2) k_query<2, NEAR><<<blocks, 256, 0, s>>>(a);
    else k_query<1, NEAR><<<blocks, 256, 0, s>>>(a);
}

}  // namespace

int query_launch(const pll_index *ix, const uint32_t *d_src, const uint32_t *d_dst, uint64_t q,
                 uint8_t *d_out, unsigned long long *err, cudaStream_t s) {
    return query_launch_strided(ix, d_src, d_dst, 1, q, d_out, err, s);
}

int query_launch_strided(const pll_index *ix, const uint32_t *d_src, const uint32_t *d_dst,
                         uint32_t stride, uint64_t q, uint8_t *d_out, unsigned long long *err,
                         cudaStream_t s) {
    if (q == 0) return PLL_OK;
    // resident blocks of k_query on this device (SMs x blocks per SM) and its L2,
    // looked up once per device: the serving loop launches it thousands of times
    static std::atomic<int> resident[64], l2_bytes[64];
    int dev = 0;
    PLL_TRY(cudaGetDevice(&dev));
    int l2 = dev < 64 ? l2_bytes[dev].load(std::memory_order_relaxed) : 0;
    int res = dev < 64 ? resident[dev].load(std::memory_order_relaxed) : 0;
    if (res == 0 || l2 == 0) {
        int sms = 0, per = 0;
        PLL_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        PLL_TRY(cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev));
        PLL_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_query<32, true>, 256, 0));
        res = (sms > 0 ? sms : 1) * (per > 0 ? per : 1);
        l2 = l2 > 0 ? l2 : 1;
        if (dev < 64) resident[dev].store(res, std::memory_order_relaxed);
        if (dev < 64) l2_bytes[dev].store(l2, std::memory_order_relaxed);
    }
    const QueryArgs a = query_args(ix, d_src, d_dst, stride, q, d_out, err);
    // Pairs one warp each would leave most of the GPU idle: give each pair G
    // warps (8, 4 or 2; 8 / G pairs per block) while the ceil(q G / 8)
    // blocks still fit in one resident wave.
    const uint64_t R = (uint64_t)res;
    if (q <= R) {
        k_query_wide<8><<<(unsigned)q, 256, 0, s>>>(a);
    } else if (q <= 2 * R) {
        k_query_wide<4><<<(unsigned)((q + 1) / 2), 256, 0, s>>>(a);
    } else if (q <= 4 * R) {
        k_query_wide<2><<<(unsigned)((q + 3) / 4), 256, 0, s>>>(a);
    } else {
        // pairs per warp group: as many as keep every resident warp busy (R
        // blocks of 8 warps), up to 32
        const uint64_t per = q / (R * 8);
        if (ix->entries * 4 > (uint64_t)l2) launch_query<true>(a, per, (unsigned)R, s);
        else launch_query<false>(a, per, (unsigned)R, s);
    }
    PLL_TRY(cudaGetLastError());
    return PLL_OK;
}

}  // namespace pll
