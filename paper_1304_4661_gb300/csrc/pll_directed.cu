// pll_directed.cu -- directed graphs (Sec. 6, "Directed Graphs").
//
// Two label sets per vertex: L_IN(v) holds (u, d(u, v)) and L_OUT(v) holds
// (u, d(v, u)); d(s, t) = min over common hubs of L_OUT(s) and L_IN(t). Each
// root v_k, in rank order, runs a pruned BFS along arcs that fills L_IN
// (u is pruned when L_OUT(v_k) and L_IN(u) already give d(v_k, u)) and one
// against arcs that fills L_OUT (pruned when L_OUT(u) and L_IN(v_k) give
// d(u, v_k)). There are no bit-parallel labels: the masks of Sec. 5 rest on
// |d(s, v) - d(r, v)| <= 1 for neighbours s of r, which one-way arcs do not
// give.
//
// Root batches, as in the undirected build: the BFSs of roots [k0, k1) run
// together, pruned only with hubs < k0, then a cleanup removes the entries an
// in-batch hub h < k covers. A forward tuple (u, k, d) is surplus iff some
// in-batch h < k has a reverse tuple (v_k, h, a) (a = d(v_k, h)) and a forward
// tuple (u, h, b) (b = d(h, u)) with a + b <= d; a reverse tuple (u, k, d)
// iff some h < k has (u, h, a) reverse and (v_k, h, b) forward with
// a + b <= d. Every emitted distance is exact (a vertex reached late would
// have been pruned), and the least such h has tuples at both ends (nothing
// of rank < k0 lies on the subpaths), so the cleanup leaves exactly the
// sequential labels.
//
// The BFSs of a batch are the undirected build's sweeps (k_pruned.cu, without
// bit-parallel labels): the level loop as one CUDA graph launch per direction,
// with the root's table made from one label set and the visited vertices'
// labels read from the other; so are sorting, cleanup (each direction's tuples
// against the other's), compaction and the label store (k_labels.cu). The host
// reads back once a batch. Kernels of their own: k_dvalidate (CSR checks),
// k_dindeg / k_ddeg (in- plus out-degree for the Degree order and the reverse
// lists' offsets; a warp per vertex) and k_dquery (warp per pair).
// R-MAT-15, arcs one way or both (1.2M): 49.3 ms for the build and 1M queries
// with a thread-serial merge of two labels per frontier entry, two read-backs a
// level and batches of 1024; 11.7 ms so. What is left is launches: two
// directions of up to ten levels a batch, and a sort and a cleanup each.
#include <algorithm>
#include <new>
#include <vector>

#include <cub/cub.cuh>

#include "pll_internal.cuh"

using namespace pll;

// The directed index: labels in rank space, [0] = L_IN, [1] = L_OUT.
struct pll_dindex {
    int device = 0;
    unsigned long long ctx = 0;   // context_id() of its arrays
    uint32_t n = 0;
    uint64_t nnz = 0;
    uint32_t *d_order = nullptr;  // rank -> caller vertex id
    uint32_t *d_inv = nullptr;    // caller vertex id -> rank
    uint64_t *d_off[2] = {nullptr, nullptr};
    uint32_t *d_lab[2] = {nullptr, nullptr};
    uint64_t entries[2] = {0, 0};
    unsigned long long *d_qerr = nullptr;  // [0] finite distance >= 255, [1] id >= n
    uint64_t batches = 0;
    uint64_t pre_cleanup = 0;
};

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr uint32_t BIG = 1u << 20;

inline int blocks_for(uint64_t items, int per_block) {
    uint64_t g = (items + per_block - 1) / per_block;
    if (g < 1) g = 1;
    if (g > 16384) g = 16384;
    return (int)g;
}

// ---------------------------------------------------------------- checks
// Offsets start at 0, never decrease and end at nnz; each row is strictly
// ascending, without self-loops or ids >= n. A row (a warp each) is read only
// behind offsets that passed.
__global__ void k_dvalidate(uint32_t n, uint64_t nnz, const uint32_t *__restrict__ off,
                            const uint32_t *__restrict__ col, uint32_t *err) {
    const uint32_t lane = threadIdx.x & 31, warps = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t v = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += warps) {
        const uint32_t b = off[v], e = off[v + 1];
        bool bad = (v == 0 && b != 0) || (v == n - 1 && e != nnz) || b > e || e > nnz;
        if (!(b > e || e > nnz))
            for (uint32_t x = b + lane; x < e; x += 32) {
                const uint32_t c = col[x];
                bad |= c >= n || c == v || (x > b && col[x - 1] >= c);
            }
        if (bad) atomicOr(err, ERR_CSR);
    }
}

// cnt[w] += arcs into w
__global__ void k_dindeg(uint32_t n, const uint32_t *__restrict__ off, const uint32_t *__restrict__ col,
                         uint32_t *cnt) {
    const uint32_t lane = threadIdx.x & 31, warps = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t v = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += warps)
        for (uint32_t x = off[v] + lane, e = off[v + 1]; x < e; x += 32) atomicAdd(&cnt[col[x]], 1u);
}

// deg[v] = out-degree + in-degree (deg[n] is left 0 for the scan)
__global__ void k_ddeg(uint32_t n, const uint32_t *__restrict__ off, uint32_t *deg) {
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
        deg[v] += off[v + 1] - off[v];
}

// ------------------------------------------------------------- query
struct DQueryArgs {
    uint32_t n;
    const uint32_t *inv;
    const uint64_t *off_in, *off_out;
    const uint32_t *lab_in, *lab_out;
    const uint32_t *src, *dst;
    uint64_t q;
    uint8_t *out;
    unsigned long long *err;
};

// One warp per pair: lanes take entries of the shorter of L_OUT(s), L_IN(t)
// and binary-search the other by hub. A warp counts its errors and adds them at the
// end: the counters may be host memory (10M pairs, every id out of range: 114 ms
// with an addition for each, 0.4 ms so).
__global__ void __launch_bounds__(256) k_dquery(DQueryArgs a) {
    const int lane = threadIdx.x & 31;
    const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    uint32_t far = 0, bad = 0;
    for (uint64_t qi = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; qi < a.q; qi += warps) {
        const uint32_t sid = a.src[qi], tid = a.dst[qi];
        if (sid >= a.n || tid >= a.n) {
            if (lane == 0) a.out[qi] = INF8;
            ++bad;
            continue;
        }
        const uint32_t s = a.inv[sid], t = a.inv[tid];
        if (s == t) {
            if (lane == 0) a.out[qi] = 0;
            continue;
        }
        const uint64_t os = a.off_out[s], ot = a.off_in[t];
        const uint32_t ls = (uint32_t)(a.off_out[s + 1] - os), lt = (uint32_t)(a.off_in[t + 1] - ot);
        const bool sa = ls <= lt;
        const uint32_t *A = sa ? a.lab_out + os : a.lab_in + ot;
        const uint32_t *B = sa ? a.lab_in + ot : a.lab_out + os;
        const uint32_t la = sa ? ls : lt, lb = sa ? lt : ls;
        uint32_t best = BIG;
        for (uint32_t j = lane; j < la; j += 32) {
            const uint32_t ea = A[j], h = entry_hub(ea);
            uint32_t lo = 0, hi = lb;
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                if (entry_hub(B[mid]) < h) lo = mid + 1; else hi = mid;
            }
            if (lo < lb && entry_hub(B[lo]) == h) best = min(best, entry_dist(ea) + entry_dist(B[lo]));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) best = min(best, __shfl_xor_sync(FULL, best, o));
        if (lane == 0) a.out[qi] = (uint8_t)min(best, (uint32_t)INF8);
        far += best >= INF8 && best < BIG;
    }
    if (lane == 0 && far) atomicAdd_system(a.err, (unsigned long long)far);
    if (lane == 0 && bad) atomicAdd_system(a.err + 1, (unsigned long long)bad);
}

// ------------------------------------------------------------- host
int read_back(const void *d, void *h, size_t bytes, cudaStream_t s) {
    PLL_TRY(cudaMemcpyAsync(h, d, bytes, cudaMemcpyDeviceToHost, s));
    PLL_TRY(cudaStreamSynchronize(s));
    return PLL_OK;
}

void dindex_release(pll_dindex *ix) {
    if (!ix) return;
    dev_free(ix->d_order);
    dev_free(ix->d_inv);
    for (int i = 0; i < 2; ++i) {
        dev_free(ix->d_off[i]);
        dev_free(ix->d_lab[i]);
    }
    dev_free(ix->d_qerr);
    delete ix;
}

// Step 1: checks, order, relabel, reverse CSR. adj_off/adj_col[0] = arcs
// (out-neighbours), [1] = reversed arcs (in-neighbours), both in rank space.
int directed_prep(pll_dindex *ix, const uint32_t *off, const uint32_t *col, const uint32_t *order,
                  PoolMem *adj_off, PoolMem *adj_col, uint32_t *d_err, cudaStream_t s) {
    const uint32_t n = ix->n;
    const uint64_t nnz = ix->nnz;
    uint32_t h_err = 0;
    const int warp_blocks = blocks_for((uint64_t)n * 32, 256);
    k_dvalidate<<<warp_blocks, 256, 0, s>>>(n, nnz, off, col, d_err);
    PLL_TRY(cudaGetLastError());
    PLL_CHECK(read_back(d_err, &h_err, 4, s));
    if (h_err) return PLL_E_INVAL;
    Graph g;
    g.n = n; g.nnz = nnz; g.off = off; g.col = col;
    if (order) {
        PLL_TRY(cudaMemcpyAsync(ix->d_order, order, (size_t)n * 4, cudaMemcpyDeviceToDevice, s));
        PLL_CHECK(prep_check_order(g, ix->d_order, d_err, s));
        PLL_CHECK(read_back(d_err, &h_err, 4, s));
        if (h_err) return PLL_E_ORDER;
    } else {
        // the Degree order by in- plus out-degree: a CSR-shaped array whose
        // row lengths are those degrees feeds the undirected order's sort
        // (differences of the wrapped 32-bit scan are exact)
        PoolMem deg(s), doff(s), temp(s);
        PLL_CHECK(deg.alloc(((size_t)n + 1) * 4));
        PLL_CHECK(doff.alloc(((size_t)n + 1) * 4));
        PLL_TRY(cudaMemsetAsync(deg.p, 0, ((size_t)n + 1) * 4, s));
        k_dindeg<<<warp_blocks, 256, 0, s>>>(n, off, col, deg.as<uint32_t>());
        k_ddeg<<<blocks_for(n, 256), 256, 0, s>>>(n, off, deg.as<uint32_t>());
        PLL_TRY(cudaGetLastError());
        size_t tb = 0;
        PLL_TRY(cub::DeviceScan::ExclusiveSum(nullptr, tb, deg.as<uint32_t>(), doff.as<uint32_t>(),
                                              (int64_t)n + 1, s));
        PLL_CHECK(temp.alloc(tb));
        PLL_TRY(cub::DeviceScan::ExclusiveSum(temp.p, tb, deg.as<uint32_t>(), doff.as<uint32_t>(),
                                              (int64_t)n + 1, s));
        Graph gd;
        gd.n = n; gd.nnz = nnz; gd.off = doff.as<uint32_t>(); gd.col = col;
        PLL_CHECK(prep_degree_order(gd, ix->d_order, s));
    }
    PLL_CHECK(adj_off[0].alloc(((size_t)n + 1) * 4));
    PLL_CHECK(adj_col[0].alloc(std::max<uint64_t>(nnz, 1) * 4));
    PLL_CHECK(adj_off[1].alloc(((size_t)n + 1) * 4));
    PLL_CHECK(adj_col[1].alloc(std::max<uint64_t>(nnz, 1) * 4));
    PoolMem heads(s), cnt(s), temp(s);
    PLL_CHECK(heads.alloc(std::max<uint64_t>(nnz, 1) * 4));
    PLL_CHECK(prep_relabel(g, ix->d_order, ix->d_inv, adj_off[0].as<uint32_t>(), adj_col[0].as<uint32_t>(),
                           heads.as<uint32_t>(), adj_col[1].as<uint32_t>(), s));
    // the reverse lists' offsets: arcs into each rank, counted and scanned
    PLL_CHECK(cnt.alloc(((size_t)n + 1) * 4));
    PLL_TRY(cudaMemsetAsync(cnt.p, 0, ((size_t)n + 1) * 4, s));
    k_dindeg<<<warp_blocks, 256, 0, s>>>(n, adj_off[0].as<uint32_t>(), adj_col[0].as<uint32_t>(), cnt.as<uint32_t>());
    PLL_TRY(cudaGetLastError());
    size_t tb = 0;
    PLL_TRY(cub::DeviceScan::ExclusiveSum(nullptr, tb, cnt.as<uint32_t>(), adj_off[1].as<uint32_t>(),
                                          (int64_t)n + 1, s));
    PLL_CHECK(temp.alloc(tb));
    PLL_TRY(cub::DeviceScan::ExclusiveSum(temp.p, tb, cnt.as<uint32_t>(), adj_off[1].as<uint32_t>(),
                                          (int64_t)n + 1, s));
    return PLL_OK;
}

struct Store {
    LabelStore st;
    PoolMem off, len, cap;
    cudaStream_t s;
    explicit Store(cudaStream_t st_) : off(st_), len(st_), cap(st_), s(st_) {}
    ~Store() {
        pool_free(st.pool, s);
        labels_near_free(st, s);
    }
    int init(uint32_t n, unsigned long long *top) {
        st.n = n;
        PLL_CHECK(off.alloc((size_t)n * 8));
        PLL_CHECK(len.alloc((size_t)n * 4));
        PLL_CHECK(cap.alloc((size_t)n * 4));
        PLL_TRY(cudaMemsetAsync(off.p, 0, (size_t)n * 8, s));
        PLL_TRY(cudaMemsetAsync(len.p, 0, (size_t)n * 4, s));
        PLL_TRY(cudaMemsetAsync(cap.p, 0, (size_t)n * 4, s));
        st.off = off.as<uint64_t>();
        st.len = len.as<uint32_t>();
        st.cap = cap.as<uint32_t>();
        const uint64_t test_cap = test_caps().pool;
        st.pool_cap = test_cap ? test_cap : std::max<uint64_t>((uint64_t)n * 64, 1ull << 20);
        PLL_TRY(pool_malloc(&st.pool, st.pool_cap * 4, s));
        st.pool_top = top;
        return PLL_OK;
    }
};

// What the two directions of a batch leave on the device for one read-back.
struct DirState {
    BatchCounters c[2];
    LevelDesc d[2];
};

// Steps 2-4: root batches, both directions, cleanup, append; then the CSR.
int directed_labels(pll_dindex *ix, PoolMem *adj_off, PoolMem *adj_col, uint32_t bmax, cudaStream_t s) {
    const uint32_t n = ix->n;
    PoolMem m_state(s), m_loop(s), m_args(s);
    PLL_CHECK(m_state.alloc(sizeof(DirState)));
    PLL_CHECK(m_loop.alloc(sizeof(LoopState)));
    PLL_CHECK(m_args.alloc(sizeof(BatchArgs)));
    PLL_TRY(cudaMemsetAsync(m_state.p, 0, sizeof(DirState), s));
    PLL_TRY(cudaMemsetAsync(m_loop.p, 0, sizeof(LoopState), s));
    DirState *d = m_state.as<DirState>();
    Store store[2] = {Store(s), Store(s)};  // [0] L_IN, [1] L_OUT
    for (int dir = 0; dir < 2; ++dir) PLL_CHECK(store[dir].init(n, &d->c[dir].pool_top));

    const uint32_t block = 256, NW = (n + 31) / 32;
    int grid[2] = {0, 0};
    PLL_CHECK(batch_grid(block, grid));
    struct Graph2 {
        cudaGraph_t g = nullptr;
        cudaGraphExec_t e = nullptr;
        ~Graph2() {
            if (e) cudaGraphExecDestroy(e);
            if (g) cudaGraphDestroy(g);
        }
    } loop;
    PLL_CHECK(batch_graph_build(block, grid, m_args.as<BatchArgs>(), &loop.g, &loop.e));
    struct Mirror {
        DirState d;
        BatchArgs args[2];  // staging of the graph's device-side arguments
    };
    Mirror *h = nullptr;
    PLL_TRY(host_malloc(&h, sizeof(Mirror)));
    struct HostGuard {
        Mirror *h;
        ~HostGuard() { host_free(h); }
    } host_guard{h};

    // buffers shared by the directions (candidates, tables, the visited rows) or
    // one each (tuples and their sorted copy, needed together by the cleanup);
    // a batch that overflows one runs again with a larger one
    PoolMem vis(s), ht(s), reach(s), tab(s), cand(s), candc(s), slices(s), inX(s), keep(s), temp(s);
    PoolMem rstart[2] = {PoolMem(s), PoolMem(s)}, out[2] = {PoolMem(s), PoolMem(s)},
            sorted[2] = {PoolMem(s), PoolMem(s)};
    PLL_CHECK(vis.alloc((size_t)bmax * NW * 4));
    PLL_CHECK(inX.alloc(n));
    PLL_TRY(cudaMemsetAsync(inX.p, 0, n, s));
    const TestCaps caps = test_caps();
    uint64_t ht_cap = caps.ht ? caps.ht : std::max<uint64_t>((uint64_t)bmax * 1024, 1ull << 18);
    auto alloc_tables = [&]() -> int {
        PLL_CHECK(ht.alloc(ht_cap * 4));
        return reach.alloc(ht_cap * 4);
    };
    PLL_CHECK(alloc_tables());
    PLL_CHECK(tab.alloc((size_t)bmax * 8));
    size_t free_b = 0, total_b = 0;
    if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) {
        (void)cudaGetLastError();
        free_b = 0;
    }
    const uint64_t slice_cap = caps.cand ? std::min<uint64_t>(caps.cand, SLICE_CAP) : slice_entries(ix->nnz, free_b);
    PLL_CHECK(slices.alloc(slice_cap * 16));
    uint64_t cand_cap = caps.cand ? caps.cand
                                  : std::max<uint64_t>(std::min<uint64_t>((uint64_t)n * 128, free_b / 16 / 24), 1ull << 16);
    uint64_t out_cap = caps.out ? caps.out
                                : std::max<uint64_t>(std::min<uint64_t>((uint64_t)n * 64, free_b / 16 / 33), 1ull << 16);
    const int end_bit = 32 + [&] { int b = 1; while (b < 24 && ((n - 1) >> b)) ++b; return b; }();
    constexpr int SORT_BEGIN_BIT = 8;  // (u, k) is unique within a batch and direction
    auto alloc_cand = [&]() -> int {
        PLL_CHECK(cand.alloc(cand_cap * 8));
        PLL_CHECK(candc.alloc(cand_cap * 16));
        return PLL_OK;
    };
    auto alloc_out = [&]() -> int {
        for (int dir = 0; dir < 2; ++dir) {
            PLL_CHECK(out[dir].alloc(out_cap * 8));
            PLL_CHECK(sorted[dir].alloc(out_cap * 8));
        }
        PLL_CHECK(keep.alloc(out_cap));
        size_t a = 0, b = 0;
        PLL_CHECK(labels_sort_tuples(nullptr, nullptr, out_cap, SORT_BEGIN_BIT, end_bit, nullptr, &a, s));
        PLL_CHECK(labels_compact(nullptr, nullptr, out_cap, nullptr, nullptr, nullptr, &b, s));
        PLL_CHECK(temp.alloc(std::max<size_t>(std::max(a, b), (size_t)bmax * 16)));
        return PLL_OK;
    };
    PLL_CHECK(alloc_cand());
    PLL_CHECK(alloc_out());
    for (int dir = 0; dir < 2; ++dir) PLL_CHECK(rstart[dir].alloc((size_t)n * 4));

    // forward: along arcs, root label L_OUT, visited labels L_IN; reverse:
    // against arcs, root label L_IN, visited labels L_OUT
    auto run_dir = [&](int dir, uint32_t k0, uint32_t B, bool cut) -> int {
        const LabelStore &from = store[1 - dir].st, &to = store[dir].st;
        BatchArgs &a = h->args[dir];
        a = BatchArgs{};
        a.n = n;
        a.roff = adj_off[dir].as<uint32_t>(); a.rcol = adj_col[dir].as<uint32_t>();
        // a batch that found depth 255 runs again over the whole lists: past the
        // cut a vertex reached earlier would look new at that depth
        a.rstart = cut ? rstart[dir].as<uint32_t>() : a.roff;
        a.inX = inX.as<uint8_t>();
        a.lab_off = from.off; a.lab_len = from.len; a.pool = from.pool;
        a.vis_off = to.off; a.vis_len = to.len; a.vis_pool = to.pool;
        a.near = to.near; a.near_lab = to.near_lab; a.near_end = to.near_end;
        a.k0 = k0; a.B = B; a.NW = NW;
        a.visited = vis.as<uint32_t>();
        a.ht = ht.as<uint32_t>(); a.tab = tab.as<uint2>(); a.ht_cap = ht_cap;
        a.reach = reach.as<uint32_t>();
        a.cand = cand.as<uint64_t>(); a.candc = candc.as<uint64_t>(); a.cand_cap = cand_cap;
        a.out = out[dir].as<uint64_t>(); a.out_cap = out_cap;
        a.slices = slices.as<uint4>(); a.slice_cap = slice_cap;
        a.ctr = &d->c[dir]; a.desc = &d->d[dir]; a.loop = m_loop.as<LoopState>();
        PLL_TRY(cudaMemsetAsync(a.ctr, 0, 16, s));             // cand_n, out_n
        PLL_TRY(cudaMemsetAsync(&a.ctr->slice_n, 0, 28, s));   // slice_n, ht_top, taken, err
        if (cut) PLL_CHECK(batch_row_starts(n, k0, a.roff, a.rcol, rstart[dir].as<uint32_t>(), grid[0], s));
        PLL_CHECK(batch_init(a, s));
        PLL_TRY(cudaMemcpyAsync(m_args.p, &a, sizeof(BatchArgs), cudaMemcpyHostToDevice, s));
        PLL_TRY(cudaGraphLaunch(loop.e, s));
        return batch_clear(a, grid[0], s);
    };
    auto read_back = [&]() -> int {
        PLL_TRY(cudaMemcpyAsync(&h->d, d, sizeof(DirState), cudaMemcpyDeviceToHost, s));
        PLL_TRY(cudaStreamSynchronize(s));
        return PLL_OK;
    };
    // the kept counts of a batch arrive with the next batch's read-back
    // allocations past this point that the build cannot do without
    LabelStore *const stores[] = {&store[0].st, &store[1].st};
    auto needed = [&](auto &&alloc) { return alloc_needed(stores, 2, s, alloc); };
    uint64_t total[2] = {0, 0};
    bool pending[2] = {false, false};
    auto settle = [&]() -> int {
        for (int dir = 0; dir < 2; ++dir) {
            if (!pending[dir]) continue;
            pending[dir] = false;
            if (h->d.c[dir].err_post & ERR_POOL) return PLL_E_NOMEM;
            total[dir] += h->d.c[dir].nkept;
        }
        return PLL_OK;
    };
    uint32_t B = next_batch(0, 0, bmax), zeroed = 0;
    bool cut = true;
    for (uint32_t k0 = 0; k0 < n;) {
        const uint32_t k1 = (uint32_t)std::min<uint64_t>((uint64_t)k0 + B, n), Bc = k1 - k0;
        if (Bc > zeroed) {  // rows used for the first time
            PLL_TRY(cudaMemsetAsync(vis.as<uint32_t>() + (size_t)zeroed * NW, 0, (size_t)(Bc - zeroed) * NW * 4, s));
            zeroed = Bc;
        }
        for (int dir = 0; dir < 2; ++dir) PLL_CHECK(run_dir(dir, k0, Bc, cut));
        PLL_CHECK(read_back());
        PLL_CHECK(settle());
        const uint32_t err = h->d.c[0].err | h->d.c[1].err;
        if (err & ERR_TABLE) {  // those roots were binary-searched; grow for later batches
            const uint64_t need = std::max(h->d.c[0].ht_top, h->d.c[1].ht_top);
            if (!caps.ht)  // the test capacity keeps the pool small for the whole build
                PLL_CHECK(grow_if_possible(ht_cap, std::max<uint64_t>(need + need / 4, ht_cap * 2), alloc_tables));
        }
        if (err & ERR_BUF) {
            const uint64_t nc = std::max(h->d.c[0].cand_n, h->d.c[1].cand_n), no = std::max(h->d.c[0].out_n, h->d.c[1].out_n);
            if (nc > cand_cap) {
                cand_cap = std::max<uint64_t>(cand_cap * 2, nc + nc / 4);
                PLL_CHECK(needed(alloc_cand));
            }
            if (no > out_cap) {
                out_cap = std::max<uint64_t>(out_cap * 2, no + no / 4);
                PLL_CHECK(needed(alloc_out));
            }
            continue;
        }
        if (err & ERR_DEPTH) {
            if (!cut) return PLL_E_RANGE;
            cut = false;
            continue;
        }
        cut = true;
        const uint64_t P[2] = {h->d.c[0].out_n, h->d.c[1].out_n};
        ix->pre_cleanup += P[0] + P[1];
        // sort both directions, then clean each against the pre-cleanup other
        for (int dir = 0; dir < 2; ++dir) {
            size_t tb = temp.bytes;
            if (P[dir])
                PLL_CHECK(labels_sort_tuples(out[dir].as<uint64_t>(), sorted[dir].as<uint64_t>(), P[dir],
                                             SORT_BEGIN_BIT, end_bit, temp.p, &tb, s));
        }
        for (int dir = 0; dir < 2; ++dir) {
            if (P[dir] == 0) continue;
            LabelStore &st = store[dir].st;
            // worst-case pool growth of one append: 2 x (entries + new) + 8 per run
            const uint64_t need = h->d.c[dir].pool_top + 2 * (total[dir] + P[dir]) + 12 * P[dir];
            if (need > st.pool_cap)
                PLL_CHECK(needed([&] {
                    return labels_regrow(st, std::max<uint64_t>(st.pool_cap * 2, 3 * (total[dir] + P[dir]) + 12 * P[dir]), s);
                }));
            PLL_CHECK(labels_cleanup(sorted[dir].as<uint64_t>(), P[dir], sorted[1 - dir].as<uint64_t>(), P[1 - dir],
                                     keep.as<uint8_t>(), k0, Bc, temp.p, temp.bytes, s));
            size_t tb = temp.bytes;
            PLL_CHECK(labels_compact(sorted[dir].as<uint64_t>(), keep.as<uint8_t>(), P[dir], out[dir].as<uint64_t>(),
                                     &d->c[dir].nkept, temp.p, &tb, s));
            PLL_CHECK(labels_append(st, out[dir].as<uint64_t>(), &d->c[dir].nkept, P[dir], &d->c[dir].err_post, s));
            if (!caps.ht) PLL_CHECK(labels_near(st, total[dir], s));
            pending[dir] = true;
        }
        ++ix->batches;
        k0 = k1;
        B = next_batch(k0, P[0] + P[1], bmax);
    }
    PLL_CHECK(read_back());
    PLL_CHECK(settle());
    for (int dir = 0; dir < 2; ++dir) {
        PLL_CHECK(needed([&]() -> int { PLL_TRY(dev_malloc(&ix->d_off[dir], ((size_t)n + 1) * 8)); return PLL_OK; }));
        PLL_CHECK(needed([&]() -> int { PLL_TRY(dev_malloc(&ix->d_lab[dir], std::max<uint64_t>(total[dir], 1) * 4)); return PLL_OK; }));
        size_t ftb = 0;
        PLL_CHECK(labels_finalize(store[dir].st, total[dir], ix->d_off[dir], ix->d_lab[dir], nullptr, &ftb, s));
        PLL_CHECK(needed([&] { return temp.alloc(std::max<size_t>(ftb, 16)); }));
        PLL_CHECK(labels_finalize(store[dir].st, total[dir], ix->d_off[dir], ix->d_lab[dir], temp.p, &ftb, s));
        ix->entries[dir] = total[dir];
    }
    PLL_TRY(cudaStreamSynchronize(s));
    return PLL_OK;
}

}  // namespace

extern "C" {

PLL_API int pll_build_directed(const uint32_t *offsets, const uint32_t *cols, uint32_t n, uint64_t nnz,
                               const uint32_t *order, const pll_build_opts *opts, void *stream,
                               pll_dindex **out) {
    if (!out) return PLL_E_INVAL;
    *out = nullptr;
    pll_build_opts o{};
    if (opts) o = *opts;
    if (o.t != 0 || o.flags != 0 || o.reserved != 0) return PLL_E_INVAL;
    if (n > MAX_N || nnz >= 0xffffffffull) return PLL_E_RANGE;
    if ((n > 0 && !offsets) || (nnz > 0 && !cols) || (n == 0 && nnz != 0)) return PLL_E_INVAL;
    // default batch: as large as the undirected build's (R-MAT-17: 84.8 ms at 1024
    // roots, 52.0 at 16384, 50.6 at 65536; R-MAT-15: 18.6, 11.4, 11.4); the visited bits
    // of any batch stay within 2 GiB
    uint32_t bmax = std::max(1u, std::min({n, o.root_batch ? o.root_batch : default_batch(n, 2ull << 30, 64), BATCH_MAX}));
    while (bmax > 64 && (uint64_t)n * bmax / 8 > (2ull << 30)) bmax >>= 1;
    cudaStream_t s = (cudaStream_t)stream;
    pll_dindex *ix = new (std::nothrow) pll_dindex();
    if (!ix) return PLL_E_NOMEM;
    struct Guard {
        pll_dindex *ix;
        ~Guard() { dindex_release(ix); }
    } guard{ix};
    PLL_TRY(cudaGetDevice(&ix->device));
    ix->n = n;
    ix->nnz = nnz;
    PLL_TRY(dev_malloc(&ix->d_order, std::max<size_t>((size_t)n * 4, 4)));
    PLL_TRY(dev_malloc(&ix->d_inv, std::max<size_t>((size_t)n * 4, 4)));
    PLL_TRY(dev_malloc(&ix->d_qerr, 16));
    PLL_TRY(cudaMemsetAsync(ix->d_qerr, 0, 16, s));
    if (n == 0) {
        for (int dir = 0; dir < 2; ++dir) {
            PLL_TRY(dev_malloc(&ix->d_off[dir], 8));
            PLL_TRY(dev_malloc(&ix->d_lab[dir], 4));
            PLL_TRY(cudaMemsetAsync(ix->d_off[dir], 0, 8, s));
        }
    } else {
        PoolMem m_err(s), adj_off[2] = {PoolMem(s), PoolMem(s)}, adj_col[2] = {PoolMem(s), PoolMem(s)};
        PLL_CHECK(m_err.alloc(4));
        PLL_TRY(cudaMemsetAsync(m_err.p, 0, 4, s));
        PLL_CHECK(directed_prep(ix, offsets, cols, order, adj_off, adj_col, m_err.as<uint32_t>(), s));
        PLL_CHECK(directed_labels(ix, adj_off, adj_col, bmax, s));
    }
    PLL_TRY(cudaStreamSynchronize(s));
    ix->ctx = context_id();
    guard.ix = nullptr;
    *out = ix;
    return PLL_OK;
}

PLL_API int pll_dquery(const pll_dindex *idx, const uint32_t *src, const uint32_t *dst, uint64_t q,
                       uint8_t *out, void *stream) {
    if (!idx) return PLL_E_INVAL;
    if (q == 0) return PLL_OK;
    if (!src || !dst || !out) return PLL_E_INVAL;
    cudaStream_t s = (cudaStream_t)stream;
    CallErrors err(s, idx->ctx);
    PLL_CHECK(err.begin(idx->d_qerr));
    const DQueryArgs a{idx->n, idx->d_inv, idx->d_off[0], idx->d_off[1], idx->d_lab[0], idx->d_lab[1],
                       src, dst, q, out, err.p};
    int dev = 0, sms = 0;
    PLL_TRY(cudaGetDevice(&dev));
    PLL_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const uint64_t want = (q + 7) / 8, most = (uint64_t)(sms > 0 ? sms : 1) * 8;
    k_dquery<<<(unsigned)std::min(want, most), 256, 0, s>>>(a);
    PLL_TRY(cudaGetLastError());
    return err.finish();
}

PLL_API int pll_dlabel_entries(const pll_dindex *idx, uint64_t *in_entries, uint64_t *out_entries) {
    if (!idx || !in_entries || !out_entries) return PLL_E_INVAL;
    *in_entries = idx->entries[0];
    *out_entries = idx->entries[1];
    return PLL_OK;
}

PLL_API int pll_dexport_labels(const pll_dindex *idx, int which, uint64_t *offsets, uint32_t *hubs,
                               uint8_t *dists) {
    if (!idx || (which != 0 && which != 1) || !offsets) return PLL_E_INVAL;
    const uint64_t E = idx->entries[which];
    if (E && (!hubs || !dists)) return PLL_E_INVAL;
    const uint32_t n = idx->n;
    std::vector<uint64_t> off((size_t)n + 1);
    std::vector<uint32_t> lab(E), inv(n);
    PLL_TRY(cudaMemcpy(off.data(), idx->d_off[which], ((size_t)n + 1) * 8, cudaMemcpyDeviceToHost));
    if (E) PLL_TRY(cudaMemcpy(lab.data(), idx->d_lab[which], E * 4, cudaMemcpyDeviceToHost));
    if (n) PLL_TRY(cudaMemcpy(inv.data(), idx->d_inv, (size_t)n * 4, cudaMemcpyDeviceToHost));
    uint64_t p = 0;
    for (uint32_t v = 0; v < n; ++v) {
        offsets[v] = p;
        const uint32_t r = inv[v];
        for (uint64_t j = off[r]; j < off[(size_t)r + 1]; ++j, ++p) {
            hubs[p] = entry_hub(lab[j]);
            dists[p] = (uint8_t)entry_dist(lab[j]);
        }
    }
    offsets[n] = p;
    return PLL_OK;
}

PLL_API int pll_dexport_order(const pll_dindex *idx, uint32_t *order) {
    if (!idx || (idx->n && !order)) return PLL_E_INVAL;
    if (idx->n) PLL_TRY(cudaMemcpy(order, idx->d_order, (size_t)idx->n * 4, cudaMemcpyDeviceToHost));
    return PLL_OK;
}

PLL_API void pll_dfree(pll_dindex *idx) { dindex_release(idx); }

}  // extern "C"
