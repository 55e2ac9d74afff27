// k_learned.cu -- a learned vertex order for the labelling.
//
// The labels are exact and minimal for ANY order (Thm 4.1, 4.2), but their
// size depends on it (Sec. 4.4, Table 4). Besides the paper's Degree order,
// a small network scores every vertex from local features, and vertices are
// taken by descending score:
//
//   features   per vertex: log(1 + deg), log(1 + sum of neighbour degrees),
//              log(1 + core number), and five statistics of the bit-parallel
//              labels of the Degree order (Alg. 3, Sec. 5.4): mean and min of
//              min(d(r_i, v), 32), the share of roots within distance 2, and
//              the mean sizes of S^-1 and S^0 over 64; every column then
//              standardised over the graph's vertices.
//   network    8 -> 64 -> 64 -> 1 with ReLU, parameters held as bfloat16 for
//              the forward and backward passes (float32 master copy, Adam),
//              all arithmetic in float32 (a dense but tiny contraction: 4.7k
//              multiply-adds per vertex; CUDA cores, weights staged in shared
//              memory).
//   target     log(1 + number of label entries whose hub is v) from builds in
//              the Degree order; vertices that get no pruned BFS are left out.
//   order      descending score, ties by ascending vertex id (one radix sort
//              of 64-bit keys).
#include <cub/cub.cuh>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>

#include "pll_internal.cuh"

namespace pll {
namespace {

constexpr int NF = 8, HID = 64;
constexpr int O_W1 = 0, O_B1 = 512, O_W2 = 576, O_B2 = 4672, O_W3 = 4736, O_B3 = 4800;
constexpr int NP = 4801;
constexpr uint32_t D_CAP = 32;

constexpr unsigned FULL = 0xffffffffu;

// ------------------------------------------------------------------ features
// deg(v) and the walks of length two, sum over neighbours of their degree;
// one warp per vertex.
__global__ void k_deg_twohop(uint32_t n, const uint32_t *__restrict__ off,
                             const uint32_t *__restrict__ col, uint32_t *deg,
                             unsigned long long *two_hop) {
    const int lane = threadIdx.x & 31;
    const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t v = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += warps) {
        const uint32_t b = off[v], e = off[v + 1];
        unsigned long long s = 0;
        for (uint32_t j = b + lane; j < e; j += 32) {
            const uint32_t u = col[j];
            s += off[u + 1] - off[u];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
        if (lane == 0) {
            deg[v] = e - b;
            two_hop[v] = s;
        }
    }
}

// Core numbers as the limit of repeated h-indices (Lu et al., Nature
// Communications 7, 2016): every vertex starts at its degree, and its value is
// replaced by the largest h such that h neighbours have a value of at least h,
// until nothing changes. Values only fall and never pass the core number, so
// they may be updated in place in any order. Only vertices that lost support
// are looked at again: a vertex that falls to h marks the neighbours above h
// for the next step. R-MAT-17 settles in 20 to 32 steps, most of them over a
// few hundred vertices, where peeling by degree takes 488 dependent passes,
// each a scan of all vertices and a read-back (pll_features with t = 64: 24.0
// ms so, 4.7 ms with the steps, 1.3 ms of it theirs). Bound by the longest
// lists of a step and the gathers of their neighbours' values (which take 64
// registers and 136 bytes of local memory a thread in lists next to CORE_BIG).
constexpr uint32_t CORE_BIG = 512;     // lists this long get a block each
constexpr int CORE_BIG_BLOCKS = 1024;
constexpr int CORE_CHUNK = 4;          // vertices a warp looks at together; it takes the marked
                                       // ones in turn (32 at a time: 0.75 ms more on R-MAT-17)

__global__ void k_core_init(uint32_t n, const uint32_t *__restrict__ deg, uint32_t *cur, uint8_t *dirty0,
                            uint8_t *dirty1, uint32_t *big, uint32_t *nbig) {
    for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (uint64_t)gridDim.x * blockDim.x) {
        cur[v] = deg[v];
        dirty0[v] = deg[v] != 0;
        dirty1[v] = 0;
        if (deg[v] >= CORE_BIG) big[atomicAdd(nbig, 1u)] = (uint32_t)v;
    }
}

struct CoreArgs {
    uint32_t n;
    const uint32_t *off, *col;
    uint32_t *cur;
    uint8_t *src, *dst;  // marked vertices of this step and of the next
    const uint32_t *big, *nbig;
    const uint32_t *prev;  // what the step before changed (null: run)
    uint32_t *changed;
};

// A vertex of at least CORE_BIG neighbours, one block: if fewer than c of them
// are at c or above, the largest h in [that count, c) by histograms of 256
// bins over the range that is left.
__device__ void core_big(const CoreArgs &a, uint32_t v) {
    __shared__ uint32_t hist[256], sum[8], pick;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t b = a.off[v], e = a.off[v + 1], c = a.cur[v];
    auto block_sum = [&](uint32_t x) {
        x = __reduce_add_sync(FULL, x);
        __syncthreads();
        if (lane == 0) sum[warp] = x;
        __syncthreads();
        uint32_t t = 0;
        for (int w = 0; w < 8; ++w) t += sum[w];
        return t;
    };
    uint32_t x = 0;
    for (uint32_t j = b + tid; j < e; j += 256) x += a.cur[a.col[j]] >= c;
    uint32_t above = block_sum(x);  // values past the range at hand
    if (above >= c) return;
    uint32_t lo = above, hi = c - 1;
    for (;;) {
        const uint32_t width = (hi - lo) / 256 + 1;
        hist[tid] = 0;
        __syncthreads();
        for (uint32_t j = b + tid; j < e; j += 256) {
            const uint32_t y = a.cur[a.col[j]];
            if (y >= lo && y <= hi) atomicAdd(&hist[(y - lo) / width], 1u);
        }
        if (tid == 0) pick = 0;
        __syncthreads();
        // values of bin tid and above: a scan over the bins from the top
        uint32_t suffix = hist[255 - tid];
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, suffix, o);
            if (lane >= o) suffix += y;
        }
        if (lane == 31) sum[warp] = suffix;
        __syncthreads();
        for (int w = 0; w < warp; ++w) suffix += sum[w];
        const uint32_t bin = 255 - tid;
        // the highest bin whose first value h has h neighbours at it or above
        const uint64_t h = (uint64_t)lo + (uint64_t)bin * width;
        if (h <= hi && (uint64_t)above + suffix >= h) atomicMax(&pick, bin);
        __syncthreads();
        const uint32_t at = pick;
        if (width == 1) {
            lo += at;
            break;
        }
        if (tid == 255 - (int)at) hist[0] = suffix - hist[at];  // values past the chosen bin
        __syncthreads();
        above += hist[0];
        lo += at * width;
        hi = min(hi, lo + width - 1);
        __syncthreads();
    }
    if (tid == 0) {
        a.cur[v] = lo;
        *a.changed = 1;
    }
    for (uint32_t j = b + tid; j < e; j += 256) {
        const uint32_t u = a.col[j];
        if (a.cur[u] > lo) a.dst[u] = 1;
    }
}

// the other marked vertices, a warp each, the neighbours' values in registers
__device__ void core_small(const CoreArgs &a, uint32_t v, uint32_t b, uint32_t d) {
    constexpr uint32_t Q = CORE_BIG / 32;
    const int lane = threadIdx.x & 31;
    const uint32_t c = a.cur[v];
    uint32_t id[Q], val[Q], x = 0;
#pragma unroll
    for (uint32_t q = 0; q < Q; ++q) {
        if (32 * q >= d) break;
        const bool in = 32 * q + lane < d;
        id[q] = in ? a.col[b + 32 * q + lane] : v;
    }
#pragma unroll
    for (uint32_t q = 0; q < Q; ++q) {
        if (32 * q >= d) break;
        val[q] = 32 * q + lane < d ? min(a.cur[id[q]], c) : 0;
        x += val[q] >= c;
    }
    uint32_t lo = __reduce_add_sync(FULL, x), hi = c - 1;
    if (lo >= c) return;
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) / 2;
        x = 0;
#pragma unroll
        for (uint32_t q = 0; q < Q; ++q) {
            if (32 * q >= d) break;
            x += val[q] >= mid;
        }
        if (__reduce_add_sync(FULL, x) >= mid) lo = mid; else hi = mid - 1;
    }
    if (lane == 0) {
        a.cur[v] = lo;
        *a.changed = 1;
    }
#pragma unroll
    for (uint32_t q = 0; q < Q; ++q) {
        if (32 * q >= d) break;
        if (val[q] > lo) a.dst[id[q]] = 1;
    }
}

// One step: the marked vertices' values. Blocks below CORE_BIG_BLOCKS take the
// long lists, the others CORE_CHUNK vertices a warp. Nothing to do (and nothing
// marked) if the step before changed nothing.
__global__ void __launch_bounds__(256) k_core_step(CoreArgs a) {
    if (a.prev && *a.prev == 0) return;
    if (blockIdx.x < CORE_BIG_BLOCKS) {
        for (uint32_t i = blockIdx.x; i < *a.nbig; i += CORE_BIG_BLOCKS) {
            const uint32_t v = a.big[i];
            const bool marked = a.src[v];  // the same on every thread
            __syncthreads();
            if (!marked) continue;
            core_big(a, v);
            __syncthreads();
            if (threadIdx.x == 0) a.src[v] = 0;
        }
        return;
    }
    const int lane = threadIdx.x & 31;
    const uint64_t warp = ((uint64_t)(blockIdx.x - CORE_BIG_BLOCKS) * blockDim.x + threadIdx.x) >> 5;
    const uint64_t warps = ((uint64_t)(gridDim.x - CORE_BIG_BLOCKS) * blockDim.x) >> 5;
    for (uint64_t v0 = warp * CORE_CHUNK; v0 < a.n; v0 += warps * CORE_CHUNK) {
        const uint64_t v = v0 + lane;
        uint32_t b = 0, d = CORE_BIG;
        if (lane < CORE_CHUNK && v < a.n && a.src[v]) {
            b = a.off[v];
            d = a.off[v + 1] - b;
        }
        for (unsigned m = __ballot_sync(FULL, d < CORE_BIG); m; m &= m - 1) {
            const int j = __ffs(m) - 1;
            core_small(a, (uint32_t)(v0 + j), __shfl_sync(FULL, b, j), __shfl_sync(FULL, d, j));
        }
        if (d < CORE_BIG) a.src[v] = 0;
    }
}

// Raw features (by caller id), a warp for 32 vertices: the bit-parallel rows
// (in rank space, row inv[v]) one vertex after the other over the lanes (roots
// lane and lane + 32), then a lane per vertex for the logarithms and quotients,
// which are in double precision: the FP64 units do two lanes a cycle, so the
// warp must not spend them on one vertex at a time (R-MAT-17, t = 64: 1173 us
// with a warp per vertex, 102 us so).
__global__ void __launch_bounds__(256) k_features_raw(uint32_t n, uint32_t t, uint32_t tp,
                                                      const uint32_t *__restrict__ inv,
                                                      const uint32_t *__restrict__ deg,
                                                      const unsigned long long *__restrict__ two_hop,
                                                      const uint32_t *__restrict__ core,
                                                      const uint8_t *__restrict__ bp_d,
                                                      const uint64_t *__restrict__ bp_m, float *X) {
    const int lane = threadIdx.x & 31;
    const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t v0 = (((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; v0 < n; v0 += warps * 32) {
        const uint64_t v = v0 + lane;
        uint32_t sum = 0, mn = D_CAP, near = 0, p1 = 0, p0 = 0;  // of vertex v
        if (t) {
            const uint32_t mine = v < n ? inv[v] : 0;
            const int cnt = n - v0 < 32 ? (int)(n - v0) : 32;
#pragma unroll 4
            for (int j = 0; j < cnt; ++j) {
                const size_t r = __shfl_sync(FULL, mine, j);
                uint32_t dn = 0, pp = 0, m = D_CAP;  // sum | near << 16, |S^-1| | |S^0| << 16
#pragma unroll
                for (uint32_t h = 0; h < 2; ++h) {
                    const uint32_t i = lane + 32 * h;
                    if (i < t) {
                        const uint32_t dc = min((uint32_t)bp_d[r * tp + i], D_CAP);
                        const ulonglong2 s = reinterpret_cast<const ulonglong2 *>(bp_m)[r * t + i];
                        m = min(m, dc);
                        dn += dc + ((uint32_t)(dc <= 2) << 16);
                        pp += __popcll(s.x) + ((uint32_t)__popcll(s.y) << 16);
                    }
                }
                dn = __reduce_add_sync(FULL, dn);  // at most 64 * 32 and 64
                pp = __reduce_add_sync(FULL, pp);  // at most 64 * 64 each
                m = __reduce_min_sync(FULL, m);
                if (lane == j) {
                    sum = dn & 0xffff;
                    near = dn >> 16;
                    p1 = pp & 0xffff;
                    p0 = pp >> 16;
                    mn = m;
                }
            }
        }
        if (v < n) {
            float *x = X + v * NF;
            x[0] = (float)log1p((double)deg[v]);
            x[1] = (float)log1p((double)two_hop[v]);
            x[2] = (float)log1p((double)core[v]);
            x[3] = t ? (float)((double)sum / t) : 0.f;
            x[4] = t ? (float)mn : 0.f;
            x[5] = t ? (float)((double)near / t) : 0.f;
            x[6] = t ? (float)((double)p1 / (64.0 * t)) : 0.f;
            x[7] = t ? (float)((double)p0 / (64.0 * t)) : 0.f;
        }
    }
}

// Column sums (pass 0) or sums of squared deviations from mean[] (pass 1),
// in double, one atomic per column per block.
__global__ void k_col_moments(uint32_t n, const float *__restrict__ X, const double *__restrict__ mean,
                              int pass, double *acc) {
    __shared__ double part[NF][33];
    double s[NF];
#pragma unroll
    for (int j = 0; j < NF; ++j) s[j] = 0;
    for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (uint64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int j = 0; j < NF; ++j) {
            const double x = X[v * NF + j];
            s[j] += pass == 0 ? x : (x - mean[j]) * (x - mean[j]);
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int j = 0; j < NF; ++j) {
        double a = s[j];
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(FULL, a, o);
        if (lane == 0) part[j][warp] = a;
    }
    __syncthreads();
    if (threadIdx.x < NF) {
        double a = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) a += part[threadIdx.x][w];
        atomicAdd(&acc[threadIdx.x], a);
    }
}

__global__ void k_mean(uint32_t n, double *acc) {
    if (threadIdx.x < NF) acc[threadIdx.x] = n ? acc[threadIdx.x] / n : 0;
}

// ssd[j] becomes the population std of column j (a square root per column, not
// per value, in double precision)
__global__ void k_std(uint32_t n, double *ssd) {
    if (threadIdx.x < NF) ssd[threadIdx.x] = sqrt(ssd[threadIdx.x] / n);
}

__global__ void k_standardise(uint32_t n, const double *__restrict__ mean, const double *__restrict__ sd,
                              float *X) {
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (uint64_t)n * NF;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const int j = (int)(i % NF);
        X[i] = sd[j] > 0 ? (float)(((double)X[i] - mean[j]) / sd[j]) : 0.f;
    }
}

// ------------------------------------------------------------------ hubs
__global__ void k_hub_counts(uint64_t entries, const uint32_t *__restrict__ lab,
                             const uint32_t *__restrict__ order, uint32_t *counts) {
    for (uint64_t e = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; e < entries;
         e += (uint64_t)gridDim.x * blockDim.x)
        atomicAdd(&counts[order[entry_hub(lab[e])]], 1u);
}

__global__ void k_log1p_counts(uint32_t n, const uint32_t *__restrict__ counts, float *target) {
    for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (uint64_t)gridDim.x * blockDim.x)
        target[v] = (float)log1p((double)counts[v]);
}

// ------------------------------------------------------------------ network
// the bf16 parameters as floats (W has room for NP + 3)
__device__ __forceinline__ void load_weights(const __nv_bfloat16 *__restrict__ w16, float *W) {
    const __nv_bfloat162 *p = reinterpret_cast<const __nv_bfloat162 *>(w16);
    for (int i = threadIdx.x; i < NP / 2; i += blockDim.x) {
        const float2 f = __bfloat1622float2(p[i]);
        W[2 * i] = f.x;
        W[2 * i + 1] = f.y;
    }
    if (threadIdx.x == 0) W[NP - 1] = __bfloat162float(w16[NP - 1]);
}

// row r of the features; vec: x is 16-byte aligned
__device__ __forceinline__ void load_features(const float *__restrict__ X, uint64_t r, bool vec, float (&x)[NF]) {
    if (vec) {
        const float4 a = __ldg(reinterpret_cast<const float4 *>(X) + 2 * r);
        const float4 b = __ldg(reinterpret_cast<const float4 *>(X) + 2 * r + 1);
        x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
        x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
    } else {
#pragma unroll
        for (int k = 0; k < NF; ++k) x[k] = X[r * NF + k];
    }
}

// y = w3 . relu(W2 relu(W1 x + b1) + b2) + b3, R rows a thread (row tid + FT a
// of the block's tile). Every output keeps one chain of multiply-adds in index
// order. Bound by the FP32 units: with one row a thread and one output unit
// at a time each multiply-add waited for the one before it and every four
// took a load of weights (2.1M rows: 980 us, 20 TFLOP/s); with four units at a
// time over two rows eight chains run together and a load of four weights
// serves eight multiply-adds: 385 us, 51 TFLOP/s (63 % of the FMA pipe and 66 %
// of the shared-memory bandwidth). The same with two-row multiply-adds
// (fma.rn.f32x2): 403 us. Three blocks an SM (168 registers).
constexpr int FT = 128;
template <int R>
__global__ void __launch_bounds__(FT, 3) k_mlp_fwd(uint64_t n, const float *__restrict__ X, bool vec,
                                                const __nv_bfloat16 *__restrict__ w16, float *y) {
    __shared__ __align__(16) float W[NP + 3];
    load_weights(w16, W);
    __syncthreads();
    for (uint64_t base = (uint64_t)blockIdx.x * FT * R; base < n; base += (uint64_t)gridDim.x * FT * R) {
        float x[R][NF], h1[R][HID];
#pragma unroll
        for (int a = 0; a < R; ++a) {
            const uint64_t r = base + FT * a + threadIdx.x;
            load_features(X, r < n ? r : n - 1, vec, x[a]);
        }
#pragma unroll
        for (int i = 0; i < HID; ++i) {
            float z[R];
#pragma unroll
            for (int a = 0; a < R; ++a) z[a] = W[O_B1 + i];
#pragma unroll
            for (int k = 0; k < NF; ++k) {
                const float w = W[O_W1 + i * NF + k];
#pragma unroll
                for (int a = 0; a < R; ++a) z[a] = fmaf(w, x[a][k], z[a]);
            }
#pragma unroll
            for (int a = 0; a < R; ++a) h1[a][i] = fmaxf(z[a], 0.f);
        }
        float out[R];
#pragma unroll
        for (int a = 0; a < R; ++a) out[a] = W[O_B3];
#pragma unroll 1
        for (int j = 0; j < HID; j += 4) {
            float z[4][R];
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int a = 0; a < R; ++a) z[c][a] = W[O_B2 + j + c];
#pragma unroll
            for (int i = 0; i < HID; i += 4) {
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float4 w = *reinterpret_cast<const float4 *>(&W[O_W2 + (j + c) * HID + i]);
#pragma unroll
                    for (int a = 0; a < R; ++a) {
                        z[c][a] = fmaf(w.x, h1[a][i], z[c][a]);
                        z[c][a] = fmaf(w.y, h1[a][i + 1], z[c][a]);
                        z[c][a] = fmaf(w.z, h1[a][i + 2], z[c][a]);
                        z[c][a] = fmaf(w.w, h1[a][i + 3], z[c][a]);
                    }
                }
            }
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int a = 0; a < R; ++a) out[a] = fmaf(W[O_W3 + j + c], fmaxf(z[c][a], 0.f), out[a]);
        }
#pragma unroll
        for (int a = 0; a < R; ++a) {
            const uint64_t r = base + FT * a + threadIdx.x;
            if (r < n) y[r] = out[a];
        }
    }
}

constexpr int GT = 64;       // rows per block of the gradient kernel
constexpr int GTH = 256;     // its threads: 16 x 16, each 4 x 4 outputs of a 64 x 64 product
constexpr int RS = HID + 4;  // padded row stride of its tiles: 16-byte loads of 16 rows without conflicts
struct GradSmem {
    float W2[HID * RS], W2t[HID * RS];    // [j][i], [i][j]
    float H1[GT * RS], H1t[HID * RS];     // [row][i] (later dZ1), [i][row]
    float D2[GT * RS], D2t[HID * RS];     // [row][j] (first H2, then dZ2), [j][row]
    float X[GT * NF], W1[HID * NF], b1[HID], b2[HID], w3[HID], dy[GT], sq[GT];
    float b3;
};

// acc[a][b] += sum over k of A[r0 + 16 a][k] B[c0 + 16 b][k], k ascending: a 4 x 4
// register tile of a product of two 64 x 64 tiles, both read along k
__device__ __forceinline__ void tile_product(const float *A, const float *B, int r0, int c0, float (&acc)[4][4]) {
#pragma unroll 4
    for (int k = 0; k < HID; k += 4) {
        float4 x[4], y[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) x[a] = *reinterpret_cast<const float4 *>(&A[(r0 + 16 * a) * RS + k]);
#pragma unroll
        for (int b = 0; b < 4; ++b) y[b] = *reinterpret_cast<const float4 *>(&B[(c0 + 16 * b) * RS + k]);
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                acc[a][b] = fmaf(x[a].x, y[b].x, acc[a][b]);
                acc[a][b] = fmaf(x[a].y, y[b].y, acc[a][b]);
                acc[a][b] = fmaf(x[a].z, y[b].z, acc[a][b]);
                acc[a][b] = fmaf(x[a].w, y[b].w, acc[a][b]);
            }
    }
}

// Gradient of the mean squared error over `batch` rows (row g of the batch is
// sample idx[g], or g without idx). Each block takes GT rows: the forward pass
// and the back-propagation to dZ2 and dZ1 as products of 64 x 64 tiles in
// shared memory (each in both layouts that its products read along), then
// the sums over the rows for the 4801 parameters, written as one partial per
// block (summed in a fixed order by k_mlp_reduce, so the result is
// deterministic). Bound by shared-memory loads (8 for 64 multiply-adds) and,
// at a batch of 16,384, by one wave of 256 blocks, two an SM: with a thread
// per row and 128 rows a block each SM had four warps. 50.6 -> 21.7 us there.
__global__ void __launch_bounds__(GTH) k_mlp_grad(uint32_t batch, const float *__restrict__ X, bool vec,
                                                  const float *__restrict__ target,
                                                  const uint32_t *__restrict__ idx,
                                                  const __nv_bfloat16 *__restrict__ w16,
                                                  float *partial, float *ploss) {
    extern __shared__ float4 grad_dyn[];
    GradSmem &s = *reinterpret_cast<GradSmem *>(grad_dyn);
    const int tid = threadIdx.x, r0 = tid >> 4, c0 = tid & 15;
    for (int o = tid; o < NP; o += GTH) {
        const float w = __bfloat162float(w16[o]);
        if (o < O_B1) s.W1[o] = w;
        else if (o < O_W2) s.b1[o - O_B1] = w;
        else if (o < O_B2) {
            const int j = (o - O_W2) / HID, i = (o - O_W2) % HID;
            s.W2[j * RS + i] = w;
            s.W2t[i * RS + j] = w;
        } else if (o < O_W3) s.b2[o - O_B2] = w;
        else if (o < O_B3) s.w3[o - O_W3] = w;
        else s.b3 = w;
    }
    uint64_t row = 0;  // of thread tid < GT
    bool valid = false;
    if (tid < GT) {
        const uint32_t g = blockIdx.x * GT + tid;
        valid = g < batch;
        row = valid ? (idx ? idx[g] : g) : 0;
        float x[NF];
        load_features(X, row, vec, x);
#pragma unroll
        for (int k = 0; k < NF; ++k) s.X[tid * NF + k] = valid ? x[k] : 0.f;
    }
    __syncthreads();

    float acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int r = r0 + 16 * a, i = c0 + 16 * b;
            float z = s.b1[i];
#pragma unroll
            for (int k = 0; k < NF; ++k) z = fmaf(s.W1[i * NF + k], s.X[r * NF + k], z);
            z = fmaxf(z, 0.f);
            s.H1[r * RS + i] = z;
            s.H1t[i * RS + r] = z;
        }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int a = 0; a < 4; ++a) acc[a][b] = s.b2[c0 + 16 * b];
    tile_product(s.H1, s.W2, r0, c0, acc);  // Z2
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            acc[a][b] = fmaxf(acc[a][b], 0.f);
            s.D2[(r0 + 16 * a) * RS + c0 + 16 * b] = acc[a][b];  // H2
        }
    __syncthreads();
    if (tid < GT) {
        float y = s.b3;
#pragma unroll
        for (int j = 0; j < HID; j += 4) {
            const float4 h = *reinterpret_cast<const float4 *>(&s.D2[tid * RS + j]);
            y = fmaf(s.w3[j], h.x, y);
            y = fmaf(s.w3[j + 1], h.y, y);
            y = fmaf(s.w3[j + 2], h.z, y);
            y = fmaf(s.w3[j + 3], h.w, y);
        }
        const float res = valid ? y - target[row] : 0.f;
        s.dy[tid] = 2.f * res / (float)batch;
        s.sq[tid] = res * res;
    }
    __syncthreads();
    float *out = partial + (size_t)blockIdx.x * NP;
    if (tid < HID) {  // dw3, from H2
        float a = 0.f;
#pragma unroll 8
        for (int r = 0; r < GT; ++r) a = fmaf(s.dy[r], s.D2[r * RS + tid], a);
        out[O_W3 + tid] = a;
    } else if (tid == HID) {
        float a = 0.f, l = 0.f;
        for (int r = 0; r < GT; ++r) {
            a += s.dy[r];
            l += s.sq[r];
        }
        out[O_B3] = a;
        ploss[blockIdx.x] = l;
    }
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int r = r0 + 16 * a, j = c0 + 16 * b;
            const float dz = acc[a][b] > 0.f ? s.dy[r] * s.w3[j] : 0.f;
            s.D2[r * RS + j] = dz;
            s.D2t[j * RS + r] = dz;
            acc[a][b] = 0.f;
        }
    __syncthreads();
    tile_product(s.D2, s.W2t, r0, c0, acc);  // dH1
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            float *h = &s.H1[(r0 + 16 * a) * RS + c0 + 16 * b];  // read and replaced by this thread only
            *h = *h > 0.f ? acc[a][b] : 0.f;
            acc[a][b] = 0.f;
        }
    tile_product(s.D2t, s.H1t, r0, c0, acc);  // dW2[j][i]
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) out[O_W2 + (r0 + 16 * a) * HID + c0 + 16 * b] = acc[a][b];
    __syncthreads();
    float w0 = 0.f, w1 = 0.f, bs = 0.f;  // dW1[i][k], dW1[i + 32][k]; db1 or db2
    const int i1 = tid / NF, k1 = tid % NF;
    const float *bsrc = tid < HID ? &s.H1[tid] : &s.D2[tid - HID];
#pragma unroll 8
    for (int r = 0; r < GT; ++r) {
        const float x = s.X[r * NF + k1];
        w0 = fmaf(s.H1[r * RS + i1], x, w0);
        w1 = fmaf(s.H1[r * RS + i1 + 32], x, w1);
        if (tid < 2 * HID) bs += bsrc[r * RS];
    }
    out[O_W1 + i1 * NF + k1] = w0;
    out[O_W1 + (i1 + 32) * NF + k1] = w1;
    if (tid < HID) out[O_B1 + tid] = bs;
    else if (tid < 2 * HID) out[O_B2 + tid - HID] = bs;
}

// grad[o] = sum over blocks of partial[b][o], eight interleaved runs of blocks
// in block order, then the runs in order; grad[NP] = loss.
__global__ void __launch_bounds__(256) k_mlp_reduce(uint32_t blocks, uint32_t batch, const float *__restrict__ partial,
                                                    const float *__restrict__ ploss, float *grad) {
    __shared__ float part[8][32];
    const int lane = threadIdx.x & 31, run = threadIdx.x >> 5, o = blockIdx.x * 32 + lane;
    float a = 0.f;
    if (o <= NP) {
        const float *src = o < NP ? partial + o : ploss;
        const size_t step = o < NP ? NP : 1;
#pragma unroll 4
        for (uint32_t b = run; b < blocks; b += 8) a += src[(size_t)b * step];
    }
    part[run][lane] = a;
    __syncthreads();
    if (run != 0 || o > NP) return;
#pragma unroll
    for (int r = 1; r < 8; ++r) a += part[r][lane];
    grad[o] = o < NP ? a : a / (float)batch;
}

// Adam (Kingma and Ba, 2015) on the float32 master parameters; c1, c2 are
// the bias corrections 1 / (1 - beta^step), and 1 - beta comes in rounded
// from double (1 - 0.999f in float32 is off by 1e-5 relative). The bf16 copy
// follows.
__global__ void k_adam(const float *__restrict__ grad, float *master, float *m, float *v,
                       __nv_bfloat16 *w16, float lr, float b1, float omb1, float b2, float omb2,
                       float eps, float c1, float c2) {
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= NP) return;
    const float g = grad[o];
    const float mo = b1 * m[o] + omb1 * g;
    const float vo = b2 * v[o] + omb2 * g * g;
    m[o] = mo;
    v[o] = vo;
    const float p = master[o] - lr * (mo * c1) / (sqrtf(vo * c2) + eps);
    master[o] = p;
    w16[o] = __float2bfloat16_rn(p);
}

__global__ void k_to_bf16(const float *__restrict__ p, __nv_bfloat16 *w16) {
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o < NP) w16[o] = __float2bfloat16_rn(p[o]);
}

// ------------------------------------------------------------------ order
// Key of a score that sorts ascending as the score descends; -0 is +0, NaN
// goes last.
__global__ void k_score_keys(uint32_t n, const float *__restrict__ score, uint64_t *keys) {
    for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (uint64_t)gridDim.x * blockDim.x) {
        const float f = score[v];
        uint32_t k;
        if (f != f) {
            k = 0xffffffffu;
        } else {
            uint32_t b = __float_as_uint(f == 0.f ? 0.f : f);
            const uint32_t asc = (b & 0x80000000u) ? ~b : (b | 0x80000000u);  // ascending in f
            k = ~asc;
        }
        keys[v] = ((uint64_t)k << 32) | v;
    }
}

__global__ void k_key_ids(uint32_t n, const uint64_t *__restrict__ keys, uint32_t *order) {
    for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (uint64_t)gridDim.x * blockDim.x)
        order[v] = (uint32_t)keys[v];
}

int grid_for(uint64_t work, int block) {
    uint64_t g = (work + block - 1) / block;
    if (g > 152ull * 32) g = 152ull * 32;
    return (int)(g ? g : 1);
}

int read_u32(const uint32_t *d, cudaStream_t s, uint32_t *h) {
    PLL_TRY(cudaMemcpyAsync(h, d, 4, cudaMemcpyDeviceToHost, s));
    PLL_TRY(cudaStreamSynchronize(s));
    return PLL_OK;
}

}  // namespace

// Core numbers of the caller-space graph (deg already computed). The steps are
// enqueued several at a time; a step that finds nothing changed before it
// returns at once.
int core_numbers(const Graph &g, const uint32_t *d_deg, uint32_t *d_core, cudaStream_t s) {
    const uint32_t n = g.n;
    if (n == 0) return PLL_OK;
    constexpr int AHEAD = 8;
    PoolMem m_d0(s), m_d1(s), m_big(s), m_ctl(s);
    PLL_CHECK(m_d0.alloc(n));
    PLL_CHECK(m_d1.alloc(n));
    PLL_CHECK(m_big.alloc(std::max<uint64_t>(g.nnz / CORE_BIG, 1) * 4));
    PLL_CHECK(m_ctl.alloc((AHEAD + 1) * 4));
    uint32_t *nbig = m_ctl.as<uint32_t>(), *changed = nbig + 1;
    PLL_TRY(cudaMemsetAsync(nbig, 0, 4, s));
    k_core_init<<<grid_for(n, 256), 256, 0, s>>>(n, d_deg, d_core, m_d0.as<uint8_t>(), m_d1.as<uint8_t>(),
                                                 m_big.as<uint32_t>(), nbig);
    PLL_TRY(cudaGetLastError());
    CoreArgs a{n, g.off, g.col, d_core, m_d0.as<uint8_t>(), m_d1.as<uint8_t>(), m_big.as<uint32_t>(), nbig,
               nullptr, nullptr};
    const int grid = CORE_BIG_BLOCKS + grid_for((uint64_t)n * 32 / CORE_CHUNK, 256);
    uint32_t h[AHEAD];
    // every step but the last lowers a value, so the loop is finite
    for (uint64_t step = 0; step <= g.nnz + AHEAD; step += AHEAD) {
        PLL_TRY(cudaMemsetAsync(changed, 0, AHEAD * 4, s));
        for (int i = 0; i < AHEAD; ++i) {
            a.prev = i ? changed + i - 1 : nullptr;
            a.changed = changed + i;
            k_core_step<<<grid, 256, 0, s>>>(a);
            std::swap(a.src, a.dst);
        }
        PLL_TRY(cudaGetLastError());
        PLL_TRY(cudaMemcpyAsync(h, changed, AHEAD * 4, cudaMemcpyDeviceToHost, s));
        PLL_TRY(cudaStreamSynchronize(s));
        if (h[AHEAD - 1] == 0) return PLL_OK;
    }
    return PLL_E_CUDA;
}

}  // namespace pll

using namespace pll;

struct pll_mlp {
    int device = 0;
    unsigned long long ctx = 0;  // context_id() of its arrays
    uint32_t wide = 0;  // blocks of k_mlp_fwd<2> that the device holds at once
    uint32_t max_batch = 0, blocks = 0;
    float *master = nullptr, *m = nullptr, *v = nullptr;
    __nv_bfloat16 *w16 = nullptr;
    float *grad = nullptr;     // [NP + 1], the last one the loss
    float *partial = nullptr;  // [blocks][NP]
    float *ploss = nullptr;    // [blocks]
    uint64_t step = 0;
    void *mem = nullptr;
};

extern "C" {

PLL_API int pll_features(const uint32_t *offsets, const uint32_t *cols, uint32_t n, uint64_t nnz,
                         uint32_t t, void *stream, float *feat, uint32_t *core,
                         uint64_t *two_hop) {
    cudaStream_t s = (cudaStream_t)stream;
    if (t > PLL_MAX_T) return PLL_E_RANGE;
    if (n > MAX_N || nnz >= 0xffffffffull) return PLL_E_RANGE;
    if ((n > 0 && (!offsets || !feat)) || (nnz > 0 && !cols) || (n == 0 && nnz)) return PLL_E_INVAL;
    if (n == 0) return PLL_OK;
    Graph g;
    g.n = n; g.nnz = nnz; g.off = offsets; g.col = cols;
    PoolMem m_err(s);
    PLL_CHECK(m_err.alloc(4));
    PLL_TRY(cudaMemsetAsync(m_err.p, 0, 4, s));
    PLL_CHECK(prep_validate_csr(g, m_err.as<uint32_t>(), s));
    uint32_t h_err = 0;
    PLL_CHECK(read_u32(m_err.as<uint32_t>(), s, &h_err));
    if (h_err) return PLL_E_INVAL;

    PoolMem m_deg(s), m_two(s), m_core(s);
    PLL_CHECK(m_deg.alloc((size_t)n * 4));
    uint64_t *d_two = two_hop;
    uint32_t *d_core = core;
    if (!d_two) { PLL_CHECK(m_two.alloc((size_t)n * 8)); d_two = m_two.as<uint64_t>(); }
    if (!d_core) { PLL_CHECK(m_core.alloc((size_t)n * 4)); d_core = m_core.as<uint32_t>(); }
    k_deg_twohop<<<grid_for((uint64_t)n * 32, 256), 256, 0, s>>>(
        n, offsets, cols, m_deg.as<uint32_t>(), reinterpret_cast<unsigned long long *>(d_two));
    PLL_TRY(cudaGetLastError());
    PLL_CHECK(core_numbers(g, m_deg.as<uint32_t>(), d_core, s));

    // bit-parallel labels of the Degree order (rank space)
    const uint32_t tp = bp_stride(t);
    PoolMem m_order(s), m_inv(s), m_roff(s), m_rcol(s), m_inX(s), m_root(s), m_cnt(s), m_S(s), m_bpd(s), m_bpm(s);
    if (t) {
        PLL_CHECK(m_order.alloc((size_t)n * 4));
        PLL_CHECK(m_inv.alloc((size_t)n * 4));
        PLL_CHECK(prep_degree_order(g, m_order.as<uint32_t>(), s));
        PLL_CHECK(m_roff.alloc(((size_t)n + 1) * 4));
        PLL_CHECK(m_rcol.alloc(std::max<uint64_t>(nnz, 1) * 4));
        PLL_CHECK(prep_relabel(g, m_order.as<uint32_t>(), m_inv.as<uint32_t>(), m_roff.as<uint32_t>(),
                               m_rcol.as<uint32_t>(), nullptr, nullptr, s));
        PLL_CHECK(m_inX.alloc(n));
        PLL_TRY(cudaMemsetAsync(m_inX.p, 0, n, s));
        PLL_CHECK(m_root.alloc((size_t)t * 4));
        PLL_CHECK(m_cnt.alloc((size_t)t * 4));
        PLL_CHECK(m_S.alloc((size_t)t * BPW * 4));
        PLL_TRY(cudaMemsetAsync(m_S.p, 0xff, (size_t)t * BPW * 4, s));
        PLL_CHECK(prep_select_bp_roots(n, t, m_roff.as<uint32_t>(), m_rcol.as<uint32_t>(),
                                       m_inX.as<uint8_t>(), m_root.as<uint32_t>(), m_cnt.as<uint32_t>(),
                                       m_S.as<uint32_t>(), s));
        PLL_CHECK(m_bpd.alloc((size_t)n * tp));
        PLL_CHECK(m_bpm.alloc((size_t)n * t * 16));
        uint32_t levels = 0;
        PLL_TRY(cudaMemsetAsync(m_err.p, 0, 4, s));
        PLL_CHECK(bp_run(n, t, 1, m_roff.as<uint32_t>(), m_rcol.as<uint32_t>(), m_root.as<uint32_t>(),
                         m_cnt.as<uint32_t>(), m_S.as<uint32_t>(), m_bpd.as<uint8_t>(),
                         m_bpm.as<uint64_t>(), nullptr, m_err.as<uint32_t>(), s, &levels));
        PLL_CHECK(read_u32(m_err.as<uint32_t>(), s, &h_err));
        if (h_err) return (h_err & ERR_DEPTH) ? PLL_E_RANGE : PLL_E_CUDA;
    }
    k_features_raw<<<grid_for(n, 256), 256, 0, s>>>(
        n, t, tp, m_inv.as<uint32_t>(), m_deg.as<uint32_t>(),
        reinterpret_cast<const unsigned long long *>(d_two), d_core, m_bpd.as<uint8_t>(),
        m_bpm.as<uint64_t>(), feat);
    PLL_TRY(cudaGetLastError());
    PoolMem m_mom(s);
    PLL_CHECK(m_mom.alloc(2 * NF * sizeof(double)));
    double *mean = m_mom.as<double>(), *ssd = mean + NF;
    PLL_TRY(cudaMemsetAsync(m_mom.p, 0, 2 * NF * sizeof(double), s));
    k_col_moments<<<grid_for(n, 256), 256, 0, s>>>(n, feat, mean, 0, mean);
    k_mean<<<1, 32, 0, s>>>(n, mean);
    k_col_moments<<<grid_for(n, 256), 256, 0, s>>>(n, feat, mean, 1, ssd);
    k_std<<<1, 32, 0, s>>>(n, ssd);
    k_standardise<<<grid_for((uint64_t)n * NF, 256), 256, 0, s>>>(n, mean, ssd, feat);
    PLL_TRY(cudaGetLastError());
    PLL_TRY(cudaStreamSynchronize(s));
    return PLL_OK;
}

PLL_API int pll_hub_counts(const pll_index *idx, uint32_t *counts, float *log1p_counts, void *stream) {
    if (!idx || !counts) return PLL_E_INVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const uint32_t n = idx->n;
    if (n == 0) return PLL_OK;
    PLL_TRY(cudaMemsetAsync(counts, 0, (size_t)n * 4, s));
    if (idx->entries) {
        k_hub_counts<<<grid_for(idx->entries, 256), 256, 0, s>>>(idx->entries, idx->d_lab, idx->d_order,
                                                                  counts);
        PLL_TRY(cudaGetLastError());
    }
    if (log1p_counts) {
        k_log1p_counts<<<grid_for(n, 256), 256, 0, s>>>(n, counts, log1p_counts);
        PLL_TRY(cudaGetLastError());
    }
    PLL_TRY(cudaStreamSynchronize(s));
    return PLL_OK;
}

PLL_API int pll_order_from_scores(const float *scores, uint32_t n, uint32_t *order, void *stream) {
    if (n && (!scores || !order)) return PLL_E_INVAL;
    if (n == 0) return PLL_OK;
    cudaStream_t s = (cudaStream_t)stream;
    PoolMem m_keys(s), m_sorted(s), m_temp(s);
    PLL_CHECK(m_keys.alloc((size_t)n * 8));
    PLL_CHECK(m_sorted.alloc((size_t)n * 8));
    k_score_keys<<<grid_for(n, 256), 256, 0, s>>>(n, scores, m_keys.as<uint64_t>());
    PLL_TRY(cudaGetLastError());
    size_t tb = 0;
    PLL_TRY(cub::DeviceRadixSort::SortKeys(nullptr, tb, m_keys.as<uint64_t>(), m_sorted.as<uint64_t>(),
                                           (int)n, 0, 64, s));
    PLL_CHECK(m_temp.alloc(tb));
    PLL_TRY(cub::DeviceRadixSort::SortKeys(m_temp.p, tb, m_keys.as<uint64_t>(), m_sorted.as<uint64_t>(),
                                           (int)n, 0, 64, s));
    k_key_ids<<<grid_for(n, 256), 256, 0, s>>>(n, m_sorted.as<uint64_t>(), order);
    PLL_TRY(cudaGetLastError());
    PLL_TRY(cudaStreamSynchronize(s));
    return PLL_OK;
}

PLL_API int pll_mlp_create(uint32_t max_batch, pll_mlp **out) {
    if (!out || max_batch == 0) return PLL_E_INVAL;
    *out = nullptr;
    pll_mlp *p = new (std::nothrow) pll_mlp();
    if (!p) return PLL_E_NOMEM;
    p->max_batch = max_batch;
    p->blocks = (max_batch + GT - 1) / GT;
    const size_t nf = 4 * (size_t)NP + (NP + 1) + (size_t)p->blocks * NP + p->blocks + 8;
    int sms = 0, per = 0;
    cudaError_t e = cudaGetDevice(&p->device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p->device);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_mlp_fwd<2>, FT, 0);
    p->wide = (uint32_t)std::max(1, sms * per);
    if (e == cudaSuccess) e = cudaMalloc(&p->mem, nf * sizeof(float));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GradSmem));
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        if (p->mem) cudaFree(p->mem);
        delete p;
        return e == cudaErrorMemoryAllocation ? PLL_E_NOMEM : cuda_status(e);
    }
    float *f = static_cast<float *>(p->mem);
    p->master = f;
    p->m = f + NP;
    p->v = f + 2 * NP;
    p->w16 = reinterpret_cast<__nv_bfloat16 *>(f + 3 * NP);  // NP bf16 fit in NP floats
    p->grad = f + 4 * NP;
    p->partial = p->grad + NP + 1;
    p->ploss = p->partial + (size_t)p->blocks * NP;
    if (cudaMemset(p->mem, 0, nf * sizeof(float)) != cudaSuccess) {
        (void)cudaGetLastError();
        cudaFree(p->mem);
        delete p;
        return PLL_E_CUDA;
    }
    p->ctx = context_id();
    *out = p;
    return PLL_OK;
}

PLL_API void pll_mlp_free(pll_mlp *p) {
    if (!p) return;
    if (p->mem) cudaFree(p->mem);
    delete p;
}

PLL_API int pll_mlp_set_params(pll_mlp *p, const float *host_params, void *stream) {
    if (!p || !host_params) return PLL_E_INVAL;
    cudaStream_t s = (cudaStream_t)stream;
    PLL_TRY(cudaMemcpyAsync(p->master, host_params, NP * sizeof(float), cudaMemcpyHostToDevice, s));
    PLL_TRY(cudaMemsetAsync(p->m, 0, 2 * NP * sizeof(float), s));
    k_to_bf16<<<(NP + 255) / 256, 256, 0, s>>>(p->master, p->w16);
    PLL_TRY(cudaGetLastError());
    PLL_TRY(cudaStreamSynchronize(s));
    p->step = 0;
    return PLL_OK;
}

PLL_API int pll_mlp_get_params(const pll_mlp *p, float *host_master, uint16_t *host_bf16) {
    if (!p || (!host_master && !host_bf16)) return PLL_E_INVAL;
    if (host_master) PLL_TRY(cudaMemcpy(host_master, p->master, NP * sizeof(float), cudaMemcpyDeviceToHost));
    if (host_bf16) PLL_TRY(cudaMemcpy(host_bf16, p->w16, NP * 2, cudaMemcpyDeviceToHost));
    return PLL_OK;
}

PLL_API int pll_mlp_forward(const pll_mlp *p, const float *x, uint64_t n, float *y, void *stream) {
    if (!p || (n && (!x || !y))) return PLL_E_INVAL;
    if (n == 0) return PLL_OK;
    cudaStream_t s = (cudaStream_t)stream;
    // two rows a thread where that still fills the GPU (three blocks an SM)
    const bool vec = reinterpret_cast<uintptr_t>(x) % 16 == 0;
    if (n >= (uint64_t)p->wide * FT * 2)
        k_mlp_fwd<2><<<p->wide, FT, 0, s>>>(n, x, vec, p->w16, y);
    else
        k_mlp_fwd<1><<<(unsigned)((n + FT - 1) / FT), FT, 0, s>>>(n, x, vec, p->w16, y);
    PLL_TRY(cudaGetLastError());
    return PLL_OK;
}

PLL_API int pll_mlp_grad(pll_mlp *p, const float *x, const float *target, const uint32_t *idx,
                         uint32_t batch, void *stream) {
    if (!p || !x || !target || batch == 0) return PLL_E_INVAL;
    if (batch > p->max_batch) return PLL_E_RANGE;
    cudaStream_t s = (cudaStream_t)stream;
    const uint32_t blocks = (batch + GT - 1) / GT;
    const bool vec = reinterpret_cast<uintptr_t>(x) % 16 == 0;
    k_mlp_grad<<<blocks, GTH, sizeof(GradSmem), s>>>(batch, x, vec, target, idx, p->w16, p->partial, p->ploss);
    PLL_TRY(cudaGetLastError());
    k_mlp_reduce<<<(NP + 1 + 31) / 32, 256, 0, s>>>(blocks, batch, p->partial, p->ploss, p->grad);
    PLL_TRY(cudaGetLastError());
    return PLL_OK;
}

PLL_API int pll_mlp_read_grad(const pll_mlp *p, float *host_grad, float *host_loss, void *stream) {
    if (!p || (!host_grad && !host_loss)) return PLL_E_INVAL;
    cudaStream_t s = (cudaStream_t)stream;
    // gradient and loss in one copy into pinned memory (two into the caller's
    // pageable arrays are staged ones, a wait each)
    static_assert((NP + 1) * sizeof(float) <= HOST_BLOCK_BYTES, "the gradient fits a host block");
    HostBlock block(s, p->ctx);
    if (!block.p) {
        if (host_grad) PLL_TRY(cudaMemcpyAsync(host_grad, p->grad, NP * sizeof(float), cudaMemcpyDeviceToHost, s));
        if (host_loss) PLL_TRY(cudaMemcpyAsync(host_loss, p->grad + NP, sizeof(float), cudaMemcpyDeviceToHost, s));
        PLL_TRY(cudaStreamSynchronize(s));
        return PLL_OK;
    }
    float *h = block.as<float>();
    const size_t first = host_grad ? 0 : NP, last = host_loss ? NP + 1 : NP;
    PLL_TRY(cudaMemcpyAsync(h + first, p->grad + first, (last - first) * sizeof(float), cudaMemcpyDeviceToHost, s));
    PLL_CHECK(block.wait());
    if (host_grad) std::memcpy(host_grad, h, NP * sizeof(float));
    if (host_loss) *host_loss = h[NP];
    return PLL_OK;
}

PLL_API int pll_mlp_adam(pll_mlp *p, float lr, void *stream) {
    if (!p || !(lr > 0)) return PLL_E_INVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const double b1 = 0.9, b2 = 0.999;
    p->step++;
    const double c1 = 1.0 / (1.0 - std::pow(b1, (double)p->step));
    const double c2 = 1.0 / (1.0 - std::pow(b2, (double)p->step));
    k_adam<<<(NP + 255) / 256, 256, 0, s>>>(p->grad, p->master, p->m, p->v, p->w16, lr, (float)b1,
                                             (float)(1.0 - b1), (float)b2, (float)(1.0 - b2), 1e-8f,
                                             (float)c1, (float)c2);
    PLL_TRY(cudaGetLastError());
    return PLL_OK;
}

PLL_API int pll_mlp_train_step(pll_mlp *p, const float *x, const float *target, const uint32_t *idx,
                               uint32_t batch, float lr, void *stream) {
    PLL_CHECK(pll_mlp_grad(p, x, target, idx, batch, stream));
    return pll_mlp_adam(p, lr, stream);
}

PLL_API int pll_learned_order(const uint32_t *offsets, const uint32_t *cols, uint32_t n, uint64_t nnz,
                              uint32_t t, const pll_mlp *p, uint32_t *order, void *stream) {
    if (!p || (n && !order)) return PLL_E_INVAL;
    if (n == 0) return PLL_OK;
    cudaStream_t s = (cudaStream_t)stream;
    PoolMem m_x(s), m_y(s);
    PLL_CHECK(m_x.alloc((size_t)n * NF * 4));
    PLL_CHECK(m_y.alloc((size_t)n * 4));
    PLL_CHECK(pll_features(offsets, cols, n, nnz, t, stream, m_x.as<float>(), nullptr, nullptr));
    PLL_CHECK(pll_mlp_forward(p, m_x.as<float>(), n, m_y.as<float>(), stream));
    PLL_CHECK(pll_order_from_scores(m_y.as<float>(), n, order, stream));
    PLL_TRY(cudaStreamSynchronize(s));
    return PLL_OK;
}

}  // extern "C"
