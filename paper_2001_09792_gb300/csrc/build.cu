// LBVH construction of the two-level acceleration structure (paper Sec. 1:
// the two-layered structure built from vertices and transformation matrices).
//
// Bottom level, per mesh: triangle boxes and centroid bounds -> Morton codes
// -> stable LSD radix sort -> Karras (HPG 2012) hierarchy -> bottom-up box
// refit with one atomic flag per node (second arriver proceeds).  Top level:
// float64 inverse of each instance transform, Arvo (Graphics Gems 1990) world
// box with directed rounding, then the same LBVH steps over instance boxes.
//
// Every float32 operation that decides a Morton code or a box is an explicit
// round-to-nearest (or directed) intrinsic, so no FMA contraction can change
// a result: codes, order, topology and boxes are reproducible bit for bit.
#include <algorithm>

#include "karras.cuh"
#include "rg_internal.cuh"

namespace rg {

namespace {

constexpr int kBlock = 256;

__device__ __forceinline__ uint32_t spread10(uint32_t x) {
    x &= 0x3FFu;
    x = (x | (x << 16)) & 0x030000FFu;
    x = (x | (x << 8)) & 0x0300F00Fu;
    x = (x | (x << 4)) & 0x030C30C3u;
    x = (x | (x << 2)) & 0x09249249u;
    return x;
}

__device__ __forceinline__ uint64_t spread21(uint64_t x) {
    x &= 0x1FFFFFull;
    x = (x | (x << 32)) & 0x1F00000000FFFFull;
    x = (x | (x << 16)) & 0x1F0000FF0000FFull;
    x = (x | (x << 8)) & 0x100F00F00F00F00Full;
    x = (x | (x << 4)) & 0x10C30C30C30C30C3ull;
    x = (x | (x << 2)) & 0x1249249249249249ull;
    return x;
}

// warp-level min/max of ordered ints, one atomic per warp
__device__ __forceinline__ void reduce_bounds(int* cb_ord, int c0, int c1, int c2, bool valid) {
    int mn[3] = {valid ? c0 : INT_MAX, valid ? c1 : INT_MAX, valid ? c2 : INT_MAX};
    int mx[3] = {valid ? c0 : INT_MIN, valid ? c1 : INT_MIN, valid ? c2 : INT_MIN};
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            mn[a] = min(mn[a], __shfl_xor_sync(0xFFFFFFFFu, mn[a], off));
            mx[a] = max(mx[a], __shfl_xor_sync(0xFFFFFFFFu, mx[a], off));
        }
    }
    if ((threadIdx.x & 31) == 0 && mn[0] != INT_MAX) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            atomicMin(cb_ord + a, mn[a]);
            atomicMax(cb_ord + 3 + a, mx[a]);
        }
    }
}

__device__ __forceinline__ float centroid(float lo, float hi) { return __fmul_rn(__fadd_rn(lo, hi), 0.5f); }

__global__ void k_init_bounds(int* cb_ord) {
    chain_wait();
    int t = threadIdx.x;
    if (t < 3) cb_ord[t] = f2ord(__int_as_float(0x7F800000));        // +inf
    else if (t < 6) cb_ord[t] = f2ord(__int_as_float(0xFF800000));   // -inf
}

// The same, and a BLAS's descriptor (its boxes come later).
__global__ void k_blas_begin(int* cb_ord, BlasDev* out, BlasDev desc) {
    chain_wait();
    const int t = threadIdx.x;
    if (t < 3) cb_ord[t] = f2ord(__int_as_float(0x7F800000));
    else if (t < 6) cb_ord[t] = f2ord(__int_as_float(0xFF800000));
    else if (t == 6) *out = desc;
}

__global__ void k_tri_bounds(const float* __restrict__ vtx, uint32_t nv, const uint32_t* __restrict__ idx,
                             uint32_t nt, float* __restrict__ lohi, int* cb_ord, DevStatus* st,
                             uint32_t* __restrict__ flags) {
    chain_wait();
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    bool valid = i < nt;
    int c[3] = {0, 0, 0};
    if (flags && i + 1 < nt) flags[i] = 0u;
    if (valid) {
        uint32_t a = idx[3 * (size_t)i], b = idx[3 * (size_t)i + 1], cc = idx[3 * (size_t)i + 2];
        if (a >= nv || b >= nv || cc >= nv) {
            record_error(st, RG_ERR_INVALID_ARG);
            a = b = cc = 0;
        }
        float lo[3], hi[3];
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            float x0 = vtx[3 * (size_t)a + ax], x1 = vtx[3 * (size_t)b + ax], x2 = vtx[3 * (size_t)cc + ax];
            lo[ax] = fminf(fminf(x0, x1), x2);
            hi[ax] = fmaxf(fmaxf(x0, x1), x2);
            lohi[6 * (size_t)i + ax] = lo[ax];
            lohi[6 * (size_t)i + 3 + ax] = hi[ax];
            c[ax] = f2ord(centroid(lo[ax], hi[ax]));
        }
    }
    if (cb_ord) reduce_bounds(cb_ord, c[0], c[1], c[2], valid);
}

__global__ void k_centroid_bounds(const float* __restrict__ lohi, uint32_t n, int* cb_ord) {
    chain_wait();
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    bool valid = i < n;
    int c[3] = {0, 0, 0};
    if (valid) {
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) c[ax] = f2ord(centroid(lohi[6 * (size_t)i + ax], lohi[6 * (size_t)i + 3 + ax]));
    }
    reduce_bounds(cb_ord, c[0], c[1], c[2], valid);
}

// Morton quantisation on one cubic grid over the centroid box: a single scale
// for all axes, so a flat mesh keeps its thin axis thin instead of being
// split across it first.
struct MortonGrid {
    float cmin[3], cmax[3], scale;
};

__device__ __forceinline__ MortonGrid morton_grid(const int* cb_ord, int bits) {
    MortonGrid g;
    const float full = (float)(1u << bits);
    float ext = 0.0f;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        g.cmin[ax] = ord2f(cb_ord[ax]);
        g.cmax[ax] = ord2f(cb_ord[3 + ax]);
        if (g.cmax[ax] > g.cmin[ax]) ext = fmaxf(ext, __fsub_rn(g.cmax[ax], g.cmin[ax]));
    }
    g.scale = ext > 0.0f ? __fdiv_rn(full, ext) : 0.0f;
    return g;
}

// Quantised centroid of box b (lo.xyz, hi.xyz).
template <int BITS>
__device__ __forceinline__ void morton_q(const MortonGrid& g, const float* b, uint32_t* q) {
    const float qmax = (float)((1u << BITS) - 1u);
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        if (!(g.cmax[ax] > g.cmin[ax])) {
            q[ax] = 0;
            continue;
        }
        float c = centroid(b[ax], b[3 + ax]);
        float f = floorf(__fmul_rn(__fsub_rn(c, g.cmin[ax]), g.scale));
        f = fminf(fmaxf(f, 0.0f), qmax);
        q[ax] = (uint32_t)f;
    }
}

__device__ __forceinline__ uint32_t morton30(const MortonGrid& g, const float* b) {
    uint32_t q[3];
    morton_q<10>(g, b, q);
    return (spread10(q[0]) << 2) | (spread10(q[1]) << 1) | spread10(q[2]);
}

template <int BITS>
__global__ void k_morton(const float* __restrict__ lohi, uint32_t n, const int* __restrict__ cb_ord,
                         void* __restrict__ codes, float* cb_out) {
    chain_wait();
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    const MortonGrid g = morton_grid(cb_ord, BITS);
    if (cb_out && i == 0) {
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            cb_out[ax] = g.cmin[ax];
            cb_out[3 + ax] = g.cmax[ax];
        }
    }
    if (i >= n) return;
    if (BITS == 10) {
        static_cast<uint32_t*>(codes)[i] = morton30(g, lohi + 6 * (size_t)i);
    } else {
        uint32_t q[3];
        morton_q<21>(g, lohi + 6 * (size_t)i, q);
        static_cast<uint64_t*>(codes)[i] = (spread21(q[0]) << 2) | (spread21(q[1]) << 1) | spread21(q[2]);
    }
}

// ---------------------------------------------------------------- radix sort
// Stable LSD radix sort, 8-bit digits.  One read of the keys counts every
// pass's digits (k_rs_hist); each pass is then one kernel (k_rs_pass): a tile
// ranks its pairs in shared memory, publishes its digit counts, adds up the
// counts of the tiles before it as they appear (decoupled look-back, Merrill &
// Garland 2016, in the one-pass-per-digit form of Adinets & Merrill 2022) and
// writes its pairs grouped by digit, so that the stores are runs.  Bound by
// memory (12 B read and written per pair and pass) where the launch is large;
// a million pairs are 245 tiles on 152 SMs and bound by each tile's chain of ranks
// and look-backs (17.7 us a pass alone, 33 % of the issue slots, 6 % of the
// DRAM rate, 12.6 warps an SM).  1,000,003 pairs of 32-bit keys: 67.6 us,
// 324.9 us with a count, a one-block scan (50 us a pass) and a scatter per
// pass.
//
// The look-back waits on nothing: a tile takes its number from a counter, so
// the tiles before it have started, and a count that has not appeared after
// kSpinMax reads is recounted from the pass's input, which no tile writes.
constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSpinMax = 1 << 14;
constexpr uint32_t kLook = 8, kSortLargeTiles = 200;
// Items per thread: 8 (tiles of kSortTilePairs), or 16 from kSortLargeTiles tiles
// of those on, 1.3 an SM of 152: with a tile and more on every SM the shorter
// chain of look-backs outweighs the longer tile.  us with 8 and 16: 1,000,003 pairs 78.7
// and 67.5 (64-bit keys 149.5, 131.9), 16M 654 and 605, 819,200 67.7 and 63.9; but
// 311,297 41.9 and 45.4, and with 64-bit keys 100,001 60.4 and 75.7, 311,297 72.1
// and 84.5.  Between 450,001 (50.2, 46.5) and the line 16 would be 4 to 8 % faster.
constexpr int kSortItems = (int)kSortTilePairs / kSortThreads;

// Ranks of a warp's ITEMS x 32 digits among its own: cnt (256 entries, this
// warp's) ends as the warp's digit counts; rank[j] counts the warp's equal
// digits before (j, lane) in that order.
template <int ITEMS, class K, class C>
__device__ __forceinline__ void rank_digits(const K (&key)[ITEMS], int shift, C* cnt, uint32_t (&rank)[ITEMS]) {
    const uint32_t lane = threadIdx.x & 31u, lt = (1u << lane) - 1u;
    for (uint32_t i = lane; i < 256u; i += 32u) cnt[i] = 0;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint32_t d = (uint32_t)(key[j] >> shift) & 0xFFu;
        uint32_t peers = 0xFFFFFFFFu;
#pragma unroll
        for (int bit = 0; bit < 8; ++bit) {
            const uint32_t bal = __ballot_sync(0xFFFFFFFFu, (d >> bit) & 1u);
            peers &= ((d >> bit) & 1u) ? bal : ~bal;
        }
        const uint32_t before = cnt[d];
        rank[j] = before + __popc(peers & lt);
        __syncwarp();
        if ((peers & lt) == 0) cnt[d] = (C)(before + __popc(peers));
        __syncwarp();
    }
}

// Exclusive prefix over the first 256 threads of the block (all threads call).
__device__ __forceinline__ uint32_t scan256(uint32_t v, uint32_t* wsum) {
    const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, off);
        if ((int)lane >= off) inc += y;
    }
    if (lane == 31 && warp < 8) wsum[warp] = inc;
    __syncthreads();
    uint32_t before = 0;
    for (uint32_t w = 0; w < 8; ++w)
        if (w < warp) before += wsum[w];
    __syncthreads();
    return before + inc - v;
}

// Digit counts of every pass in one read of the keys; hist: 256 per pass, zeroed.
template <class K>
__global__ void __launch_bounds__(kSortThreads) k_rs_hist(const K* __restrict__ keys, uint32_t n,
                                                           uint32_t* __restrict__ hist) {
    chain_wait();
    constexpr int P = (int)sizeof(K);
    __shared__ uint32_t cnt[P][256];
#pragma unroll
    for (int q = 0; q < P; ++q) cnt[q][threadIdx.x] = 0;
    __syncthreads();
    const size_t step = (size_t)gridDim.x * kSortThreads;
#pragma unroll 4
    for (size_t i = (size_t)blockIdx.x * kSortThreads + threadIdx.x; i < n; i += step) {
        const K k = keys[i];
#pragma unroll
        for (int q = 0; q < P; ++q) atomicAdd(&cnt[q][(uint32_t)(k >> (8 * q)) & 0xFFu], 1u);
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < P; ++q)
        if (cnt[q][threadIdx.x]) atomicAdd(hist + 256 * q + threadIdx.x, cnt[q][threadIdx.x]);
}

// One pass.  status: per tile and digit a count with two flag bits on top (0:
// none yet, 1: the tile's own, 2: with all tiles before it); W holds counts
// below 2^30 in 32 bits.  next: the other pass's status, cleared here for the
// pass that follows.
template <class K, class W, int ITEMS>
__global__ void __launch_bounds__(kSortThreads) k_rs_pass(const K* __restrict__ keys, const uint32_t* __restrict__ vals,
                                                           uint32_t n, int shift, const uint32_t* __restrict__ hist,
                                                           W* status, W* __restrict__ next, uint32_t* ticket,
                                                           K* __restrict__ keys_out, uint32_t* __restrict__ vals_out) {
    chain_wait();
    constexpr int kTile = kSortThreads * ITEMS;
    constexpr int kFlag = (int)sizeof(W) * 8 - 2;
    constexpr W kOwn = W(1) << kFlag, kAll = W(2) << kFlag, kCount = kOwn - 1;
    __shared__ uint32_t s_cnt[kSortWarps][256];
    __shared__ K s_pair[kTile];  // the keys in digit order, then the values
    __shared__ uint32_t s_off[256], s_dst[256], s_wsum[8], s_tile;
    const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
    if (t == 0) s_tile = atomicAdd(ticket, 1u);
    __syncthreads();
    const uint32_t tile = s_tile;
    const size_t base = (size_t)tile * kTile;
    const uint32_t m = (uint32_t)min((size_t)kTile, (size_t)n - base);
    K key[ITEMS];
    uint32_t val[ITEMS], rank[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {  // past the end: the largest key, which stays last
        const uint32_t p = warp * (32u * ITEMS) + 32u * j + lane;
        key[j] = p < m ? keys[base + p] : ~K(0);
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint32_t p = warp * (32u * ITEMS) + 32u * j + lane;
        val[j] = p < m ? (vals ? vals[base + p] : (uint32_t)(base + p)) : 0u;
    }
    rank_digits<ITEMS>(key, shift, s_cnt[warp], rank);
    __syncthreads();
    uint32_t total = 0;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) {
        const uint32_t c = s_cnt[w][t];
        s_cnt[w][t] = total;
        total += c;
    }
    W* mine = status + (size_t)tile * 256 + t;
    *reinterpret_cast<volatile W*>(mine) = (tile == 0 ? kAll : kOwn) | (W)total;
    if (next) next[(size_t)tile * 256 + t] = 0;
    const uint32_t off = scan256(total, s_wsum);
    const uint32_t first = scan256(hist[t], s_wsum);  // the digit's place over all tiles
    // the pairs of this digit in the tiles before
    // (kLook tiles are read at a time, for the chain of reads is what a pass waits
    // on: before the launches were chained 1,000,003 pairs took 95.6 us with one at a
    // time, 88.9 with 8, and 78.7 with 8 and the larger tiles, 86.0 and 98.4 with 16
    // and 32)
    uint32_t before = 0;
    for (uint32_t q = tile;; q -= kLook) {
        W v[kLook];
#pragma unroll
        for (uint32_t k = 0; k < kLook; ++k)
            v[k] = q > k ? *reinterpret_cast<const volatile W*>(status + (size_t)(q - 1 - k) * 256 + t) : kAll;
        bool done = false;
#pragma unroll
        for (uint32_t k = 0; k < kLook; ++k) {
            if (done) continue;
            if (!(v[k] >> kFlag)) {
                const size_t p = q - 1 - k;
                for (int spin = 0; !(v[k] >> kFlag) && spin < kSpinMax; ++spin)
                    v[k] = *reinterpret_cast<const volatile W*>(status + p * 256 + t);
                if (!(v[k] >> kFlag)) {
                    uint32_t c = 0;
                    for (uint32_t i = 0; i < (uint32_t)kTile; ++i)
                        c += ((uint32_t)(keys[p * kTile + i] >> shift) & 0xFFu) == t;
                    v[k] = kOwn | (W)c;
                }
            }
            before += (uint32_t)(v[k] & kCount);
            done = (v[k] & kAll) != 0;
        }
        if (done) break;
    }
    if (tile) *reinterpret_cast<volatile W*>(mine) = kAll | (W)(before + total);
    s_off[t] = off;
    s_dst[t] = first + before - off;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint32_t d = (uint32_t)(key[j] >> shift) & 0xFFu;
        rank[j] += s_off[d] + s_cnt[warp][d];
        s_pair[rank[j]] = key[j];
    }
    __syncthreads();
    uint32_t dst[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint32_t p = j * kSortThreads + t;
        dst[j] = n;
        if (p < m) {
            const K k = s_pair[p];
            dst[j] = s_dst[(uint32_t)(k >> shift) & 0xFFu] + p;
            if (dst[j] < n) keys_out[dst[j]] = k;
        }
    }
    __syncthreads();
    uint32_t* s_val = reinterpret_cast<uint32_t*>(s_pair);
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) s_val[rank[j]] = val[j];
    __syncthreads();
#pragma unroll
    for (int j = 0; j < ITEMS; ++j)
        if (dst[j] < n) vals_out[dst[j]] = s_val[j * kSortThreads + t];
}

// All passes of up to kSortOneMax pairs in one block, the pairs in registers
// between the passes: one launch where the tiles would take six.
constexpr int kSortOneThreads = 512, kSortOneItems = 8;
constexpr uint32_t kSortOneMax = kSortOneThreads * kSortOneItems;
template <class K>
__global__ void __launch_bounds__(kSortOneThreads) k_rs_one(const K* keys, const uint32_t* vals, uint32_t n,
                                                             K* keys_out, uint32_t* vals_out) {
    chain_wait();
    constexpr int ITEMS = kSortOneItems, kW = kSortOneThreads / 32;
    __shared__ uint16_t s_cnt[kW][256];
    __shared__ K s_pair[kSortOneMax];
    __shared__ uint32_t s_off[256], s_wsum[8];
    uint32_t* s_val = reinterpret_cast<uint32_t*>(s_pair);
    const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
    K key[ITEMS];
    uint32_t val[ITEMS], rank[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint32_t p = warp * (32u * ITEMS) + 32u * j + lane;
        key[j] = p < n ? keys[p] : ~K(0);
        val[j] = p < n ? (vals ? vals[p] : p) : 0u;
    }
    for (int shift = 0; shift < (int)sizeof(K) * 8; shift += 8) {
        rank_digits<ITEMS>(key, shift, s_cnt[warp], rank);
        __syncthreads();
        uint32_t total = 0;
        if (t < 256) {
#pragma unroll
            for (int w = 0; w < kW; ++w) {
                const uint32_t c = s_cnt[w][t];
                s_cnt[w][t] = (uint16_t)total;
                total += c;
            }
        }
        const uint32_t off = scan256(total, s_wsum);
        if (t < 256) s_off[t] = off;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const uint32_t d = (uint32_t)(key[j] >> shift) & 0xFFu;
            rank[j] += s_off[d] + s_cnt[warp][d];
            s_pair[rank[j]] = key[j];
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) key[j] = s_pair[warp * (32u * ITEMS) + 32u * j + lane];
        __syncthreads();
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) s_val[rank[j]] = val[j];
        __syncthreads();
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) val[j] = s_val[warp * (32u * ITEMS) + 32u * j + lane];
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint32_t p = warp * (32u * ITEMS) + 32u * j + lane;
        if (p < n) {
            keys_out[p] = key[j];
            vals_out[p] = val[j];
        }
    }
}

// ---------------------------------------------------------------- Karras
// (delta, karras_node: karras.cuh)

// One thread per internal node of all segments: the segment by binary search
// over the segments' first thread numbers.
template <class K>
__global__ void k_karras_segments(const K* __restrict__ keys, const KarrasSeg* __restrict__ segs, uint32_t n_segs,
                                  uint32_t n_threads, uint32_t n_leaves, uint32_t* __restrict__ child_base,
                                  uint32_t* __restrict__ parents, uint32_t* __restrict__ ranges) {
    chain_wait();
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n_threads) return;
    uint32_t lo = 0, hi = n_segs - 1;
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) / 2;
        if (segs[mid].first <= g)
            lo = mid;
        else
            hi = mid - 1;
    }
    const KarrasSeg S = segs[lo];
    karras_node(keys + S.begin, S.count, (int64_t)(g - S.first), child_base, 16, parents, ranges, S.node, S.begin,
                n_leaves);
}

template <class K>
__global__ void k_karras(const K* __restrict__ keys, uint32_t n, uint32_t* __restrict__ child_base, int stride,
                         uint32_t* __restrict__ parents, uint32_t* __restrict__ ranges) {
    chain_wait();
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)n - 1) return;
    karras_node(keys, n, i, child_base, stride, parents, ranges);
}

// ---------------------------------------------------------------- refit
// Write one child box into slot `side` of node p (see the node layout).
__device__ __forceinline__ void store_slot(float4* nodes, uint32_t p, int side, const float* b) {
    float* f = reinterpret_cast<float*>(nodes + 4 * (size_t)p);
    if (side == 0) {
        *reinterpret_cast<float4*>(f) = make_float4(b[0], b[1], b[2], b[3]);
        *reinterpret_cast<float2*>(f + 4) = make_float2(b[4], b[5]);
    } else {
        *reinterpret_cast<float2*>(f + 6) = make_float2(b[0], b[1]);
        *reinterpret_cast<float4*>(f + 8) = make_float4(b[2], b[3], b[4], b[5]);
    }
}
__device__ __forceinline__ void load_slot_cg(const float4* nodes, uint32_t p, int side, float* b) {
    const float* f = reinterpret_cast<const float*>(nodes + 4 * (size_t)p);
    if (side == 0) {
        float4 x = __ldcg(reinterpret_cast<const float4*>(f));
        float2 y = __ldcg(reinterpret_cast<const float2*>(f + 4));
        b[0] = x.x; b[1] = x.y; b[2] = x.z; b[3] = x.w; b[4] = y.x; b[5] = y.y;
    } else {
        float2 x = __ldcg(reinterpret_cast<const float2*>(f + 6));
        float4 y = __ldcg(reinterpret_cast<const float4*>(f + 8));
        b[0] = x.x; b[1] = x.y; b[2] = y.x; b[3] = y.y; b[4] = y.z; b[5] = y.w;
    }
}

// Climb from leaf j to the root; the second thread to reach a node unions its
// two child boxes and continues.  Writes the root box to root_box (6 floats).
__device__ void climb(uint32_t j, uint32_t n, float* box, const uint32_t* __restrict__ parents, float4* nodes,
                      uint32_t* flags, float* root_box, DevStatus* st) {
    if (n == 1) {
        for (int a = 0; a < 6; ++a) root_box[a] = box[a];
        return;
    }
    uint32_t cur = kLeaf | j;
    uint32_t p = parents[(size_t)(n - 1) + j];
    for (uint32_t step = 0; step < n; ++step) {
        const uint32_t* n3 = reinterpret_cast<const uint32_t*>(nodes + 4 * (size_t)p + 3);
        int side = (n3[0] == cur) ? 0 : 1;
        store_slot(nodes, p, side, box);
        __threadfence();
        uint32_t old = atomicAdd(flags + p, 1u);
        if (old == 0) return;
        __threadfence();
        float other[6];
        load_slot_cg(nodes, p, 1 - side, other);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            box[a] = fminf(box[a], other[a]);
            box[3 + a] = fmaxf(box[3 + a], other[3 + a]);
        }
        if (p == 0) {
            for (int a = 0; a < 6; ++a) root_box[a] = box[a];
            return;
        }
        cur = p;
        p = parents[p];
    }
    record_error(st, RG_ERR_TIMEOUT);
}

__global__ void k_blas_leaves_refit(const float* __restrict__ vtx, uint32_t nv, const uint32_t* __restrict__ idx,
                                    const uint32_t* __restrict__ perm, const float* __restrict__ lohi, uint32_t n,
                                    const uint32_t* __restrict__ parents, float4* nodes, uint32_t* flags,
                                    float4* __restrict__ tris, uint32_t* __restrict__ leaf_of_prim, BlasDev* blas_out,
                                    DevStatus* st, const uint32_t* __restrict__ boxes_done) {
    chain_wait();
    uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    uint32_t prim = perm[j];
    leaf_of_prim[prim] = j;
    uint32_t vi[3] = {idx[3 * (size_t)prim], idx[3 * (size_t)prim + 1], idx[3 * (size_t)prim + 2]};
    // (a bad index was reported by k_tri_bounds, which boxed vertex 0 in its place)
    if (vi[0] >= nv || vi[1] >= nv || vi[2] >= nv) vi[0] = vi[1] = vi[2] = 0u;
    // the triangle record: its vertices in the axis orders (x, y, z), (y, z, x)
    // and (z, x, y), prim in the first vertex's w of each
    float4* t = tris + 9 * (size_t)j;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        float x = vtx[3 * (size_t)vi[c]], y = vtx[3 * (size_t)vi[c] + 1], z = vtx[3 * (size_t)vi[c] + 2];
        const float w = c == 0 ? __uint_as_float(prim) : 0.0f;
        t[c] = make_float4(x, y, z, w);
        t[3 + c] = make_float4(y, z, x, w);
        t[6 + c] = make_float4(z, x, y, w);
    }
    if (boxes_done && *boxes_done) {  // the build wrote every node's boxes
        if (j == 0) {
            const float* f = reinterpret_cast<const float*>(nodes);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                blas_out->lo[a] = fminf(f[a], f[6 + a]);
                blas_out->hi[a] = fmaxf(f[3 + a], f[9 + a]);
            }
        }
        return;
    }
    float box[6];
#pragma unroll
    for (int a = 0; a < 6; ++a) box[a] = lohi[6 * (size_t)prim + a];
    climb(j, n, box, parents, nodes, flags, blas_out->lo, st);
}

// check_blas: a refit; the BLAS id of instance k must equal the one stored in
// tmp[k] by the build (read before tmp[k] is overwritten by the same thread).
// Bounding sphere: the largest upward-rounded squared distance of a vertex
// from the root box centre, reduced per warp, one atomicMax per warp.
__global__ void k_bound_sphere(const float* __restrict__ vtx, uint32_t nv, BlasDev* blas) {
    chain_wait();
    float c[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) c[q] = __fmul_rn(__fadd_rn(blas->lo[q], blas->hi[q]), 0.5f);
    uint32_t best = 0;  // bits of a non-negative float: integer order = float order
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < nv; v += gridDim.x * blockDim.x) {
        float e[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const float x = vtx[3 * (size_t)v + q];
            e[q] = x >= c[q] ? __fsub_ru(x, c[q]) : __fsub_ru(c[q], x);
        }
        const float d2 = __fadd_ru(__fadd_ru(__fmul_ru(e[0], e[0]), __fmul_ru(e[1], e[1])), __fmul_ru(e[2], e[2]));
        best = max(best, __float_as_uint(d2));
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) best = max(best, __shfl_xor_sync(0xFFFFFFFFu, best, off));
    if ((threadIdx.x & 31) == 0 && best) atomicMax(&blas->r2_bits, best);
}

// Instance k: float64 inverse, InstDev record into tmp[k], world box into
// wbox[k]; c receives the box centroid as ordered ints.
__device__ __forceinline__ void instance_prep_one(const rg_instance* __restrict__ in, uint32_t k,
                                                  const BlasDev* __restrict__ blas, uint32_t nblas, InstDev* tmp,
                                                  float* __restrict__ wbox, bool check_blas, DevStatus* st, int* c) {
    {
        const rg_instance& I = in[k];
        float m[12];
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q) m[4 * r + q] = I.m[r][q];
        uint32_t b = I.blas_id;
        if (b >= nblas || (check_blas && tmp[k].blas != b)) {
            record_error(st, RG_ERR_INVALID_ARG);
            b = 0;
        }
        const BlasDev B = blas[b];
        // float64 inverse of A = m[0..2 | 4..6 | 8..10]: adjugate / det
        double a0 = m[0], a1 = m[1], a2 = m[2], a3 = m[4], a4 = m[5], a5 = m[6], a6 = m[8], a7 = m[9], a8 = m[10];
        double c00 = a4 * a8 - a5 * a7, c01 = -(a3 * a8 - a5 * a6), c02 = a3 * a7 - a4 * a6;
        double det = a0 * c00 + a1 * c01 + a2 * c02;
        double inv[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
        if (det == 0.0 || !isfinite(det)) {
            record_error(st, RG_ERR_SINGULAR);
        } else {
            double id = 1.0 / det;
            inv[0] = c00 * id;
            inv[1] = -(a1 * a8 - a2 * a7) * id;
            inv[2] = (a1 * a5 - a2 * a4) * id;
            inv[3] = c01 * id;
            inv[4] = (a0 * a8 - a2 * a6) * id;
            inv[5] = -(a0 * a5 - a2 * a3) * id;
            inv[6] = c02 * id;
            inv[7] = -(a0 * a7 - a1 * a6) * id;
            inv[8] = (a0 * a4 - a1 * a3) * id;
        }
        InstDev D;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            double tr = -(inv[3 * r] * (double)m[3] + inv[3 * r + 1] * (double)m[7] + inv[3 * r + 2] * (double)m[11]);
            D.inv[r] = make_float4(__double2float_rn(inv[3 * r]), __double2float_rn(inv[3 * r + 1]),
                                   __double2float_rn(inv[3 * r + 2]), __double2float_rn(tr));
            D.m[r] = make_float4(m[4 * r], m[4 * r + 1], m[4 * r + 2], m[4 * r + 3]);
        }
        D.nodes = B.nodes;
        D.tris = B.tris;
        D.root = B.root;
        D.id = k;
        D.material = I.material_id;
        D.blas = b;
        tmp[k] = D;
        // Arvo box of the BLAS root box, outward rounded
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            float lo = 0.f, hi = 0.f;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                float mn = fminf(__fmul_rd(m[4 * r + q], B.lo[q]), __fmul_rd(m[4 * r + q], B.hi[q]));
                float mx = fmaxf(__fmul_ru(m[4 * r + q], B.lo[q]), __fmul_ru(m[4 * r + q], B.hi[q]));
                lo = q == 0 ? mn : __fadd_rd(lo, mn);
                hi = q == 0 ? mx : __fadd_ru(hi, mx);
            }
            lo = __fadd_rd(lo, m[4 * r + 3]);
            hi = __fadd_ru(hi, m[4 * r + 3]);
            // intersect with the box of the transformed bounding sphere:
            // A c + t -/+ r |row_r(A)|, outward rounded (a rotation leaves a
            // sphere's box unchanged, where it inflates the Arvo box)
            const float* row = m + 4 * r;
            float cx[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) cx[q] = __fmul_rn(__fadd_rn(B.lo[q], B.hi[q]), 0.5f);
            float cl = __fadd_rd(__fadd_rd(__fadd_rd(__fmul_rd(row[0], cx[0]), __fmul_rd(row[1], cx[1])),
                                           __fmul_rd(row[2], cx[2])), row[3]);
            float ch = __fadd_ru(__fadd_ru(__fadd_ru(__fmul_ru(row[0], cx[0]), __fmul_ru(row[1], cx[1])),
                                           __fmul_ru(row[2], cx[2])), row[3]);
            const float norm = __fsqrt_ru(__fadd_ru(__fadd_ru(__fmul_ru(row[0], row[0]), __fmul_ru(row[1], row[1])),
                                                    __fmul_ru(row[2], row[2])));
            const float R = __fmul_ru(__fsqrt_ru(__uint_as_float(B.r2_bits)), norm);
            lo = fmaxf(lo, __fsub_rd(cl, R));
            hi = fminf(hi, __fadd_ru(ch, R));
            wbox[6 * (size_t)k + r] = lo;
            wbox[6 * (size_t)k + 3 + r] = hi;
            c[r] = f2ord(centroid(lo, hi));
        }
    }
}

__global__ void k_instance_prep(const rg_instance* __restrict__ in, uint32_t n, const BlasDev* __restrict__ blas,
                                uint32_t nblas, InstDev* tmp, float* __restrict__ wbox, int* cb_ord, bool check_blas,
                                uint32_t* __restrict__ flags, DevStatus* st) {
    chain_wait();
    uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    bool valid = k < n;
    int c[3] = {0, 0, 0};
    if (k + 1 < n) flags[k] = 0u;
    if (valid) instance_prep_one(in, k, blas, nblas, tmp, wbox, check_blas, st, c);
    if (cb_ord) reduce_bounds(cb_ord, c[0], c[1], c[2], valid);
}

__global__ void k_tlas_leaves_refit(const InstDev* __restrict__ tmp, const float* __restrict__ wbox,
                                    const uint32_t* __restrict__ perm, uint32_t n, const uint32_t* __restrict__ parents,
                                    float4* nodes, uint32_t* flags, InstDev* __restrict__ inst_out,
                                    uint32_t* __restrict__ leaf_of_inst, DevStatus* st,
                                    const uint32_t* __restrict__ boxes_done) {
    chain_wait();
    uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    uint32_t k = perm[j];
    inst_out[j] = tmp[k];
    if (leaf_of_inst) leaf_of_inst[k] = j;
    if (boxes_done && *boxes_done) return;
    float box[6];
#pragma unroll
    for (int a = 0; a < 6; ++a) box[a] = wbox[6 * (size_t)k + a];
    float root_box[6];
    climb(j, n, box, parents, nodes, flags, root_box, st);
}

// The whole TLAS build (or refit) of up to kTlasSmallMax instances in one
// block, thread k = instance k: instance prep, centroid bounds, Morton codes,
// a stable sort, the Karras hierarchy and the bottom-up box refit.  Same
// per-element code and the same results as the multi-kernel path; a small
// TLAS is otherwise bound by the issue of its 17 launches.  The sort is an
// LSD sort by single bits (30 stable splits, each a block-wide prefix count
// of zeros), which starting from instance order gives the (key, index) order.
__global__ void __launch_bounds__(kTlasSmallMax) k_tlas_small(const rg_instance* __restrict__ in, uint32_t n,
                                                              const BlasDev* __restrict__ blas, uint32_t nblas,
                                                              InstDev* tmp, float* wbox, bool refit, float4* nodes,
                                                              uint32_t* perm, uint32_t* parents, uint32_t* flags,
                                                              uint32_t* ranges, InstDev* inst_out,
                                                              uint32_t* leaf_of_inst, DevStatus* st) {
    chain_wait();
    __shared__ int s_cb[6];
    __shared__ uint32_t s_key[kTlasSmallMax], s_val[kTlasSmallMax];
    __shared__ uint32_t s_warp[32], s_total;
    const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
    const uint32_t n_warps = blockDim.x >> 5;
    const bool valid = t < n;
    if (t < 3) s_cb[t] = f2ord(__int_as_float(0x7F800000));
    else if (t < 6) s_cb[t] = f2ord(__int_as_float(0xFF800000));
    __syncthreads();
    int c[3] = {INT_MAX, INT_MAX, INT_MAX};
    if (valid) instance_prep_one(in, t, blas, nblas, tmp, wbox, refit, st, c);
    if (!refit) {
        int mn[3] = {c[0], c[1], c[2]}, mx[3] = {valid ? c[0] : INT_MIN, valid ? c[1] : INT_MIN, valid ? c[2] : INT_MIN};
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                mn[a] = min(mn[a], __shfl_xor_sync(0xFFFFFFFFu, mn[a], off));
                mx[a] = max(mx[a], __shfl_xor_sync(0xFFFFFFFFu, mx[a], off));
            }
        if (lane == 0 && mn[0] != INT_MAX)
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                atomicMin(s_cb + a, mn[a]);
                atomicMax(s_cb + 3 + a, mx[a]);
            }
        __syncthreads();
        const MortonGrid g = morton_grid(s_cb, 10);
        if (valid) {
            float b[6];
#pragma unroll
            for (int a = 0; a < 6; ++a) b[a] = wbox[6 * (size_t)t + a];
            s_key[t] = morton30(g, b);
            s_val[t] = t;
        }
        // stable LSD sort by single bits
        for (int bit = 0; bit < 30; ++bit) {
            __syncthreads();
            const uint32_t k = valid ? s_key[t] : 0u, v = valid ? s_val[t] : 0u;
            const bool zero = valid && !((k >> bit) & 1u);
            const uint32_t zb = __ballot_sync(0xFFFFFFFFu, zero);
            if (lane == 0) s_warp[warp] = __popc(zb);
            __syncthreads();
            if (warp == 0) {
                const uint32_t x = lane < n_warps ? s_warp[lane] : 0u;
                uint32_t inc = x;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, off);
                    if ((int)lane >= off) inc += y;
                }
                if (lane < n_warps) s_warp[lane] = inc - x;
                if (lane == 31) s_total = inc;
            }
            __syncthreads();
            // (every read of s_key in this pass came before the barrier above)
            const uint32_t zeros_before = s_warp[warp] + __popc(zb & ((1u << lane) - 1u));
            const uint32_t pos = zero ? zeros_before : s_total + (t - zeros_before);
            if (valid) {
                s_key[pos] = k;
                s_val[pos] = v;
            }
        }
        __syncthreads();
        if (valid) perm[t] = s_val[t];
        if (t + 1 < n) karras_node(s_key, n, t, reinterpret_cast<uint32_t*>(nodes) + 12, 16, parents, ranges);
    }
    if (t + 1 < n) flags[t] = 0;
    __syncthreads();
    __threadfence();
    if (valid) {
        const uint32_t k = perm[t];
        inst_out[t] = tmp[k];
        leaf_of_inst[k] = t;
        float box[6];
#pragma unroll
        for (int a = 0; a < 6; ++a) box[a] = wbox[6 * (size_t)k + a];
        float root_box[6];
        climb(t, n, box, parents, nodes, flags, root_box, st);
    }
}

inline unsigned grid_for(size_t n, int block = kBlock) { return (unsigned)((n + block - 1) / block); }

}  // namespace

cudaError_t launch_init_bounds(int* cb_ord, cudaStream_t s) {
    launch_chain(k_init_bounds, 1, 32, 0, s, cb_ord);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_blas_begin(int* cb_ord, BlasDev* out, const BlasDev& desc, cudaStream_t s) {
    launch_chain(k_blas_begin, 1, 32, 0, s, cb_ord, out, desc);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_tri_bounds(const float* vtx, uint32_t nv, const uint32_t* idx, uint32_t nt, float* lohi,
                              int* cb_ord, DevStatus* st, cudaStream_t s, uint32_t* flags) {
    if (nt == 0) return cudaSuccess;
    launch_chain(k_tri_bounds, grid_for(nt), kBlock, 0, s, vtx, nv, idx, nt, lohi, cb_ord, st, flags);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_centroid_bounds(const float* lohi, uint32_t n, int* cb_ord, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    launch_chain(k_centroid_bounds, grid_for(n), kBlock, 0, s, lohi, n, cb_ord);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_morton(const float* lohi, uint32_t n, const int* cb_ord, int bits, void* codes, float* cb_out,
                          cudaStream_t s) {
    unsigned g = grid_for(n > 0 ? n : 1);
    if (bits == 10)
        launch_chain(k_morton<10>, g, kBlock, 0, s, lohi, n, cb_ord, codes, cb_out);
    else
        launch_chain(k_morton<21>, g, kBlock, 0, s, lohi, n, cb_ord, codes, cb_out);
    count_launches(1);
    return cudaGetLastError();
}

template <class K, class W>
static cudaError_t radix_sort_impl(const K* keys_in, const uint32_t* vals_in, uint32_t n, K* keys_out,
                                   uint32_t* vals_out, void* scratch, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    if (n <= kSortOneMax) {
        launch_chain(k_rs_one<K>, 1, kSortOneThreads, 0, s, keys_in, vals_in, n, keys_out, vals_out);
        count_launches(1);
        return cudaGetLastError();
    }
    constexpr int passes = (int)sizeof(K);
    const bool large = n / (2 * kSortTilePairs) >= kSortLargeTiles;
    const uint32_t tile = large ? 2 * kSortTilePairs : kSortTilePairs;
    const uint32_t nb = (uint32_t)(((size_t)n + tile - 1) / tile);
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    char* p = static_cast<char*>(scratch);
    K* kt = reinterpret_cast<K*>(p);
    p += al((size_t)n * sizeof(K));
    uint32_t* vt = reinterpret_cast<uint32_t*>(p);
    p += al((size_t)n * 4);
    uint32_t* hist = reinterpret_cast<uint32_t*>(p);  // 256 per pass, then a tile counter per pass
    uint32_t* ticket = hist + 256 * 8;
    W* status[2];
    status[0] = reinterpret_cast<W*>(ticket + 64);
    status[1] = status[0] + (size_t)256 * nb;
    cudaError_t e = cudaMemsetAsync(hist, 0, (256 * 8 + 64) * 4 + (size_t)256 * nb * sizeof(W), s);
    if (e != cudaSuccess) return e;
    launch_chain(k_rs_hist<K>, std::min(nb, (uint32_t)device_sm_count() * 4u), kSortThreads, 0, s, keys_in, n, hist);
    // even pass count: in -> tmp -> out -> tmp ... ends in `out`
    const K* ksrc = keys_in;
    const uint32_t* vsrc = vals_in;
    for (int pass = 0; pass < passes; ++pass) {
        const bool to_out = (pass & 1) != 0;
        K* kdst = to_out ? keys_out : kt;
        uint32_t* vdst = to_out ? vals_out : vt;
        auto* pass_kernel = large ? k_rs_pass<K, W, 2 * kSortItems> : k_rs_pass<K, W, kSortItems>;
        launch_chain(pass_kernel, nb, kSortThreads, 0, s, ksrc, vsrc, n, 8 * pass, hist + 256 * pass, status[pass & 1],
                     pass + 1 < passes ? status[(pass + 1) & 1] : nullptr, ticket + pass, kdst, vdst);
        ksrc = kdst;
        vsrc = vdst;
    }
    count_launches(1 + passes);
    return cudaGetLastError();
}

cudaError_t radix_sort_pairs(const void* keys_in, const uint32_t* vals_in, uint32_t n, int key_bits, void* keys_out,
                             uint32_t* vals_out, void* scratch, cudaStream_t s) {
    const bool big = n >= (1u << 30);  // counts that need more than 30 bits
    if (key_bits == 64) {
        auto* f = big ? radix_sort_impl<uint64_t, uint64_t> : radix_sort_impl<uint64_t, uint32_t>;
        return f(static_cast<const uint64_t*>(keys_in), vals_in, n, static_cast<uint64_t*>(keys_out), vals_out, scratch, s);
    }
    auto* f = big ? radix_sort_impl<uint32_t, uint64_t> : radix_sort_impl<uint32_t, uint32_t>;
    return f(static_cast<const uint32_t*>(keys_in), vals_in, n, static_cast<uint32_t*>(keys_out), vals_out, scratch, s);
}

cudaError_t launch_karras(const void* keys, uint32_t n, int key_bits, uint32_t* child_base, int stride,
                          uint32_t* parents, cudaStream_t s, uint32_t* ranges) {
    if (n < 2) return cudaSuccess;
    if (key_bits == 64)
        launch_chain(k_karras<uint64_t>, grid_for(n - 1), kBlock, 0, s, static_cast<const uint64_t*>(keys), n, child_base,
                     stride, parents, ranges);
    else
        launch_chain(k_karras<uint32_t>, grid_for(n - 1), kBlock, 0, s, static_cast<const uint32_t*>(keys), n, child_base,
                     stride, parents, ranges);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_karras_segments(const void* keys, int key_bits, const KarrasSeg* segs, uint32_t n_segs,
                                   uint32_t n_threads, uint32_t n_leaves, float4* nodes, uint32_t* parents,
                                   uint32_t* ranges, cudaStream_t s) {
    if (n_segs == 0 || n_threads == 0) return cudaSuccess;
    uint32_t* child_base = reinterpret_cast<uint32_t*>(nodes) + 12;
    if (key_bits == 64)
        launch_chain(k_karras_segments<uint64_t>, grid_for(n_threads), kBlock, 0, s, static_cast<const uint64_t*>(keys), segs,
                     n_segs, n_threads, n_leaves, child_base, parents, ranges);
    else
        launch_chain(k_karras_segments<uint32_t>, grid_for(n_threads), kBlock, 0, s, static_cast<const uint32_t*>(keys), segs,
                     n_segs, n_threads, n_leaves, child_base, parents, ranges);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_blas_leaves_refit(const float* vtx, uint32_t nv, const uint32_t* idx, const uint32_t* perm,
                                     const float* lohi, uint32_t n, const uint32_t* parents, float4* nodes, uint32_t* flags,
                                     float4* tris, uint32_t* leaf_of_prim, BlasDev* blas_out, DevStatus* st,
                                     cudaStream_t s, const uint32_t* boxes_done) {
    launch_chain(k_blas_leaves_refit, grid_for(n), kBlock, 0, s, vtx, nv, idx, perm, lohi, n, parents, nodes, flags,
                 tris, leaf_of_prim, blas_out, st, boxes_done);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_bound_sphere(const float* vtx, uint32_t nv, BlasDev* blas, cudaStream_t s) {
    if (nv == 0) return cudaSuccess;
    const uint32_t blocks = (uint32_t)min((nv + 255u) / 256u, (uint32_t)device_sm_count() * 4u);
    launch_chain(k_bound_sphere, blocks, 256, 0, s, vtx, nv, blas);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_instance_prep(const rg_instance* in, uint32_t n, const BlasDev* blas, uint32_t nblas,
                                 InstDev* tmp, float* wbox, int* cb_ord, bool check_blas, uint32_t* flags,
                                 DevStatus* st, cudaStream_t s) {
    launch_chain(k_instance_prep, grid_for(n), kBlock, 0, s, in, n, blas, nblas, tmp, wbox, cb_ord, check_blas, flags, st);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_tlas_leaves_refit(const InstDev* tmp, const float* wbox, const uint32_t* perm, uint32_t n,
                                     const uint32_t* parents, float4* nodes, uint32_t* flags, InstDev* inst_out,
                                     uint32_t* leaf_of_inst, DevStatus* st, cudaStream_t s,
                                     const uint32_t* boxes_done) {
    launch_chain(k_tlas_leaves_refit, grid_for(n), kBlock, 0, s, tmp, wbox, perm, n, parents, nodes, flags,
                 inst_out, leaf_of_inst, st, boxes_done);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_tlas_small(const rg_instance* in, uint32_t n, const BlasDev* blas, uint32_t nblas, InstDev* tmp,
                              float* wbox, bool refit, float4* nodes, uint32_t* perm, uint32_t* parents,
                              uint32_t* flags, uint32_t* ranges, InstDev* inst_out, uint32_t* leaf_of_inst,
                              DevStatus* st, cudaStream_t s) {
    if (n == 0 || n > kTlasSmallMax) return cudaErrorInvalidValue;
    const uint32_t threads = (n + 31u) & ~31u;
    launch_chain(k_tlas_small, 1, threads, 0, s, in, n, blas, nblas, tmp, wbox, refit, nodes, perm, parents, flags, ranges,
                 inst_out, leaf_of_inst, st);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace rg
