// Binned surface-area-heuristic (SAH) topology: the trace-speed build of a
// bottom-level BVH (RG_BLAS_SAH) and of a TLAS of up to kSahOneMax instances
// (RG_SCENE_SAH_TLAS).  The items start in Morton order (the LBVH's sort); a
// segment of that order is one subtree.  Level by level, every segment of more
// than two items is split by the binned SAH (kSahBins bins of the centroid
// bounds on each axis, the split of least area(left) * count(left) +
// area(right) * count(right)), and partitioned stably, so each side keeps its
// Morton order.  Every segment below kSahMaxLevels levels gets the Karras
// hierarchy of its Morton codes.  (Stopping the SAH at segments of 16 or 4
// triangles measured 3-4 % and 1 % slower traversal.)  The internal nodes of a
// segment of c items whose root is node d are d .. d + c - 2 (depth-first
// numbering: left subtree from d + 1, right from d + count(left)), so no
// allocation is needed and the root is node 0, as in the LBVH.  Every choice
// comes from atomic minima, maxima and counts, which do not depend on the
// order of the atomics, so the build is deterministic.
//
// Three ways of splitting, by segment size, all on the device:
//   more than kSahMid items: three launches per level over all such segments
//     (bins, splits, partition), blocks of kSahChunk positions;
//   kSahTiny + 1 .. kSahMid items: a block per segment builds its levels in
//     shared memory (k_sah_block);
//   at most kSahTiny items: a warp or three per segment build it to the end
//     (k_sah_tiny), an item a lane.
// Bound by latency: the levels are a serial chain, and a level of one block
// waits on its barriers and atomics, not on memory.  The splits' bins also
// give the exact boxes of both children, which are written into the node; only
// position halvings (no valid split), Karras segments and NaN boxes leave the
// boxes to the bottom-up refit, which the build then asks for.
#include <algorithm>
#include <climits>
#include <atomic>
#include <string>
#include <vector>

#include "karras.cuh"
#include "rg_internal.cuh"

namespace rg {

namespace {

constexpr int kBinVals = 7;  // per bin: count, box lo (3), box hi (3) as ordered ints
constexpr int kTaskBins = 3 * kSahBins * kBinVals;
constexpr int kTaskAcc = 6 + kTaskBins;  // centroid bounds (lo 3, hi 3), then the bins
constexpr int kAcc = (kTaskAcc + 3) & ~3;  // a segment's accumulators, padded to 16 bytes
constexpr int kSahBlock = 256;
constexpr int kSahItems = (int)kSahChunk / kSahBlock;  // consecutive positions of a thread

__device__ __forceinline__ float centroid_of(const float* __restrict__ lohi, uint32_t prim, int a) {
    return __fmul_rn(0.5f, __fadd_rn(lohi[6 * (size_t)prim + a], lohi[6 * (size_t)prim + 3 + a]));
}

// Bin of a centroid coordinate: floor((c - cmin) * scale) clamped to the
// bins (NaN to bin 0); the binning and the partition use this one function.
__device__ __forceinline__ int bin_of(float c, float cmin, float scale) {
    const float f = __fmul_rn(__fsub_rn(c, cmin), scale);
    if (!(f >= 0.0f)) return 0;
    return f < (float)kSahBins ? (int)f : kSahBins - 1;
}

__device__ __forceinline__ int ord_inf() { return f2ord(__int_as_float(0x7F800000)); }
__device__ __forceinline__ int ord_ninf() { return f2ord(__int_as_float(0xFF800000)); }


// A segment of more than kSahMid items at its level.
struct SahTask {
    uint32_t begin, count, node, first_block;
};
// What its split came to.
struct SahSplit {
    float cmin, scale;                   // the axis's binning frame
    int axis, split;                     // axis -1: halved by position
    uint32_t nl;                         // items on the left
    uint32_t child[2];                   // next-level task of each side, or kNone
    uint32_t pad;
};
// A segment left to a block or a warp; its items are in buffer `buf`.
struct SahPending {
    uint32_t begin, count, node;
    uint16_t level, buf;
};

// Counters: per level {tasks, blocks}, then the pending lists' lengths.
constexpr uint32_t kCntMid = 4 * (kSahMaxLevels + 1), kCntTiny = kCntMid + 1, kCntKarras = kCntMid + 2;
constexpr uint32_t kCntAll = kCntMid + 4;

// Everything the build's kernels share (device pointers).
struct SahBuild {
    const float* lohi;                   // item boxes (lo xyz, hi xyz)
    uint32_t n;
    uint32_t* prim[2];                   // item at each position; [0] is the result
    void* key[2];                        // its Morton code
    uint32_t* cnt;                       // kCntAll
    SahTask* tasks[2];                   // of even and odd levels
    uint2* blk[2];                       // per block of a level: task, first position
    int* acc[2];                         // per task: centroid bounds and bins
    SahSplit* split;                     // per task
    uint32_t *blk_cnt, *blk_off;         // per block: 16 bin counts per axis; left items before it
    SahPending *mid, *tiny;
    KarrasSeg* karras;
    float4* nodes;
    uint32_t *parents, *ranges;          // ranges may be null
    uint32_t* boxes_done;                // 1 until something leaves boxes to the refit
};

__device__ __forceinline__ int acc_init(int v) {
    if (v < 6) return v < 3 ? ord_inf() : ord_ninf();
    const int w = (v - 6) % kBinVals;
    return w == 0 ? 0 : (w < 4 ? ord_inf() : ord_ninf());
}

// The binning frame of an axis with centroid bounds lo, hi (scale 0, every
// centroid in bin 0, when they are a point).
__device__ __forceinline__ float bin_scale(float lo, float hi) {
    const float ext = __fsub_rn(hi, lo);
    return ext > 0.0f ? fminf(__fdiv_rn((float)kSahBins, ext), 3.0e38f) : 0.0f;
}

__device__ __forceinline__ unsigned long long split_key(float cost, int a, int s) {
    return ((unsigned long long)__float_as_uint(cost) << 32) | (uint32_t)(a * (kSahBins - 1) + s - 1);
}

__device__ __forceinline__ float half_area(const float* lo, const float* hi) {
    const float dx = __fsub_rn(hi[0], lo[0]), dy = __fsub_rn(hi[1], lo[1]), dz = __fsub_rn(hi[2], lo[2]);
    return __fadd_rn(__fadd_rn(__fmul_rn(dx, dy), __fmul_rn(dy, dz)), __fmul_rn(dz, dx));
}

// Node `node` over leaves b .. b + c - 1 with nl on the left: its children
// (a leaf when one side holds one item), their parent entries, its range.
__device__ __forceinline__ void emit_sah_node(uint32_t node, uint32_t b, uint32_t c, uint32_t nl, uint32_t n_leaves,
                                              float4* nodes, uint32_t* parents, uint32_t* ranges) {
    const uint32_t nr = c - nl;
    const uint32_t left = nl == 1 ? (kLeaf | b) : node + 1;
    const uint32_t right = nr == 1 ? (kLeaf | (b + nl)) : node + nl;
    uint32_t* ch = reinterpret_cast<uint32_t*>(nodes + 4 * (size_t)node + 3);
    ch[0] = left;
    ch[1] = right;
    parents[(left & kLeaf) ? (size_t)(n_leaves - 1) + (left & ~kLeaf) : left] = node;
    parents[(right & kLeaf) ? (size_t)(n_leaves - 1) + (right & ~kLeaf) : right] = node;
    if (node == 0) parents[0] = kNone;
    if (ranges) {
        ranges[2 * (size_t)node] = b;
        ranges[2 * (size_t)node + 1] = b + c - 1;
    }
}

// The boxes of a node's two children (lo xyz, hi xyz each), in the node's
// layout: floats 0-5 the left child's, 6-11 the right child's.
__device__ __forceinline__ void put_child_boxes(float4* nodes, uint32_t node, const float* l, const float* r) {
    float4* f = nodes + 4 * (size_t)node;
    f[0] = make_float4(l[0], l[1], l[2], l[3]);
    f[1] = make_float4(l[4], l[5], r[0], r[1]);
    f[2] = make_float4(r[2], r[3], r[4], r[5]);
}


// The least cost over the boundaries of one axis, by 16 lanes: lane s of the
// group holds bin s (g: the axis's bins); the left side of boundary s is the
// prefix of bins 0 .. s - 1, the right side the suffix s .. 15, both scanned
// across the lanes.  All lanes of the warp call; every lane of a group gets its
// least packed key (cost bits, then the candidate's index a * 15 + s - 1, so
// the first of equal costs; -0 taken as +0), ~0 if no boundary is valid.  The
// minima and maxima of each side are exact in any order.
__device__ __forceinline__ unsigned long long sweep16(const int* g, int a, uint32_t s, bool valid) {
    const int* e = g + (int)s * kBinVals;
    int pc = valid ? e[0] : 0, sc = pc;
    int pv[6], sv[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) pv[k] = sv[k] = valid ? e[1 + k] : (k < 3 ? ord_inf() : ord_ninf());
#pragma unroll
    for (int d = 1; d < 16; d <<= 1) {
        const int yc = __shfl_up_sync(0xFFFFFFFFu, pc, d, 16);
        const int zc = __shfl_down_sync(0xFFFFFFFFu, sc, d, 16);
        if ((int)s >= d) pc += yc;
        if ((int)s + d < 16) sc += zc;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, pv[k], d, 16);
            const int z = __shfl_down_sync(0xFFFFFFFFu, sv[k], d, 16);
            if ((int)s >= d) pv[k] = k < 3 ? min(pv[k], y) : max(pv[k], y);
            if ((int)s + d < 16) sv[k] = k < 3 ? min(sv[k], z) : max(sv[k], z);
        }
    }
    const int lc = __shfl_up_sync(0xFFFFFFFFu, pc, 1, 16);
    float lo[3], hi[3], rlo[3], rhi[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        lo[k] = ord2f(__shfl_up_sync(0xFFFFFFFFu, pv[k], 1, 16));
        hi[k] = ord2f(__shfl_up_sync(0xFFFFFFFFu, pv[3 + k], 1, 16));
        rlo[k] = ord2f(sv[k]);
        rhi[k] = ord2f(sv[3 + k]);
    }
    unsigned long long key = ~0ull;
    if (valid && s >= 1u && lc != 0 && sc != 0) {
        const float cost = __fadd_rn(__fadd_rn(__fmul_rn(half_area(lo, hi), (float)(uint32_t)lc),
                                               __fmul_rn(half_area(rlo, rhi), (float)(uint32_t)sc)),
                                     0.0f);
        if (cost < INFINITY) key = split_key(cost, a, (int)s);
    }
#pragma unroll
    for (int d = 8; d > 0; d >>= 1) {
        const unsigned long long y = __shfl_xor_sync(0xFFFFFFFFu, key, d, 16);
        key = y < key ? y : key;
    }
    return key;
}

// Both children's boxes from the bins of the winning axis; returns the left count.
__device__ __forceinline__ uint32_t side_boxes(const int* g, int sp, float* l, float* r) {
    int lb[6], rb[6];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        lb[k] = rb[k] = ord_inf();
        lb[3 + k] = rb[3 + k] = ord_ninf();
    }
    uint32_t nl = 0;
    for (int b = 0; b < kSahBins; ++b) {
        const int* e = g + b * kBinVals;
        int* d = b < sp ? lb : rb;
        if (b < sp) nl += (uint32_t)e[0];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            d[k] = min(d[k], e[1 + k]);
            d[3 + k] = max(d[3 + k], e[4 + k]);
        }
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        l[k] = ord2f(lb[k]);
        r[k] = ord2f(rb[k]);
    }
    return nl;
}

__device__ __forceinline__ bool has_nan(const float* b) {
    return b[0] != b[0] || b[1] != b[1] || b[2] != b[2] || b[3] != b[3] || b[4] != b[4] || b[5] != b[5];
}

__device__ __forceinline__ void push_pending(const SahBuild& B, uint32_t begin, uint32_t count, uint32_t node,
                                             uint32_t level, uint32_t buf) {
    const SahPending T{begin, count, node, (uint16_t)level, (uint16_t)buf};
    if (count <= kSahTiny)
        B.tiny[atomicAdd(B.cnt + kCntTiny, 1u)] = T;
    else
        B.mid[atomicAdd(B.cnt + kCntMid, 1u)] = T;
}

// The counters, and the root segment (its centroid bounds cb_ord are known).
__global__ void k_sah_start(SahBuild B, const int* __restrict__ cb_ord) {
    chain_wait();
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    for (uint32_t k = i; blockIdx.x == 0 && k < kCntAll; k += blockDim.x) B.cnt[k] = 0u;
    __syncthreads();
    if (i == 0) *B.boxes_done = 1u;
    if (B.n <= kSahMid) {
        if (i == 0) push_pending(B, 0, B.n, 0, 0, 0);
        return;
    }
    const uint32_t chunks = (B.n + kSahChunk - 1) / kSahChunk;
    if (i == 0) {
        B.tasks[0][0] = SahTask{0u, B.n, 0u, 0u};
        B.cnt[0] = 1u;
        B.cnt[1] = chunks;
    }
    for (uint32_t b = i; b < chunks; b += gridDim.x * blockDim.x) B.blk[0][b] = make_uint2(0u, b * kSahChunk);
    if (i < (uint32_t)kAcc) B.acc[0][i] = i < 6 ? cb_ord[i] : acc_init((int)i);
}

// Bins of a level: each block its chunk in shared memory (a thread merges its
// consecutive positions, Morton neighbours, per run of one bin before the
// atomics), then merged into the task's bins once per non-empty bin; the
// chunk's counts are kept for the partition.
__global__ void __launch_bounds__(kSahBlock) k_sah_bin(SahBuild B, uint32_t level) {
    chain_wait();
    __shared__ int sb[kTaskBins];
    __shared__ float s_cmin[3], s_scale[3];
    const uint32_t cur = level & 1u;
    if (blockIdx.x >= B.cnt[4 * level + 1]) return;
    const uint2 e = B.blk[cur][blockIdx.x];
    const SahTask T = B.tasks[cur][e.x];
    int* acc = B.acc[cur] + (size_t)e.x * kAcc;
    for (int v = threadIdx.x; v < kTaskBins; v += kSahBlock) sb[v] = acc_init(v + 6);
    if (threadIdx.x < 3) {
        const float lo = ord2f(acc[threadIdx.x]);
        s_cmin[threadIdx.x] = lo;
        s_scale[threadIdx.x] = bin_scale(lo, ord2f(acc[3 + threadIdx.x]));
    }
    __syncthreads();
    const uint32_t p0 = e.y + threadIdx.x * kSahItems, p1 = min(e.y + kSahChunk, T.begin + T.count);
    int rb[3] = {-1, -1, -1}, st[3][7] = {};
    auto flush = [&](int a) {
        int* d = sb + (a * kSahBins + rb[a]) * kBinVals;
        atomicAdd(d, st[a][0]);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            atomicMin(d + 1 + k, st[a][1 + k]);
            atomicMax(d + 4 + k, st[a][4 + k]);
        }
    };
    bool nan = false;
#pragma unroll
    for (int j = 0; j < kSahItems; ++j) {
        if (p0 + j >= p1) break;
        const uint32_t prim = B.prim[cur][p0 + j];
        float bx[6];
        int v[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            bx[k] = B.lohi[6 * (size_t)prim + k];
            v[k] = f2ord(bx[k]);
        }
        nan |= has_nan(bx);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int b = bin_of(centroid_of(bx, 0, a), s_cmin[a], s_scale[a]);
            if (b == rb[a]) {
                st[a][0] += 1;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    st[a][1 + k] = min(st[a][1 + k], v[k]);
                    st[a][4 + k] = max(st[a][4 + k], v[3 + k]);
                }
            } else {
                if (rb[a] >= 0) flush(a);
                rb[a] = b;
                st[a][0] = 1;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    st[a][1 + k] = v[k];
                    st[a][4 + k] = v[3 + k];
                }
            }
        }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a)
        if (rb[a] >= 0) flush(a);
    if (nan) *B.boxes_done = 0u;
    __syncthreads();
    for (int v = threadIdx.x; v < kTaskBins; v += kSahBlock) {
        const int w = v % kBinVals;
        if (w == 0) B.blk_cnt[(size_t)blockIdx.x * (3 * kSahBins) + v / kBinVals] = (uint32_t)sb[v];
        if (sb[v - w] == 0) continue;  // empty bin
        if (w == 0)
            atomicAdd(acc + 6 + v, sb[v]);
        else if (w < 4)
            atomicMin(acc + 6 + v, sb[v]);
        else
            atomicMax(acc + 6 + v, sb[v]);
    }
}

// Splits of a level, a block per task: the split of least cost (axis, then
// boundary; the first of equal costs), without one (every axis' centroids in
// one bin) the halves by position; the node and its children's boxes; what
// becomes of the children; and the left items before each block of the task.
constexpr int kSplitBlock = 128;
__global__ void __launch_bounds__(kSplitBlock) k_sah_split(SahBuild B, uint32_t level) {
    chain_wait();
    __shared__ int sb[kTaskBins];
    __shared__ unsigned long long s_best;
    __shared__ SahSplit s_split;
    __shared__ SahTask s_child[2];
    __shared__ uint32_t s_warp[kSplitBlock / 32];
    const uint32_t cur = level & 1u, nxt = cur ^ 1u, t = threadIdx.x, lane = t & 31u, warp = t >> 5;
    if (blockIdx.x >= B.cnt[4 * level]) return;
    const SahTask T = B.tasks[cur][blockIdx.x];
    const int* acc = B.acc[cur] + (size_t)blockIdx.x * kAcc;
    for (int v = t; v < kTaskBins; v += kSplitBlock) sb[v] = acc[6 + v];
    if (t == 0) s_best = ~0ull;
    __syncthreads();
    if (t < 64) {
        const int a = (int)(t >> 4);
        const unsigned long long key = sweep16(sb + min(a, 2) * kSahBins * kBinVals, a, t & 15u, a < 3);
        if ((t & 15u) == 0u && key != ~0ull) atomicMin(&s_best, key);
    }
    __syncthreads();
    if (t == 0) {
        SahSplit R{};
        R.axis = -1;
        R.nl = T.count / 2;
        if (s_best != ~0ull) {
            const uint32_t c = (uint32_t)s_best;
            R.axis = (int)(c / (kSahBins - 1));
            R.split = (int)(c % (kSahBins - 1)) + 1;
            float l[6], r[6];
            R.nl = side_boxes(sb + R.axis * kSahBins * kBinVals, R.split, l, r);
            put_child_boxes(B.nodes, T.node, l, r);
            R.cmin = ord2f(acc[R.axis]);
            R.scale = bin_scale(R.cmin, ord2f(acc[3 + R.axis]));
        } else {
            *B.boxes_done = 0u;
        }
        emit_sah_node(T.node, T.begin, T.count, R.nl, B.n, B.nodes, B.parents, B.ranges);
        for (int side = 0; side < 2; ++side) {
            const uint32_t b = side ? T.begin + R.nl : T.begin, c = side ? T.count - R.nl : R.nl;
            const uint32_t nd = side ? T.node + R.nl : T.node + 1;
            R.child[side] = kNone;
            s_child[side] = SahTask{b, c, nd, 0u};
            if (c >= 3 && level + 1 >= kSahMaxLevels) {  // (level kSahMaxLevels is even: its items are in buffer 0)
                B.karras[atomicAdd(B.cnt + kCntKarras, 1u)] = KarrasSeg{b, c, nd, 0u};
                *B.boxes_done = 0u;
            } else if (c <= kSahMid) {
                push_pending(B, b, c, nd, level + 1, nxt);
            } else {
                const uint32_t slot = atomicAdd(B.cnt + 4 * (level + 1), 1u);
                s_child[side].first_block =
                    atomicAdd(B.cnt + 4 * (level + 1) + 1, (c + kSahChunk - 1) / kSahChunk);
                B.tasks[nxt][slot] = s_child[side];
                R.child[side] = slot;
            }
        }
        s_split = R;
        B.split[blockIdx.x] = R;
    }
    __syncthreads();
    const SahSplit R = s_split;
    for (int side = 0; side < 2; ++side) {
        if (R.child[side] == kNone) continue;
        const SahTask C = s_child[side];
        int* ca = B.acc[nxt] + (size_t)R.child[side] * kAcc;
        for (int v = t; v < kAcc; v += kSplitBlock) ca[v] = acc_init(v);
        const uint32_t chunks = (C.count + kSahChunk - 1) / kSahChunk;
        for (uint32_t b = t; b < chunks; b += kSplitBlock)
            B.blk[nxt][C.first_block + b] = make_uint2(R.child[side], C.begin + b * kSahChunk);
    }
    const uint32_t chunks = (T.count + kSahChunk - 1) / kSahChunk;
    uint32_t carry = 0;
    for (uint32_t b0 = 0; b0 < chunks; b0 += kSplitBlock) {
        const uint32_t b = b0 + t;
        uint32_t left = 0;
        if (b < chunks) {
            if (R.axis < 0) {
                const uint32_t o = b * kSahChunk;
                left = R.nl > o ? min(R.nl - o, kSahChunk) : 0u;
            } else {
                const uint32_t* c = B.blk_cnt + (size_t)(T.first_block + b) * (3 * kSahBins) + R.axis * kSahBins;
                for (int q = 0; q < R.split; ++q) left += c[q];
            }
        }
        uint32_t inc = left;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, off);
            if ((int)lane >= off) inc += y;
        }
        if (lane == 31) s_warp[warp] = inc;
        __syncthreads();
        uint32_t before = carry, total = 0;
        for (uint32_t w = 0; w < kSplitBlock / 32; ++w) {
            if (w < warp) before += s_warp[w];
            total += s_warp[w];
        }
        if (b < chunks) B.blk_off[T.first_block + b] = before + inc - left;
        carry += total;
        __syncthreads();
    }
}

// Stable partition of a level into the other buffer; the centroid bounds of
// the children that are split at the next level.
template <class K>
__global__ void __launch_bounds__(kSahBlock) k_sah_scatter(SahBuild B, uint32_t level) {
    chain_wait();
    __shared__ uint32_t s_warp[kSahBlock / 32];
    __shared__ int s_cb[2][6];
    const uint32_t cur = level & 1u, nxt = cur ^ 1u, t = threadIdx.x, lane = t & 31u, warp = t >> 5;
    if (blockIdx.x >= B.cnt[4 * level + 1]) return;
    const uint2 e = B.blk[cur][blockIdx.x];
    const SahTask T = B.tasks[cur][e.x];
    const SahSplit R = B.split[e.x];
    const K* key_in = static_cast<const K*>(B.key[cur]);
    K* key_out = static_cast<K*>(B.key[nxt]);
    if (t < 12) s_cb[t / 6][t % 6] = acc_init((int)(t % 6));
    const uint32_t p0 = e.y + t * kSahItems, p1 = min(e.y + kSahChunk, T.begin + T.count);
    uint32_t prim[kSahItems], mine = 0;
    K key[kSahItems];
    bool left[kSahItems];
    int mn[2][3], mx[2][3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        mn[0][k] = mn[1][k] = ord_inf();
        mx[0][k] = mx[1][k] = ord_ninf();
    }
#pragma unroll
    for (int j = 0; j < kSahItems; ++j) {
        left[j] = false;
        if (p0 + j >= p1) continue;
        prim[j] = B.prim[cur][p0 + j];
        key[j] = key_in[p0 + j];
        float c[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) c[k] = centroid_of(B.lohi, prim[j], k);
        const float ca = R.axis == 0 ? c[0] : (R.axis == 1 ? c[1] : c[2]);
        left[j] = R.axis < 0 ? (p0 + j - T.begin < R.nl) : bin_of(ca, R.cmin, R.scale) < R.split;
        mine += left[j];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int v = f2ord(c[k]);
            if (left[j]) {
                mn[0][k] = min(mn[0][k], v);
                mx[0][k] = max(mx[0][k], v);
            } else {
                mn[1][k] = min(mn[1][k], v);
                mx[1][k] = max(mx[1][k], v);
            }
        }
    }
    uint32_t inc = mine;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, off);
        if ((int)lane >= off) inc += y;
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    uint32_t run = B.blk_off[blockIdx.x] + inc - mine;
    for (uint32_t w = 0; w < warp; ++w) run += s_warp[w];
#pragma unroll
    for (int j = 0; j < kSahItems; ++j) {
        if (p0 + j >= p1) break;
        const uint32_t dest = T.begin + (left[j] ? run : R.nl + ((p0 + j - T.begin) - run));
        run += left[j];
        B.prim[nxt][dest] = prim[j];
        key_out[dest] = key[j];
    }
    if (R.child[0] == kNone && R.child[1] == kNone) return;
#pragma unroll
    for (int side = 0; side < 2; ++side)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int a = __reduce_min_sync(0xFFFFFFFFu, mn[side][k]);
            const int b = __reduce_max_sync(0xFFFFFFFFu, mx[side][k]);
            if (lane == 0) {
                atomicMin(&s_cb[side][k], a);
                atomicMax(&s_cb[side][3 + k], b);
            }
        }
    __syncthreads();
    if (t < 12) {
        const int side = (int)t / 6, k = (int)t % 6;
        if (R.child[side] != kNone) {
            int* d = B.acc[nxt] + (size_t)R.child[side] * kAcc + k;
            if (k < 3)
                atomicMin(d, s_cb[side][k]);
            else
                atomicMax(d, s_cb[side][k]);
        }
    }
}

// ---------------------------------------------------------------- segments in a block
constexpr uint16_t kSegNone = 0xFFFF;

struct OneSeg {
    uint16_t begin, count, node, pad;    // block-local first position, items, internal node past the segment's
};
struct OneRes {
    uint16_t nl;                         // items on the left
    int8_t axis, split;                  // the split (axis -1: halving by position)
    float cmin, scale;                   // the axis's binning frame
    uint16_t child[2];                   // next-level segment of each side, or kSegNone
};

// Shared state of a block that builds a segment of up to NMAX items, at most
// SEGS subsegments split per level.  Items are named by their position in the
// segment as it came: the box of each, and the item at each position now.
template <int NMAX, int SEGS>
struct BlockSah {
    float box[NMAX][6];
    uint16_t idx[2][NMAX];               // item at each position (two buffers)
    uint16_t seg_of[NMAX];               // this level's segment of each position, or kSegNone
    uint16_t excl[NMAX];                 // left items before each position
    OneSeg seg[2][SEGS];
    OneRes res[SEGS];
    alignas(16) int acc[SEGS * kAcc];    // per segment: centroid bounds and bins
    float par[SEGS * 6];                 // per segment: cmin and scale of each axis
    unsigned long long best[SEGS];       // per segment: least (cost, candidate)
    alignas(16) int pat[kAcc];           // the accumulators' initial values of one segment
    uint32_t m, mnext, wsum[32];
};
constexpr int kMidThreads = 512, kTopThreads = 1024;
using BlockMid = BlockSah<(int)kSahMid, (int)(kSahMid / (kSahTiny + 1) + 1)>;
using BlockTop = BlockSah<(int)kSahOneMax, (int)(kSahOneMax / (kSahMid + 1) + 1)>;
static_assert(sizeof(BlockTop) <= 227 * 1024 && 2 * (sizeof(BlockMid) + 1024) <= 227 * 1024, "shared memory of the SAH blocks");
static_assert(kSahOneMax <= 0xFFFFu, "16-bit positions");

// Keys of a segment through its positions' items.
template <class K>
struct LocalKeys {
    const K* keys;
    const uint16_t* idx;
    __device__ __forceinline__ K operator[](int64_t i) const { return keys[idx[i]]; }
};

// Builds segment T to the end, or with subsegments of at most `stop` items left
// to the pending lists; the final order of its items and codes goes to buffer 0
// (the buffers' contents may be in place: every read comes before the writes).
template <int NT, int NMAX, int SEGS, class K>
__device__ void sah_block(BlockSah<NMAX, SEGS>& S, const SahBuild& B, const SahPending T, uint32_t stop) {
    const uint32_t base = T.begin, cnt = T.count;
    const uint32_t* src = B.prim[T.buf];
    const K* skey = static_cast<const K*>(B.key[T.buf]);
    float4* nodes = B.nodes;
    constexpr uint32_t P = (NMAX + NT - 1) / NT;  // positions per thread in the partition's scan
    constexpr int W = NT / 32;
    const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
    bool nan = false;
    for (uint32_t i = t; i < cnt; i += NT) {
        const uint32_t prim = src[base + i];
#pragma unroll
        for (int k = 0; k < 6; ++k) S.box[i][k] = B.lohi[6 * (size_t)prim + k];
        nan |= has_nan(S.box[i]);
        S.idx[0][i] = (uint16_t)i;
        S.seg_of[i] = 0;
    }
    if (nan) *B.boxes_done = 0u;
    for (uint32_t w = t; w < (uint32_t)kAcc; w += NT) S.pat[w] = w < (uint32_t)kTaskAcc ? acc_init((int)w) : 0;
    if (t == 0) {
        S.seg[0][0] = OneSeg{0, (uint16_t)cnt, 0, 0};
        S.m = 1;
    }
    __syncthreads();
    int cb = 0;
    for (uint32_t level = T.level;; ++level) {
        const uint32_t m = S.m;
        if (m == 0) break;
        OneSeg* cur = S.seg[cb];
        OneSeg* nxt = S.seg[cb ^ 1];
        const uint16_t* ix = S.idx[cb];
        uint16_t* ix2 = S.idx[cb ^ 1];
        __syncthreads();
        if (t == 0) S.mnext = 0;
        for (uint32_t v = t; v < m * (uint32_t)(kAcc / 4); v += NT) {
            const uint32_t q = v / (uint32_t)(kAcc / 4), w = v - q * (uint32_t)(kAcc / 4);
            reinterpret_cast<int4*>(S.acc)[v] = reinterpret_cast<const int4*>(S.pat)[w];
        }
        __syncthreads();
        // centroid bounds: each thread's P consecutive positions merged per run
        // of one segment; one warp reduction when the warp holds one segment
        {
            uint32_t rq = kSegNone;
            bool multi = false;
            int mn[3] = {0, 0, 0}, mx[3] = {0, 0, 0};
#pragma unroll
            for (uint32_t j = 0; j < P; ++j) {
                const uint32_t p = P * t + j;
                const uint32_t q = p < cnt ? S.seg_of[p] : kSegNone;
                if (q == kSegNone) continue;
                const float* bx = S.box[ix[p]];
                int c[3];
#pragma unroll
                for (int k = 0; k < 3; ++k) c[k] = f2ord(centroid_of(bx, 0, k));
                if (q != rq) {
                    if (rq != kSegNone) {
                        int* ac = S.acc + (size_t)rq * kAcc;
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            atomicMin(ac + k, mn[k]);
                            atomicMax(ac + 3 + k, mx[k]);
                        }
                        multi = true;
                    }
                    rq = q;
#pragma unroll
                    for (int k = 0; k < 3; ++k) mn[k] = mx[k] = c[k];
                } else {
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        mn[k] = min(mn[k], c[k]);
                        mx[k] = max(mx[k], c[k]);
                    }
                }
            }
            const uint32_t q0 = __shfl_sync(0xFFFFFFFFu, rq, 0);
            const bool uni = __all_sync(0xFFFFFFFFu, rq == q0 && !multi);
            if (uni) {
                if (q0 != kSegNone) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        mn[k] = __reduce_min_sync(0xFFFFFFFFu, mn[k]);
                        mx[k] = __reduce_max_sync(0xFFFFFFFFu, mx[k]);
                    }
                    if (lane == 0) {
                        int* ac = S.acc + (size_t)q0 * kAcc;
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            atomicMin(ac + k, mn[k]);
                            atomicMax(ac + 3 + k, mx[k]);
                        }
                    }
                }
            } else if (rq != kSegNone) {
                int* ac = S.acc + (size_t)rq * kAcc;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    atomicMin(ac + k, mn[k]);
                    atomicMax(ac + 3 + k, mx[k]);
                }
            }
        }
        __syncthreads();
        for (uint32_t q = t; q < m; q += NT) {
            const int* a = S.acc + (size_t)q * kAcc;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float lo = ord2f(a[k]), hi = ord2f(a[3 + k]);
                S.par[6 * q + k] = lo;
                S.par[6 * q + 3 + k] = bin_scale(lo, hi);
            }
            S.best[q] = ~0ull;
        }
        __syncthreads();
        // bins: each thread's P consecutive positions merged per run of one
        // segment and bin on each axis, one set of atomics per run
        {
            uint32_t rq = kSegNone;
            int rb[3] = {0, 0, 0};
            int st[3][7];
#pragma unroll
            for (uint32_t j = 0; j < P; ++j) {
                const uint32_t p = P * t + j;
                const uint32_t q = p < cnt ? S.seg_of[p] : kSegNone;
                if (q == kSegNone) continue;
                const float* bx = S.box[ix[p]];
                int v[6];
#pragma unroll
                for (int k = 0; k < 6; ++k) v[k] = f2ord(bx[k]);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const int b = bin_of(centroid_of(bx, 0, a), S.par[6 * q + a], S.par[6 * q + 3 + a]);
                    if (q == rq && b == rb[a]) {
                        st[a][0] += 1;
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            st[a][1 + k] = min(st[a][1 + k], v[k]);
                            st[a][4 + k] = max(st[a][4 + k], v[3 + k]);
                        }
                    } else {
                        if (rq != kSegNone) {
                            int* e = S.acc + (size_t)rq * kAcc + 6 + (a * kSahBins + rb[a]) * kBinVals;
                            atomicAdd(e, st[a][0]);
#pragma unroll
                            for (int k = 0; k < 3; ++k) {
                                atomicMin(e + 1 + k, st[a][1 + k]);
                                atomicMax(e + 4 + k, st[a][4 + k]);
                            }
                        }
                        rb[a] = b;
                        st[a][0] = 1;
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            st[a][1 + k] = v[k];
                            st[a][4 + k] = v[3 + k];
                        }
                    }
                }
                rq = q;
            }
            if (rq != kSegNone) {
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    int* e = S.acc + (size_t)rq * kAcc + 6 + (a * kSahBins + rb[a]) * kBinVals;
                    atomicAdd(e, st[a][0]);
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        atomicMin(e + 1 + k, st[a][1 + k]);
                        atomicMax(e + 4 + k, st[a][4 + k]);
                    }
                }
            }
        }
        __syncthreads();
        // the least cost of each segment, 16 lanes per (segment, axis)
        for (uint32_t v = t; v < ((m * 48u + 31u) & ~31u); v += NT) {
            const uint32_t g = v >> 4;
            const bool valid = g < m * 3u;
            const uint32_t q = valid ? g / 3u : 0u;
            const int a = valid ? (int)(g % 3u) : 0;
            const unsigned long long key =
                sweep16(S.acc + (size_t)q * kAcc + 6 + a * kSahBins * kBinVals, a, v & 15u, valid);
            if (valid && (v & 15u) == 0u && key != ~0ull) atomicMin(&S.best[q], key);
        }
        __syncthreads();
        // the split of each segment, its node, and its children's boxes from
        // the bins of each side
        for (uint32_t q = t; q < m; q += NT) {
            const unsigned long long key = S.best[q];
            const uint32_t count = cur[q].count;
            OneRes R;
            R.axis = -1;
            R.split = 0;
            R.nl = (uint16_t)(count / 2);
            R.cmin = R.scale = 0.0f;
            if (key != ~0ull) {
                const uint32_t c = (uint32_t)key;
                const int a = (int)(c / (kSahBins - 1)), sp = (int)(c % (kSahBins - 1)) + 1;
                float l[6], r[6];
                const uint32_t nl = side_boxes(S.acc + (size_t)q * kAcc + 6 + a * kSahBins * kBinVals, sp, l, r);
                put_child_boxes(nodes, T.node + cur[q].node, l, r);
                R.axis = (int8_t)a;
                R.split = (int8_t)sp;
                R.nl = (uint16_t)nl;
                R.cmin = S.par[6 * q + a];
                R.scale = S.par[6 * q + 3 + a];
            } else {
                *B.boxes_done = 0u;  // halved by position: the children's boxes come from the refit
            }
            R.child[0] = R.child[1] = kSegNone;
            S.res[q] = R;
            emit_sah_node(T.node + cur[q].node, base + cur[q].begin, count, R.nl, B.n, nodes, B.parents, B.ranges);
        }
        __syncthreads();
        // stable partition: exclusive left counts over the positions (thread t
        // owns positions P t .. P t + P - 1)
        bool left[P];
        uint32_t mine = 0;
#pragma unroll
        for (uint32_t j = 0; j < P; ++j) {
            const uint32_t p = P * t + j;
            left[j] = false;
            if (p < cnt && S.seg_of[p] != kSegNone) {
                const uint16_t q = S.seg_of[p];
                const OneRes R = S.res[q];
                left[j] = R.axis < 0 ? (p - cur[q].begin < R.nl)
                                     : bin_of(centroid_of(S.box[ix[p]], 0, R.axis), R.cmin, R.scale) < R.split;
            }
            mine += left[j];
        }
        uint32_t inc = mine;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, off);
            if ((int)lane >= off) inc += y;
        }
        if (lane == 31) S.wsum[warp] = inc;
        __syncthreads();
        if (warp == 0) {
            const uint32_t x = lane < (uint32_t)W ? S.wsum[lane] : 0u;
            uint32_t winc = x;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, winc, off);
                if ((int)lane >= off) winc += y;
            }
            if (lane < (uint32_t)W) S.wsum[lane] = winc - x;
        }
        __syncthreads();
        uint32_t run = S.wsum[warp] + inc - mine;
#pragma unroll
        for (uint32_t j = 0; j < P; ++j) {
            const uint32_t p = P * t + j;
            if (p < cnt) S.excl[p] = (uint16_t)run;
            run += left[j];
        }
        __syncthreads();
#pragma unroll
        for (uint32_t j = 0; j < P; ++j) {
            const uint32_t p = P * t + j;
            if (p >= cnt) continue;
            const uint16_t q = S.seg_of[p];
            if (q == kSegNone) {
                ix2[p] = ix[p];
                continue;
            }
            const uint32_t b = cur[q].begin;
            const uint32_t lr = (uint32_t)S.excl[p] - (uint32_t)S.excl[b];
            ix2[b + (left[j] ? lr : (uint32_t)S.res[q].nl + ((p - b) - lr))] = ix[p];
        }
        __syncthreads();
        // children: pairs, the Karras hierarchy below the depth cap, pending
        // segments, or the next level
        for (uint32_t q = t; q < m; q += NT) {
            const OneSeg G = cur[q];
            const uint32_t nl = S.res[q].nl;
            for (int side = 0; side < 2; ++side) {
                const uint32_t b = side ? G.begin + nl : G.begin;
                const uint32_t c = side ? G.count - nl : nl;
                const uint32_t nd = side ? G.node + nl : G.node + 1;
                if (c == 2) {
                    emit_sah_node(T.node + nd, base + b, 2, 1, B.n, nodes, B.parents, B.ranges);
                    put_child_boxes(nodes, T.node + nd, S.box[ix2[b]], S.box[ix2[b + 1]]);
                } else if (c >= 3 && level + 1 >= kSahMaxLevels) {
                    const LocalKeys<K> ks{skey + base, ix2 + b};
                    for (uint32_t i = 0; i + 1 < c; ++i)
                        karras_node(ks, c, (int64_t)i, reinterpret_cast<uint32_t*>(nodes) + 12, 16, B.parents, B.ranges,
                                    T.node + nd, base + b, B.n);
                    *B.boxes_done = 0u;  // the Karras nodes' boxes come from the refit
                } else if (c >= 3 && c <= stop) {
                    push_pending(B, base + b, c, T.node + nd, level + 1, 0u);
                } else if (c >= 3) {
                    const uint32_t slot = atomicAdd(&S.mnext, 1u);
                    nxt[slot] = OneSeg{(uint16_t)b, (uint16_t)c, (uint16_t)nd, 0};
                    S.res[q].child[side] = (uint16_t)slot;
                }
            }
        }
        __syncthreads();
        for (uint32_t p = t; p < cnt; p += NT) {
            const uint16_t q = S.seg_of[p];
            if (q == kSegNone) continue;
            S.seg_of[p] = S.res[q].child[p - cur[q].begin >= S.res[q].nl ? 1 : 0];
        }
        if (t == 0) S.m = S.mnext;
        cb ^= 1;
        __syncthreads();

    }
    uint32_t prim[P];
    K key[P];
#pragma unroll
    for (uint32_t j = 0; j < P; ++j) {
        const uint32_t p = NT * j + t;
        if (p >= cnt) continue;
        const uint32_t i = base + S.idx[cb][p];
        prim[j] = src[i];
        key[j] = skey[i];
    }
    __syncthreads();
#pragma unroll
    for (uint32_t j = 0; j < P; ++j) {
        const uint32_t p = NT * j + t;
        if (p >= cnt) continue;
        B.prim[0][base + p] = prim[j];
        static_cast<K*>(B.key[0])[base + p] = key[j];
    }
    __syncthreads();
}

// A block per pending segment of kSahTiny + 1 .. kSahMid items.
template <class K>
__global__ void __launch_bounds__(kMidThreads) k_sah_block(SahBuild B) {
    chain_wait();
    extern __shared__ __align__(16) unsigned char sm[];
    BlockMid& S = *reinterpret_cast<BlockMid*>(sm);
    const uint32_t m = B.cnt[kCntMid];
    for (uint32_t k = blockIdx.x; k < m; k += gridDim.x)
        sah_block<kMidThreads, (int)kSahMid, (int)(kSahMid / (kSahTiny + 1) + 1), K>(S, B, B.mid[k], kSahTiny);
}

// The tasks left at `level` when the host does not look (n <= kSahOneMax):
// usually none.
template <class K>
__global__ void __launch_bounds__(kTopThreads, 1) k_sah_rest(SahBuild B, uint32_t level) {
    chain_wait();
    extern __shared__ __align__(16) unsigned char sm[];
    BlockTop& S = *reinterpret_cast<BlockTop*>(sm);
    const uint32_t m = B.cnt[4 * level];
    for (uint32_t k = blockIdx.x; k < m; k += gridDim.x) {
        const SahTask T = B.tasks[level & 1u][k];
        sah_block<kTopThreads, (int)kSahOneMax, (int)(kSahOneMax / (kSahMid + 1) + 1), K>(
            S, B, SahPending{T.begin, T.count, T.node, (uint16_t)level, (uint16_t)(level & 1u)}, kSahMid);
    }
}

// A warp (W = 1), or three with an axis each (W = 3), per pending segment of at
// most kSahTiny items, an item a lane.  A split of few items has few distinct
// partitions: each lane tries, on each axis, the boundary above its item's bin
// (the first boundary of every distinct partition is one of these), going over
// the items of its subsegment; no bins are kept, and no barrier is wider than the
// segment's warps.  Same costs, order of candidates and results as the binned
// sweep.  Bound by the latency of the lanes' loops in a small build, where
// three warps shorten them (a tick of 4,096 instances 286 -> 264 us, the four
// medium meshes 1,733 -> 1,721), by issue in a large one, where they repeat
// the rest (400,000 triangles 1,254 -> 1,321 us): see the launch.
constexpr int kTinyBlock = 96;
constexpr uint32_t kSahWideMax = 65536;
template <class K, int W>
__global__ void __launch_bounds__(kTinyBlock) k_sah_tiny(SahBuild B) {
    chain_wait();
    constexpr int A = 3 / W, GROUPS = kTinyBlock / (32 * W);  // axes of a warp, segments of a block
    struct Group {
        int box[2][32][6];               // ordered ints of each position's box (two buffers)
        unsigned long long key[W][32], best[W][32];
        uint32_t prim[2][32];
        uint16_t item[2][32];            // its position in the segment as it came
        uint8_t bin[3][32];
    };
    __shared__ Group sg[GROUPS];
    const uint32_t lane = threadIdx.x & 31u, lt = (1u << lane) - 1u;
    const int warp = (int)(threadIdx.x >> 5), part = W == 1 ? 0 : warp, axis0 = part * A;
    Group& S = sg[W == 1 ? warp : 0];
    const auto sync = [] {
        if (W == 1)
            __syncwarp();
        else
            __syncthreads();
    };
    const uint32_t m = B.cnt[kCntTiny];
    for (uint32_t w = blockIdx.x * GROUPS + (W == 1 ? warp : 0); w < m; w += gridDim.x * GROUPS) {
        const SahPending T = B.tiny[w];
        const bool valid = lane < T.count;
        int cb = 0;
        sync();
        if (part == 0) {
            S.item[0][lane] = (uint16_t)lane;
            if (valid) {
                const uint32_t prim = B.prim[T.buf][T.begin + lane];
                float f[6];
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    f[k] = B.lohi[6 * (size_t)prim + k];
                    S.box[0][lane][k] = f2ord(f[k]);
                }
                S.prim[0][lane] = prim;
                if (has_nan(f)) *B.boxes_done = 0u;
            }
        }
        sync();
        // this lane's subsegment: positions sb .. sb + sc - 1, root node sn
        uint32_t sb = 0, sc = valid && T.count > 1 ? T.count : 0u, sn = T.node;
        for (uint32_t level = T.level;; ++level) {
            const int(*box)[6] = S.box[cb];
            if (sc == 2) {
                if (part == 0 && lane == sb) {
                    float l[6], r[6];
#pragma unroll
                    for (int k = 0; k < 6; ++k) {
                        l[k] = ord2f(box[lane][k]);
                        r[k] = ord2f(box[lane + 1][k]);
                    }
                    emit_sah_node(sn, T.begin + sb, 2, 1, B.n, B.nodes, B.parents, B.ranges);
                    put_child_boxes(B.nodes, sn, l, r);
                }
                sc = 0;
            }
            if (sc >= 3 && level >= kSahMaxLevels) {
                if (part == 0 && lane == sb) {
                    const LocalKeys<K> ks{static_cast<const K*>(B.key[T.buf]) + T.begin, S.item[cb] + sb};
                    for (uint32_t i = 0; i + 1 < sc; ++i)
                        karras_node(ks, sc, (int64_t)i, reinterpret_cast<uint32_t*>(B.nodes) + 12, 16, B.parents,
                                    B.ranges, sn, T.begin + sb, B.n);
                    *B.boxes_done = 0u;
                }
                sc = 0;
            }
            const bool active = sc >= 3;
            if (!__any_sync(0xFFFFFFFFu, active)) break;  // (the same in all the segment's warps)
            // per axis: the frame of the subsegment, and this item's bin
            int bin[A];
#pragma unroll
            for (int q = 0; q < A; ++q) {
                const int axis = axis0 + q;
                int mn = ord_inf(), mx = ord_ninf();
                for (uint32_t j = sb; j < sb + sc; ++j) {
                    const int c = f2ord(__fmul_rn(0.5f, __fadd_rn(ord2f(box[j][axis]), ord2f(box[j][3 + axis]))));
                    mn = min(mn, c);
                    mx = max(mx, c);
                }
                const float cmin = ord2f(mn);
                bin[q] = 0;
                if (active)
                    bin[q] = bin_of(__fmul_rn(0.5f, __fadd_rn(ord2f(box[lane][axis]), ord2f(box[lane][3 + axis]))),
                                    cmin, bin_scale(cmin, ord2f(mx)));
                S.bin[axis][lane] = (uint8_t)bin[q];
            }
            __syncwarp();
            // both sides of this item's boundary on each axis
            int lb[A][6], rb[A][6];
            uint32_t nl[A];
#pragma unroll
            for (int q = 0; q < A; ++q) {
                nl[q] = 0;
#pragma unroll
                for (int k = 0; k < 6; ++k) lb[q][k] = rb[q][k] = k < 3 ? ord_inf() : ord_ninf();
            }
            for (uint32_t j = sb; j < sb + sc; ++j) {
                int v[6];
#pragma unroll
                for (int k = 0; k < 6; ++k) v[k] = box[j][k];
#pragma unroll
                for (int q = 0; q < A; ++q) {
                    const bool l = (int)S.bin[axis0 + q][j] <= bin[q];
                    nl[q] += l;
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        if (l) {
                            lb[q][k] = min(lb[q][k], v[k]);
                            lb[q][3 + k] = max(lb[q][3 + k], v[3 + k]);
                        } else {
                            rb[q][k] = min(rb[q][k], v[k]);
                            rb[q][3 + k] = max(rb[q][3 + k], v[3 + k]);
                        }
                    }
                }
            }
            unsigned long long mine = ~0ull;
#pragma unroll
            for (int q = 0; q < A; ++q) {
                if (nl[q] == 0 || nl[q] >= sc) continue;
                float l[6], r[6];
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    l[k] = ord2f(lb[q][k]);
                    r[k] = ord2f(rb[q][k]);
                }
                const float cost = __fadd_rn(__fadd_rn(__fmul_rn(half_area(l, l + 3), (float)nl[q]),
                                                       __fmul_rn(half_area(r, r + 3), (float)(sc - nl[q]))),
                                             0.0f);
                if (!(cost < INFINITY)) continue;
                const unsigned long long key = split_key(cost, axis0 + q, bin[q] + 1);
                mine = key < mine ? key : mine;
            }
            S.key[part][lane] = mine;
            __syncwarp();
            unsigned long long best = ~0ull;
            for (uint32_t j = sb; j < sb + sc; ++j) best = S.key[part][j] < best ? S.key[part][j] : best;
            S.best[part][lane] = best;
            sync();
#pragma unroll
            for (int a = 0; a < W; ++a) best = S.best[a][lane] < best ? S.best[a][lane] : best;
            const bool cut = active && best != ~0ull;
            const int ax = cut ? (int)((uint32_t)best / (kSahBins - 1)) : 0;
            const int split = (int)((uint32_t)best % (kSahBins - 1)) + 1;
            const bool left = active && (cut ? (int)S.bin[ax][lane] < split : lane - sb < sc / 2);
            const uint32_t seg = active ? (0xFFFFFFFFu >> (32u - sc)) << sb : 0u;
            const uint32_t bal = __ballot_sync(0xFFFFFFFFu, left) & seg;
            const uint32_t own = __ballot_sync(0xFFFFFFFFu, cut && mine == best) & seg;
            const uint32_t nleft = (uint32_t)__popc(bal);
            if (cut && mine == best && (own & lt) == 0u) {  // (a key names its axis: one warp has it)
                float l[6], r[6];
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    int x = lb[0][k], y = rb[0][k];
#pragma unroll
                    for (int q = 1; q < A; ++q)
                        if (ax == q) {
                            x = lb[q][k];
                            y = rb[q][k];
                        }
                    l[k] = ord2f(x);
                    r[k] = ord2f(y);
                }
                put_child_boxes(B.nodes, sn, l, r);
            }
            uint32_t dest = lane;
            if (active) {
                if (part == 0 && lane == sb) {
                    emit_sah_node(sn, T.begin + sb, sc, nleft, B.n, B.nodes, B.parents, B.ranges);
                    if (!cut) *B.boxes_done = 0u;
                }
                const uint32_t lr = (uint32_t)__popc(bal & lt);
                dest = left ? sb + lr : sb + nleft + ((lane - sb) - lr);
            }
#pragma unroll
            for (int c = 0; c < 2 * A; ++c) S.box[cb ^ 1][dest][2 * axis0 + c] = box[lane][2 * axis0 + c];
            if (part == 0) S.prim[cb ^ 1][dest] = S.prim[cb][lane];
            if (part == W - 1) S.item[cb ^ 1][dest] = S.item[cb][lane];
            cb ^= 1;
            sync();
            if (active) {
                if (lane - sb < nleft) {
                    sc = nleft;
                    sn = sn + 1;
                } else {
                    sb += nleft;
                    sc -= nleft;
                    sn += nleft;
                }
                if (sc < 2) sc = 0;
            }
        }
        if (valid && part == 0) B.prim[0][T.begin + lane] = S.prim[cb][lane];
    }
}

template <class K>
cudaError_t set_block_smem() {
    cudaError_t e = cudaFuncSetAttribute(k_sah_block<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BlockMid));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_sah_rest<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BlockTop));
    return e;
}

rg_status sah_cuda_fail(cudaError_t e, const char* what) {
    cudaGetLastError();  // clear a sticky launch error
    return report_error(e == cudaErrorMemoryAllocation ? RG_ERR_OOM : RG_ERR_CUDA,
                        (std::string(what) + ": " + cudaGetErrorString(e)).c_str());
}

#define SAH_CK(call)                                             \
    do {                                                         \
        cudaError_t e_ = (call);                                 \
        if (e_ != cudaSuccess) return sah_cuda_fail(e_, #call);  \
    } while (0)

template <class K>
rg_status sah_build(SahBuild B, const int* cb_ord, cudaStream_t s) {
    // a bit per device, for the attribute holds for the current one only
    // (concurrent first callers set the same values; devices past 63 set them each time)
    static std::atomic<uint64_t> attr_set{0};
    int dev = 0;
    SAH_CK(cudaGetDevice(&dev));
    const uint64_t bit = dev < 64 ? 1ull << dev : 0ull;
    if (!(attr_set.load(std::memory_order_acquire) & bit)) {
        SAH_CK(set_block_smem<K>());
        attr_set.fetch_or(bit, std::memory_order_release);
    }
    const uint32_t n = B.n, sms = (uint32_t)device_sm_count();
    const uint32_t chunks = (n + kSahChunk - 1) / kSahChunk;
    launch_chain(k_sah_start, std::min(chunks / 512u + 1u, 1024u), 512, 0, s, B, cb_ord);
    count_launches(1);
    const uint32_t max_tasks = n / (kSahMid + 1) + 1;
    auto run_level = [&](uint32_t level) {
        const uint32_t tasks = level < 31 ? std::min(1u << level, max_tasks) : max_tasks;
        const uint32_t blocks = n / kSahChunk + tasks;
        launch_chain(k_sah_bin, blocks, kSahBlock, 0, s, B, level);
        launch_chain(k_sah_split, tasks, kSplitBlock, 0, s, B, level);
        launch_chain(k_sah_scatter<K>, blocks, kSahBlock, 0, s, B, level);
        count_launches(3);
    };
    // levels for a balanced tree and one more; then the host looks whether
    // large segments are left (small builds leave that to the device)
    uint32_t levels = 0;
    if (n > kSahMid) {
        for (uint32_t c = n; c > kSahMid; c = (c + 1) / 2) ++levels;
        ++levels;
        for (uint32_t l = 0; l < levels; ++l) run_level(l);
    }
    if (n > kSahOneMax) {
        uint32_t h[kCntAll];
        for (;;) {
            SAH_CK(cudaMemcpyAsync(h, B.cnt, sizeof h, cudaMemcpyDeviceToHost, s));
            SAH_CK(cudaStreamSynchronize(s));
            if (levels >= kSahMaxLevels || h[4 * levels] == 0) break;
            const uint32_t more = std::min(levels + 4, kSahMaxLevels);
            for (; levels < more; ++levels) run_level(levels);
        }
        if (h[kCntKarras]) {  // segments of more than kSahMid items at the depth cap
            std::vector<KarrasSeg> segs(h[kCntKarras]);
            SAH_CK(cudaMemcpyAsync(segs.data(), B.karras, segs.size() * sizeof(KarrasSeg), cudaMemcpyDeviceToHost, s));
            SAH_CK(cudaStreamSynchronize(s));
            uint32_t threads = 0;
            for (KarrasSeg& g : segs) {
                g.first = threads;
                threads += g.count - 1;
            }
            SAH_CK(cudaMemcpyAsync(B.karras, segs.data(), segs.size() * sizeof(KarrasSeg), cudaMemcpyHostToDevice, s));
            SAH_CK(launch_karras_segments(B.key[0], 8 * (int)sizeof(K), B.karras, (uint32_t)segs.size(), threads, n,
                                          B.nodes, B.parents, B.ranges, s));
            SAH_CK(cudaStreamSynchronize(s));  // segs is this frame's
        }
    } else if (n > kSahMid) {
        launch_chain(k_sah_rest<K>, std::min(max_tasks, sms), kTopThreads, sizeof(BlockTop), s, B, levels);
        count_launches(1);
    }
    if (n > kSahTiny) {
        launch_chain(k_sah_block<K>, std::min(n / (kSahTiny + 1) + 1, 4 * sms), kMidThreads, sizeof(BlockMid), s, B);
        count_launches(1);
    }
    // three warps per segment while the chip holds all segments at once that way
    if (n <= kSahWideMax)
        launch_chain(k_sah_tiny<K, 3>, std::min(n / 16u + 1u, 16 * sms), kTinyBlock, 0, s, B);
    else
        launch_chain(k_sah_tiny<K, 1>, 8 * sms, kTinyBlock, 0, s, B);
    count_launches(1);
    SAH_CK(cudaGetLastError());
    return RG_OK;
}

}  // namespace

rg_status sah_topology(const ScratchAlloc& tmp, const float* lohi, uint32_t n, const int* cb_ord, int bits, float4* nodes,
                       uint32_t* perm, uint32_t* parents, cudaStream_t s, uint32_t* ranges, uint32_t* boxes_done) {
    const int key_bits = bits == 21 ? 64 : 32;
    const size_t kb = key_bits / 8;
    const size_t max_tasks = n > kSahMid ? n / (kSahMid + 1) + 1 : 1, max_blocks = n / kSahChunk + max_tasks;
    // every split leaves at most two pending segments, each of its own items
    const size_t max_tiny = n, max_mid = n / (kSahTiny + 1) + 1;
    // one allocation, its parts 256-byte aligned
    size_t total = 0;
    auto part = [&](size_t bytes) {
        const size_t at = total;
        total += (bytes + 255) & ~(size_t)255;
        return at;
    };
    const size_t o_codes = part(n * kb), o_sorted = part(n * kb), o_sort = part(radix_sort_scratch_bytes(n, key_bits));
    const size_t o_prim = part(n * 4ull), o_key = part(n * kb), o_cnt = part(kCntAll * 4);
    const size_t o_tasks = part(2 * max_tasks * sizeof(SahTask)), o_blk = part(2 * max_blocks * sizeof(uint2));
    const size_t o_acc = part(2 * max_tasks * kAcc * 4), o_split = part(max_tasks * sizeof(SahSplit));
    const size_t o_bc = part(max_blocks * 3 * kSahBins * 4), o_bo = part(max_blocks * 4);
    const size_t o_mid = part(max_mid * sizeof(SahPending)), o_tiny = part(max_tiny * sizeof(SahPending));
    const size_t o_karras = part(2 * max_tasks * sizeof(KarrasSeg));
    void* mem;
    rg_status r;
    if ((r = tmp.get(tmp.ctx, &mem, total, "SAH build scratch"))) return r;
    char* m = static_cast<char*>(mem);
    SAH_CK(launch_morton(lohi, n, cb_ord, bits, m + o_codes, nullptr, s));
    SAH_CK(radix_sort_pairs(m + o_codes, nullptr, n, key_bits, m + o_sorted, perm, m + o_sort, s));
    SahBuild B{};
    B.lohi = lohi;
    B.n = n;
    B.prim[0] = perm;
    B.prim[1] = reinterpret_cast<uint32_t*>(m + o_prim);
    B.key[0] = m + o_sorted;
    B.key[1] = m + o_key;
    B.cnt = reinterpret_cast<uint32_t*>(m + o_cnt);
    for (int k = 0; k < 2; ++k) {
        B.tasks[k] = reinterpret_cast<SahTask*>(m + o_tasks) + k * max_tasks;
        B.blk[k] = reinterpret_cast<uint2*>(m + o_blk) + k * max_blocks;
        B.acc[k] = reinterpret_cast<int*>(m + o_acc) + k * max_tasks * kAcc;
    }
    B.split = reinterpret_cast<SahSplit*>(m + o_split);
    B.blk_cnt = reinterpret_cast<uint32_t*>(m + o_bc);
    B.blk_off = reinterpret_cast<uint32_t*>(m + o_bo);
    B.mid = reinterpret_cast<SahPending*>(m + o_mid);
    B.tiny = reinterpret_cast<SahPending*>(m + o_tiny);
    B.karras = reinterpret_cast<KarrasSeg*>(m + o_karras);
    B.nodes = nodes;
    B.parents = parents;
    B.ranges = ranges;
    B.boxes_done = boxes_done;
    return key_bits == 64 ? sah_build<uint64_t>(B, cb_ord, s) : sah_build<uint32_t>(B, cb_ord, s);
}

}  // namespace rg
