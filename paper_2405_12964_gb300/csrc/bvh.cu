// Linear BVH over boundary elements, built on the device:
//   element boxes + scene bounds -> Morton codes -> radix sort (CUB) ->
//   binary radix tree (Karras, "Maximizing parallelism in the construction of
//   BVHs, octrees and k-d trees", HPG 2012) -> leaf primitives written in Morton
//   order -> boxes over the nodes' ranges of leaves -> wide tree collapsed from the
//   binary one (2D: 32 axis-aligned slots, 3D: 8 oriented ones).
// Plus the batched closest-point, ray-parity inside test and Philox kernels.
#include <cub/device/device_radix_sort.cuh>

#include <cstring>

#include "dwos_device.cuh"
#include "dwos_internal.h"

namespace dwos {

namespace {

__device__ __forceinline__ unsigned int float_to_ordered(float f) {
    const unsigned int u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ordered_to_float(unsigned int u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

template <int DIM>
__device__ __forceinline__ void elem_box(const float* vert, const int* elem, int e, float* lo, float* hi) {
#pragma unroll
    for (int k = 0; k < DIM; ++k) { lo[k] = kInf; hi[k] = -kInf; }
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        const int v = elem[DIM * e + a];
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            const float x = vert[DIM * v + k];
            lo[k] = fminf(lo[k], x);
            hi[k] = fmaxf(hi[k], x);
        }
    }
}

template <int DIM>
__device__ __forceinline__ float elem_diag(const float* vert, const int* elem, int e) {
    float lo[DIM], hi[DIM];
    elem_box<DIM>(vert, elem, e, lo, hi);
    float s = 0.0f;
#pragma unroll
    for (int k = 0; k < DIM; ++k) s += (hi[k] - lo[k]) * (hi[k] - lo[k]);
    return sqrtf(s);
}

// Sum of element box diagonals (stats[0]) for the mean size.
template <int DIM>
__global__ void size_kernel(const float* vert, const int* elem, int n, float* stats) {
    float s = 0.0f;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x)
        s += elem_diag<DIM>(vert, elem, e);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(stats, s);
}

// Elements whose box diagonal exceeds kBigFactor x the mean: count (stats[1]).
constexpr float kBigFactor = 16.0f;

// Also the largest half box diagonal over the elements that stay in the tree
// (stats_i[1]) and over all elements (stats_i[2]), as float bits.
template <int DIM>
__global__ void count_big_kernel(const float* vert, const int* elem, int n, float* stats, int* count) {
    const float thr = kBigFactor * stats[0] / (float)n;
    int c = 0;
    float r_small = 0.0f, r_all = 0.0f;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        const float dgn = elem_diag<DIM>(vert, elem, e);
        const bool big = dgn > thr;
        c += big ? 1 : 0;
        r_all = fmaxf(r_all, 0.5f * dgn);
        if (!big) r_small = fmaxf(r_small, 0.5f * dgn);
    }
    for (int o = 16; o > 0; o >>= 1) {
        c += __shfl_xor_sync(0xffffffffu, c, o);
        r_small = fmaxf(r_small, __shfl_xor_sync(0xffffffffu, r_small, o));
        r_all = fmaxf(r_all, __shfl_xor_sync(0xffffffffu, r_all, o));
    }
    if ((threadIdx.x & 31) == 0) {
        if (c) atomicAdd(count, c);
        atomicMax(count + 1, __float_as_int(r_small));   // non-negative floats order as ints
        atomicMax(count + 2, __float_as_int(r_all));
    }
}

// Scene bounds of the tree elements' centroids (ordered-uint encoding).
template <int DIM>
__global__ void bounds_kernel(const float* vert, const int* elem, int n, const float* stats, int split,
                              unsigned int* bounds) {
    const float thr = split ? kBigFactor * stats[0] / (float)n : kInf;
    float lo[DIM], hi[DIM];
#pragma unroll
    for (int k = 0; k < DIM; ++k) { lo[k] = kInf; hi[k] = -kInf; }
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        float l[DIM], h[DIM];
        elem_box<DIM>(vert, elem, e, l, h);
        float d2 = 0.0f;
#pragma unroll
        for (int k = 0; k < DIM; ++k) d2 += (h[k] - l[k]) * (h[k] - l[k]);
        if (sqrtf(d2) > thr) continue;
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            const float c = 0.5f * (l[k] + h[k]);
            lo[k] = fminf(lo[k], c);
            hi[k] = fmaxf(hi[k], c);
        }
    }
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        for (int o = 16; o > 0; o >>= 1) {
            lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], o));
            hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], o));
        }
    }
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            atomicMin(bounds + k, float_to_ordered(lo[k]));
            atomicMax(bounds + DIM + k, float_to_ordered(hi[k]));
        }
    }
}

__device__ __forceinline__ unsigned int spread2(unsigned int x) {   // 16 bits -> even bits
    x &= 0xffffu;
    x = (x | (x << 8)) & 0x00ff00ffu;
    x = (x | (x << 4)) & 0x0f0f0f0fu;
    x = (x | (x << 2)) & 0x33333333u;
    x = (x | (x << 1)) & 0x55555555u;
    return x;
}
__device__ __forceinline__ unsigned int spread3(unsigned int x) {   // 10 bits -> every third bit
    x &= 0x3ffu;
    x = (x | (x << 16)) & 0x030000ffu;
    x = (x | (x << 8)) & 0x0300f00fu;
    x = (x | (x << 4)) & 0x030c30c3u;
    x = (x | (x << 2)) & 0x09249249u;
    return x;
}

// 30-bit Morton code of the centroid (15 bits per axis in 2D, 10 in 3D);
// outsized elements get 0xFFFFFFFF so that the sort puts them last, in index order.
template <int DIM>
__global__ void morton_kernel(const float* vert, const int* elem, int n, const unsigned int* bounds,
                              const float* stats, int split, unsigned int* keys, int* vals) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    vals[e] = e;
    float l[DIM], h[DIM];
    elem_box<DIM>(vert, elem, e, l, h);
    float d2 = 0.0f;
#pragma unroll
    for (int k = 0; k < DIM; ++k) d2 += (h[k] - l[k]) * (h[k] - l[k]);
    if (split && sqrtf(d2) > kBigFactor * stats[0] / (float)n) { keys[e] = 0xFFFFFFFFu; return; }
    unsigned int q[DIM];
    const float levels = DIM == 2 ? 32767.0f : 1023.0f;
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        const float lo = ordered_to_float(bounds[k]);
        const float hi = ordered_to_float(bounds[DIM + k]);
        const float ext = hi - lo;
        float t = ext > 0.0f ? (0.5f * (l[k] + h[k]) - lo) / ext : 0.5f;
        t = fminf(fmaxf(t, 0.0f), 1.0f);
        q[k] = (unsigned int)(t * levels + 0.5f);
    }
    keys[e] = DIM == 2 ? (spread2(q[0]) | (spread2(q[1]) << 1))
                       : (spread3(q[0]) | (spread3(q[1]) << 1) | (spread3(q[2]) << 2));
}

// Length of the common prefix of keys i and j, with the index as tie-breaker;
// -1 outside [0, n).
__device__ __forceinline__ int delta(const unsigned int* k, int n, int i, int j) {
    if (j < 0 || j >= n) return -1;
    const unsigned int a = k[i], b = k[j];
    if (a == b) return 32 + __clz((unsigned int)(i ^ j));
    return __clz(a ^ b);
}

// Box of centroids admitted by a Morton prefix: the top p bits of the 30-bit
// code fix the top bits of each axis; q = floor(t * levels + 0.5) lies in
// [q_lo, q_hi] iff t lies in [(q_lo - 0.5)/levels, (q_hi + 0.5)/levels).
template <int DIM>
__device__ void morton_cell(unsigned int key, int p, const unsigned int* bounds, float* cell) {
    const int B = DIM == 2 ? 15 : 10;
    const float levels = DIM == 2 ? 32767.0f : 1023.0f;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        int n_a = 0;
        for (int b = 29; b >= 30 - p; --b) n_a += (b % DIM == a) ? 1 : 0;
        unsigned int q = 0;
        for (int k = 0; k < B; ++k) q |= ((key >> (DIM * k + a)) & 1u) << k;
        const unsigned int q_lo = n_a > 0 ? ((q >> (B - n_a)) << (B - n_a)) : 0u;
        const unsigned int q_hi = q_lo + (1u << (B - n_a)) - 1u;
        const float lo = ordered_to_float(bounds[a]);
        const float ext = ordered_to_float(bounds[DIM + a]) - lo;
        if (!(ext > 0.0f)) {              // flat axis: the code does not separate along it
            cell[a] = -kInf;
            cell[DIM + a] = kInf;
            continue;
        }
        cell[a] = lo + (((float)q_lo - 0.5f) / levels) * ext;
        cell[DIM + a] = lo + (((float)q_hi + 0.5f) / levels) * ext;
    }
}

template <int DIM>
__global__ void radix_tree_kernel(const unsigned int* keys, int n, int* node_child, int* node_parent,
                                  int* leaf_parent, const unsigned int* bounds, float* node_cell, int* node_count,
                                  int* node_first) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n - 1) return;
    const int dir = (delta(keys, n, i, i + 1) - delta(keys, n, i, i - 1)) >= 0 ? 1 : -1;
    const int dmin = delta(keys, n, i, i - dir);
    int lmax = 2;
    while (delta(keys, n, i, i + lmax * dir) > dmin) lmax <<= 1;
    int l = 0;
    for (int t = lmax >> 1; t >= 1; t >>= 1)
        if (delta(keys, n, i, i + (l + t) * dir) > dmin) l += t;
    const int j = i + l * dir;
    const int dnode = delta(keys, n, i, j);
    int s = 0, t = l;
    do {
        t = (t + 1) >> 1;
        if (delta(keys, n, i, i + (s + t) * dir) > dnode) s += t;
    } while (t > 1);
    const int split = i + s * dir + min(dir, 0);
    const int first = min(i, j), last = max(i, j);
    node_count[i] = last - first + 1;               // leaves under node i: first .. last
    node_first[i] = first;
    int left, right;
    if (first == split) { left = ~split; leaf_parent[split] = i; }
    else { left = split; node_parent[split] = i; }
    if (last == split + 1) { right = ~(split + 1); leaf_parent[split + 1] = i; }
    else { right = split + 1; node_parent[split + 1] = i; }
    node_child[2 * i] = left;
    node_child[2 * i + 1] = right;
    if (i == 0) node_parent[0] = -1;
    // keys of this node's range share dnode leading bits (>= 32: all equal)
    const int p = dnode >= 32 ? 30 : dnode - 2;
    morton_cell<DIM>(keys[i], p, bounds, node_cell + 2 * DIM * i);
}

template <int DIM>
__device__ __forceinline__ void write_child_box(float4* nodes, int node, int slot, const float* lo,
                                                const float* hi) {
    float* f = reinterpret_cast<float*>(nodes + BvhLayout<DIM>::kNodeF4 * node);
    if (DIM == 2) {
        float* b = f + 4 * slot;
        b[0] = lo[0]; b[1] = lo[1]; b[2] = hi[0]; b[3] = hi[1];
    } else {
        float* b = f + 6 * slot;
        b[0] = lo[0]; b[1] = lo[1]; b[2] = lo[2]; b[3] = hi[0]; b[4] = hi[1]; b[5] = hi[2];
    }
}

// ---- boxes ----------------------------------------------------------------
// A node's box is the union over its contiguous range of leaves.  Climbing from every
// leaf with an arrival counter per node, a fence and an atomic per level, the boxes of
// 4,100 segments took 35 us, all of it the chain of a dozen dependent levels.  Instead
// one launch writes the leaves and the boxes of their aligned blocks of 8, 64 and 512,
// and a second covers each node's range by at most seven leaves or blocks on each side
// per level, all loaded independently: 9 us.
constexpr int kLeafBlock = 512;      // leaves of a block, and of the highest level's boxes

// Box k of level 1..3 (8, 64, 512 leaves) among nt leaves.
template <int DIM>
__device__ __forceinline__ float4* level_box(float4* boxes, int nt, int level, int k) {
    const int n8 = (nt + 7) / 8, n64 = (nt + 63) / 64;
    return boxes + (DIM == 2 ? 1 : 2) * ((level > 1 ? n8 : 0) + (level > 2 ? n64 : 0) + (size_t)k);
}
__host__ inline size_t level_boxes(size_t n) { return (n + 7) / 8 + (n + 63) / 64 + (n + 511) / 512; }

template <int DIM>
__device__ __forceinline__ void store_level_box(float4* b, const float* lo, const float* hi) {
    if (DIM == 2) {
        *b = make_float4(lo[0], lo[1], hi[0], hi[1]);
    } else {
        b[0] = make_float4(lo[0], lo[1], lo[DIM - 1], 0.0f);
        b[1] = make_float4(hi[0], hi[1], hi[DIM - 1], 0.0f);
    }
}
template <int DIM>
__device__ __forceinline__ void add_level_box(const float4* b, float* lo, float* hi) {
    const float4 p = __ldg(b);
    const float4 q = DIM == 2 ? make_float4(p.z, p.w, 0.0f, 0.0f) : __ldg(b + 1);
    lo[0] = fminf(lo[0], p.x); lo[1] = fminf(lo[1], p.y);
    hi[0] = fmaxf(hi[0], q.x); hi[1] = fmaxf(hi[1], q.y);
    if (DIM == 3) { lo[DIM - 1] = fminf(lo[DIM - 1], p.z); hi[DIM - 1] = fmaxf(hi[DIM - 1], q.z); }
}

// Union over groups of eight lanes.
template <int DIM>
__device__ __forceinline__ void union8(unsigned mask, float* lo, float* hi) {
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            lo[k] = fminf(lo[k], __shfl_xor_sync(mask, lo[k], o));
            hi[k] = fmaxf(hi[k], __shfl_xor_sync(mask, hi[k], o));
        }
    }
}

// The leaves (vertices, elements), the nodes' links and, over the nt >= 2 leaves of a
// tree, the leaves' own boxes in their parents and the level boxes.
template <int DIM>
__global__ void __launch_bounds__(kLeafBlock)
    leaves_kernel(const float* vert, const int* elem, const int* sorted_elem, int n, int nt, const int* node_child,
                  const int* node_parent, const int* leaf_parent, float4* nodes, float4* prims, int* prim_elem,
                  int* leaf_of_elem, float4* boxes) {
    const int i = blockIdx.x * kLeafBlock + threadIdx.x, t = threadIdx.x;
    const bool tree = nt >= 2;
    if (tree && i < nt - 1) {
        float4* m = nodes + BvhLayout<DIM>::kNodeF4 * i + (BvhLayout<DIM>::kNodeF4 - 1);
        *m = make_float4(__int_as_float(node_child[2 * i]), __int_as_float(node_child[2 * i + 1]),
                         __int_as_float(node_parent[i]), 0.0f);
    }
    float lo[DIM], hi[DIM];
#pragma unroll
    for (int k = 0; k < DIM; ++k) { lo[k] = kInf; hi[k] = -kInf; }
    if (i < n) {
        const int e = sorted_elem[i];
        prim_elem[i] = e;
        leaf_of_elem[e] = i;
        if (DIM == 2) {
            const int a = elem[2 * e], b = elem[2 * e + 1];
            prims[i] = make_float4(vert[2 * a], vert[2 * a + 1], vert[2 * b], vert[2 * b + 1]);
        } else {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int v = elem[3 * e + c];
                prims[3 * i + c] = make_float4(vert[3 * v], vert[3 * v + 1], vert[3 * v + 2], 0.0f);
            }
        }
        if (tree && i < nt) {
            elem_box<DIM>(vert, elem, e, lo, hi);
            const int parent = leaf_parent[i];
            write_child_box<DIM>(nodes, parent, node_child[2 * parent] == ~i ? 0 : 1, lo, hi);
        }
    }
    if (!tree || blockIdx.x * kLeafBlock >= nt) return;      // whole blocks
    __shared__ float sb[kLeafBlock / 8][2 * DIM];
    union8<DIM>(0xffffffffu, lo, hi);
    auto put = [&](int level, int k, int slot) {
        if (k * (level == 1 ? 8 : level == 2 ? 64 : 512) < nt) store_level_box<DIM>(level_box<DIM>(boxes, nt, level, k), lo, hi);
#pragma unroll
        for (int j = 0; j < DIM; ++j) { sb[slot][j] = lo[j]; sb[slot][DIM + j] = hi[j]; }
    };
    auto get = [&](int slot) {
#pragma unroll
        for (int j = 0; j < DIM; ++j) { lo[j] = sb[slot][j]; hi[j] = sb[slot][DIM + j]; }
    };
    if (t % 8 == 0) put(1, i / 8, t / 8);
    __syncthreads();
    if (t < 64) {
        get(t);
        union8<DIM>(0xffffffffu, lo, hi);
    }
    __syncthreads();
    if (t < 64 && t % 8 == 0) put(2, blockIdx.x * 8 + t / 8, t / 8);
    __syncthreads();
    if (t < 8) {
        get(t);
        union8<DIM>(0xffu, lo, hi);
        if (t == 0) store_level_box<DIM>(level_box<DIM>(boxes, nt, 3, blockIdx.x), lo, hi);
    }
}

// The inner nodes' boxes in their parents: eight lanes to a node.
template <int DIM>
__global__ void node_boxes_kernel(const float4* prims, float4* boxes, int nt, const int* node_child,
                                  const int* node_parent, const int* node_count, const int* node_first,
                                  float4* nodes) {
    const int c = (blockIdx.x * blockDim.x + threadIdx.x) / 8 + 1, j = threadIdx.x % 8;   // the root has no parent
    float lo[DIM], hi[DIM];
#pragma unroll
    for (int k = 0; k < DIM; ++k) { lo[k] = kInf; hi[k] = -kInf; }
    if (c < nt - 1) {
        int a = node_first[c], b = a + node_count[c];
        auto add = [&](int level, int k) {
            if (level == 0) {
                float l[DIM], h[DIM];
                prim_box<DIM>(prims, k, l, h);
#pragma unroll
                for (int q = 0; q < DIM; ++q) { lo[q] = fminf(lo[q], l[q]); hi[q] = fmaxf(hi[q], h[q]); }
            } else {
                add_level_box<DIM>(level_box<DIM>(boxes, nt, level, k), lo, hi);
            }
        };
#pragma unroll
        for (int level = 0; level < 4; ++level) {
            const int na = (a + 7) >> 3, nb = b >> 3;
            if (level == 3 || na >= nb) {
                for (int k = a + j; k < b; k += 8) add(level, k);
                break;
            }
            if (a + j < 8 * na) add(level, a + j);
            if (8 * nb + j < b) add(level, 8 * nb + j);
            a = na;
            b = nb;
        }
    }
    __syncwarp();
    union8<DIM>(0xffffffffu, lo, hi);
    if (c < nt - 1 && j == 0) {
        const int parent = node_parent[c];
        write_child_box<DIM>(nodes, parent, node_child[2 * parent] == c ? 0 : 1, lo, hi);
    }
}

// One tree element: a single node whose right child is empty.
template <int DIM>
__global__ void single_leaf_kernel(const float* vert, const int* elem, const int* sorted_elem, float4* nodes,
                                   int* leaf_parent, float* node_cell) {
    leaf_parent[0] = 0;
#pragma unroll
    for (int k = 0; k < DIM; ++k) { node_cell[k] = -kInf; node_cell[DIM + k] = kInf; }
    float lo[DIM], hi[DIM], elo[DIM], ehi[DIM];
    elem_box<DIM>(vert, elem, sorted_elem[0], lo, hi);
#pragma unroll
    for (int k = 0; k < DIM; ++k) { elo[k] = kInf; ehi[k] = -kInf; }
    write_child_box<DIM>(nodes, 0, 0, lo, hi);
    write_child_box<DIM>(nodes, 0, 1, elo, ehi);
    nodes[BvhLayout<DIM>::kNodeF4 - 1] =
        make_float4(__int_as_float(~0), __int_as_float(kEmptyChild), __int_as_float(-1), 0.0f);
}

// ---- wide tree --------------------------------------------------------------
// Built top-down, one level per launch.  A wide node starts from its binary
// root's two children; it first opens, largest first, the inner children with
// more than W leaves (they cannot become one leaf-level node), then absorbs
// whole inner children that still fit as their leaves, largest first.  Its
// remaining inner children become the next level's wide nodes.  (Opening
// every child by size alone cuts small subtrees into pieces, each a nearly
// empty wide node: 37 % of 32 slots used on a 32 k-element test set against
// 71 % with this rule.)

// The children of the wide node whose binary root is r: their codes (>= 0: binary
// node, < 0: ~leaf) and the binary tree's slots of their boxes ((parent << 1) |
// side); returns their number.
template <int W>
__device__ __forceinline__ int wide_children(const int* node_child, const int* node_count, const int* node_first,
                                             const int* leaf_parent, int r, int* code, int* src) {
    int cnt = 0;
    for (int side = 0; side < 2; ++side) {
        code[cnt] = node_child[2 * r + side];
        src[cnt] = (r << 1) | side;
        ++cnt;
    }
    auto leaves = [&](int c) { return c >= 0 ? node_count[c] : 1; };
    while (cnt < W) {                          // open the largest child with more than W leaves
        int pick = -1, best = W;
        for (int i = 0; i < cnt; ++i)
            if (code[i] >= 0 && leaves(code[i]) > best) { best = leaves(code[i]); pick = i; }
        if (pick < 0) break;
        const int c = code[pick];
        for (int i = cnt; i > pick + 1; --i) { code[i] = code[i - 1]; src[i] = src[i - 1]; }
        for (int side = 0; side < 2; ++side) {
            code[pick + side] = node_child[2 * c + side];
            src[pick + side] = (c << 1) | side;
        }
        ++cnt;
    }
    while (cnt < W) {                          // absorb the largest inner child that fits
        const int room = W - cnt + 1;
        int pick = -1, best = 0;
        for (int i = 0; i < cnt; ++i)
            if (code[i] >= 0 && leaves(code[i]) <= room && leaves(code[i]) > best) { best = leaves(code[i]); pick = i; }
        if (pick < 0) break;
        const int c = code[pick], k = node_count[c], f = node_first[c];
        for (int i = cnt - 1; i > pick; --i) { code[i + k - 1] = code[i]; src[i + k - 1] = src[i]; }
        for (int t = 0; t < k; ++t) {
            const int leaf = f + t, par = leaf_parent[leaf];
            code[pick + t] = ~leaf;
            src[pick + t] = (par << 1) | (node_child[2 * par] == ~leaf ? 0 : 1);
        }
        cnt += k - 1;
    }
    return cnt;
}

// lev[L]: wide nodes of level L.  A level's kernel reads its own count, which the
// kernel before it finished, so the host enqueues every level without waiting
// and reads the counts once (a copy, a wait and six allocations per level took
// longer than the levels themselves).  Per wide node: its binary root and its first
// inner child's id (the inner children of a node have consecutive ids).  Ids are
// given out by an atomic counter: a node's number varies from build to build, its
// children and their order do not.
template <int W>
__global__ void wide_level_kernel(const int* node_child, const int* node_count, const int* node_first,
                                  const int* leaf_parent, int level, int* lev, int* wroot, int* wnext) {
    int base = 0;
    for (int l = 0; l < level; ++l) base += lev[l];
    const int m = lev[level];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
        int code[W], src[W];
        const int cnt = wide_children<W>(node_child, node_count, node_first, leaf_parent, wroot[base + i], code, src);
        int inner = 0;
        for (int k = 0; k < cnt; ++k) inner += code[k] >= 0 ? 1 : 0;
        int id = base + m + (inner ? atomicAdd(lev + level + 1, inner) : 0);
        wnext[base + i] = id;
        for (int k = 0; k < cnt; ++k)
            if (code[k] >= 0) wroot[id++] = code[k];
    }
}

// Per slot: the child's code in the wide tree and the binary tree's slot of its box (-1:
// unused); per wide node, the slot that holds it.
template <int W>
__global__ void wide_codes_kernel(const int* node_child, const int* node_count, const int* node_first,
                                  const int* leaf_parent, int n_wide, const int* wroot, const int* wnext, int* wcode,
                                  int* wsrc, int* wslot) {
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= n_wide) return;
    int code[W], src[W];
    const int cnt = wide_children<W>(node_child, node_count, node_first, leaf_parent, wroot[w], code, src);
    int id = wnext[w];
    if (w == 0) wslot[0] = -1;
    for (int k = 0; k < W; ++k) {
        const bool in = k < cnt && code[k] >= 0;
        wsrc[W * w + k] = k < cnt ? src[k] : -1;
        if (in) wslot[id] = W * w + k;
        wcode[W * w + k] = in ? id++ : (k < cnt ? code[k] : kEmptyChild);
    }
}

// The 2D tree's slots: inner children's boxes gathered from the binary tree (its refit
// already ran), leaf children's segments, and the codes.
__global__ void wide_refit_kernel(const float4* nodes, const float4* prims, const int* wsrc, const int* wcode,
                                  int n_wide, float* wnodes) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_wide * kWide) return;
    float* f = wnodes + (size_t)(t / kWide) * kWideFloats;
    const int j = t % kWide, src = wsrc[t], code = wcode[t];
    float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (code < 0) v = prims[~code];
    else if (src >= 0) v = nodes[BvhLayout<2>::kNodeF4 * (src >> 1) + (src & 1)];
    reinterpret_cast<float4*>(f)[j] = v;
    f[4 * kWide + j] = __int_as_float(code);
}

__device__ __forceinline__ float warp_fsum(float v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float warp_fmin(float v) {
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float warp_fmax(float v) { return -warp_fmin(-v); }

// Up to this many leaves a node gets a box oriented by its elements' mean normal;
// above it the axis-aligned box of the binary tree (a patch that large is curved, and
// the pass over its leaves would dominate the refit).  On spheres, limits of 256 / 512 / 1024:
// walk kernel over 50,000 triangles 3.32 / 3.28 / 3.41 ms, 200,000 12.80 / 12.90 / 13.06;
// this kernel 11.7 / 12.6 / 18.1 and 40.0 / 40.3 / 41.1 us.  (64: 18.8 visits per query over
// 200,000 triangles, 1024 15.2, none 15.7.)
constexpr int kOrientMax = 512;

// Vertex a of triangle leaf p.
__device__ __forceinline__ void leaf_vertex(const float4* prims, int p, int a, float* v) {
    const float4 s = __ldg(prims + 3 * p + a);
    v[0] = s.x; v[1] = s.y; v[2] = s.z;
}

// Its normal, of twice its area's length.
__device__ __forceinline__ void leaf_normal(const float4* prims, int p, float* n) {
    float a[3], b[3], c[3];
    leaf_vertex(prims, p, 0, a);
    leaf_vertex(prims, p, 1, b);
    leaf_vertex(prims, p, 2, c);
    const float u[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]};
    const float v[3] = {c[0] - a[0], c[1] - a[1], c[2] - a[2]};
    n[0] = u[1] * v[2] - u[2] * v[1];
    n[1] = u[2] * v[0] - u[0] * v[2];
    n[2] = u[0] * v[1] - u[1] * v[0];
}

// v over its length; false, with v as it was, without a direction.  (Scaled by the largest
// component first: squares of a small or large mesh's cross products leave FP32's range.)
__device__ __forceinline__ bool unit(float* v) {
    const float m = fmaxf(fabsf(v[0]), fmaxf(fabsf(v[1]), fabsf(v[2])));
    if (!(m > 1e-37f && m < 1e37f)) return false;
    const float r = 1.0f / m, s[3] = {v[0] * r, v[1] * r, v[2] * r};
    const float il = rsqrtf(s[0] * s[0] + s[1] * s[1] + s[2] * s[2]);
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] = s[k] * il;
    return true;
}

// A unit vector t perpendicular to the unit vector n, from the axis least aligned with n.
__device__ __forceinline__ void perpendicular(const float* n, float* t) {
    const float ax = fabsf(n[0]), ay = fabsf(n[1]), az = fabsf(n[2]);
    if (ax <= ay && ax <= az) { t[0] = 0.0f; t[1] = n[2]; t[2] = -n[1]; }
    else if (ay <= az) { t[0] = -n[2]; t[1] = 0.0f; t[2] = n[0]; }
    else { t[0] = n[1]; t[1] = -n[0]; t[2] = 0.0f; }
    const float il = rsqrtf(t[0] * t[0] + t[1] * t[1] + t[2] * t[2]);
#pragma unroll
    for (int k = 0; k < 3; ++k) t[k] *= il;
}

// The frame of the unit normal n (row 0) and the unit tangent t (row 1), perpendicular to
// each other: a box bounds distances only if its rows are orthonormal.
__device__ __forceinline__ void frame_rows(const float* n, const float* t, float (*R)[3]) {
#pragma unroll
    for (int k = 0; k < 3; ++k) { R[0][k] = n[k]; R[1][k] = t[k]; }
    R[2][0] = n[1] * t[2] - n[2] * t[1];
    R[2][1] = n[2] * t[0] - n[0] * t[2];
    R[2][2] = n[0] * t[1] - n[1] * t[0];
}

// A triangle's frame, from its normal n (any length) and first edge t (R as it was without
// one).  The thinner the triangle, the more of n is the cross product's rounding, along t as
// well: what lies along t is taken out (with it left in, boxes of triangles thinner than 1e-3
// of their length exceeded squared distances by up to |n . t|, beyond what the search allows), and
// where little else is left any perpendicular serves.
__device__ __forceinline__ void leaf_frame(float* n, float* t, float (*R)[3]) {
    if (!unit(t)) return;
    const bool ok = unit(n);
    const float d = n[0] * t[0] + n[1] * t[1] + n[2] * t[2];
    if (ok && d * d < 0.5f) {
#pragma unroll
        for (int k = 0; k < 3; ++k) n[k] = fmaf(-d, t[k], n[k]);
        const float il = rsqrtf(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
#pragma unroll
        for (int k = 0; k < 3; ++k) n[k] *= il;
    } else {
        perpendicular(t, n);
    }
    frame_rows(n, t, R);
}

// Row r of a frame times (v - o), in the order of the search's box test.
__device__ __forceinline__ float along(const float* r, const float* v, const float* o) {
    return fmaf(r[0], v[0] - o[0], fmaf(r[1], v[1] - o[1], r[2] * (v[2] - o[2])));
}

// Box slot `slot` (node * kOriented + j): centre c, rows R, half extents h with the
// margin for the rounding of the search's box test (2e-6 of the largest), the code.
__device__ __forceinline__ void store_box(float4* wnodes, int slot, const float* c, const float (*R)[3],
                                          const float* h, int code) {
    const float m = 2e-6f * fmaxf(h[0], fmaxf(h[1], h[2]));
    float4* o = wnodes + (size_t)(slot / kOriented) * kOrientedF4 + slot % kOriented;
    o[0] = make_float4(c[0], c[1], c[2], __int_as_float(code));
#pragma unroll
    for (int k = 0; k < 3; ++k) o[(1 + k) * kOriented] = make_float4(R[k][0], R[k][1], R[k][2], h[k] + m);
}

// The oriented boxes of a 3D tree, one warp per wide node: the node's own box, in its
// parent's slot, and the boxes of its leaf children and empty slots, one per lane.  A
// box's frame is the mean normal of the elements under it (each counted along the
// first one's side; a leaf's own normal and first edge, made perpendicular); its extents are
// taken about its rounded centre, so that only relative rounding is left.
__global__ void oriented_fill_kernel(const float4* nodes, const float4* prims, const int* node_count,
                                     const int* node_first, const int* wcode, const int* wroot, const int* wslot,
                                     int n_wide, float4* wnodes) {
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= n_wide) return;                      // whole warps exit together
    const int my_code = lane < kOriented ? wcode[kOriented * w + lane] : 0;
    if (lane < kOriented && (my_code < 0 || my_code == kEmptyChild)) {
        float c[3] = {0.0f, 0.0f, 0.0f}, h[3] = {0.0f, 0.0f, 0.0f};
        float R[3][3] = {{1.0f, 0.0f, 0.0f}, {0.0f, 1.0f, 0.0f}, {0.0f, 0.0f, 1.0f}};
        if (my_code < 0) {
            float v[3][3], n[3], t[3];
            for (int a = 0; a < 3; ++a) leaf_vertex(prims, ~my_code, a, v[a]);
            leaf_normal(prims, ~my_code, n);
#pragma unroll
            for (int k = 0; k < 3; ++k) t[k] = v[1][k] - v[0][k];
            leaf_frame(n, t, R);
            float m[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                float lo = kInf, hi = -kInf;
                for (int a = 0; a < 3; ++a) {
                    const float y = along(R[k], v[a], v[0]);
                    lo = fminf(lo, y);
                    hi = fmaxf(hi, y);
                }
                m[k] = 0.5f * (lo + hi);
            }
#pragma unroll
            for (int i = 0; i < 3; ++i) c[i] = v[0][i] + (R[0][i] * m[0] + R[1][i] * m[1] + R[2][i] * m[2]);
#pragma unroll
            for (int k = 0; k < 3; ++k)
                for (int a = 0; a < 3; ++a) h[k] = fmaxf(h[k], fabsf(along(R[k], v[a], c)));
        }
        store_box(wnodes, kOriented * w + lane, c, R, h, my_code);
    }
    const int slot = wslot[w];
    if (slot < 0) return;                         // the root is in no slot
    const int b = wroot[w], cnt = node_count[b], first = node_first[b];
    float R[3][3] = {{1.0f, 0.0f, 0.0f}, {0.0f, 1.0f, 0.0f}, {0.0f, 0.0f, 1.0f}};
    float c[3], h[3];
    {                                             // axis-aligned frame and box
        float lo0[3], hi0[3], lo1[3], hi1[3];
        int c0, c1, parent;
        load_node<3>(nodes, b, lo0, hi0, lo1, hi1, c0, c1, parent);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float lo = fminf(lo0[k], lo1[k]), hi = fmaxf(hi0[k], hi1[k]);
            c[k] = 0.5f * (lo + hi);
            h[k] = fmaxf(hi - c[k], c[k] - lo);
        }
    }
    if (cnt <= kOrientMax) {
        float ref[3], n[3] = {0.0f, 0.0f, 0.0f}, area = 0.0f;
        leaf_normal(prims, first, ref);
#pragma unroll 4
        for (int p = first + lane; p < first + cnt; p += 32) {
            float m[3];
            leaf_normal(prims, p, m);
            const float d = m[0] * ref[0] + m[1] * ref[1] + m[2] * ref[2];
#pragma unroll
            for (int k = 0; k < 3; ++k) n[k] += d < 0.0f ? -m[k] : m[k];
            area += sqrtf(m[0] * m[0] + m[1] * m[1] + m[2] * m[2]);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) n[k] = warp_fsum(n[k]);
        area = warp_fsum(area);
        const float len = sqrtf(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
        // a patch whose normals spread too far keeps the axis-aligned box
        if (len > 0.7f * area && area < kInf && unit(n)) {
            float t[3], o[3], lo[3], hi[3];
            perpendicular(n, t);
            frame_rows(n, t, R);
            leaf_vertex(prims, first, 0, o);
#pragma unroll
            for (int k = 0; k < 3; ++k) { lo[k] = kInf; hi[k] = -kInf; }
#pragma unroll 2
            for (int p = first + lane; p < first + cnt; p += 32)
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    float v[3];
                    leaf_vertex(prims, p, a, v);
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        const float y = along(R[k], v, o);
                        lo[k] = fminf(lo[k], y);
                        hi[k] = fmaxf(hi[k], y);
                    }
                }
            float m[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) { m[k] = 0.5f * (warp_fmin(lo[k]) + warp_fmax(hi[k])); h[k] = 0.0f; }
#pragma unroll
            for (int i = 0; i < 3; ++i) c[i] = o[i] + (R[0][i] * m[0] + R[1][i] * m[1] + R[2][i] * m[2]);
#pragma unroll 2
            for (int p = first + lane; p < first + cnt; p += 32)
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    float v[3];
                    leaf_vertex(prims, p, a, v);
#pragma unroll
                    for (int k = 0; k < 3; ++k) h[k] = fmaxf(h[k], fabsf(along(R[k], v, c)));
                }
#pragma unroll
            for (int k = 0; k < 3; ++k) h[k] = warp_fmax(h[k]);
        }
    }
    if (lane == 0) store_box(wnodes, slot, c, R, h, w);
}

// ---- queries --------------------------------------------------------------
template <int DIM>
__global__ void closest_kernel(BvhView bvh, const int* prim_elem, const int* leaf_of_elem, int n, const float* p,
                               const int* hint_elem, float* dist, int* elem_out, float* bary, int* err,
                               DevCounters* ctr) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float q[DIM];
#pragma unroll
    for (int k = 0; k < DIM; ++k) q[k] = p[DIM * i + k];
    float best2 = kInf;
    int best = -1;
    if (hint_elem) {   // seed with the caller's element, as a walk seeds with its previous hit
        const int h = hint_elem[i];
        if (h >= 0 && h < bvh.n_tree + bvh.n_big) {
            best = leaf_of_elem[h];
            best2 = prim_dist2<DIM>(bvh.prims, best, q);
        }
    }
    unsigned nn = 0, np = 0;
    if (!closest_leaf<DIM>(bvh, q, best2, best, nn, np)) atomicOr(err, 1);
    if (ctr) {
        atomicAdd(&ctr->nodes, (unsigned long long)nn);
        atomicAdd(&ctr->prims, (unsigned long long)np);
    }
    float w1 = 0.0f, w2 = 0.0f;
    if (best >= 0) {
        if (DIM == 2) {
            const float4 s = bvh.prims[best];
            best2 = seg_closest(q, s.x, s.y, s.z, s.w, w1);
        } else {
            const float4 a = bvh.prims[3 * best], b = bvh.prims[3 * best + 1], c = bvh.prims[3 * best + 2];
            best2 = tri_closest(q, make_float3(a.x, a.y, a.z), make_float3(b.x, b.y, b.z),
                                make_float3(c.x, c.y, c.z), w1, w2);
        }
    }
    dist[i] = sqrtf(best2);
    elem_out[i] = best >= 0 ? prim_elem[best] : -1;
    bary[2 * i] = w1;
    bary[2 * i + 1] = w2;
}

// The same query with the warp's search of the wide tree: all lanes of a
// block take part (a lane past n only helps), so there is no early return.
template <int DIM>
__global__ void closest_wide_kernel(BvhView bvh, WideView wv, const int* prim_elem, const int* leaf_of_elem, int n,
                                    const float* p, const int* hint_elem, float* dist, int* elem_out, float* bary,
                                    int* err, DevCounters* ctr, int stk_cap) {
    extern __shared__ float2 wide_stack[];
    float2* stk = wide_stack + (size_t)(threadIdx.x >> 5) * (wide_smem_bytes(DIM, stk_cap) / sizeof(float2));
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const bool act = i < n;
    float q[DIM];
#pragma unroll
    for (int k = 0; k < DIM; ++k) q[k] = act ? p[DIM * i + k] : 0.0f;
    float best2 = kInf;
    int best = -1;
    unsigned nn = 0, np = 0;
    if (act) {
        if (hint_elem) {
            const int h = hint_elem[i];
            if (h >= 0 && h < bvh.n_tree + bvh.n_big) {
                best = leaf_of_elem[h];
                best2 = prim_dist2<DIM>(bvh.prims, best, q);
            }
        }
        big_closest<DIM>(bvh.prims, bvh.n_tree, bvh.n_big, q, best2, best, np);
    }
    const int e = wide_search<DIM>(wv, __ballot_sync(kWarpAll, act), q, best2, best, stk, stk_cap, nn, np);
    if (e) atomicOr(err, 1);
    if (ctr) {
        atomicAdd(&ctr->wnodes, (unsigned long long)nn);
        atomicAdd(&ctr->prims, (unsigned long long)np);
    }
    if (!act) return;
    float w1 = 0.0f, w2 = 0.0f;
    if (best >= 0) {
        if (DIM == 2) {
            const float4 s = bvh.prims[best];
            best2 = seg_closest(q, s.x, s.y, s.z, s.w, w1);
        } else {
            const float4 a = bvh.prims[3 * best], b = bvh.prims[3 * best + 1], c = bvh.prims[3 * best + 2];
            best2 = tri_closest(q, make_float3(a.x, a.y, a.z), make_float3(b.x, b.y, b.z),
                                make_float3(c.x, c.y, c.z), w1, w2);
        }
    }
    dist[i] = sqrtf(best2);
    elem_out[i] = best >= 0 ? prim_elem[best] : -1;
    bary[2 * i] = w1;
    bary[2 * i + 1] = w2;
}

// Inside test by ray parity along a fixed generic direction.  The ray from
// each point is cut into 32 sub-intervals [t_s, t_s+1) up to the far corner of
// the scene box; lane s of the point's warp counts the crossings in its
// interval with an any-order traversal (pruning boxes its interval
// misses) plus the outsized elements, and the warp sums the counts.
template <int DIM>
__device__ __forceinline__ bool seg_hits_box(const float* o, const float* inv, float ta, float tb, const float* lo,
                                             const float* hi) {
    float t0 = ta, t1 = tb;
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        const float a = (lo[k] - o[k]) * inv[k], b = (hi[k] - o[k]) * inv[k];
        t0 = fmaxf(t0, fminf(a, b));
        t1 = fminf(t1, fmaxf(a, b));
    }
    // a prefilter only: a ray through a box corner (a shared vertex) must not be
    // rejected by rounding, so the overlap test allows a small relative slack
    return t0 <= t1 + 1e-5f * fmaxf(1.0f, fabsf(t1));
}

// Ray parameter of the crossing with leaf p, or -1.  Watertight: a crossing
// through a vertex or edge shared by two elements is counted exactly once.
//  2D: crossing-number rule; each vertex's side of the ray's line is computed
//      from that vertex alone, so both segments sharing it agree.
//  3D: vertices are projected on the plane orthogonal to the ray (per-vertex
//      arithmetic, identical in every triangle); the 2D edge functions are
//      evaluated without contraction, so the two triangles of a shared edge get
//      exactly opposite values, and a zero value is broken by the edge's
//      direction, which the two triangles also see reversed.
struct RayFrame {
    float dir[3];
    float e1[3], e2[3];   // 3D: orthonormal basis of the plane orthogonal to dir
};

__device__ __forceinline__ float side2(const float* o, const float* dir, float vx, float vy) {
    return __fsub_rn(__fmul_rn(dir[0], __fsub_rn(vy, o[1])), __fmul_rn(dir[1], __fsub_rn(vx, o[0])));
}

__device__ __forceinline__ float edge_fn(float px, float py, float qx, float qy) {
    return __fsub_rn(__fmul_rn(px, qy), __fmul_rn(py, qx));
}

__device__ __forceinline__ bool edge_positive(float px, float py, float qx, float qy) {
    const float e = edge_fn(px, py, qx, qy);
    if (e != 0.0f) return e > 0.0f;
    return (qx > px) || (qx == px && qy > py);
}

__device__ __forceinline__ void project(const RayFrame& F, const float* o, float4 v, float& x, float& y, float& z) {
    const float dx = __fsub_rn(v.x, o[0]), dy = __fsub_rn(v.y, o[1]), dz = __fsub_rn(v.z, o[2]);
    x = __fadd_rn(__fadd_rn(__fmul_rn(dx, F.e1[0]), __fmul_rn(dy, F.e1[1])), __fmul_rn(dz, F.e1[2]));
    y = __fadd_rn(__fadd_rn(__fmul_rn(dx, F.e2[0]), __fmul_rn(dy, F.e2[1])), __fmul_rn(dz, F.e2[2]));
    z = __fadd_rn(__fadd_rn(__fmul_rn(dx, F.dir[0]), __fmul_rn(dy, F.dir[1])), __fmul_rn(dz, F.dir[2]));
}

__device__ __forceinline__ float ray_segment_t(float4 s, const float* o, const float* dir) {
    const float sa = side2(o, dir, s.x, s.y), sb = side2(o, dir, s.z, s.w);
    if ((sa >= 0.0f) == (sb >= 0.0f)) return -1.0f;
    const float lam = sa / (sa - sb);
    const float ax = s.x - o[0], ay = s.y - o[1];
    return (ax + lam * (s.z - s.x)) * dir[0] + (ay + lam * (s.w - s.y)) * dir[1];
}

template <int DIM>
__device__ __forceinline__ float ray_prim_t(const float4* prims, int p, const float* o, const RayFrame& F) {
    if (DIM == 2) {
        return ray_segment_t(prims[p], o, F.dir);
    } else {
        float ax, ay, az, bx, by, bz, cx, cy, cz;
        project(F, o, prims[3 * p], ax, ay, az);
        project(F, o, prims[3 * p + 1], bx, by, bz);
        project(F, o, prims[3 * p + 2], cx, cy, cz);
        // the projected origin is (0, 0): inside iff all edge functions share a sign
        const bool pa = edge_positive(bx, by, cx, cy);   // edge b -> c (weight of a)
        const bool pb = edge_positive(cx, cy, ax, ay);   // edge c -> a (weight of b)
        const bool pc = edge_positive(ax, ay, bx, by);   // edge a -> b (weight of c)
        if (!((pa && pb && pc) || (!pa && !pb && !pc))) return -1.0f;
        const float wa = edge_fn(bx, by, cx, cy), wb = edge_fn(cx, cy, ax, ay), wc = edge_fn(ax, ay, bx, by);
        const float den = wa + wb + wc;
        if (den == 0.0f) return -1.0f;
        return (wa * az + wb * bz + wc * cz) / den;
    }
}

template <int DIM>
__global__ void inside_kernel(BvhView bvh, int n, const float* p, int* inside, const float* prev, float* prev_out) {
    const int pt = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (pt >= n) return;    // whole warps exit together
    float o[DIM], inv[DIM];
    RayFrame F;
    if (DIM == 2) {
        F.dir[0] = 0.8191520443f; F.dir[1] = 0.5735764364f; F.dir[2] = 0.0f;
    } else {
        // generic unit direction and an orthonormal basis of its normal plane
        F.dir[0] = 0.5144957554f; F.dir[1] = 0.6859943406f; F.dir[2] = 0.5144957554f;
        F.e1[0] = 0.7071067812f; F.e1[1] = 0.0f; F.e1[2] = -0.7071067812f;
        F.e2[0] = -0.4850712500f; F.e2[1] = 0.7276068751f; F.e2[2] = -0.4850712500f;
    }
    const float* dir = F.dir;
#pragma unroll
    for (int k = 0; k < DIM; ++k) { o[k] = p[DIM * pt + k]; inv[k] = 1.0f / dir[k]; }
    if (prev) {   // the same point as last time: its flag stands
        bool same = true;
#pragma unroll
        for (int k = 0; k < DIM; ++k) same = same && __float_as_uint(o[k]) == __float_as_uint(prev[DIM * pt + k]);
        if (same) return;
    }
    // scene box: the root's two children and the outsized elements
    float slo[DIM], shi[DIM];
#pragma unroll
    for (int k = 0; k < DIM; ++k) { slo[k] = o[k]; shi[k] = o[k]; }
    if (bvh.n_internal > 0) {
        float lo0[DIM], hi0[DIM], lo1[DIM], hi1[DIM];
        int c0, c1, parent;
        load_node<DIM>(bvh.nodes, bvh.root, lo0, hi0, lo1, hi1, c0, c1, parent);
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            slo[k] = fminf(slo[k], lo0[k]); shi[k] = fmaxf(shi[k], hi0[k]);
            if (c1 != kEmptyChild) { slo[k] = fminf(slo[k], lo1[k]); shi[k] = fmaxf(shi[k], hi1[k]); }
        }
    }
    for (int q = bvh.n_tree; q < bvh.n_tree + bvh.n_big; ++q) {
        float lo[DIM], hi[DIM];
        prim_box<DIM>(bvh.prims, q, lo, hi);
#pragma unroll
        for (int k = 0; k < DIM; ++k) { slo[k] = fminf(slo[k], lo[k]); shi[k] = fmaxf(shi[k], hi[k]); }
    }
    float tmax2 = 0.0f;
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        const float e = fmaxf(o[k] - slo[k], shi[k] - o[k]);
        tmax2 += e * e;
    }
    const float tmax = 1.001f * sqrtf(tmax2) + 1e-6f;
    const float ta = tmax * (float)lane / 32.0f;
    const float tb = lane == 31 ? 2.0f * tmax : tmax * (float)(lane + 1) / 32.0f;
    int count = 0;
    for (int q = bvh.n_tree; q < bvh.n_tree + bvh.n_big; ++q) {
        const float t = ray_prim_t<DIM>(bvh.prims, q, o, F);
        count += (t > 0.0f && t >= ta && t < tb) ? 1 : 0;
    }
    if (bvh.n_internal > 0) {
        int st[kLaneStack], sp = 0, node = bvh.root;
        int budget = bvh.n_internal + 8;
        while (--budget >= 0) {
            float lo0[DIM], hi0[DIM], lo1[DIM], hi1[DIM];
            int c0, c1, parent;
            load_node<DIM>(bvh.nodes, node, lo0, hi0, lo1, hi1, c0, c1, parent);
            int next = kNoNode;
#pragma unroll
            for (int side = 0; side < 2; ++side) {
                const int c = side == 0 ? c0 : c1;
                if (c == kEmptyChild || !(side == 0 ? seg_hits_box<DIM>(o, inv, ta, tb, lo0, hi0)
                                                    : seg_hits_box<DIM>(o, inv, ta, tb, lo1, hi1))) continue;
                if (c < 0) {
                    const float t = ray_prim_t<DIM>(bvh.prims, ~c, o, F);
                    count += (t > 0.0f && t >= ta && t < tb) ? 1 : 0;
                } else if (next == kNoNode) {
                    next = c;
                } else if (sp < kLaneStack) {     // (a path has at most 62 nodes)
                    st[sp++] = c;
                }
            }
            if (next == kNoNode) {
                if (sp == 0) break;
                next = st[--sp];
            }
            node = next;
        }
    }
    for (int off = 16; off > 0; off >>= 1) count += __shfl_xor_sync(0xffffffffu, count, off);
    if (lane == 0) {
        inside[pt] = count & 1;
        if (prev_out) {
#pragma unroll
            for (int k = 0; k < DIM; ++k) prev_out[DIM * pt + k] = o[k];
        }
    }
}

// The same for segments with a wide tree: a warp per point, one child of the current
// node per lane, in any order (every leaf that the ray's line can cross is counted once).
// Bound by the chain of node fetches, three levels of them for 4096 segments instead of
// a dozen (256 points: 29 us by intervals of the ray on the binary tree).
constexpr int kInsideBlock = 128;

__global__ void __launch_bounds__(kInsideBlock) inside_wide_kernel(const float* wnodes, const float4* prims, int n_tree,
                                                                   int n_big, int n, const float* p, int* inside,
                                                                   const float* prev, float* prev_out) {
    __shared__ int stacks[kInsideBlock / 32][kWideStack];
    const int pt = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    int* stk = stacks[threadIdx.x >> 5];
    if (pt >= n) return;    // whole warps exit together
    const float dir[2] = {0.8191520443f, 0.5735764364f};
    const float o[2] = {p[2 * pt], p[2 * pt + 1]}, inv[2] = {1.0f / dir[0], 1.0f / dir[1]};
    if (prev && __float_as_uint(o[0]) == __float_as_uint(prev[2 * pt]) &&
        __float_as_uint(o[1]) == __float_as_uint(prev[2 * pt + 1])) return;   // the same point as last time: its flag stands
    int count = 0;
    for (int q = n_tree + lane; q < n_tree + n_big; q += 32) count += ray_segment_t(prims[q], o, dir) > 0.0f ? 1 : 0;
    int top = 0, cur = 0;
    for (;;) {
        const float* f = wnodes + (size_t)cur * kWideFloats;
        const float4 s = __ldg(reinterpret_cast<const float4*>(f) + lane);
        const int code = __float_as_int(__ldg(f + 4 * kWide + lane));
        if (code < 0) count += ray_segment_t(s, o, dir) > 0.0f ? 1 : 0;
        const float lo[2] = {s.x, s.y}, hi[2] = {s.z, s.w};
        const bool hit = code >= 0 && code != kEmptyChild && seg_hits_box<2>(o, inv, 0.0f, kInf, lo, hi);
        const unsigned m = __ballot_sync(0xffffffffu, hit);
        __syncwarp();
        if (hit) {
            const int at = top + __popc(m & ((1u << lane) - 1u));
            if (at < kWideStack) stk[at] = code;       // (31 x the depth + 1 entries at most)
        }
        top = min(top + __popc(m), kWideStack);
        __syncwarp();
        if (top == 0) break;
        cur = stk[--top];
    }
    count = __reduce_add_sync(0xffffffffu, count);
    if (lane == 0) {
        inside[pt] = count & 1;
        if (prev_out) { prev_out[2 * pt] = o[0]; prev_out[2 * pt + 1] = o[1]; }
    }
}

__global__ void philox_kernel(int n, const uint32_t* ctr, uint32_t k0, uint32_t k1, uint32_t* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const U4 r = philox(U4{ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]}, k0, k1);
    out[4 * i] = r.x; out[4 * i + 1] = r.y; out[4 * i + 2] = r.z; out[4 * i + 3] = r.w;
}

// v = v_ref + J theta, one thread per (vertex, coordinate) row.
__global__ void apply_params_kernel(const float* vert_ref, const float* jac, const float* theta, float* vert,
                                    int n_rows, int n_param) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n_rows) return;
    float s = vert_ref[r];
    const float* J = jac + (size_t)r * n_param;
    for (int j = 0; j < n_param; ++j) s = fmaf(J[j], theta[j], s);
    vert[r] = s;
}

inline int nblk(long long n, int b) { return (int)((n + b - 1) / b); }

}  // namespace

constexpr int kWideLevels = 16;   // level counts kept by a wide tree's build

cudaError_t bvh_reserve(BvhBuffers& b, int dim, int n_elem) {
    if (n_elem <= b.capacity && dim == b.dim) return cudaSuccess;
    bvh_free(b);
    const int n_int = n_elem > 1 ? n_elem - 1 : 1;
    const int nf4 = dim == 2 ? 3 : 4, pf4 = dim == 2 ? 1 : 3;
    cudaError_t e;
#define DW_TRY(x) do { e = (x); if (e != cudaSuccess) { bvh_free(b); return e; } } while (0)
    DW_TRY(cudaMalloc(&b.nodes, sizeof(float4) * nf4 * (size_t)n_int));
    DW_TRY(cudaMalloc(&b.prims, sizeof(float4) * pf4 * (size_t)n_elem));
    DW_TRY(cudaMalloc(&b.prim_elem, sizeof(int) * (size_t)n_elem));
    DW_TRY(cudaMalloc(&b.leaf_of_elem, sizeof(int) * (size_t)n_elem));
    DW_TRY(cudaMalloc(&b.keys, sizeof(unsigned int) * (size_t)n_elem));
    DW_TRY(cudaMalloc(&b.keys_sorted, sizeof(unsigned int) * (size_t)n_elem));
    DW_TRY(cudaMalloc(&b.vals, sizeof(int) * (size_t)n_elem));
    DW_TRY(cudaMalloc(&b.vals_sorted, sizeof(int) * (size_t)n_elem));
    DW_TRY(cudaMalloc(&b.leaf_parent, sizeof(int) * (size_t)n_elem));
    DW_TRY(cudaMalloc(&b.node_parent, sizeof(int) * (size_t)n_int));
    DW_TRY(cudaMalloc(&b.node_child, sizeof(int) * 2 * (size_t)n_int));
    DW_TRY(cudaMalloc(&b.boxes, sizeof(float4) * (dim == 2 ? 1 : 2) * level_boxes((size_t)n_elem)));
    DW_TRY(cudaMalloc(&b.node_count, sizeof(int) * 2 * (size_t)n_int));   // leaf counts, then first leaves
    DW_TRY(cudaMalloc(&b.node_cell, sizeof(float) * 2 * dim * (size_t)n_int));
    DW_TRY(cudaMalloc(&b.wroot, sizeof(int) * 2 * (size_t)n_int));        // roots, then first inner children
    DW_TRY(cudaMalloc(&b.wlev, sizeof(int) * kWideLevels));
    DW_TRY(cudaMalloc(&b.bounds, sizeof(unsigned int) * 6));
    DW_TRY(cudaMalloc(&b.stats, sizeof(float) * 2 + sizeof(int) * 4));
    size_t tmp = 0;
    DW_TRY(cub::DeviceRadixSort::SortPairs(nullptr, tmp, b.keys, b.keys_sorted, b.vals, b.vals_sorted, n_elem));
    DW_TRY(cudaMalloc(&b.sort_tmp, tmp));
#undef DW_TRY
    b.sort_tmp_bytes = tmp;
    b.capacity = n_elem;
    b.dim = dim;
    return cudaSuccess;
}

void bvh_free(BvhBuffers& b) {
    cudaFree(b.nodes); cudaFree(b.prims); cudaFree(b.prim_elem); cudaFree(b.leaf_of_elem); cudaFree(b.keys); cudaFree(b.keys_sorted);
    cudaFree(b.vals); cudaFree(b.vals_sorted); cudaFree(b.leaf_parent); cudaFree(b.node_parent);
    cudaFree(b.node_child); cudaFree(b.boxes); cudaFree(b.bounds); cudaFree(b.stats); cudaFree(b.node_cell);
    cudaFree(b.sort_tmp);
    cudaFree(b.wnodes); cudaFree(b.wsrc); cudaFree(b.wroot); cudaFree(b.wlev); cudaFree(b.node_count);
    b = BvhBuffers();
}

constexpr int kMaxBig = 64;

// Leaves, links and, for a tree of two leaves or more, all boxes of the binary tree.
template <int DIM>
static void fill_boxes(BvhBuffers& b, const float* vert, const int* elem, cudaStream_t s) {
    const int nt = b.n_tree;
    leaves_kernel<DIM><<<nblk(b.n_elem, kLeafBlock), kLeafBlock, 0, s>>>(
        vert, elem, b.vals_sorted, b.n_elem, nt, b.node_child, b.node_parent, b.leaf_parent, b.nodes, b.prims,
        b.prim_elem, b.leaf_of_elem, b.boxes);
    if (nt >= 3)
        node_boxes_kernel<DIM><<<nblk(8LL * (nt - 2), 256), 256, 0, s>>>(b.prims, b.boxes, nt, b.node_child,
                                                                         b.node_parent, b.node_count,
                                                                         b.node_count + (nt - 1), b.nodes);
}

// The wide tree's boxes (and, in 2D, leaf children's vertices) from the binary tree.
template <int DIM>
static cudaError_t fill_wide(BvhBuffers& b, cudaStream_t s) {
    if constexpr (DIM == 2) {
        wide_refit_kernel<<<nblk((long long)b.n_wide * kWide, 256), 256, 0, s>>>(
            b.nodes, b.prims, b.wsrc, b.wsrc + kWide * (size_t)b.n_wide, b.n_wide, b.wnodes);
    } else {
        oriented_fill_kernel<<<nblk(32LL * b.n_wide, 128), 128, 0, s>>>(
            b.nodes, b.prims, b.node_count, b.node_count + b.n_internal, b.wsrc + kOriented * (size_t)b.n_wide,
            b.wroot, b.wsrc + 2 * kOriented * (size_t)b.n_wide, b.n_wide, reinterpret_cast<float4*>(b.wnodes));
    }
    return cudaGetLastError();
}

// Collapse the binary tree (n_internal >= 1 nodes, boxes refit) into the
// wide tree.  Nodes are numbered level by level, the root first.
template <int DIM>
static cudaError_t build_wide(BvhBuffers& b, cudaStream_t s) {
    constexpr int W = DIM == 2 ? kWide : kOriented;
    constexpr int kNodeFloats = DIM == 2 ? kWideFloats : 4 * kOrientedF4;
    constexpr int kMax = DIM == 2 ? (kWideStack - 1) / (kWide - 1) : kOrientedDepthMax;   // levels the search takes
    static_assert(kMax < kWideLevels, "level counts");
    const int n_int = b.n_internal;
    // level counts: one node (the binary root, id 0) at level 0
    cudaError_t e = cudaMemsetAsync(b.wlev, 0, sizeof(int) * kWideLevels, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(b.wroot, 0, sizeof(int), s);
    int lev[kWideLevels] = {1};
    if (e == cudaSuccess) e = cudaMemcpyAsync(b.wlev, lev, sizeof(int), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    int done = 0;
    while (done < kMax && lev[done] > 0) {        // a few levels at a time (200k triangles have eight, 4k segments three)
        for (const int to = done + (DIM == 2 ? 4 : 9); done < to && done < kMax; ++done) {
            long long most = 1;
            for (int k = 0; k < done && most < n_int; ++k) most *= W;
            const int blocks = min(nblk(most < n_int ? most : n_int, 128), 1024);
            wide_level_kernel<W><<<blocks, 128, 0, s>>>(b.node_child, b.node_count, b.node_count + n_int,
                                                        b.leaf_parent, done, b.wlev, b.wroot, b.wroot + n_int);
        }
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(lev, b.wlev, sizeof(lev), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return e;
    }
    b.n_wide = 0;
    b.wide_depth = 0;
    for (int l = 0; l < done && lev[l] > 0; ++l) { b.n_wide += lev[l]; b.wide_depth = l + 1; }
    b.wide_ok = lev[kMax] == 0;
    if (!b.wide_ok) { b.n_wide = 0; return cudaSuccess; }     // too deep: the binary tree serves every query
    if (b.n_wide > b.wide_cap) {
        cudaFree(b.wnodes); cudaFree(b.wsrc);
        b.wnodes = nullptr; b.wsrc = nullptr; b.wide_cap = 0;
        e = cudaMalloc(&b.wnodes, sizeof(float) * kNodeFloats * (size_t)b.n_wide);
        if (e == cudaSuccess) e = cudaMalloc(&b.wsrc, sizeof(int) * (2 * W + 1) * (size_t)b.n_wide);
        if (e != cudaSuccess) return e;
        b.wide_cap = b.n_wide;
    }
    wide_codes_kernel<W><<<nblk(b.n_wide, 128), 128, 0, s>>>(
        b.node_child, b.node_count, b.node_count + n_int, b.leaf_parent, b.n_wide, b.wroot, b.wroot + n_int,
        b.wsrc + W * (size_t)b.n_wide, b.wsrc, b.wsrc + 2 * W * (size_t)b.n_wide);
    return fill_wide<DIM>(b, s);
}

template <int DIM>
static cudaError_t build_impl(BvhBuffers& b, const float* vert, const int* elem, int n, cudaStream_t s) {
    b.n_elem = n;
    float* stats = b.stats;
    int* count = reinterpret_cast<int*>(b.stats + 2);
    cudaError_t e = cudaMemsetAsync(b.stats, 0, sizeof(float) * 2 + sizeof(int) * 4, s);
    if (e != cudaSuccess) return e;
    const int gb = min(nblk(n, 256), 1024);
    size_kernel<DIM><<<gb, 256, 0, s>>>(vert, elem, n, stats);
    count_big_kernel<DIM><<<gb, 256, 0, s>>>(vert, elem, n, stats, count);
    int host[3] = {0, 0, 0};
    e = cudaMemcpyAsync(host, count, sizeof(int) * 3, cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return e;
    e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    int n_big = host[0];
    const int split = (n_big > 0 && n_big <= kMaxBig && n_big < n) ? 1 : 0;
    if (!split) n_big = 0;
    float r_small, r_all;
    memcpy(&r_small, &host[1], sizeof(float));
    memcpy(&r_all, &host[2], sizeof(float));
    // margin for the FP32 rounding of the Morton quantisation
    b.r_max = (split ? r_small : r_all) * 1.0001f + 1e-6f;
    const int nt = n - n_big;
    b.n_big = n_big;
    b.n_tree = nt;
    e = cudaMemsetAsync(b.bounds, 0xff, sizeof(unsigned int) * DIM, s);   // min slots
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(b.bounds + DIM, 0, sizeof(unsigned int) * DIM, s);             // max slots
    if (e != cudaSuccess) return e;
    bounds_kernel<DIM><<<gb, 256, 0, s>>>(vert, elem, n, stats, split, b.bounds);
    morton_kernel<DIM><<<nblk(n, 256), 256, 0, s>>>(vert, elem, n, b.bounds, stats, split, b.keys, b.vals);
    size_t tmp = b.sort_tmp_bytes;
    e = cub::DeviceRadixSort::SortPairs(b.sort_tmp, tmp, b.keys, b.keys_sorted, b.vals, b.vals_sorted, n, 0, 32, s);
    if (e != cudaSuccess) return e;
    if (nt >= 2) {
        b.n_internal = nt - 1;
        radix_tree_kernel<DIM><<<nblk(nt - 1, 256), 256, 0, s>>>(b.keys_sorted, nt, b.node_child, b.node_parent,
                                                                 b.leaf_parent, b.bounds, b.node_cell,
                                                                 b.node_count, b.node_count + (nt - 1));
        fill_boxes<DIM>(b, vert, elem, s);
        e = build_wide<DIM>(b, s);
        if (e != cudaSuccess) return e;
    } else {
        b.n_wide = 0;
        b.wide_depth = 0;
        b.wide_ok = true;     // nothing to search beyond the single leaf
        b.n_internal = nt;    // 1: a single-leaf node; 0: no tree
        if (nt == 1) single_leaf_kernel<DIM><<<1, 1, 0, s>>>(vert, elem, b.vals_sorted, b.nodes, b.leaf_parent,
                                                             b.node_cell);
        fill_boxes<DIM>(b, vert, elem, s);
    }
    return cudaGetLastError();
}

cudaError_t bvh_build(BvhBuffers& b, int dim, const float* vert, const int* elem, int n_elem, cudaStream_t s) {
    cudaError_t e = bvh_reserve(b, dim, n_elem);
    if (e != cudaSuccess) return e;
    b.cells_ok = false;
    e = dim == 2 ? build_impl<2>(b, vert, elem, n_elem, s) : build_impl<3>(b, vert, elem, n_elem, s);
    b.cells_ok = e == cudaSuccess;
    return e;
}

template <int DIM>
static cudaError_t refit_impl(BvhBuffers& b, const float* vert, const int* elem, cudaStream_t s) {
    const int n = b.n_elem, nt = b.n_tree;
    if (n <= 0) return cudaSuccess;
    if (nt >= 2) {
        fill_boxes<DIM>(b, vert, elem, s);
        if (b.n_wide > 0) {
            const cudaError_t e = fill_wide<DIM>(b, s);
            if (e != cudaSuccess) return e;
        }
    } else {
        if (nt == 1) single_leaf_kernel<DIM><<<1, 1, 0, s>>>(vert, elem, b.vals_sorted, b.nodes, b.leaf_parent,
                                                             b.node_cell);
        fill_boxes<DIM>(b, vert, elem, s);
    }
    b.cells_ok = false;
    return cudaGetLastError();
}

cudaError_t bvh_refit(BvhBuffers& b, const float* vert, const int* elem, cudaStream_t s) {
    return b.dim == 2 ? refit_impl<2>(b, vert, elem, s) : refit_impl<3>(b, vert, elem, s);
}

static BvhView view_of(const BvhBuffers& b) {
    BvhView v;
    v.nodes = b.nodes;
    v.prims = b.prims;
    v.root = 0;
    v.n_internal = b.n_internal;
    v.n_tree = b.n_tree;
    v.n_big = b.n_big;
    v.climb = 0;
    v.leaf_parent = b.leaf_parent;
    v.node_cell = b.node_cell;
    v.r_max = b.r_max;
    return v;
}

cudaError_t launch_closest(const BvhBuffers& b, int n, const float* p, const int* hint_elem, float* dist,
                           int* elem_out, float* bary, int* err, DevCounters* ctr, int traversal, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    BvhView v = view_of(b);
    if (traversal == 2 && b.wide_ok) {
        const WideView wv{b.wnodes, b.prims, b.n_wide, b.n_tree};
        const int cap = wide_stack_entries(b.dim, b.wide_depth);
        const size_t smem = wide_smem_bytes(b.dim, cap) * (128 / 32);
        if (b.dim == 2) closest_wide_kernel<2><<<nblk(n, 128), 128, smem, s>>>(v, wv, b.prim_elem, b.leaf_of_elem, n, p, hint_elem, dist, elem_out, bary, err, ctr, cap);
        else closest_wide_kernel<3><<<nblk(n, 128), 128, smem, s>>>(v, wv, b.prim_elem, b.leaf_of_elem, n, p, hint_elem, dist, elem_out, bary, err, ctr, cap);
        return cudaGetLastError();
    }
    v.climb = traversal == 1 ? 1 : 0;
    if (b.dim == 2) closest_kernel<2><<<nblk(n, 128), 128, 0, s>>>(v, b.prim_elem, b.leaf_of_elem, n, p, hint_elem, dist, elem_out, bary, err, ctr);
    else closest_kernel<3><<<nblk(n, 128), 128, 0, s>>>(v, b.prim_elem, b.leaf_of_elem, n, p, hint_elem, dist, elem_out, bary, err, ctr);
    return cudaGetLastError();
}

cudaError_t launch_inside(const BvhBuffers& b, int n, const float* p, int* inside, cudaStream_t s,
                          const float* prev, float* prev_out) {
    if (n <= 0) return cudaSuccess;
    if (b.dim == 2 && b.wide_ok && b.n_wide > 0)
        inside_wide_kernel<<<nblk(32LL * n, kInsideBlock), kInsideBlock, 0, s>>>(b.wnodes, b.prims, b.n_tree, b.n_big, n, p,
                                                                                 inside, prev, prev_out);
    else if (b.dim == 2) inside_kernel<2><<<nblk(32LL * n, 128), 128, 0, s>>>(view_of(b), n, p, inside, prev, prev_out);
    else inside_kernel<3><<<nblk(32LL * n, 128), 128, 0, s>>>(view_of(b), n, p, inside, prev, prev_out);
    return cudaGetLastError();
}

cudaError_t launch_philox(int n, const uint32_t* ctr, uint32_t k0, uint32_t k1, uint32_t* out, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    philox_kernel<<<nblk(n, 256), 256, 0, s>>>(n, ctr, k0, k1, out);
    return cudaGetLastError();
}

cudaError_t launch_apply_params(const float* vert_ref, const float* jac, const float* theta, float* vert,
                                int n_rows, int n_param, cudaStream_t s) {
    if (n_rows <= 0) return cudaSuccess;
    apply_params_kernel<<<nblk(n_rows, 256), 256, 0, s>>>(vert_ref, jac, theta, vert, n_rows, n_param);
    return cudaGetLastError();
}

}  // namespace dwos
