// lbvh.cu -- LBVH construction on the device: FP32 Morton codes of triangle
// centroids, a stable LSD radix sort of (code, index), the Karras (HPG 2012)
// radix tree, and a bottom-up AABB refit that packs 64-byte nodes and 48-byte
// triangles.  Integer results (codes, order, topology) and the FP32 min/max
// boxes are exact and reproducible.
#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"

namespace dpcs {

namespace {

constexpr int kSortTile = 256;  // items (and threads) per radix-sort block

// floats as unsigned integers in the same order, for atomic min / max
__device__ __forceinline__ uint32_t ordered(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : u | 0x80000000u;
}
__device__ __forceinline__ float unordered(uint32_t u) {
    return __uint_as_float((u & 0x80000000u) ? u & 0x7fffffffu : ~u);
}

// centroids (v0 + v1 + v2) * (1/3) in FP32 without contraction, and their
// bounds -> bounds[0..2] lo (set to all ones before), [3..5] hi (set to zero
// before), as ordered integers.  min and max do not depend on the order.
__global__ void __launch_bounds__(256) k_centroids(const float *__restrict__ verts, const int32_t *__restrict__ tris,
                                                   int T, float *__restrict__ cen, uint32_t *__restrict__ bounds) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const float third = 1.0f / 3.0f;
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    if (i < T) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float a = verts[3 * tris[3 * i] + k], b = verts[3 * tris[3 * i + 1] + k],
                        c = verts[3 * tris[3 * i + 2] + k];
            lo[k] = hi[k] = cen[3 * i + k] = __fmul_rn(__fadd_rn(__fadd_rn(a, b), c), third);
        }
    }
    __shared__ float slo[3][8], shi[3][8];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        for (int off = 16; off; off >>= 1) {
            lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], off));
            hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], off));
        }
        if (l == 0) {
            slo[k][w] = lo[k];
            shi[k][w] = hi[k];
        }
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        const int k = threadIdx.x;
        float a = INFINITY, b = -INFINITY;
        for (int j = 0; j < 8; ++j) {
            a = fminf(a, slo[k][j]);
            b = fmaxf(b, shi[k][j]);
        }
        atomicMin(bounds + k, ordered(a));
        atomicMax(bounds + 3 + k, ordered(b));
    }
}

__device__ __forceinline__ uint32_t expand10(uint32_t v) {
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000FFu;
    v = (v | (v << 8)) & 0x0300F00Fu;
    v = (v | (v << 4)) & 0x030C30C3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

// 30-bit Morton code of the centroid normalised into the centroid bounds
__global__ void k_morton(const float *__restrict__ cen, const uint32_t *__restrict__ bounds, int T,
                         uint32_t *__restrict__ codes, int32_t *__restrict__ idx) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= T) return;
    uint32_t q[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float lo = unordered(bounds[k]), ext = __fsub_rn(unordered(bounds[3 + k]), lo);
        const float inv = ext > 0.0f ? __frcp_rn(ext) : 0.0f;
        const float nrm = __fmul_rn(__fsub_rn(cen[3 * i + k], lo), inv);
        float f = floorf(__fmul_rn(nrm, 1024.0f));
        f = fminf(fmaxf(f, 0.0f), 1023.0f);
        q[k] = (uint32_t)f;
    }
    codes[i] = (expand10(q[0]) << 2) | (expand10(q[1]) << 1) | expand10(q[2]);
    idx[i] = i;
}

// --- stable LSD radix sort, 8-bit digits -----------------------------------
__global__ void k_radix_hist(const uint32_t *__restrict__ keys, int n, int shift, int nblocks,
                             uint32_t *__restrict__ hist) {
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int i = blockIdx.x * kSortTile + threadIdx.x;
    if (i < n) atomicAdd(&h[(keys[i] >> shift) & 0xffu], 1u);
    __syncthreads();
    hist[threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

// exclusive prefix of v over a block of 256 threads; total: the block's sum
__device__ __forceinline__ uint32_t block_prefix(uint32_t v, uint32_t &total) {
    __shared__ uint32_t ws[8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t x = v;
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    __syncthreads();  // ws may still be read from the call before
    if (lane == 31) ws[w] = x;
    __syncthreads();
    uint32_t before = 0;
    total = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        if (j < w) before += ws[j];
        total += ws[j];
    }
    return before + x - v;
}

// Exclusive scan of each digit's counters over the blocks, one block per
// digit, and the digit's total; the scatter adds the digits before it.
__global__ void __launch_bounds__(256) k_radix_rows(uint32_t *__restrict__ hist, int nblocks, uint32_t *__restrict__ total) {
    uint32_t *row = hist + (size_t)blockIdx.x * nblocks;
    uint32_t carry = 0;
    for (int i0 = 0; i0 < nblocks; i0 += 256) {
        const int i = i0 + threadIdx.x;
        const uint32_t v = i < nblocks ? row[i] : 0u;
        uint32_t t;
        const uint32_t e = block_prefix(v, t);
        if (i < nblocks) row[i] = carry + e;
        carry += t;
    }
    if (threadIdx.x == 0) total[blockIdx.x] = carry;
}

__global__ void k_radix_scatter(const uint32_t *__restrict__ kin, const int32_t *__restrict__ vin,
                                uint32_t *__restrict__ kout, int32_t *__restrict__ vout, int n, int shift,
                                int nblocks, const uint32_t *__restrict__ offs, const uint32_t *__restrict__ total) {
    __shared__ uint32_t cnt[kSortTile / 32][256], first[256];
    uint32_t all;
    first[threadIdx.x] = block_prefix(total[threadIdx.x], all);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int j = threadIdx.x; j < (kSortTile / 32) * 256; j += blockDim.x) (&cnt[0][0])[j] = 0u;
    __syncthreads();
    const int i = blockIdx.x * kSortTile + threadIdx.x;
    const bool valid = i < n;
    const uint32_t key = valid ? kin[i] : 0u;
    const uint32_t digit = valid ? ((key >> shift) & 0xffu) : 0x100u;
    const unsigned peers = __match_any_sync(0xffffffffu, digit);
    const unsigned lt = (1u << lane) - 1u;
    const uint32_t rank = __popc(peers & lt);
    if (valid && (peers & lt) == 0u) cnt[w][digit] = __popc(peers);
    __syncthreads();
    if (valid) {
        uint32_t off = rank;
        for (int ww = 0; ww < w; ++ww) off += cnt[ww][digit];
        const uint32_t dst = first[digit] + (offs ? offs[digit * nblocks + blockIdx.x] : 0u) + off;
        kout[dst] = key;
        vout[dst] = vin[i];
    }
}

// --- Karras radix tree -------------------------------------------------------
__device__ __forceinline__ int delta(const uint32_t *__restrict__ c, int T, int i, int j) {
    if (j < 0 || j > T - 1) return -1;
    const uint32_t a = c[i], b = c[j];
    if (a == b) return 32 + __clz((uint32_t)(i ^ j));
    return __clz(a ^ b);
}

__global__ void k_karras(const uint32_t *__restrict__ codes, int T, float4 *__restrict__ nodes,
                         int32_t *__restrict__ parent) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= T - 1) return;
    const int d = (delta(codes, T, i, i + 1) - delta(codes, T, i, i - 1)) >= 0 ? 1 : -1;
    const int dmin = delta(codes, T, i, i - d);
    int lmax = 2;
    while (delta(codes, T, i, i + lmax * d) > dmin) lmax <<= 1;
    int l = 0;
    for (int t = lmax >> 1; t >= 1; t >>= 1)
        if (delta(codes, T, i, i + (l + t) * d) > dmin) l += t;
    const int j = i + l * d;
    const int dnode = delta(codes, T, i, j);
    int s = 0, t = l;
    do {
        t = (t + 1) >> 1;
        if (delta(codes, T, i, i + (s + t) * d) > dnode) s += t;
    } while (t > 1);
    const int g = i + s * d + min(d, 0);
    const int left = (min(i, j) == g) ? ~g : g;
    const int right = (max(i, j) == g + 1) ? ~(g + 1) : g + 1;
    nodes[4 * i + 3] = make_float4(__int_as_float(left), __int_as_float(right), 0.0f, 0.0f);
    if (left >= 0) parent[left] = i; else parent[T - 1 + g] = i;
    if (right >= 0) parent[right] = i; else parent[T - 1 + g + 1] = i;
}

__device__ __forceinline__ void store_box(float *nd, bool right, const float b[6]) {
    // node float layout: [0..3] left x/y, [4..7] right x/y, [8..11] z of left, right
    float *xy = nd + (right ? 4 : 0);
    float *z = nd + 8 + (right ? 2 : 0);
    __stcg(xy + 0, b[0]);
    __stcg(xy + 1, b[3]);
    __stcg(xy + 2, b[1]);
    __stcg(xy + 3, b[4]);
    __stcg(z + 0, b[2]);
    __stcg(z + 1, b[5]);
}

// one thread per leaf: pack the triangle, then walk up; the second thread to
// reach a node forms the union of its two child boxes and continues
__global__ void k_refit(const float *__restrict__ verts, const int32_t *__restrict__ tris,
                        const float *__restrict__ uv, const int32_t *__restrict__ order, int T,
                        float4 *__restrict__ nodes, const int32_t *__restrict__ parent,
                        int32_t *__restrict__ flags, float4 *__restrict__ tout, float2 *__restrict__ tuv) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= T) return;
    const int t = order[p];
    const int i0 = tris[3 * t], i1 = tris[3 * t + 1], i2 = tris[3 * t + 2];
    const float x0 = verts[3 * i0], y0 = verts[3 * i0 + 1], z0 = verts[3 * i0 + 2];
    const float x1 = verts[3 * i1], y1 = verts[3 * i1 + 1], z1 = verts[3 * i1 + 2];
    const float x2 = verts[3 * i2], y2 = verts[3 * i2 + 1], z2 = verts[3 * i2 + 2];
    // the three vertices as uploaded: a vertex shared by two triangles has
    // the same bits in both, which the watertight hit test relies on
    tout[3 * p + 0] = make_float4(x0, y0, z0, __int_as_float(t));
    tout[3 * p + 1] = make_float4(x1, y1, z1, 0.0f);
    tout[3 * p + 2] = make_float4(x2, y2, z2, 0.0f);
    tuv[3 * p + 0] = make_float2(uv[2 * i0], uv[2 * i0 + 1]);
    tuv[3 * p + 1] = make_float2(uv[2 * i1], uv[2 * i1 + 1]);
    tuv[3 * p + 2] = make_float2(uv[2 * i2], uv[2 * i2 + 1]);
    if (T < 2) return;
    float b[6] = {fminf(fminf(x0, x1), x2), fminf(fminf(y0, y1), y2), fminf(fminf(z0, z1), z2),
                  fmaxf(fmaxf(x0, x1), x2), fmaxf(fmaxf(y0, y1), y2), fmaxf(fmaxf(z0, z1), z2)};
    int child = ~p;
    int node = parent[T - 1 + p];
    while (true) {
        float *nd = reinterpret_cast<float *>(nodes + 4 * node);
        const int cl = __float_as_int(__ldcg(nd + 12));
        store_box(nd, cl != child, b);
        __threadfence();
        if (atomicAdd(&flags[node], 1) == 0) return;
        __threadfence();
        // both children are final: union
        const float lx0 = __ldcg(nd + 0), lx1 = __ldcg(nd + 1), ly0 = __ldcg(nd + 2), ly1 = __ldcg(nd + 3);
        const float rx0 = __ldcg(nd + 4), rx1 = __ldcg(nd + 5), ry0 = __ldcg(nd + 6), ry1 = __ldcg(nd + 7);
        const float lz0 = __ldcg(nd + 8), lz1 = __ldcg(nd + 9), rz0 = __ldcg(nd + 10), rz1 = __ldcg(nd + 11);
        b[0] = fminf(lx0, rx0); b[3] = fmaxf(lx1, rx1);
        b[1] = fminf(ly0, ry0); b[4] = fmaxf(ly1, ry1);
        b[2] = fminf(lz0, rz0); b[5] = fmaxf(lz1, rz1);
        if (node == 0) return;
        child = node;
        node = parent[node];
    }
}

// Clusters left and the number of the next node to make, kept on the device:
// round r reads state[r] and writes state[r + 1], so that the host need not
// wait for a round to launch the next (its grids fit the clusters the host
// last saw, and blocks past the present count do nothing).
struct PlocState {
    int32_t n, next;
};

__device__ __forceinline__ bool ploc_done(const PlocState *s) { return s->n == 1 && s->next == 0; }

// parent of every internal node and leaf, read back from the child
// references the Karras pass stored in the nodes
__global__ void k_parents(const float4 *__restrict__ nodes, int T, int32_t *__restrict__ parent,
                          const PlocState *state) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= T - 1 || (state && !ploc_done(state))) return;
    const float4 r = nodes[4 * i + 3];
    const int left = __float_as_int(r.x), right = __float_as_int(r.y);
    parent[left >= 0 ? left : T - 1 + ~left] = i;
    parent[right >= 0 ? right : T - 1 + ~right] = i;
}

inline size_t align256(size_t n) { return (n + 255) & ~size_t(255); }

// --- PLOC: agglomerative clustering over the Morton order -------------------
// (Meister & Bittner, "Parallel Locally-Ordered Clustering for Bounding
// Volume Hierarchy Construction", IEEE TVCG 2018.)  Clusters sit in Morton
// order; each finds its nearest neighbour -- the one whose union with it has
// the smallest surface area -- among the kPlocRadius clusters on either side;
// mutual nearest neighbours merge into a new node, and the survivors are
// compacted in order, until one cluster is left.  Ties go to the smaller
// index, which orders every pair by (area, lower index, higher index): the
// least pair of a round is always mutual, so every round merges.  New nodes
// are numbered downwards from T - 2 by a prefix sum of the merge flags, so
// the last merge (the root) is node 0 and the build is deterministic.
#ifndef DPCS_PLOC_RADIUS
#define DPCS_PLOC_RADIUS 16
#endif
constexpr int kPlocRadius = DPCS_PLOC_RADIUS;
constexpr int kPlocBlock = 128;

__device__ __forceinline__ float union_area(float4 alo, float4 ahi, float4 blo, float4 bhi) {
    const float dx = fmaxf(ahi.x, bhi.x) - fminf(alo.x, blo.x);
    const float dy = fmaxf(ahi.y, bhi.y) - fminf(alo.y, blo.y);
    const float dz = fmaxf(ahi.z, bhi.z) - fminf(alo.z, blo.z);
    return 2.0f * (dx * dy + dy * dz + dz * dx);
}

// leaf clusters: the boxes of the triangle records, in leaf order
__global__ void k_ploc_init(const float4 *__restrict__ tris, int T, int32_t *__restrict__ cid,
                            float4 *__restrict__ cbox) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= T) return;
    const float4 a = tris[3 * p], b = tris[3 * p + 1], c = tris[3 * p + 2];
    cid[p] = ~p;
    cbox[2 * p] = make_float4(fminf(fminf(a.x, b.x), c.x), fminf(fminf(a.y, b.y), c.y), fminf(fminf(a.z, b.z), c.z), 0.f);
    cbox[2 * p + 1] =
        make_float4(fmaxf(fmaxf(a.x, b.x), c.x), fmaxf(fmaxf(a.y, b.y), c.y), fmaxf(fmaxf(a.z, b.z), c.z), 0.f);
}

// nearest neighbour of each of the n clusters within the radius; the block's
// clusters and the radius on either side are staged in shared memory
__global__ void __launch_bounds__(kPlocBlock) k_ploc_nn(const float4 *__restrict__ cbox,
                                                       const PlocState *__restrict__ state, int32_t *__restrict__ nn) {
    const int n = state->n;
    if (n < 2 || blockIdx.x * kPlocBlock >= n) return;
    __shared__ float4 sb[2 * (kPlocBlock + 2 * kPlocRadius)];
    const int base = blockIdx.x * kPlocBlock - kPlocRadius;
    for (int k = threadIdx.x; k < kPlocBlock + 2 * kPlocRadius; k += blockDim.x) {
        const int j = base + k;
        if (j >= 0 && j < n) {
            sb[2 * k] = cbox[2 * j];
            sb[2 * k + 1] = cbox[2 * j + 1];
        }
    }
    __syncthreads();
    const int i = blockIdx.x * kPlocBlock + threadIdx.x;
    if (i >= n) return;
    const int li = i - base;
    const float4 lo = sb[2 * li], hi = sb[2 * li + 1];
    float best = INFINITY;
    int bj = i > 0 ? i - 1 : i + 1;
    const int j0 = max(0, i - kPlocRadius), j1 = min(n - 1, i + kPlocRadius);
    for (int j = j0; j <= j1; ++j) {
        if (j == i) continue;
        const float a = union_area(lo, hi, sb[2 * (j - base)], sb[2 * (j - base) + 1]);
        if (a < best) {  // ascending j with a strict comparison: ties to the smaller index
            best = a;
            bj = j;
        }
    }
    nn[i] = bj;
}

// per block of 256 clusters: merges (lower of a mutual pair) and survivors
// (not the higher of one)
__global__ void __launch_bounds__(256) k_ploc_count(const int32_t *__restrict__ nn, const PlocState *__restrict__ state,
                                                    uint2 *__restrict__ counts) {
    const int n = state->n;
    if (n < 2 || blockIdx.x * 256 >= n) return;
    const int i = blockIdx.x * 256 + threadIdx.x;
    const int j = i < n ? nn[i] : 0;
    const bool mutual = i < n && nn[j] == i;
    const int m = __syncthreads_count(mutual && i < j), k = __syncthreads_count(i < n && !(mutual && i > j));
    if (threadIdx.x == 0) counts[blockIdx.x] = make_uint2((uint32_t)m, (uint32_t)k);
}

__device__ __forceinline__ void ploc_merge(float4 *nodes, int id, int ca, int cb, float4 lo, float4 hi, float4 rlo,
                                           float4 rhi) {
    float4 *nd = nodes + 4 * (int64_t)id;
    nd[0] = make_float4(lo.x, hi.x, lo.y, hi.y);
    nd[1] = make_float4(rlo.x, rhi.x, rlo.y, rhi.y);
    nd[2] = make_float4(lo.z, hi.z, rlo.z, rhi.z);
    nd[3] = make_float4(__int_as_float(ca), __int_as_float(cb), 0.0f, 0.0f);
}

// New nodes (numbers next - 1 - rank of the merge) and the surviving clusters
// in order.  Every block adds up the counts of the blocks before it itself:
// up to 780 of them at 200k triangles, read once by each block in one sweep,
// where a scan in a kernel of its own with a single block took longer than
// the rest of the round.
__global__ void __launch_bounds__(256) k_ploc_compact(const int32_t *__restrict__ nn, PlocState *__restrict__ state,
                                                      const uint2 *__restrict__ counts, const int32_t *__restrict__ cid,
                                                      const float4 *__restrict__ cbox, int32_t *__restrict__ cid_out,
                                                      float4 *__restrict__ cbox_out, float4 *__restrict__ nodes) {
    const int n = state->n, next = state->next;
    if (n < 2) {
        if (blockIdx.x == 0 && threadIdx.x == 0) state[1] = state[0];
        return;
    }
    if (blockIdx.x * 256 >= n) return;
    uint32_t pm = 0, pk = 0;
    for (int j = threadIdx.x; j < (int)blockIdx.x; j += 256) {
        const uint2 c = counts[j];
        pm += c.x;
        pk += c.y;
    }
    uint32_t mbase, kbase, tm, tk;
    block_prefix(pm, mbase);
    block_prefix(pk, kbase);
    const int i = blockIdx.x * 256 + threadIdx.x;
    const int j = i < n ? nn[i] : 0;
    const bool mutual = i < n && nn[j] == i, merge = mutual && i < j, keep = i < n && !(mutual && i > j);
    const uint32_t m = mbase + block_prefix(merge ? 1u : 0u, tm), o = kbase + block_prefix(keep ? 1u : 0u, tk);
    if (i == n - 1) state[1] = PlocState{(int32_t)(kbase + tk), next - (int32_t)(mbase + tm)};
    if (!keep) return;  // merged into j
    const float4 lo = cbox[2 * i], hi = cbox[2 * i + 1];
    if (merge) {
        const int id = next - 1 - (int)m;
        const float4 rlo = cbox[2 * j], rhi = cbox[2 * j + 1];
        ploc_merge(nodes, id, cid[i], cid[j], lo, hi, rlo, rhi);
        cid_out[o] = id;
        cbox_out[2 * o] = make_float4(fminf(lo.x, rlo.x), fminf(lo.y, rlo.y), fminf(lo.z, rlo.z), 0.f);
        cbox_out[2 * o + 1] = make_float4(fmaxf(hi.x, rhi.x), fmaxf(hi.y, rhi.y), fmaxf(hi.z, rhi.z), 0.f);
    } else {
        cid_out[o] = cid[i];
        cbox_out[2 * o] = lo;
        cbox_out[2 * o + 1] = hi;
    }
}

// The last rounds, from kPlocSmall clusters on, in one block with the clusters
// in shared memory: the same rounds without the launches (a round of so few
// clusters is all launch latency).  Stops at the first round that merges
// nothing, which the host sees from the count left.
constexpr int kPlocSmall = 1024;
__global__ void __launch_bounds__(kPlocSmall) k_ploc_small(PlocState *__restrict__ state, const int32_t *__restrict__ cid,
                                                           const float4 *__restrict__ cbox, float4 *__restrict__ nodes) {
    __shared__ float4 slo[kPlocSmall], shi[kPlocSmall];
    __shared__ int32_t sid[kPlocSmall], snn[kPlocSmall];
    __shared__ uint32_t wm[32], wk[32];
    int n = state->n, next = state->next;
    const int i = threadIdx.x, lane = i & 31, w = i >> 5;
    if (i < n) {
        sid[i] = cid[i];
        slo[i] = cbox[2 * i];
        shi[i] = cbox[2 * i + 1];
    }
    __syncthreads();
    while (n > 1) {
        float4 lo, hi;
        int32_t id = 0;
        if (i < n) {
            lo = slo[i];
            hi = shi[i];
            id = sid[i];
            float best = INFINITY;
            int bj = i > 0 ? i - 1 : i + 1;
            const int j0 = max(0, i - kPlocRadius), j1 = min(n - 1, i + kPlocRadius);
            for (int j = j0; j <= j1; ++j) {
                if (j == i) continue;
                const float a = union_area(lo, hi, slo[j], shi[j]);
                if (a < best) {
                    best = a;
                    bj = j;
                }
            }
            snn[i] = bj;
        }
        __syncthreads();
        const int j = i < n ? snn[i] : 0;
        const bool mutual = i < n && snn[j] == i, merge = mutual && i < j, keep = i < n && !(mutual && i > j);
        const unsigned bm = __ballot_sync(0xffffffffu, merge), bk = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) {
            wm[w] = __popc(bm);
            wk[w] = __popc(bk);
        }
        float4 rlo, rhi;
        int32_t rid = 0;
        if (merge) {
            rlo = slo[j];
            rhi = shi[j];
            rid = sid[j];
        }
        __syncthreads();
        uint32_t m = __popc(bm & ((1u << lane) - 1u)), o = __popc(bk & ((1u << lane) - 1u)), tm = 0, tk = 0;
        for (int q = 0; q < 32; ++q) {
            if (q < w) {
                m += wm[q];
                o += wk[q];
            }
            tm += wm[q];
            tk += wk[q];
        }
        if (keep) {
            if (merge) {
                const int node = next - 1 - (int)m;
                ploc_merge(nodes, node, id, rid, lo, hi, rlo, rhi);
                id = node;
                lo = make_float4(fminf(lo.x, rlo.x), fminf(lo.y, rlo.y), fminf(lo.z, rlo.z), 0.f);
                hi = make_float4(fmaxf(hi.x, rhi.x), fmaxf(hi.y, rhi.y), fmaxf(hi.z, rhi.z), 0.f);
            }
            sid[o] = id;
            slo[o] = lo;
            shi[o] = hi;
        }
        __syncthreads();
        if (tm == 0) break;
        n = (int)tk;
        next -= (int)tm;
    }
    if (i == 0) *state = PlocState{n, next};
}

// deepest leaf: internal nodes on its path from the root (stops counting
// past `limit`, so a malformed tree cannot loop)
__global__ void k_tree_depth(const int32_t *__restrict__ parent, int T, int limit, int32_t *__restrict__ depth,
                             const PlocState *state) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= T || !ploc_done(state)) return;
    int d = 1, node = parent[T - 1 + p];
    while (node != 0 && d <= limit) {
        node = parent[node];
        ++d;
    }
    atomicMax(depth, d);
}

constexpr int kPlocBatch = 8;  // rounds launched before the host looks at the count

}  // namespace

size_t ploc_scratch_bytes(int32_t T) {
    const size_t n = (size_t)(T > 0 ? T : 1);
    return 2 * align256(n * 4) + 2 * align256(n * 32) + align256(n * 4) + 2 * align256(n * 4) +
           align256(n * 64) + align256(2 * n * 4) + align256((kPlocBatch + 2) * sizeof(PlocState));
}

int launch_ploc(Scene &sc, void *scratch, size_t scratch_bytes, int max_depth, cudaStream_t st, int32_t *depth_out) {
    const int T = sc.T;
    *depth_out = 0;
    if (T < 3) return 0;  // the radix tree of two leaves is already optimal
    if (scratch_bytes < ploc_scratch_bytes(T)) return DPCS_ERR_INVALID_ARG;
    const size_t n = (size_t)T;
    char *q = (char *)scratch;
    auto take = [&](size_t bytes) {
        char *r = q;
        q += align256(bytes);
        return (void *)r;
    };
    int32_t *cid[2] = {(int32_t *)take(n * 4), (int32_t *)take(n * 4)};
    float4 *cbox[2] = {(float4 *)take(n * 32), (float4 *)take(n * 32)};
    int32_t *nn = (int32_t *)take(n * 4);
    uint2 *bcount = (uint2 *)take(2 * align256(n * 4));
    float4 *nodes = (float4 *)take(n * 64);
    int32_t *parent = (int32_t *)take(2 * n * 4);
    PlocState *state = (PlocState *)take((kPlocBatch + 2) * sizeof(PlocState));
    int32_t *depth = (int32_t *)(state + kPlocBatch + 1);
    const int tb = 256;
    int launches = 0;
    k_ploc_init<<<(T + tb - 1) / tb, tb, 0, st>>>(sc.tris, T, cid[0], cbox[0]);
    ++launches;
    PlocState h{T, T - 1};
    int cur = 0;
    cudaError_t e = cudaMemcpyAsync(state, &h, sizeof h, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return DPCS_ERR_CUDA;
    while (h.n > kPlocSmall) {
        // a round leaves about two thirds of the clusters: stop the batch where
        // the small kernel can take over
        int rounds = 0;
        for (double left = h.n; rounds < kPlocBatch && left > kPlocSmall; ++rounds) left *= 0.66;
        const int g = (h.n + tb - 1) / tb;
        for (int r = 0; r < rounds; ++r) {
            k_ploc_nn<<<(h.n + kPlocBlock - 1) / kPlocBlock, kPlocBlock, 0, st>>>(cbox[cur], state + r, nn);
            k_ploc_count<<<g, tb, 0, st>>>(nn, state + r, bcount);
            k_ploc_compact<<<g, tb, 0, st>>>(nn, state + r, bcount, cid[cur], cbox[cur], cid[1 - cur], cbox[1 - cur], nodes);
            launches += 3;
            cur = 1 - cur;
        }
        const int32_t before = h.n;
        e = cudaMemcpyAsync(&h, state + rounds, sizeof h, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return DPCS_ERR_CUDA;
        // every round merges; each merge takes one cluster and makes one node
        if (h.n < 1 || h.n >= before || h.next != h.n - 1) return DPCS_ERR_DEVICE_CHECK;
        e = cudaMemcpyAsync(state, state + rounds, sizeof h, cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) return DPCS_ERR_CUDA;
    }
    if (h.n > 1) {
        k_ploc_small<<<1, kPlocSmall, 0, st>>>(state, cid[cur], cbox[cur], nodes);
        ++launches;
    }
    // depth of the new tree against the traversal stack (only a finished tree is walked)
    k_parents<<<(T - 1 + tb - 1) / tb, tb, 0, st>>>(nodes, T, parent, state);
    cudaMemsetAsync(depth, 0, 4, st);
    k_tree_depth<<<(T + tb - 1) / tb, tb, 0, st>>>(parent, T, max_depth + 1, depth, state);
    launches += 2;
    int32_t d = 0;
    e = cudaMemcpyAsync(&h, state, sizeof h, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&d, depth, 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return DPCS_ERR_CUDA;
    if (h.n != 1 || h.next != 0) return DPCS_ERR_DEVICE_CHECK;
    *depth_out = d;
    if (d > max_depth) return launches;  // too deep for the traversal stack: the radix tree stays
    e = cudaMemcpyAsync(sc.nodes, nodes, (n - 1) * 64, cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return DPCS_ERR_CUDA;
    sc.root = 0;
    return launches;
}

size_t lbvh_scratch_bytes(int32_t T) {
    const size_t n = (size_t)(T > 0 ? T : 1);
    const size_t nb = (n + kSortTile - 1) / kSortTile;
    return align256(3 * n * 4) + align256(6 * 4) + 4 * align256(n * 4) + align256(256 * nb * 4) +
           align256((2 * n) * 4) + align256(n * 4);
}

size_t lbvh_refit_scratch_bytes(int32_t T) {
    const size_t n = (size_t)(T > 0 ? T : 1);
    return align256((2 * n) * 4) + align256(n * 4);
}

int launch_lbvh_refit(const float *d_verts, Scene &sc, void *scratch, size_t scratch_bytes, cudaStream_t st) {
    const int T = sc.T;
    if (T <= 0) return 0;
    if (scratch_bytes < lbvh_refit_scratch_bytes(T)) return DPCS_ERR_INVALID_ARG;
    const size_t n = (size_t)T;
    int32_t *parent = (int32_t *)scratch;
    int32_t *flags = (int32_t *)((char *)scratch + align256(2 * n * 4));
    const int tb = 256, gb = (T + tb - 1) / tb;
    int launches = 0;
    if (T >= 2) {
        cudaMemsetAsync(flags, 0, n * 4, st);
        k_parents<<<(T - 1 + tb - 1) / tb, tb, 0, st>>>(sc.nodes, T, parent, nullptr);
        ++launches;
    }
    k_refit<<<gb, tb, 0, st>>>(d_verts, sc.vidx, sc.uv, sc.order, T, sc.nodes, parent, flags, sc.tris, sc.tuv);
    return launches + 1;
}

namespace {
struct Rigid {
    float R[9], t[3];
};
__global__ void k_rigid(const float *__restrict__ in, int32_t V, const Rigid m, float *__restrict__ out) {
    const int32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= V) return;
    const float x = in[3 * v], y = in[3 * v + 1], z = in[3 * v + 2];
    out[3 * v] = m.R[0] * x + m.R[1] * y + m.R[2] * z + m.t[0];
    out[3 * v + 1] = m.R[3] * x + m.R[4] * y + m.R[5] * z + m.t[1];
    out[3 * v + 2] = m.R[6] * x + m.R[7] * y + m.R[8] * z + m.t[2];
}
}  // namespace

int launch_rigid_transform(const float *in, int32_t V, const float R[9], const float t[3], float *out,
                           cudaStream_t st) {
    if (V <= 0) return 0;
    Rigid m;
    for (int i = 0; i < 9; ++i) m.R[i] = R[i];
    for (int i = 0; i < 3; ++i) m.t[i] = t[i];
    k_rigid<<<(V + 255) / 256, 256, 0, st>>>(in, V, m, out);
    return 1;
}

int launch_lbvh_build(const float *d_verts, int32_t V, const int32_t *d_tris, int32_t T, const float *d_uv,
                      Scene &sc, void *scratch, size_t scratch_bytes, cudaStream_t st) {
    (void)V;
    if (T <= 0) {
        sc.root = kEmptyRoot;
        return 0;
    }
    if (scratch_bytes < lbvh_scratch_bytes(T)) return DPCS_ERR_INVALID_ARG;
    const size_t n = (size_t)T;
    const int nb = (int)((n + kSortTile - 1) / kSortTile);
    char *p = (char *)scratch;
    auto take = [&](size_t bytes) {
        char *r = p;
        p += align256(bytes);
        return (void *)r;
    };
    float *cen = (float *)take(3 * n * 4);
    uint32_t *bounds = (uint32_t *)take(6 * 4);
    uint32_t *ka = (uint32_t *)take(n * 4), *kb = (uint32_t *)take(n * 4);
    int32_t *va = (int32_t *)take(n * 4), *vb = (int32_t *)take(n * 4);
    uint32_t *hist = (uint32_t *)take(256 * (size_t)nb * 4);
    int32_t *parent = (int32_t *)take(2 * n * 4);
    int32_t *flags = (int32_t *)take(n * 4);
    // digit totals of a sort pass: the counters themselves when there is one
    // block, else 1 KB of the flags, which only the refit uses
    uint32_t *dtotal = nb == 1 ? hist : (uint32_t *)flags;
    int launches = 0;
    const int tb = 256, gb = (T + tb - 1) / tb;
    cudaMemsetAsync(bounds, 0xff, 3 * 4, st);
    cudaMemsetAsync(bounds + 3, 0, 3 * 4, st);
    k_centroids<<<gb, tb, 0, st>>>(d_verts, d_tris, T, cen, bounds);
    k_morton<<<gb, tb, 0, st>>>(cen, bounds, T, ka, va);
    launches += 2;
    for (int shift = 0; shift < 32; shift += 8) {
        k_radix_hist<<<nb, kSortTile, 0, st>>>(ka, T, shift, nb, hist);
        if (nb > 1) k_radix_rows<<<256, 256, 0, st>>>(hist, nb, dtotal);
        k_radix_scatter<<<nb, kSortTile, 0, st>>>(ka, va, kb, vb, T, shift, nb, nb > 1 ? hist : nullptr, dtotal);
        launches += nb > 1 ? 3 : 2;
        uint32_t *tk = ka; ka = kb; kb = tk;
        int32_t *tv = va; va = vb; vb = tv;
    }
    // after 4 passes the sorted data is back in (ka, va)
    cudaMemcpyAsync(sc.codes, ka, n * 4, cudaMemcpyDeviceToDevice, st);
    cudaMemcpyAsync(sc.order, va, n * 4, cudaMemcpyDeviceToDevice, st);
    if (T >= 2) {
        cudaMemsetAsync(flags, 0, n * 4, st);
        k_karras<<<(T - 1 + tb - 1) / tb, tb, 0, st>>>(ka, T, sc.nodes, parent);
        ++launches;
    }
    k_refit<<<gb, tb, 0, st>>>(d_verts, d_tris, d_uv, va, T, sc.nodes, parent, flags, sc.tris, sc.tuv);
    ++launches;
    sc.root = T >= 2 ? 0 : ~0;
    return launches;
}

}  // namespace dpcs
