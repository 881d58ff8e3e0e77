// tile.cuh -- path tracing over block tiles.
//
// A block owns S path lanes ("slots": the L lanes of its pixels, as in
// render.cu) whose state lives in shared memory, and runs them one bounce at
// a time in three phases with a barrier between them:
//
//   trace   the extension rays of the live slots and the shadow rays of the
//           vertices shaded last, 32 rays per warp at a time;
//   shade   every hit: surface, light, continuation;
//   sort    the new extension rays by direction (octant and dominant axis).
//
// What bounds a path kernel here is instruction issue with few lanes active:
// with one path per lane throughout, lanes wait for the longest traversal of
// their warp, and lanes whose path has ended wait for the others' (13.5 of
// 32 lanes active).  Phases compact both: a warp gets 32 live rays, neighbours
// in direction, so their walks down the tree have similar lengths, and 32
// hits to shade (22 of 32 lanes active, 0.83 G warp instructions instead of
// 1.19 G; corner 256 x 256 at 64 spp, 3 bounces: 1.367 -> 1.048 ms on GB300;
// 640 x 360 at 35 spp, whose second round has 3 lanes of 32: 4.12 -> 2.55 ms).
// Of that the direction sort gives 5 %.  Tiles of one or three slots a thread
// were 15 and 9 % slower than of two; letting a slot take its next sample as
// soon as its path ended mixed bounces in the phases and was 9 % slower.
//
// Every slot runs its samples in order and adds its lit vertices in vertex
// order, and the per-vertex arithmetic is device.cuh's, so a pixel's result
// does not depend on the schedule.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "device.cuh"
#include "internal.h"

namespace dpcs {

constexpr unsigned kFull = 0xffffffffu;
constexpr int32_t kDone = kEmptyRoot;  // no leaf reference: positions stay below 2^28
constexpr int kBins = 24;              // directions: octant x dominant axis

template <int S>
struct Tile {
    float o[3][S];         // origin of the slot's extension and shadow rays
    float d[3][S];         // extension direction
    float h[3][S];         // (leaf position, u, v) of the extension ray's hit
    float beta[3][S];      // throughput entering the next vertex
    float c[3][S];         // contribution waiting for its shadow ray
    float sum[3][S];       // lane sum over the samples so far
    uint16_t ext[S];       // slots with an extension ray to trace, by direction
    uint16_t shadow[S];    // slots with a shadow ray to trace
    uint16_t hits[S];      // slots to shade
    uint16_t rank[S];      // rank of the slot's extension ray within its bin
    uint8_t key[S];        // its bin, or 255: the path has ended
    int bin[32];           // extension rays per bin
    int next;              // 32-ray chunks taken by the trace phase
    int nhit, nshadow;
    int work;              // persistent kernels: the tile in hand
};

__device__ __forceinline__ f3 ld3(const float *p, int n, int i) { return mk3(p[i], p[n + i], p[2 * n + i]); }
__device__ __forceinline__ void st3(float *p, int n, int i, f3 v) {
    p[i] = v.x;
    p[n + i] = v.y;
    p[2 * n + i] = v.z;
}

// append v of the lanes with `take` to a list shared by the block
__device__ __forceinline__ void tile_append(uint16_t *list, int *n, int v, bool take) {
    const unsigned m = __ballot_sync(kFull, take);
    if (!m) return;
    const int lane = threadIdx.x & 31;
    int base = 0;
    if (lane == 0) base = atomicAdd(n, __popc(m));
    base = __shfl_sync(kFull, base, 0);
    if (take) list[base + __popc(m & ((1u << lane) - 1u))] = (uint16_t)v;
}

__device__ __forceinline__ int dir_bin(f3 d) {
    const float ax = fabsf(d.x), ay = fabsf(d.y), az = fabsf(d.z);
    const int k = ax > ay ? (ax > az ? 0 : 2) : (ay > az ? 1 : 2);
    return 8 * k + (d.x < 0.f ? 1 : 0) + (d.y < 0.f ? 2 : 0) + (d.z < 0.f ? 4 : 0);
}

// ---------------------------------------------------------------------------
// traversal
// ---------------------------------------------------------------------------
// One step down the tree: 50 instructions against the 54 of trav_resume's with
// plain slabs (a chain of nodes with one child hit each).  The stack grows down from
// stack[kStack]; its last place, which no tree the library builds needs, leaves
// room = -1, and the caller ends the ray.
__device__ __forceinline__ void tree_node(const RenderArgs &a, const Ray &ray, float ht, int &node, int &room, int *stack,
                                          Cnt &cnt) {
    cnt.add_warp(kCntTravWarpIter);
    cnt.add(kCntNode);
    const float4 *nd = reinterpret_cast<const float4 *>(reinterpret_cast<const char *>(a.nodes) +
                                                        (size_t)(uint32_t)node * 64u);
    float4 n0, n1, n2, n3;
    ldg8(nd, n0, n1);
    ldg8(nd + 2, n2, n3);
    float tl, tr;
#if DPCS_SLAB_FMA
    const u64 ix = pk2(ray.inv.x, ray.inv.x), iy = pk2(ray.inv.y, ray.inv.y), iz = pk2(ray.inv.z, ray.inv.z);
    const u64 ox = pk2(-ray.oinv.x, -ray.oinv.x), oy = pk2(-ray.oinv.y, -ray.oinv.y),
              oz = pk2(-ray.oinv.z, -ray.oinv.z);
    const bool hl = slab2(pk2(n0.x, n0.y), pk2(n0.z, n0.w), pk2(n2.x, n2.y), ix, iy, iz, ox, oy, oz, ray.err, ht, tl);
    const bool hr = slab2(pk2(n1.x, n1.y), pk2(n1.z, n1.w), pk2(n2.z, n2.w), ix, iy, iz, ox, oy, oz, ray.err, ht, tr);
#else
    const bool hl = slab(ray, n0.x, n0.y, n0.z, n0.w, n2.x, n2.y, ht, tl);
    const bool hr = slab(ray, n1.x, n1.y, n1.z, n1.w, n2.z, n2.w, ht, tr);
#endif
    const int cl = __float_as_int(n3.x), cr = __float_as_int(n3.y);
    const bool lf = tl <= tr;
    if (hl | hr) {
        const bool takel = hl & (lf | !hr);
        node = takel ? cl : cr;
        if (hl & hr) stack[room--] = takel ? cr : cl;
    } else {
        node = room < kStack ? stack[++room] : kDone;
    }
}

// Closest hit (any = false; ht = infinity at the start) or any hit before ht,
// from node = a.root; lanes with node = kDone only take part in the warp's
// votes.  hpos < 0: nothing hit.
//
// A lane takes up to kBurst steps down the tree, then the warp meets and the
// lanes at a leaf test it.  Without the limit all lanes wait for the one that
// is longest on its way to a leaf, which curved surfaces, whose boxes overlap,
// make long.  384 x 384 x 16 spp, 4 bounces, in parts of the lanes kernel's time
// before there were tiles, without a limit and in bursts of 1 / 2 / 3 / 4 / 6:
// closed sphere of 1,280 triangles 1.24, 1.09 / 0.98 / 0.97 / 0.97 / 0.99; half
// sphere of 1,600 0.97, 0.87 / 0.80 / 0.80 / 0.80 / 0.83; corner 0.73, 0.82 / 0.77 /
// 0.76 / 0.75 / 0.75, whose flat walls need no limit.  (With the triangle test's
// present form bursts of 4 take 0.94, 0.78 and 0.73.)  Unrolled, renders are 2 to
// 4 % faster, the kernels that record 1 to 5 % slower.
//
// As in trav_resume every step, node or leaf, counts towards the visit cap: a
// ray that would take one more reports it and ends as a miss, so a walk ends
// whatever the tree holds.  The inner loop's one comparison tests the node, the
// burst (which the cap cuts) and the stack together; tested one by one they
// cost 1.3 to 2.4 % more.
constexpr int kBurst = 4;
template <bool kUnrolled>
__device__ __forceinline__ void tree_walk(const RenderArgs &a, const Ray &ray, bool any, int node, int &hpos, float &ht,
                                          float &hu, float &hv, Cnt &cnt) {
    int stack[kStack + 1];
    int room = kStack, left = (a.visit_cap > 0 ? a.visit_cap : 2 * a.T + 16) - 1;  // steps after the next one
    while (true) {
        const int most = min(kBurst - 1, left);
        int go = most;
#pragma unroll (kUnrolled ? kBurst : 1)
        while ((node | go | room) >= 0) {
            --go;
#ifdef DPCS_CHECK
            if (node >= a.T - 1) {
                atomicOr(a.status, kStatusBoundsCheck);
                hpos = -1;
                node = kDone;
                break;
            }
#endif
            tree_node(a, ray, ht, node, room, stack, cnt);
        }
        __syncwarp();
        left -= most - go;
        if (node != kDone && (left | room) < 0) {
            atomicOr(a.status, kStatusTraversalLimit);
            hpos = -1;
            node = kDone;
        }
#ifdef DPCS_CHECK
        if (node < 0 && node != kDone && ~node >= a.T) {
            atomicOr(a.status, kStatusBoundsCheck);
            hpos = -1;
            node = kDone;
        }
#endif
        if (node < 0 && node != kDone) {
            --left;
            cnt.add_warp(kCntTravWarpIter);
            cnt.add(kCntTri);
            const int pos = ~node;
            const float4 A = __ldg(a.tris + 3 * pos + 0);
            const float4 B = __ldg(a.tris + 3 * pos + 1);
            const float4 C = __ldg(a.tris + 3 * pos + 2);
            float t, u, v;
            if (tri_isect(ray, xyz(A), xyz(B), xyz(C), ht, t, u, v)) {
                // ties in t to the lowest original triangle index
                if (t < ht || (!any && hpos >= 0 && __float_as_int(A.w) < __float_as_int(__ldg(a.tris + 3 * hpos).w))) {
                    hpos = pos;
                    ht = t;
                    hu = u;
                    hv = v;
                    if (any) room = kStack;
                }
            }
            node = room < kStack ? stack[++room] : kDone;
        }
        if (__all_sync(kFull, node == kDone)) break;
    }
}

// Trace the tile's ne extension rays and ns shadow rays, 32 of a kind per warp
// at a time: closest hits into h and the list of hits; shadow rays (from o to
// the projector's centre) add their contribution c to the slot's sum, or tell
// the core that vertex v of round k is dark.
template <int S, class Core>
__device__ __forceinline__ void tile_trace(const RenderArgs &a, Core &core, Tile<S> &P, int ne, int ns, int k, int v,
                                           Cnt &cnt) {
    const int lane = threadIdx.x & 31;
    const int ce = (ne + 31) >> 5, chunks = ce + ((ns + 31) >> 5);
    while (true) {
        int c = 0;
        if (lane == 0) c = atomicAdd(&P.next, 1);
        c = __shfl_sync(kFull, c, 0);
        if (c >= chunks) break;
        const bool any = c >= ce;
        const int i = 32 * (any ? c - ce : c) + lane;
        const bool on = i < (any ? ns : ne);
        const int slot = on ? (any ? P.shadow[i] : P.ext[i]) : 0;
        int node = kDone, hpos = -1;
        float ht = INFINITY, hu = 0.f, hv = 0.f;
        Ray ray;
        if (on) {
            const f3 o = ld3(&P.o[0][0], S, slot);
            f3 d = ld3(&P.d[0][0], S, slot);
            if (any) {  // nee_prepare's shadow ray from its origin
                const f3 sv = mk3(a.cp[0], a.cp[1], a.cp[2]) - o;
                const float sd = sqrtf(dot(sv, sv));
                d = sv * (1.0f / sd);
                ht = sd - kRayEps;
            }
            cnt.add(any ? kCntShadow : kCntRay);
            ray = make_ray(o, d);
            node = a.root;
        }
        cnt.add_warp(kCntPathWarpIter);
        __syncwarp();
        tree_walk<Core::kUnrolled>(a, ray, any, node, hpos, ht, hu, hv, cnt);
        if (any) {
            if (on) {
                if (hpos < 0) {
                    st3(&P.sum[0][0], S, slot, ld3(&P.sum[0][0], S, slot) + ld3(&P.c[0][0], S, slot));
                    cnt.add(kCntLit);
                } else {
                    core.dark(a, slot, k, v);
                }
            }
        } else {
            if (hpos >= 0) st3(&P.h[0][0], S, slot, mk3(__int_as_float(hpos), hu, hv));
            tile_append(P.hits, &P.nhit, slot, hpos >= 0);
        }
        __syncwarp();
    }
}

// What shading a vertex hands back to the tile.
struct Shaded {
    bool cand, ext;  // a shadow ray carrying c is due; the path goes on along wi with throughput beta
    f3 c, so, wi, beta;
};

// Round k of the tile's slots: sample sl + k L of pixel `pix` for every slot
// whose live(slot, pix) is true.  `lane0` is the first slot's lane among the
// launch's (pixel, lane) pairs, `pix0` the pixel of lane 0, `nlane` the lanes
// there are.  Every thread of the block calls it; it ends with a barrier.
template <int B, int S, class Core>
__device__ __forceinline__ void tile_round(const RenderArgs &a, Core &core, Tile<S> &P, int64_t pix0, int64_t lane0,
                                           int64_t nlane, int k, Cnt &cnt) {
    const int L = 1 << a.log2L, tid = threadIdx.x, lane = tid & 31;
    if (tid == 0) P.next = P.nhit = P.nshadow = 0;
    if (tid < 32) P.bin[tid] = 0;
    __syncthreads();
#pragma unroll 1
    for (int slot = tid; slot < S; slot += B) {
        const int64_t gt = lane0 + slot;
        const uint32_t pix = (uint32_t)(pix0 + (gt >> a.log2L));
        const int s = (int)(gt & (L - 1)) + k * L;
        const bool live = gt < nlane && s < a.spp && core.begin(a, slot, pix, k);
        if (live) {
            f3 o, d;
            camera_ray(a, pix, (uint32_t)s, o, d);
            st3(&P.o[0][0], S, slot, o);
            st3(&P.d[0][0], S, slot, d);
            st3(&P.beta[0][0], S, slot, mk3(1.f, 1.f, 1.f));
            cnt.add(kCntPath);
        }
        tile_append(P.ext, &P.bin[0], slot, live);
    }
    __syncthreads();
    int ne = P.bin[0], ns = 0;
    __syncthreads();
    // Three barriers a bounce.  Each counter is cleared in a phase that
    // neither adds to it nor reads it: the bins and the shadow count while
    // the rays are traced, the hit count and the chunk counter after shading.
    for (int b = 1;; ++b) {
        if (tid < 32) P.bin[tid] = 0;
        if (tid == 32) P.nshadow = 0;
        tile_trace<S>(a, core, P, ne, ns, k, b - 2, cnt);
        __syncthreads();
        const int nh = P.nhit;
        if (nh == 0) break;
#pragma unroll 1
        for (int i0 = tid & ~31; i0 < nh; i0 += B) {
            const int i = i0 + lane;
            const bool on = i < nh;
            const int slot = on ? P.hits[i] : 0;
            bool cand = false;
            if (on) {
                cnt.add(kCntVert);
                const int64_t gt = lane0 + slot;
                Hit h;
                h.pos = __float_as_int(P.h[0][slot]);
                h.u = P.h[1][slot];
                h.v = P.h[2][slot];
                Shaded R;
                core.shade(a, slot, (uint32_t)(pix0 + (gt >> a.log2L)), (uint32_t)((int)(gt & (L - 1)) + k * L), k, b, h,
                           ld3(&P.d[0][0], S, slot), ld3(&P.beta[0][0], S, slot), R);
                cand = R.cand;
                if (cand) st3(&P.c[0][0], S, slot, R.c);
                int key = 255;
                if (R.ext) {
                    cnt.add(kCntCont);
                    st3(&P.beta[0][0], S, slot, R.beta);
                    st3(&P.d[0][0], S, slot, R.wi);
                    key = dir_bin(R.wi);
                    P.rank[slot] = (uint16_t)atomicAdd(&P.bin[key], 1);
                }
                P.key[slot] = (uint8_t)key;
                st3(&P.o[0][0], S, slot, R.so);
            }
            __syncwarp();
            tile_append(P.shadow, &P.nshadow, slot, cand);
        }
        __syncthreads();
        if (tid == 0) P.nhit = P.next = 0;
        // every warp scans the bins (one a lane) and places its share of the rays
        const int count = P.bin[lane];
        int end = count;
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(kFull, end, off);
            if (lane >= off) end += y;
        }
        ne = __shfl_sync(kFull, end, 31);
        ns = P.nshadow;
#pragma unroll 1
        for (int i0 = tid & ~31; i0 < nh; i0 += B) {
            const int slot = i0 + lane < nh ? P.hits[i0 + lane] : 0;
            const int key = i0 + lane < nh ? P.key[slot] : 255;
            const int first = __shfl_sync(kFull, end - count, key & 31);
            if (key != 255) P.ext[first + P.rank[slot]] = (uint16_t)slot;
        }
        __syncthreads();
    }
    __syncthreads();
}

template <int S>
__device__ __forceinline__ void tile_clear_sums(Tile<S> &P, int B) {
#pragma unroll 1
    for (int slot = threadIdx.x; slot < S; slot += B) st3(&P.sum[0][0], S, slot, mk3(0.f, 0.f, 0.f));
}

// the slot's lane sum combined over the L lanes of its pixel (the xor tree of
// render_lanes); every thread of the warp calls it with its slot
template <int S>
__device__ __forceinline__ f3 tile_pixel_sum(const Tile<S> &P, int slot, int L) {
    f3 sum = ld3(&P.sum[0][0], S, slot);
    for (int off = L >> 1; off > 0; off >>= 1) {
        sum.x += __shfl_xor_sync(kFull, sum.x, off);
        sum.y += __shfl_xor_sync(kFull, sum.y, off);
        sum.z += __shfl_xor_sync(kFull, sum.z, off);
    }
    return sum;
}

// the Lambert + GGX material, nothing recorded
struct PlainCore {
    static constexpr bool kUnrolled = true;  // tree_walk
    __device__ __forceinline__ bool begin(const RenderArgs &, int, uint32_t, int) { return true; }
    __device__ __forceinline__ void dark(const RenderArgs &, int, int, int) {}
    __device__ __forceinline__ void shade(const RenderArgs &a, int, uint32_t pix, uint32_t s, int, int b, const Hit &h,
                                          f3 d, f3 beta, Shaded &R) {
        const Surf F = surface_at(a, h, d);
        Nee Q;
        R.cand = nee_prepare(a, F, Q);
        if (R.cand) {
            unsigned unc;
            R.c = nee_contrib(a, beta, Q, unc);
        }
        R.ext = false;
        if (b < a.bounces) {
            Cont C;
            R.ext = continue_prepare(a, pix, s, b, F, C);
            if (R.ext) {
                R.beta = beta * C.w;
                R.wi = C.wi;
            }
        }
        R.so = madd(F.x, F.n, kRayEps);
    }
};

// ---------------------------------------------------------------------------
// pixels
// ---------------------------------------------------------------------------
__device__ __forceinline__ float crf(float ec, float gain, float wb, float gamma) {
    const float a = gain * wb * ec;
    return a > 0.0f ? powf(a, gamma) : 0.0f;
}

// Eqs. 4 and 5 of one pixel from the sum over its samples
__device__ __forceinline__ void write_pixel(const RenderArgs &a, int64_t pix, f3 sum) {
    const float inv = 1.0f / (float)a.spp;
    const float ex = sum.x * inv, ey = sum.y * inv, ez = sum.z * inv;
    if (a.Ec) {
        a.Ec[3 * pix] = ex;
        a.Ec[3 * pix + 1] = ey;
        a.Ec[3 * pix + 2] = ez;
    }
    a.Ic[3 * pix] = crf(ex, a.gain_c, a.wb[0], a.gamma_c[0]);
    a.Ic[3 * pix + 1] = crf(ey, a.gain_c, a.wb[1], a.gamma_c[1]);
    a.Ic[3 * pix + 2] = crf(ez, a.gain_c, a.wb[2], a.gamma_c[2]);
}

// The one-trace step's pixel: Eqs. 4 and 5, the loss, and through Eq. 5 the
// gradient of each sample's radiance (gb_in); the pixel's first lane (sl = 0)
// also writes Ec and Ic and adds to v: gamma_c(3), Gc, wb(3), loss.
__device__ __forceinline__ void pixel_loss_grad(const RenderArgs &a, const LossArgs &l, int64_t pix, int sl, f3 sum,
                                                float gb_in[3], float v[8]) {
    const float inv = 1.0f / (float)a.spp;
    const float ec[3] = {sum.x * inv, sum.y * inv, sum.z * inv};
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        gb_in[j] = 0.0f;
        const float ic = crf(ec[j], a.gain_c, a.wb[j], a.gamma_c[j]);
        if (sl == 0) {
            if (a.Ec) a.Ec[3 * pix + j] = ec[j];
            a.Ic[3 * pix + j] = ic;
        }
        const float d = ic - l.target[3 * pix + j];
        const float g = l.kind == 0 ? l.scale * d : (d > 0.0f ? l.scale : (d < 0.0f ? -l.scale : 0.0f));
        const float w = a.gain_c * a.wb[j] * ec[j];
        if (w > 0.0f) {
            const float da = a.gamma_c[j] * powf(w, a.gamma_c[j] - 1.0f);
            gb_in[j] = g * da * a.gain_c * a.wb[j] * inv;
            if (sl == 0) {
                v[j] += g * ic * logf(w);
                v[3] += g * da * a.wb[j] * ec[j];
                v[4 + j] += g * da * a.gain_c * ec[j];
            }
        }
        if (sl == 0) v[7] += l.kind == 0 ? 0.5f * l.scale * d * d : l.scale * fabsf(d);
    }
}

// ---------------------------------------------------------------------------
// block reduction of NV floats into FP64 accumulators
// ---------------------------------------------------------------------------
template <int NV>
__device__ __forceinline__ void block_reduce_add(float (&v)[NV], double *acc) {
    __shared__ float red[NV][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k)
        for (int off = 16; off; off >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], off);
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < NV; ++k) red[k][w] = v[k];
    __syncthreads();
    if (threadIdx.x < NV) {
        float s = 0.0f;
        for (int j = 0; j < (int)(blockDim.x >> 5); ++j) s += red[threadIdx.x][j];
        if (s != 0.0f) atomicAdd(acc + threadIdx.x, (double)s);
    }
}

// The image of a tile: every round of its S lanes from lane0 on, then their
// pixels.  Lane 0 belongs to pixel pix0, and there are nlane lanes.
template <int B, int S, class Core>
__device__ __forceinline__ void tile_image(const RenderArgs &a, Core &core, Tile<S> &P, int64_t pix0, int64_t lane0,
                                           int64_t nlane) {
    const int L = 1 << a.log2L;
    Cnt cnt;
    tile_clear_sums<S>(P, B);
    const int rounds = a.root != kEmptyRoot ? (a.spp + L - 1) / L : 0;
    for (int k = 0; k < rounds; ++k) tile_round<B, S>(a, core, P, pix0, lane0, nlane, k, cnt);
    cnt.flush(a.counters);
    __syncthreads();
#pragma unroll 1
    for (int slot = threadIdx.x; slot < S; slot += B) {
        const int64_t gt = lane0 + slot;
        const f3 sum = tile_pixel_sum<S>(P, slot, L);
        if (gt < nlane && (gt & (L - 1)) == 0) write_pixel(a, pix0 + (gt >> a.log2L), sum);
    }
}

// The one-trace step (l.target set) or the replay (l.target null: a.gE holds
// dLoss/dEc) over block tiles.  Persistent: a block takes tiles from a counter
// and keeps its records (`chunks` 16-byte chunks a vertex) in its own part of
// `scratch`.  The gain over the lanes kernels is the compaction's, and that a
// record is written once to its place where those spill it to local memory: 512
// x 512 at 16 spp, gradient of Ip, 2.07 -> 1.50 ms.  The records of the blocks
// in flight (90 MB at three vertices a lane, 360 at most) do not stay in L2:
// nearly every byte goes to DRAM and most come back.  sweep(k, slot, gb) sweeps the slot's path of round k.
template <int B, int S, class Core, class Sweep>
__device__ __forceinline__ void tile_adjoint(const RenderArgs &a, Core &core, Tile<S> &P, const LossArgs &l, char *scratch,
                                             size_t per_block, int64_t ntile, unsigned long long *counter, int chunks,
                                             Sweep sweep) {
    const int L = 1 << a.log2L, tid = threadIdx.x;
    const int64_t nlane = ((int64_t)a.Hc * a.Wc) << a.log2L;
    const bool replay = l.target == nullptr;
    const int rounds = (a.spp + L - 1) / L, spl = replay ? 1 : rounds;
    Cnt cnt;
    core.chunks = reinterpret_cast<uint4 *>(scratch + blockIdx.x * per_block);
    core.nvs = reinterpret_cast<uint8_t *>(core.chunks + (size_t)chunks * spl * a.bounces * S);
    core.nthr = S;
    core.t0 = 0;
    core.spl = spl;
    core.replay = replay;
    const float inv = 1.0f / (float)a.spp;
    while (true) {
        if (tid == 0) {
            const unsigned long long t = atomicAdd(counter, 1ull);
            P.work = t < (unsigned long long)ntile ? (int)t : -1;
        }
        tile_clear_sums<S>(P, B);
        __syncthreads();
        const int tile = P.work;
        if (tile < 0) break;
        const int64_t lane0 = (int64_t)tile * S;
        for (int k = 0; k < rounds; ++k) {
            tile_round<B, S>(a, core, P, 0, lane0, nlane, k, cnt);
            if (!replay) continue;
#pragma unroll 1
            for (int slot = tid; slot < S; slot += B) {
                const int64_t gt = lane0 + slot, pix = gt >> a.log2L;
                if (gt >= nlane || (int)(gt & (L - 1)) + k * L >= a.spp) continue;
                const float gb_in[3] = {a.gE[3 * pix] * inv, a.gE[3 * pix + 1] * inv, a.gE[3 * pix + 2] * inv};
                sweep(k, slot, gb_in);
            }
            __syncthreads();
        }
        if (replay) continue;
        float v[8] = {0, 0, 0, 0, 0, 0, 0, 0};  // gamma_c(3), Gc, wb(3), loss
#pragma unroll 1
        for (int slot = tid; slot < S; slot += B) {
            const int64_t gt = lane0 + slot, pix = gt >> a.log2L;
            const int sl = (int)(gt & (L - 1));
            const f3 sum = tile_pixel_sum<S>(P, slot, L);
            if (gt >= nlane) continue;
            float gb_in[3];
            pixel_loss_grad(a, l, pix, sl, sum, gb_in, v);
            if (gb_in[0] == 0.0f && gb_in[1] == 0.0f && gb_in[2] == 0.0f) continue;
            for (int k = 0; sl + k * L < a.spp; ++k) sweep(k, slot, gb_in);
        }
        __syncthreads();
        block_reduce_add<8>(v, l.acc + 4);  // acc[4..10]: gamma_c, Gc, wb; acc[11]: the loss
        __syncthreads();
    }
    cnt.flush(a.counters);
}

// ---------------------------------------------------------------------------
// dispatch
// ---------------------------------------------------------------------------
// Where the tiles pay (GB300; in parts of the time that the lanes kernels took
// before there were tiles, of which today's take 0.85 to 0.98).
//
// Paths of one bounce have nothing to compact (plane 512 x 512 at 16 spp 206 /
// 230 us).  With two there is little, and images of 0.5 to 2 M lanes, whose last
// wave of large tiles is long, took 0.94 to 1.06 (corner, heightfields, rooms,
// spheres) where every round of samples is full: lanes there, 0.90 to 0.98.
// (Samples that leave part of the last round's lanes idle cost tiles nothing:
// 0.74 of the corner with 35 samples on 32 lanes, 1.2 M.)  Longer paths, 2.4 M
// lanes, 4 bounces: corner walls of 1,026 / 8,226 triangles 0.73 / 0.75, a room of
// 2,352 / 8,112 0.90 / 0.88, a half sphere of 1,600 / 6,400 0.78 / 0.79, closed
// spheres of 1,280 / 5,120 0.94 / 0.92, heightfields of 2,048 / 7,200 0.91 / 0.91.
// A tree of some MB no longer sits in the L1 that the tiles' shared memory
// leaves: heightfields of 20,000 and 51,200 in lanes 0.93, in tiles 0.96 and more.
//
// Kernels that keep vertex records win for longer, since a tile writes them
// once: one-trace steps, 4 bounces, lanes / tiles, at 147 k and 2.4 M lanes:
// corner 0.88 / 0.87 and 0.92 / 0.70, closed spheres of 1,280 / 20,480 triangles
// 0.84 / 0.87 and 0.86 / 1.00, 0.85 / 0.88 and 0.89 / 0.96, heightfields of 20,000 /
// 51,200 0.96 / 1.03 and 0.94 / 0.81, 0.91 / 0.90 and 0.94 / 0.83.
//
// Small images want more, smaller tiles: steps in tiles of 64 / 256 lanes take
// 0.87 / 1.08 (corner), 0.87 / 1.30 (sphere), 0.87 / 1.09 (heightfield of 7,200) at
// 147 k lanes, 0.91 / 0.82, 0.89 / 0.98, 0.95 / 0.87 at 590 k and 0.92 / 0.73, 0.88 /
// 1.03, 0.98 / 0.89 at 1 M.
constexpr int32_t kTileTriangles = 10240;
constexpr int32_t kRecordTriangles = 65536;
constexpr int64_t kTileLanes = 500000;
inline int64_t path_lanes(const RenderArgs &a) { return ((int64_t)a.Hc * a.Wc) << a.log2L; }
// do these arguments run in the small tiles?
inline bool small_tiles(const RenderArgs &a) { return path_lanes(a) < kTileLanes; }
// do the samples fill the rounds of a pixel's lanes (35 samples on 32 lanes do not)?
inline bool full_rounds(const RenderArgs &a) {
    const int64_t L = int64_t(1) << a.log2L;
    return 10 * (int64_t)a.spp >= 9 * ((a.spp + L - 1) / L) * L;
}
// renders
inline bool tiled(const RenderArgs &a) {
    const bool middle = path_lanes(a) >= kTileLanes && path_lanes(a) < 4 * kTileLanes;
    return a.bounces > 1 && a.T <= kTileTriangles && !(a.bounces == 2 && middle && full_rounds(a));
}
// kernels that record every vertex
inline bool tiled_records(const RenderArgs &a) { return a.bounces > 1 && a.T <= kRecordTriangles; }
// blocks of b threads that the GPU holds at once: the persistent grid
inline int resident_blocks(int b) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms * (1024 / b);
}

// one block's records: S slots of `words` 32-bit words a vertex
inline size_t tile_block_bytes(const RenderArgs &a, bool replay, int S, int words) {
    const int L = 1 << a.log2L;
    const size_t spl = replay ? 1 : (size_t)((a.spp + L - 1) / L);
    return (spl * S * ((size_t)words * 4 * a.bounces + 1) + 255) & ~size_t(255);
}

// blocks of B threads that take the tiles of S lanes from their counter
inline int64_t tile_blocks(const RenderArgs &a, int B, int S) {
    const int64_t ntile = (path_lanes(a) + S - 1) / S, most = resident_blocks(B);
    return ntile < most ? ntile : most;
}

inline size_t tile_scratch_bytes(const RenderArgs &a, bool replay, int words) {
    if (!tiled_records(a) || a.root == kEmptyRoot) return 0;
    return small_tiles(a) ? (size_t)tile_blocks(a, 64, 64) * tile_block_bytes(a, replay, 64, words)
                          : (size_t)tile_blocks(a, 128, 256) * tile_block_bytes(a, replay, 256, words);
}

struct TileGrid {
    unsigned grid;
    int64_t ntile;
    size_t per_block;
    unsigned long long *counter;
};
inline TileGrid tile_grid(const RenderArgs &a, const LossArgs &l, int B, int S, int words) {
    TileGrid g;
    g.ntile = (path_lanes(a) + S - 1) / S;
    g.grid = (unsigned)tile_blocks(a, B, S);
    g.per_block = tile_block_bytes(a, l.target == nullptr, S, words);
    g.counter = reinterpret_cast<unsigned long long *>(l.acc + kTileCounter);
    return g;
}

}  // namespace dpcs
