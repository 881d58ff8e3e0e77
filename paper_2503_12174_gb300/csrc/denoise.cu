// denoise.cu -- the differentiable denoiser of Eq. 11, Ic' = D(Ic), as a
// cross-bilateral filter guided by noise-free first-hit features.
//
//   guide g(p): albedo (3), normal towards the camera (3), hit distance, hit
//               flag of the ray through pixel centre p (k_gbuffer);
//   D(I)(p)   = sum_q w(p,q) I(q) / W(p),   W(p) = sum_q w(p,q);
//   w(p,q)    = exp(-|p-q|^2 ks - |da|^2 ka - |dn|^2 kn - dt^2 kd),
//               k = 1 / (2 sigma^2), or 0 for a feature that is switched off,
//               q over the (2r+1)^2 window around p inside the image.
//
// The weights depend on the guide only, so D is linear in I and, because
// w(p,q) = w(q,p) over a symmetric window, its adjoint is the same gather
// applied to dD / W without the normalisation:
//   dI(q) = sum_p w(q,p) (dD(p) / W(p)).
// Both directions run one kernel: a 16 x 16 output tile per CTA with its
// (16 + 2r)^2 halo of guide and image staged in shared memory, so each input
// is read from HBM once per tile instead of (2r+1)^2 times; each thread
// computes a vertical strip of outputs that share the taps they load.
#include <cuda_runtime.h>
#include <stdint.h>

#include "device.cuh"
#include "internal.h"

namespace dpcs {

namespace {

constexpr int kTile = 16;
constexpr int kMaxRadius = 8;  // (16 + 16)^2 pixels x 40 B = 40 KiB of shared memory

// First-hit guide through each camera pixel centre (a.jitter must be 0).
__global__ void k_gbuffer(const RenderArgs a, float4 *__restrict__ guide) {
    const int64_t pix = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (pix >= (int64_t)a.Hc * a.Wc) return;
    f3 o, d;
    camera_ray(a, (uint32_t)pix, 0u, o, d);
    const Ray ray = make_ray(o, d);
    Hit h;
    Cnt cnt;
    float4 g0 = make_float4(0.f, 0.f, 0.f, 0.f), g1 = g0;
    if (traverse(a.nodes, a.tris, a.root, a.T, ray, INFINITY, false, h, a.status, cnt)) {
        const Surf S = surface_at(a, h, ray.d);
        g0 = make_float4(S.rho.x, S.rho.y, S.rho.z, S.n.x);
        g1 = make_float4(S.n.y, S.n.z, h.t, 1.0f);
    }
    guide[2 * pix] = g0;
    guide[2 * pix + 1] = g1;
}

struct Widths {
    float ks, ka, kn, kd;  // 1 / (2 sigma^2) per term; 0 = term off
};

// two FP32 lanes in one instruction (each rounded as the scalar operation)
typedef unsigned long long u64;
__device__ __forceinline__ u64 pair(float a, float b) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ u64 pair(float2 v) { return pair(v.x, v.y); }
__device__ __forceinline__ float2 unpair(u64 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
    u64 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
    u64 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
    u64 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ float ex2(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// The filter, two vertically stacked outputs per thread.
// kAdjoint = false: out = D(img), wsum = W (wsum may be null).
// kAdjoint = true : out += D^T(img), where img is dD and wsum the forward W.
//
// The taps are FP32 work on shared memory (121 taps x 24 operations an output
// at r = 5; DRAM traffic is 4 % of the time), so the kernel counts
// instructions.  The guide and the image sit in shared memory one feature a
// plane, and a thread takes two horizontally adjacent taps at a time: one
// 8-byte load a feature and packed FP32 operations, half the instructions of
// one tap at a time.  Pairs start on even columns, so a window row is r pairs
// and one tap left over at its right (even outputs) or left end, which runs as
// a pair of its guide with itself, a distance term that makes the second weight
// 0 and no image beside it (0 times an infinite one would be NaN); it loads
// nothing outside the window, whose NaN would otherwise count.  The
// widths carry log2(e), and a weight is one ex2 of the whole exponent
// (against 64 bits the filter's error is 1.8e-7, with expf it was 2.7e-7).
// 1024 x 1024 at r = 5, forward / adjoint, one tap at a time -> pairs: 0.193 /
// 0.191 -> 0.148 / 0.165 ms; r = 8, 1000 x 700: 0.344 / 0.333 -> 0.216 / 0.231
// ms (the packed FP32 pipe is 61 % busy).  Four outputs a thread instead of
// two 2 to 8 % slower at r = 8 and as fast at 5; 64 registers (8 blocks an
// SM) 16 % slower.
constexpr int kFeat = 10;   // albedo 3, normal 3, depth, image 3
constexpr int kStrip = 2;   // outputs per thread (the window tests below are written for two)
constexpr float kFar = 1e30f;

template <bool kAdjoint>
__global__ void __launch_bounds__(kTile *kTile / kStrip)
    k_bilateral(const float *__restrict__ img, const float4 *__restrict__ guide, const float *__restrict__ wsum_in,
                int H, int W, int r, Widths k, float *__restrict__ out, float *__restrict__ wsum_out) {
    extern __shared__ float smem[];
    const int S = kTile + 2 * r, N = S * S;  // S is even
    float2 *dist = reinterpret_cast<float2 *>(smem + kFeat * N);  // [parity][pair]: -dx^2 ks of the pair's taps
    constexpr int kThreads = kTile * kTile / kStrip;
    constexpr float kLog2e = 1.44269504088896340736f;
    const float nks = -k.ks * kLog2e;
    const int tid = threadIdx.y * kTile + threadIdx.x;
    const int y0 = blockIdx.y * kTile - r, x0 = blockIdx.x * kTile - r;
    for (int i = tid; i < N; i += kThreads) {
        // a column beside the image repeats the guide of the nearest one, a tap
        // of every window that reaches past it, with no image
        const int gy = y0 + i / S, gx = x0 + i % S, cx = min(max(gx, 0), W - 1);
        float f[kFeat] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (gy >= 0 && gy < H) {
            const int64_t p = (int64_t)gy * W + cx;
            const float4 g0 = __ldg(guide + 2 * p), g1 = __ldg(guide + 2 * p + 1);
            const float s = kAdjoint ? 1.0f / __ldg(wsum_in + p) : 1.0f;
            f[0] = g0.x; f[1] = g0.y; f[2] = g0.z; f[3] = g0.w;
            f[4] = g1.x; f[5] = g1.y; f[6] = g1.z;
            if (cx == gx) {
                f[7] = __ldg(img + 3 * p) * s;
                f[8] = __ldg(img + 3 * p + 1) * s;
                f[9] = __ldg(img + 3 * p + 2) * s;
            }
        }
#pragma unroll
        for (int q = 0; q < kFeat; ++q) smem[q * N + i] = f[q];
    }
    if (tid < 2 * r) {
        const int d = 2 * (tid % r) - r + tid / r;  // first tap's dx
        dist[tid] = make_float2((float)(d * d) * nks, (float)((d + 1) * (d + 1)) * nks);
    }
    __syncthreads();
    const int px = blockIdx.x * kTile + threadIdx.x;
    if (px >= W) return;
    const int par = threadIdx.x & 1;
    const int ry = threadIdx.y * kStrip;  // the strip's first output row in the tile
    const int py = blockIdx.y * kTile + ry;
    u64 c[kStrip][7];
    u64 ax[kStrip], ay[kStrip], az[kStrip], den[kStrip];
#pragma unroll
    for (int o = 0; o < kStrip; ++o) {
        const int at = (ry + o + r) * S + threadIdx.x + r;
#pragma unroll
        for (int q = 0; q < 7; ++q) c[o][q] = pair(smem[q * N + at], smem[q * N + at]);
        ax[o] = ay[o] = az[o] = den[o] = 0ull;
    }
    const float ka = -k.ka * kLog2e, kn = -k.kn * kLog2e, kd = -k.kd * kLog2e;
    const u64 nka = pair(ka, ka), nkn = pair(kn, kn), nkd = pair(kd, kd), neg = pair(-1.0f, -1.0f);
    const bool edge = x0 < 0 || x0 + S > W;  // some taps fall off the image's sides
    // window rows, relative to the first output, inside the image
    const int j0 = max(-r, -py), j1 = min(r + kStrip - 1, H - 1 - py);
    for (int j = j0; j <= j1; ++j) {
        const float *row = smem + (ry + j + r) * S + threadIdx.x;
        const bool on[kStrip] = {j <= r, j > -r};  // is the row in the output's window?
        const u64 dy[kStrip] = {pair((float)(j * j) * nks, (float)(j * j) * nks),
                                pair((float)((j - 1) * (j - 1)) * nks, (float)((j - 1) * (j - 1)) * nks)};
        auto taps = [&](const u64 (&f)[kFeat], u64 dx) {
#pragma unroll
            for (int o = 0; o < kStrip; ++o) {
                if (!on[o]) continue;
                u64 d[7];
#pragma unroll
                for (int n = 0; n < 7; ++n) d[n] = fma2(f[n], neg, c[o][n]);
                const u64 da = fma2(d[2], d[2], fma2(d[1], d[1], mul2(d[0], d[0])));
                const u64 dn = fma2(d[5], d[5], fma2(d[4], d[4], mul2(d[3], d[3])));
                u64 e = add2(dx, dy[o]);
                e = fma2(da, nka, e);
                e = fma2(dn, nkn, e);
                e = fma2(mul2(d[6], d[6]), nkd, e);
                const float2 x = unpair(e);
                const u64 w = pair(ex2(x.x), ex2(x.y));
                ax[o] = fma2(w, f[7], ax[o]);
                ay[o] = fma2(w, f[8], ay[o]);
                az[o] = fma2(w, f[9], az[o]);
                den[o] = add2(den[o], w);
            }
        };
        u64 f[kFeat];
        for (int p = 0; p < r; ++p) {
            const float2 *q = reinterpret_cast<const float2 *>(row + par + 2 * p);
            float2 dx = dist[par * r + p];
            if (edge) {
                const int gx = x0 + (int)threadIdx.x + par + 2 * p;
                if (gx < 0 || gx >= W) dx.x = -kFar;
                if (gx + 1 < 0 || gx + 1 >= W) dx.y = -kFar;
            }
#pragma unroll
            for (int n = 0; n < kFeat; ++n) f[n] = pair(q[n * (N / 2)]);
            taps(f, pair(dx));
        }
        {  // the tap left over, at the window's right or left end
            const int at = par ? 0 : 2 * r, gx = x0 + (int)threadIdx.x + at;
#pragma unroll
            for (int n = 0; n < kFeat; ++n) f[n] = pair(row[n * N + at], n < 7 ? row[n * N + at] : 0.0f);
            taps(f, pair(gx < 0 || gx >= W ? -kFar : (float)(r * r) * nks, -kFar));
        }
    }
#pragma unroll
    for (int o = 0; o < kStrip; ++o) {
        if (py + o >= H) break;
        const int64_t p = (int64_t)(py + o) * W + px;
        const float2 x = unpair(ax[o]), y = unpair(ay[o]), z = unpair(az[o]), n = unpair(den[o]);
        if (kAdjoint) {
            out[3 * p] += x.x + x.y;
            out[3 * p + 1] += y.x + y.y;
            out[3 * p + 2] += z.x + z.y;
        } else {
            const float dn = n.x + n.y, inv = 1.0f / dn;
            out[3 * p] = (x.x + x.y) * inv;
            out[3 * p + 1] = (y.x + y.y) * inv;
            out[3 * p + 2] = (z.x + z.y) * inv;
            if (wsum_out) wsum_out[p] = dn;
        }
    }
}

}  // namespace

}  // namespace dpcs

using namespace dpcs;

namespace {

dpcs_status check_denoise_args(dpcs_ctx *c, const float *img, const float *guide, int32_t Hc, int32_t Wc,
                               const dpcs_denoise_params *prm, const float *out, Widths &k) {
    if (!img || !guide || !out || !prm || Hc <= 0 || Wc <= 0)
        return ctx_fail(c, DPCS_ERR_INVALID_ARG, "denoise: null pointer or empty image");
    if (((uintptr_t)guide & 15u) != 0)
        return ctx_fail(c, DPCS_ERR_INVALID_ARG, "denoise: guide must be 16-byte aligned");
    if (prm->radius < 0 || prm->radius > kMaxRadius || !(prm->sigma_s > 0.0f))
        return ctx_fail(c, DPCS_ERR_INVALID_ARG, "denoise: radius must be in [0, 8] and sigma_s > 0");
    auto inv2 = [](float s) { return s > 0.0f ? 0.5f / (s * s) : 0.0f; };
    k.ks = inv2(prm->sigma_s);
    k.ka = inv2(prm->sigma_albedo);
    k.kn = inv2(prm->sigma_normal);
    k.kd = inv2(prm->sigma_depth);
    return cudaSetDevice(ctx_device(c)) == cudaSuccess ? DPCS_OK
                                                        : ctx_fail(c, DPCS_ERR_CUDA, "denoise: cudaSetDevice");
}

template <bool kAdjoint>
dpcs_status launch_bilateral(dpcs_ctx *c, const float *img, const float *guide, const float *wsum_in, int32_t Hc,
                             int32_t Wc, int r, const Widths &k, float *out, float *wsum_out, cudaStream_t st) {
    const int S = kTile + 2 * r;
    const size_t shm = ((size_t)kFeat * S * S + 4 * r) * sizeof(float);
    const dim3 grid((Wc + kTile - 1) / kTile, (Hc + kTile - 1) / kTile);
    k_bilateral<kAdjoint><<<grid, dim3(kTile, kTile / kStrip), shm, st>>>(img, (const float4 *)guide, wsum_in, Hc, Wc, r, k,
                                                                         out, wsum_out);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return ctx_fail(c, DPCS_ERR_CUDA, cudaGetErrorString(e));
    ctx_add_launches(c, 1);
    return DPCS_OK;
}

}  // namespace

extern "C" {

dpcs_status dpcs_gbuffer(dpcs_ctx *c, dpcs_scene scene, const float *albedo, const float *rough, int32_t Ht,
                         int32_t Wt, const dpcs_view *view, float *guide, void *stream) {
    if (!c) return DPCS_ERR_INVALID_ARG;
    if (!guide || ((uintptr_t)guide & 15u) != 0)
        return ctx_fail(c, DPCS_ERR_INVALID_ARG, "gbuffer: guide must be a 16-byte aligned device pointer");
    dpcs_params prm{};
    prm.gamma_p[0] = prm.gamma_p[1] = prm.gamma_p[2] = 1.0f;
    prm.gamma_c[0] = prm.gamma_c[1] = prm.gamma_c[2] = 1.0f;
    prm.wb[0] = prm.wb[1] = prm.wb[2] = 1.0f;
    prm.gain_p = prm.gain_c = prm.k_proj = 1.0f;
    prm.rr_q = 1.0f;
    RenderArgs a;
    dpcs_status s = ctx_render_args(c, scene, albedo, rough, Ht, Wt, albedo, view, &prm, 1, 1, 0, a);
    if (s) return s;
    if (cudaSetDevice(ctx_device(c)) != cudaSuccess) return ctx_fail(c, DPCS_ERR_CUDA, "gbuffer: cudaSetDevice");
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t nt = (int64_t)Ht * Wt, npix = (int64_t)view->Hc * view->Wc;
    float4 *tex = nullptr;  // the packed texture, only for this call
    cudaError_t e = cudaMallocAsync((void **)&tex, (size_t)nt * 16, st);
    if (e != cudaSuccess) return ctx_fail(c, DPCS_ERR_OOM, "gbuffer: texture allocation failed");
    int nl = launch_pack_tex(albedo, rough, nt, tex, st);
    a.tex = tex;
    a.jitter = 0;  // rays through pixel centres
    a.counters = nullptr;
    k_gbuffer<<<(unsigned)((npix + 127) / 128), 128, 0, st>>>(a, (float4 *)guide);
    e = cudaGetLastError();
    cudaFreeAsync(tex, st);
    if (nl < 0 || e != cudaSuccess) return ctx_fail(c, DPCS_ERR_CUDA, "gbuffer: launch failed");
    ctx_add_launches(c, nl + 1);
    return DPCS_OK;
}

dpcs_status dpcs_denoise(dpcs_ctx *c, const float *Ic, const float *guide, int32_t Hc, int32_t Wc,
                         const dpcs_denoise_params *prm, float *out, float *wsum, void *stream) {
    if (!c) return DPCS_ERR_INVALID_ARG;
    Widths k;
    dpcs_status s = check_denoise_args(c, Ic, guide, Hc, Wc, prm, out, k);
    if (s) return s;
    if (out == Ic) return ctx_fail(c, DPCS_ERR_INVALID_ARG, "denoise: out must not alias the input");
    return launch_bilateral<false>(c, Ic, guide, nullptr, Hc, Wc, prm->radius, k, out, wsum, (cudaStream_t)stream);
}

dpcs_status dpcs_denoise_backward(dpcs_ctx *c, const float *dOut, const float *guide, const float *wsum, int32_t Hc,
                                  int32_t Wc, const dpcs_denoise_params *prm, float *dIc, void *stream) {
    if (!c) return DPCS_ERR_INVALID_ARG;
    Widths k;
    dpcs_status s = check_denoise_args(c, dOut, guide, Hc, Wc, prm, dIc, k);
    if (s) return s;
    if (!wsum) return ctx_fail(c, DPCS_ERR_INVALID_ARG, "denoise_backward: wsum from dpcs_denoise is required");
    if (dIc == dOut) return ctx_fail(c, DPCS_ERR_INVALID_ARG, "denoise_backward: dIc must not alias dOut");
    return launch_bilateral<true>(c, dOut, guide, wsum, Hc, Wc, prm->radius, k, dIc, nullptr, (cudaStream_t)stream);
}

}  // extern "C"
