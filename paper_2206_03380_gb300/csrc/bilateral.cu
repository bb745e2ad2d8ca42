// Cross-bilateral denoiser (App. B "Bilateral Denoiser": the spatial part of
// SVGF, evaluated densely over the footprint, gradients to the colours only):
//   c_hat(p) = sum_q c(q) w(p, q) / W(p),   W(p) = sum_q w(p, q)
//   w(p, q)  = exp(-|p - q|^2 / (2 sigma^2))
//            * exp(-|z(p) - z(q)| / (sigma_z |grad z(p) . (p - q)| + 1e-3 z(p)))
//            * max(0, n(p) . n(q))^128,  sigma_z = 1
// z is camera-space depth, grad z the central difference over covered
// neighbours (one-sided at borders and coverage edges), n the normalised
// G-buffer normal; uncovered pixels pass through and are never neighbours.
// Forward: one pass over the footprint accumulates every image of a view with
// the same weights.  Backward: the transpose as a gather, g(q) = sum_p g(p)
// w(p, q) / W(p) over the footprint of q, with W saved by the forward (no
// atomics, so the gradient is deterministic).
//
// A CTA owns a tile of one view, 32 pixels wide, each thread two pixels of a
// column; depth, normal and the colours of all images over the tile plus its
// halo are staged in shared memory.  What bounds it is three things at about the
// same level, per weight and warp: some 30 issued instructions, 2 MUFU
// operations (16 cycles of a scheduler) and shared-memory wavefronts (12 per
// neighbour for two images), then the staging's latency.  So a neighbour loaded
// once meets two pixels, their arithmetic goes in packed pairs, the two
// exponentials are one (base 2), slopes are
// staged in the backward instead of formed per weight, and uncovered neighbours
// (zero normal and colours) take no branch.  Measured, two images: 512 x 512,
// sigma 2: forward 45 us, backward 50; 3 x 700 x 611, sigma 3.9: 324 and 410
// (a pixel per thread, two exponentials and a division per weight, a branch per
// neighbour: 63 and 81, 630 and 816).  Four pixels per thread halve the loads
// but leave too few warps: 56 and 57, 377 and 480.
#include "internal.h"

namespace mcdi {
namespace {

constexpr int kTileW = 32;
constexpr int kRows = 2;  // pixels of a thread, in one column
constexpr int kPairs = kRows / 2;
constexpr int kUnroll = 3;
// Warps of a CTA: 4, or 8 from radius 7, where the staged halo leaves an SM room
// for 12 warps in CTAs of 4 and 16 in CTAs of 8.  Measured (4 / 8 warps, forward
// and backward): radius 8, 3 x 700 x 611: 385 + 438 / 328 + 373 us; radius 4,
// 512 x 512: 45 + 47 / 52 + 53 us (fewer, larger CTAs level the coverage less).
constexpr int kMaxWarps = 8, kWideRadius = 6;
constexpr int kMaxImgPerView = 4;
constexpr float kEpsRel = 1e-3f;  // sigma_z = 1
constexpr float kLog2E = 1.44269504088896341f;

struct Guide {  // one staged pixel
    float z;    // camera-space depth, < 0: uncovered or outside the image
    float nx, ny, nz;
};

__device__ __forceinline__ Guide load_guide(const float4* pos, const float4* nrm, const mcdi_camera& C, int H, int W,
                                            size_t base, int x, int y) {
    Guide g{-1.0f, 0.0f, 0.0f, 0.0f};
    const bool inside = x >= 0 && y >= 0 && x < W && y < H;
    const size_t i = base + (inside ? (size_t)y * W + x : 0);
    const float4 p = pos[i], n = nrm[i];  // together: the staging waits for memory once
    if (!inside || !(p.w > 0.0f)) return g;
    const float l = sqrtf(fmaf(n.z, n.z, fmaf(n.x, n.x, __fmul_rn(n.y, n.y))));
    const float inv = l > 0.0f ? 1.0f / l : 0.0f;
    g.z = fmaf(p.z - C.origin[2], C.forward[2],
               fmaf(p.y - C.origin[1], C.forward[1], __fmul_rn(p.x - C.origin[0], C.forward[0])));
    g.nx = n.x * inv;
    g.ny = n.y * inv;
    g.nz = n.z * inv;
    return g;
}

// central difference over covered neighbours, one-sided where one is missing
__device__ __forceinline__ float depth_slope(float zm, float z0, float zp) {
    const bool cm = zm >= 0.0f, cp = zp >= 0.0f;
    return cm && cp ? 0.5f * (zp - zm) : (cp ? zp - z0 : (cm ? z0 - zm : 0.0f));
}

// slopes of the staged pixel at sg[0] (rows gw apart)
__device__ __forceinline__ float2 slopes_of(const Guide* sg, int gw) {
    return make_float2(depth_slope(sg[-1].z, sg[0].z, sg[1].z), depth_slope(sg[-gw].z, sg[0].z, sg[gw].z));
}
__device__ __forceinline__ float eps_of(float z) { return kEpsRel * fabsf(z); }

__device__ __forceinline__ float exp2_approx(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Two weights: spatial part of the argument (base 2) `ws`, depth change that the
// slope predicts over the offset `pred`, depth offset `eps`, depth difference
// `dz`, cosine of the normals `nn`.  Where the slopes are steep and cancel along
// the offset, pred's rounding decides the weight: it is gx dx + gy dy with the
// first product fused, in the forward and in the backward.
__device__ __forceinline__ float2 weight_pair(float2 ws, float2 pred, float2 eps, float2 dz, float2 nn) {
    const float ax = fmaf(-kLog2E * fabsf(dz.x), __fdividef(1.0f, fabsf(pred.x) + eps.x), ws.x);
    const float ay = fmaf(-kLog2E * fabsf(dz.y), __fdividef(1.0f, fabsf(pred.y) + eps.y), ws.y);
    float2 v = make_float2(fmaxf(nn.x, 0.0f), fmaxf(nn.y, 0.0f));
#pragma unroll
    for (int i = 0; i < 7; ++i) v = mul2(v, v);
    return mul2(v, make_float2(exp2_approx(ax), exp2_approx(ay)));
}

__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }

struct Tile {  // staged extents: the guides one ring wider (slopes) than the colours
    int gw, gh, cw, ch;
    __host__ __device__ Tile(int R, int warps)
        : gw(kTileW + 2 * R + 2), gh(kRows * warps + 2 * R + 2), cw(kTileW + 2 * R), ch(kRows * warps + 2 * R) {}
};

// kRows weights of staged row s (relative to the thread's first pixel) are used
// by pixels i with |s - i| <= R; the others' colours are left out (an infinity
// outside the footprint must not meet a zero weight).
template <int K, bool kBackward, bool kEdge>
__device__ __forceinline__ void filter_row(const Guide* g, const float2* slope, const float4* c, size_t cplane, int R,
                                           int s, float spatial, const float2 (&z)[kPairs], const float2 (&nx)[kPairs],
                                           const float2 (&ny)[kPairs], const float2 (&nz)[kPairs], const float2 (&gx)[kPairs],
                                           const float2 (&gy)[kPairs], const float2 (&eps)[kPairs], float2 (&acc)[K][3][kPairs],
                                           float2 (&wt)[kPairs]) {
    float2 ws_row[kPairs], pred_row[kPairs], dy[kPairs];
#pragma unroll
    for (int h = 0; h < kPairs; ++h) {
        dy[h] = make_float2((float)(s - 2 * h), (float)(s - 2 * h - 1));
        ws_row[h] = mul2(mul2(dy[h], dy[h]), both(spatial));
        if (!kBackward) pred_row[h] = mul2(gy[h], dy[h]);
    }
#pragma unroll kUnroll
    for (int dx = -R; dx <= R; ++dx) {
        const Guide q = g[dx];
        const float fx = (float)dx;
        const float ws_col = spatial * (fx * fx);
        float2 sl = make_float2(0.0f, 0.0f);
        float ep = 0.0f;
        if (kBackward) {  // the neighbour is the weight's centre; the offset's sign drops out
            sl = slope[dx];
            ep = eps_of(q.z);
        }
#pragma unroll
        for (int h = 0; h < kPairs; ++h) {
            const bool v0 = !kEdge || abs(s - 2 * h) <= R, v1 = !kEdge || abs(s - 2 * h - 1) <= R;
            if (kEdge && !v0 && !v1) continue;
            const float2 pred = kBackward ? fma2(both(sl.x), both(fx), mul2(both(sl.y), dy[h])) : fma2(gx[h], both(fx), pred_row[h]);
            const float2 nn = fma2(nx[h], both(q.nx), fma2(ny[h], both(q.ny), mul2(nz[h], both(q.nz))));
            float2 w = weight_pair(add2(ws_row[h], both(ws_col)), pred, kBackward ? both(ep) : eps[h],
                                   make_float2(z[h].x - q.z, z[h].y - q.z), nn);
            if (kEdge) w = make_float2(v0 ? w.x : 0.0f, v1 ? w.y : 0.0f);
            if (!kBackward) wt[h] = add2(wt[h], w);
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const float4 v = c[k * cplane + dx];
                const float2 cx = kEdge ? make_float2(v0 ? v.x : 0.0f, v1 ? v.x : 0.0f) : both(v.x);
                const float2 cy = kEdge ? make_float2(v0 ? v.y : 0.0f, v1 ? v.y : 0.0f) : both(v.y);
                const float2 cz = kEdge ? make_float2(v0 ? v.z : 0.0f, v1 ? v.z : 0.0f) : both(v.z);
                acc[k][0][h] = fma2(w, cx, acc[k][0][h]);
                acc[k][1][h] = fma2(w, cy, acc[k][1][h]);
                acc[k][2][h] = fma2(w, cz, acc[k][2][h]);
            }
        }
    }
}

// Forward: in = colours, wsum written.  Backward: in = upstream gradients,
// divided by wsum as they are staged.
template <int K, bool kBackward>
__global__ void __launch_bounds__(32 * kMaxWarps) bilateral_kernel(const float4* __restrict__ pos,
                                                             const float4* __restrict__ nrm,
                                                             const mcdi_camera* __restrict__ cams, int N, int H, int W,
                                                             const float4* __restrict__ in, float inv2s2, int R,
                                                             const float* __restrict__ wsum_in,
                                                             float4* __restrict__ out, float* __restrict__ wsum_out) {
    pdl_prologue();
    extern __shared__ float4 smem[];
    const int threads = blockDim.x;
    const Tile T(R, threads >> 5);
    const int view = blockIdx.z;
    const int x0 = blockIdx.x * kTileW, y0 = blockIdx.y * kRows * (threads >> 5);
    Guide* sg = reinterpret_cast<Guide*>(smem);
    const size_t cplane = (size_t)T.cw * T.ch;
    float4* sc = smem + T.gw * T.gh;                               // K planes
    float2* ss = reinterpret_cast<float2*>(sc + K * cplane);       // slopes (backward)
    const mcdi_camera C = cams[view];
    const size_t plane = (size_t)H * W, gbase = (size_t)view * plane;
#pragma unroll 4
    for (int i = threadIdx.x; i < T.gw * T.gh; i += threads) {
        const int sy = i / T.gw, sx = i - sy * T.gw;
        sg[i] = load_guide(pos, nrm, C, H, W, gbase, x0 + sx - (R + 1), y0 + sy - (R + 1));
    }
#pragma unroll 4
    for (int i = threadIdx.x; i < (int)cplane; i += threads) {
        const int sy = i / T.cw, x = x0 + i - sy * T.cw - R, y = y0 + sy - R;
        const bool inside = x >= 0 && y >= 0 && x < W && y < H;
        const size_t p = inside ? (size_t)y * W + x : 0;
        const float w = kBackward ? wsum_in[gbase + p] : 1.0f;
        const float iw = 1.0f / w;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            float4 v = in[(size_t)(view + k * N) * plane + p];
            if (kBackward) v = make_float4(v.x * iw, v.y * iw, v.z * iw, 0.0f);
            sc[k * cplane + i] = inside && w > 0.0f ? v : make_float4(0, 0, 0, 0);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < (int)cplane; i += threads) {
        const int sy = i / T.cw, sx = i - sy * T.cw;
        const Guide* g = sg + (sy + 1) * T.gw + sx + 1;
        const bool covered = !(g->z < 0.0f);
        if (!covered) {
#pragma unroll
            for (int k = 0; k < K; ++k) sc[k * cplane + i] = make_float4(0, 0, 0, 0);
        }
        if (kBackward) ss[i] = covered ? slopes_of(g, T.gw) : make_float2(0.0f, 0.0f);
    }
    __syncthreads();
    const int tx = threadIdx.x & 31, ty = (threadIdx.x >> 5) * kRows;
    const int x = x0 + tx, y = y0 + ty;
    if (x >= W || y >= H) return;
    const Guide* g0 = sg + (ty + R + 1) * T.gw + tx + R + 1;  // the thread's first pixel
    const float4* c0 = sc + (ty + R) * T.cw + tx + R;
    const float2* s0 = ss + (ty + R) * T.cw + tx + R;
    float2 z[kPairs], nx[kPairs], ny[kPairs], nz[kPairs], gx[kPairs], gy[kPairs], eps[kPairs], acc[K][3][kPairs], wt[kPairs];
    bool any = false;
#pragma unroll
    for (int h = 0; h < kPairs; ++h) {
        const Guide a = g0[2 * h * T.gw], b = g0[(2 * h + 1) * T.gw];
        any |= !(a.z < 0.0f) || !(b.z < 0.0f);
        z[h] = make_float2(a.z, b.z);
        nx[h] = make_float2(a.nx, b.nx);
        ny[h] = make_float2(a.ny, b.ny);
        nz[h] = make_float2(a.nz, b.nz);
        if (!kBackward) {
            const float2 sa = slopes_of(g0 + 2 * h * T.gw, T.gw), sb = slopes_of(g0 + (2 * h + 1) * T.gw, T.gw);
            gx[h] = make_float2(sa.x, sb.x);
            gy[h] = make_float2(sa.y, sb.y);
            eps[h] = make_float2(eps_of(a.z), eps_of(b.z));
        }
        wt[h] = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int k = 0; k < K; ++k)
#pragma unroll
            for (int c = 0; c < 3; ++c) acc[k][c][h] = make_float2(0.0f, 0.0f);
    }
    if (any) {
        const float spatial = -inv2s2 * kLog2E;
        for (int s = -R; s <= R + kRows - 1; ++s) {
            const Guide* g = g0 + s * T.gw;
            const float4* c = c0 + s * T.cw;
            const float2* sl = s0 + s * T.cw;
            if (s >= kRows - 1 - R && s <= R)
                filter_row<K, kBackward, false>(g, sl, c, cplane, R, s, spatial, z, nx, ny, nz, gx, gy, eps, acc, wt);
            else
                filter_row<K, kBackward, true>(g, sl, c, cplane, R, s, spatial, z, nx, ny, nz, gx, gy, eps, acc, wt);
        }
    }
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
        const int h = i >> 1;
        if (y + i >= H) break;
        const size_t p = (size_t)(y + i) * W + x;
        const bool covered = !((i & 1 ? z[h].y : z[h].x) < 0.0f);
        const float w = i & 1 ? wt[h].y : wt[h].x;
        const float inv = kBackward ? 1.0f : 1.0f / w;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const size_t o = (size_t)(view + k * N) * plane + p;
            float3 v;
            if (covered) {
                v.x = (i & 1 ? acc[k][0][h].y : acc[k][0][h].x) * inv;
                v.y = (i & 1 ? acc[k][1][h].y : acc[k][1][h].x) * inv;
                v.z = (i & 1 ? acc[k][2][h].y : acc[k][2][h].x) * inv;
            } else {  // pass through
                const float4 t = in[o];
                v = make_float3(t.x, t.y, t.z);
            }
            out[o] = make_float4(v.x, v.y, v.z, 0.0f);
        }
        if (!kBackward) wsum_out[gbase + p] = covered ? w : 0.0f;
    }
}

template <int K, bool kBackward>
cudaError_t launch_k_images(const float4* pos, const float4* nrm, const mcdi_camera* cams, int N, int H, int W,
                            const float4* in, float sigma, int R, const float* wsum_in, float4* out, float* wsum_out,
                            cudaStream_t s) {
    const int warps = R > kWideRadius ? kMaxWarps : kMaxWarps / 2;
    const Tile T(R, warps);
    const size_t smem = (size_t)T.gw * T.gh * sizeof(Guide) + (size_t)K * T.cw * T.ch * sizeof(float4) +
                        (kBackward ? (size_t)T.cw * T.ch * sizeof(float2) : 0);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute((const void*)bilateral_kernel<K, kBackward>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const dim3 grid((W + kTileW - 1) / kTileW, (H + kRows * warps - 1) / (kRows * warps), N);
    launch_k(bilateral_kernel<K, kBackward>, grid, 32 * warps, smem, s, pos, nrm, cams, N, H, W, in,
             1.0f / (2.0f * sigma * sigma), R, wsum_in, out, wsum_out);
    return cudaGetLastError();
}

template <bool kBackward, typename... A>
cudaError_t launch_images(int K, A... a) {
    switch (K) {
        case 1: return launch_k_images<1, kBackward>(a...);
        case 2: return launch_k_images<2, kBackward>(a...);
        case 3: return launch_k_images<3, kBackward>(a...);
        default: return launch_k_images<4, kBackward>(a...);
    }
}

}  // namespace

int bilateral_max_images_per_view() { return kMaxImgPerView; }

cudaError_t launch_bilateral(bool backward, const float* gb_pos, const float* gb_nrm, const mcdi_camera* cams, int N,
                             int H, int W, int n_img, const float* in, float sigma, int R, const float* wsum_in,
                             float* out, float* wsum_out, cudaStream_t s) {
    const int K = n_img / N;
    const auto* pos = reinterpret_cast<const float4*>(gb_pos);
    const auto* nrm = reinterpret_cast<const float4*>(gb_nrm);
    const auto* src = reinterpret_cast<const float4*>(in);
    auto* dst = reinterpret_cast<float4*>(out);
    return backward ? launch_images<true>(K, pos, nrm, cams, N, H, W, src, sigma, R, wsum_in, dst, wsum_out, s)
                    : launch_images<false>(K, pos, nrm, cams, N, H, W, src, sigma, R, wsum_in, dst, wsum_out, s);
}

}  // namespace mcdi
