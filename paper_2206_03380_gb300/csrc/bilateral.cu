// Cross-bilateral denoiser (App. B "Bilateral Denoiser": the spatial part of
// SVGF, evaluated densely over the footprint, gradients to the colours only):
//   c_hat(p) = sum_q c(q) w(p, q) / W(p),   W(p) = sum_q w(p, q)
//   w(p, q)  = exp(-|p - q|^2 / (2 sigma^2))
//            * exp(-|z(p) - z(q)| / (sigma_z |grad z(p) . (p - q)| + 1e-3 z(p)))
//            * max(0, n(p) . n(q))^128,  sigma_z = 1
// z is camera-space depth, grad z the central difference over covered
// neighbours (one-sided at borders and coverage edges), n the normalised
// G-buffer normal; uncovered pixels pass through and are never neighbours.
// Forward: one CTA per 16 x 16 tile of one view; depth, normal and the colours
// of all images of that view over the tile plus its halo are staged in shared
// memory, and one pass over the footprint accumulates every image with the
// same weights.  Backward: the transpose as a gather, g(q) = sum_p g(p) w(p, q)
// / W(p) over the footprint of q, with W saved by the forward (no atomics, so
// the gradient is deterministic).
#include <type_traits>

#include "internal.h"

namespace mcdi {
namespace {

constexpr int kTile = 16;
constexpr int kMaxImgPerView = 4;
constexpr float kSigmaZ = 1.0f;
constexpr float kEpsRel = 1e-3f;

struct Guide {  // one staged pixel
    float z;    // camera-space depth, < 0: uncovered or outside the image
    float nx, ny, nz;
};

__device__ __forceinline__ Guide load_guide(const float4* pos, const float4* nrm, const mcdi_camera& C, int H, int W,
                                            size_t base, int x, int y) {
    Guide g{-1.0f, 0.0f, 0.0f, 0.0f};
    if (x < 0 || y < 0 || x >= W || y >= H) return g;
    const float4 p = pos[base + (size_t)y * W + x];
    if (!(p.w > 0.0f)) return g;
    const float4 n = nrm[base + (size_t)y * W + x];
    const float l = sqrtf(n.x * n.x + n.y * n.y + n.z * n.z);
    const float inv = l > 0.0f ? 1.0f / l : 0.0f;
    g.z = (p.x - C.origin[0]) * C.forward[0] + (p.y - C.origin[1]) * C.forward[1] + (p.z - C.origin[2]) * C.forward[2];
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

__device__ __forceinline__ float pow128(float d) {
    float v = fmaxf(d, 0.0f);
#pragma unroll
    for (int i = 0; i < 7; ++i) v *= v;
    return v;
}

struct Center {  // the pixel p of a weight w(p, q)
    float z, gx, gy, eps, nx, ny, nz;
};

// (the sums' roundings written out: weight_pair forms the same bits)
__device__ __forceinline__ float bilateral_weight(const Center& p, const Guide& q, int dx, int dy, float inv2s2) {
    const float ws = expf(-(float)(dx * dx + dy * dy) * inv2s2);
    const float pred = fabsf(__fmaf_rn(p.gy, (float)dy, __fmul_rn(p.gx, (float)dx)));
    const float wz = expf(-fabsf(p.z - q.z) / (kSigmaZ * pred + p.eps));
    const float wn = pow128(__fmaf_rn(p.nz, q.nz, __fmaf_rn(p.ny, q.ny, __fmul_rn(p.nx, q.nx))));
    return ws * wz * wn;
}

__device__ __forceinline__ Center center_of(const Guide* s, int sw, int sx, int sy) {
    const Guide g = s[sy * sw + sx];
    Center c;
    c.z = g.z;
    c.gx = depth_slope(s[sy * sw + sx - 1].z, g.z, s[sy * sw + sx + 1].z);
    c.gy = depth_slope(s[(sy - 1) * sw + sx].z, g.z, s[(sy + 1) * sw + sx].z);
    c.eps = kEpsRel * fabsf(g.z);
    c.nx = g.nx;
    c.ny = g.ny;
    c.nz = g.nz;
    return c;
}

// Forward.  Shared memory: guides over tile + halo R + 1 (the slopes of the
// tile's pixels need one more ring), colours over tile + halo R.
__global__ void __launch_bounds__(kTile* kTile) bilateral_fwd_kernel(const float4* __restrict__ pos,
                                                                     const float4* __restrict__ nrm,
                                                                     const mcdi_camera* __restrict__ cams, int N, int H,
                                                                     int W, int K, const float4* __restrict__ c_in,
                                                                     float inv2s2, int R, float4* __restrict__ c_out,
                                                                     float* __restrict__ wsum) {
    pdl_prologue();
    extern __shared__ float4 smem[];
    const int view = blockIdx.z;
    const int x0 = blockIdx.x * kTile, y0 = blockIdx.y * kTile;
    const int gw = kTile + 2 * (R + 1), cw = kTile + 2 * R;
    Guide* sg = reinterpret_cast<Guide*>(smem);
    float4* sc = smem + gw * gw;  // K planes of cw * cw colours
    const mcdi_camera C = cams[view];
    const size_t plane = (size_t)H * W;
    const size_t gbase = (size_t)view * plane;
    for (int i = threadIdx.x; i < gw * gw; i += blockDim.x) {
        const int sx = i % gw, sy = i / gw;
        sg[i] = load_guide(pos, nrm, C, H, W, gbase, x0 + sx - (R + 1), y0 + sy - (R + 1));
    }
    for (int k = 0; k < K; ++k) {
        const size_t cbase = (size_t)(view + k * N) * plane;
        for (int i = threadIdx.x; i < cw * cw; i += blockDim.x) {
            const int x = x0 + i % cw - R, y = y0 + i / cw - R;
            sc[k * cw * cw + i] =
                (x >= 0 && y >= 0 && x < W && y < H) ? c_in[cbase + (size_t)y * W + x] : make_float4(0, 0, 0, 0);
        }
    }
    __syncthreads();
    const int tx = threadIdx.x % kTile, ty = threadIdx.x / kTile;
    const int x = x0 + tx, y = y0 + ty;
    if (x >= W || y >= H) return;
    const size_t pix = (size_t)y * W + x;
    const Center p = center_of(sg, gw, tx + R + 1, ty + R + 1);
    if (p.z < 0.0f) {  // uncovered: pass through
        for (int k = 0; k < K; ++k) {
            const float4 c = sc[k * cw * cw + (ty + R) * cw + tx + R];
            c_out[(size_t)(view + k * N) * plane + pix] = make_float4(c.x, c.y, c.z, 0.0f);
        }
        wsum[gbase + pix] = 0.0f;
        return;
    }
    float acc[kMaxImgPerView][3] = {};
    float wt = 0.0f;
    for (int dy = -R; dy <= R; ++dy) {
        for (int dx = -R; dx <= R; ++dx) {
            const Guide q = sg[(ty + R + 1 + dy) * gw + tx + R + 1 + dx];
            if (q.z < 0.0f) continue;
            const float w = bilateral_weight(p, q, dx, dy, inv2s2);
            wt += w;
            const int ci = (ty + R + dy) * cw + tx + R + dx;
#pragma unroll
            for (int k = 0; k < kMaxImgPerView; ++k) {
                if (k >= K) break;
                const float4 c = sc[k * cw * cw + ci];
                acc[k][0] += w * c.x;
                acc[k][1] += w * c.y;
                acc[k][2] += w * c.z;
            }
        }
    }
    const float inv = 1.0f / wt;
    for (int k = 0; k < K; ++k)
        c_out[(size_t)(view + k * N) * plane + pix] = make_float4(acc[k][0] * inv, acc[k][1] * inv, acc[k][2] * inv, 0.0f);
    wsum[gbase + pix] = wt;
}

// Backward for radii 0 and 1 on images up to about 600 x 600: a pixel per thread, in
// the forward's tiles.  With at most nine weights a pixel the other form's table,
// slopes and second barrier cost more than its pairs save, until loads and
// arithmetic outweigh them.  Measured (this / the other), two images, radius 1: 100 x
// 90: 7.2 / 9.7 us, 400 x 400: 11.0 / 13.1, 640 x 640: 21.5 / 21.7, 2 x 800 x 800: 70 /
// 66; radius 2: 100 x 90: 11.4 / 11.1, 320 x 300: 19.5 / 13.9.
constexpr int kNearRadius = 1, kNearTiles = 10;  // tiles of the other form per SM
__global__ void __launch_bounds__(kTile* kTile) bilateral_bwd_near_kernel(
    const float4* __restrict__ pos, const float4* __restrict__ nrm, const mcdi_camera* __restrict__ cams, int N, int H,
    int W, int K, const float* __restrict__ wsum, const float4* __restrict__ g_out, float inv2s2, int R,
    float4* __restrict__ g_in) {
    pdl_prologue();
    extern __shared__ float4 smem[];
    const int view = blockIdx.z;
    const int x0 = blockIdx.x * kTile, y0 = blockIdx.y * kTile;
    const int gw = kTile + 2 * (R + 1), cw = kTile + 2 * R;
    Guide* sg = reinterpret_cast<Guide*>(smem);
    float4* sgw = smem + gw * gw;  // K planes of g / W over cw * cw
    const mcdi_camera C = cams[view];
    const size_t plane = (size_t)H * W;
    const size_t gbase = (size_t)view * plane;
    for (int i = threadIdx.x; i < gw * gw; i += blockDim.x) {
        const int sx = i % gw, sy = i / gw;
        sg[i] = load_guide(pos, nrm, C, H, W, gbase, x0 + sx - (R + 1), y0 + sy - (R + 1));
    }
    for (int k = 0; k < K; ++k) {
        const size_t cbase = (size_t)(view + k * N) * plane;
        for (int i = threadIdx.x; i < cw * cw; i += blockDim.x) {
            const int x = x0 + i % cw - R, y = y0 + i / cw - R;
            float4 v = make_float4(0, 0, 0, 0);
            if (x >= 0 && y >= 0 && x < W && y < H) {
                const float w = wsum[gbase + (size_t)y * W + x];
                if (w > 0.0f) {
                    const float4 g = g_out[cbase + (size_t)y * W + x];
                    const float iw = 1.0f / w;
                    v = make_float4(g.x * iw, g.y * iw, g.z * iw, 0.0f);
                }
            }
            sgw[k * cw * cw + i] = v;
        }
    }
    __syncthreads();
    const int tx = threadIdx.x % kTile, ty = threadIdx.x / kTile;
    const int x = x0 + tx, y = y0 + ty;
    if (x >= W || y >= H) return;
    const size_t pix = (size_t)y * W + x;
    const Guide q = sg[(ty + R + 1) * gw + tx + R + 1];
    if (q.z < 0.0f) {  // uncovered: pass through
        for (int k = 0; k < K; ++k) {
            const size_t i = (size_t)(view + k * N) * plane + pix;
            const float4 g = g_out[i];
            g_in[i] = make_float4(g.x, g.y, g.z, 0.0f);
        }
        return;
    }
    float acc[kMaxImgPerView][3] = {};
    // p = q + (ox, oy); the offset of q seen from p is (-ox, -oy)
    for (int oy = -R; oy <= R; ++oy) {
        for (int ox = -R; ox <= R; ++ox) {
            const int sx = tx + R + 1 + ox, sy = ty + R + 1 + oy;
            if (sg[sy * gw + sx].z < 0.0f) continue;
            const Center p = center_of(sg, gw, sx, sy);
            const float w = bilateral_weight(p, q, -ox, -oy, inv2s2);
            const int ci = (ty + R + oy) * cw + tx + R + ox;
#pragma unroll
            for (int k = 0; k < kMaxImgPerView; ++k) {
                if (k >= K) break;
                const float4 g = sgw[k * cw * cw + ci];
                acc[k][0] += w * g.x;
                acc[k][1] += w * g.y;
                acc[k][2] += w * g.z;
            }
        }
    }
    for (int k = 0; k < K; ++k)
        g_in[(size_t)(view + k * N) * plane + pix] = make_float4(acc[k][0], acc[k][1], acc[k][2], 0.0f);
}

size_t bilateral_smem(int R, int K) {
    const int gw = kTile + 2 * (R + 1), cw = kTile + 2 * R;
    return (size_t)gw * gw * sizeof(Guide) + (size_t)K * cw * cw * sizeof(float4);
}

// ---- backward
// A CTA owns a tile of one view, 32 pixels wide, each thread two pixels of a
// column; guides and the upstream gradients divided by W(p) over the tile plus its
// halo are staged in shared memory, and from the guides every staged pixel's
// slopes.  What bounds it is three things at about the same level, per pair of
// weights and warp: some 50 issued instructions, 4 MUFU operations and 15
// shared-memory wavefronts (for two images), then the staging's latency.  So a
// neighbour loaded once meets two pixels, their arithmetic goes in packed pairs,
// the spatial factors come from a table, the division takes no branch, and
// uncovered neighbours (zero normal and gradients) take none either.  Every
// operation is rounded as in bilateral_weight, so the weights are the forward's,
// bit for bit.  Measured, two images: 512 x 512, sigma 2: 36 us; 3 x 700 x 611,
// sigma 3.9: 408 (a pixel per thread, slopes formed per weight, two exponentials,
// a division and a branch: 68 and 824; with an approximate quotient and one
// approximate exponential 34 and 377, whose weights are off by up to twice as
// much: not taken).  The gradient's error against 64 bits, with the loss before
// it, is 0.5 to 12% below either of theirs over ten shapes.  The forward is not
// built this way: two pixels per thread gain it nothing (66 and 503 us against 63
// and 631, 27 against 22 at 133 x 77).
constexpr int kTileW = 32;
constexpr int kRows = 2;  // pixels of a thread, in one column
constexpr int kUnroll = 4;  // 3: 3 to 8% slower, 5 and 6: 2 to 10%
// Warps of a CTA: 4, or from radius 4 on, where the halo is as large as the tile, 8,
// unless CTAs of 4 do not outnumber the SMs and fewer would leave some idle.
// Measured (4 / 8 warps), two images: 133 x 77, radius 8: 34 / 41 us, radius 4: 15.7 /
// 17.4; 256 x 256: 18.9 / 17.5; 512 x 512: 35.8 / 36.0; 3 x 700 x 611, radius 8: 469 /
// 408; 4 x 800 x 800, radius 5: 366 / 320; 320 x 300, radius 2: 13.9 / 15.1, radius 3:
// 17.6 / 20.0; 512 x 512, radius 3: 27.5 / 27.7.
constexpr int kMaxWarps = 8, kWideRadius = 4;
// Depths for which weight_pair's divisors (from 1e-3 of one to 17 times the largest) stay in div_pair's range.
constexpr float kPlainMin = 0x1p-40f, kPlainMax = 0x1p40f;

__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// n / d of two pairs, rounded as the operator / rounds it, without its branch: a
// reciprocal with one Newton step, and the quotient corrected by its exact
// remainder (P. Markstein, "Computation of elementary functions on the IBM RISC
// System/6000 processor", 1990).  For d in [2^-60, 2^60] and |n| up to 2^60: no
// step leaves the normal range, or the quotient is too small to matter beside 1.
__device__ __forceinline__ float2 div_pair(float2 n, float2 d) {
    const float2 nd = make_float2(-d.x, -d.y);
    float2 r = make_float2(rcp_approx(d.x), rcp_approx(d.y));
    r = fma2(r, fma2(nd, r, both(1.0f)), r);
    const float2 q = mul2(n, r);
    return fma2(fma2(nd, q, n), r, q);
}

// Two of bilateral_weight's weights, rounded as there: spatial factors `ws`,
// depth change that the slope predicts over the offset `pred`, depth offset
// `eps`, depth difference `dz`, cosine of the normals `nn`.
template <bool kPlain>
__device__ __forceinline__ float2 weight_pair(float2 ws, float2 pred, float eps, float2 dz, float2 nn) {
    const float2 n = make_float2(-fabsf(dz.x), -fabsf(dz.y));
    const float2 d = make_float2(kSigmaZ * fabsf(pred.x) + eps, kSigmaZ * fabsf(pred.y) + eps);
    const float2 a = kPlain ? div_pair(n, d) : make_float2(n.x / d.x, n.y / d.y);
    float2 v = make_float2(fmaxf(nn.x, 0.0f), fmaxf(nn.y, 0.0f));
#pragma unroll
    for (int i = 0; i < 7; ++i) v = mul2(v, v);
    return mul2(mul2(ws, make_float2(expf(a.x), expf(a.y))), v);
}

struct Tile {  // staged extents: the guides one ring wider (slopes) than the gradients
    int gw, gh, cw, ch;
    __host__ __device__ Tile(int R, int warps)
        : gw(kTileW + 2 * R + 2), gh(kRows * warps + 2 * R + 2), cw(kTileW + 2 * R), ch(kRows * warps + 2 * R) {}
};

// The weights of staged row s (relative to the thread's first pixel) for its two
// pixels, s and s - 1 rows away; kEdge: one of them is beyond the footprint, and
// its gradients are left out (an infinity there must not meet a zero weight).
template <int K, bool kPlain, bool kEdge>
__device__ __forceinline__ void gather_row(const Guide* g, const float2* slope, const float4* c, int cplane, int R, int s,
                                           const float2* ws, float2 z, float2 nx, float2 ny, float2 nz, float2 (&acc)[K][3]) {
    const float2 dy = make_float2((float)s, (float)(s - 1));
    const bool v0 = !kEdge || abs(s) <= R, v1 = !kEdge || abs(s - 1) <= R;
#pragma unroll kUnroll
    for (int dx = -R; dx <= R; ++dx) {
        const Guide p = g[dx];  // the weight's centre; the offset's sign drops out
        const float2 sl = slope[dx];
        const float2 pred = fma2(both(sl.y), dy, both(__fmul_rn(sl.x, (float)dx)));
        const float2 nn = fma2(nz, both(p.nz), fma2(ny, both(p.ny), mul2(nx, both(p.nx))));
        float2 w = weight_pair<kPlain>(ws[dx], pred, kEpsRel * fabsf(p.z),
                               make_float2(z.x - p.z, z.y - p.z), nn);
        if (kEdge) w = make_float2(v0 ? w.x : 0.0f, v1 ? w.y : 0.0f);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float4 v = c[k * cplane + dx];
            const float2 cx = kEdge ? make_float2(v0 ? v.x : 0.0f, v1 ? v.x : 0.0f) : both(v.x);
            const float2 cy = kEdge ? make_float2(v0 ? v.y : 0.0f, v1 ? v.y : 0.0f) : both(v.y);
            const float2 cz = kEdge ? make_float2(v0 ? v.z : 0.0f, v1 ? v.z : 0.0f) : both(v.z);
            acc[k][0] = fma2(w, cx, acc[k][0]);
            acc[k][1] = fma2(w, cy, acc[k][1]);
            acc[k][2] = fma2(w, cz, acc[k][2]);
        }
    }
}

template <int K>
__global__ void __launch_bounds__(32 * kMaxWarps) bilateral_bwd_kernel(const float4* __restrict__ pos,
                                                                       const float4* __restrict__ nrm,
                                                                       const mcdi_camera* __restrict__ cams, int N, int H,
                                                                       int W, const float* __restrict__ wsum,
                                                                       const float4* __restrict__ g_out, float inv2s2,
                                                                       int R, float4* __restrict__ g_in) {
    pdl_prologue();
    extern __shared__ float4 smem[];
    const int threads = blockDim.x;
    const Tile T(R, threads >> 5);
    const int view = blockIdx.z;
    const int tiles_x = (W + kTileW - 1) / kTileW, tile_y = blockIdx.x / tiles_x;  // (rows of tiles may outnumber a grid's y)
    const int x0 = (blockIdx.x - tile_y * tiles_x) * kTileW, y0 = tile_y * kRows * (threads >> 5);
    Guide* sg = reinterpret_cast<Guide*>(smem);
    const int cplane = T.cw * T.ch;
    float4* sc = smem + T.gw * T.gh;                          // K planes of g / W
    float2* ss = reinterpret_cast<float2*>(sc + K * cplane);  // slopes
    float2* s_ws = ss + cplane;                               // spatial factors of rows s and s - 1, [s + R][dx + R]
    const mcdi_camera C = cams[view];
    const size_t plane = (size_t)H * W, gbase = (size_t)view * plane;
    bool plain = true;
#pragma unroll 4
    for (int i = threadIdx.x; i < T.gw * T.gh; i += threads) {
        const int sy = i / T.gw, sx = i - sy * T.gw;
        const Guide g = load_guide(pos, nrm, C, H, W, gbase, x0 + sx - (R + 1), y0 + sy - (R + 1));
        sg[i] = g;
        plain &= g.z < 0.0f || (g.z >= kPlainMin && g.z <= kPlainMax);
    }
#pragma unroll 4
    for (int i = threadIdx.x; i < cplane; i += threads) {
        const int sy = i / T.cw, x = x0 + i - sy * T.cw - R, y = y0 + sy - R;
        const bool inside = x >= 0 && y >= 0 && x < W && y < H;
        const size_t p = inside ? (size_t)y * W + x : 0;
        const float w = wsum[gbase + p];
        const float iw = 1.0f / w;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float4 v = g_out[(size_t)(view + k * N) * plane + p];
            sc[k * cplane + i] =
                inside && w > 0.0f ? make_float4(v.x * iw, v.y * iw, v.z * iw, 0.0f) : make_float4(0, 0, 0, 0);
        }
    }
    plain = __syncthreads_and(plain);
    for (int i = threadIdx.x; i < (2 * R + 2) * (2 * R + 1); i += threads) {
        const int row = i / (2 * R + 1), dx = i - row * (2 * R + 1) - R, s = row - R;
        s_ws[i] = make_float2(expf(-(float)(dx * dx + s * s) * inv2s2),
                              expf(-(float)(dx * dx + (s - 1) * (s - 1)) * inv2s2));
    }
    for (int i = threadIdx.x; i < cplane; i += threads) {
        const int sy = i / T.cw, sx = i - sy * T.cw;
        const Guide* g = sg + (sy + 1) * T.gw + sx + 1;
        const bool covered = !(g->z < 0.0f);
        if (!covered) {
#pragma unroll
            for (int k = 0; k < K; ++k) sc[k * cplane + i] = make_float4(0, 0, 0, 0);
        }
        ss[i] = covered ? make_float2(depth_slope(g[-1].z, g->z, g[1].z), depth_slope(g[-T.gw].z, g->z, g[T.gw].z))
                        : make_float2(0.0f, 0.0f);
    }
    __syncthreads();
    const int tx = threadIdx.x & 31, ty = (threadIdx.x >> 5) * kRows;
    const int x = x0 + tx, y = y0 + ty;
    if (x >= W || y >= H) return;
    const Guide* g0 = sg + (ty + R + 1) * T.gw + tx + R + 1;  // the thread's first pixel
    const int o0 = (ty + R) * T.cw + tx + R;
    const Guide a = g0[0], b = g0[T.gw];
    const bool cov[2] = {!(a.z < 0.0f), !(b.z < 0.0f)};
    float2 acc[K][3];
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k][0] = acc[k][1] = acc[k][2] = make_float2(0.0f, 0.0f);
    if (cov[0] || cov[1]) {
        const float2 z = make_float2(a.z, b.z), nx = make_float2(a.nx, b.nx), ny = make_float2(a.ny, b.ny),
                     nz = make_float2(a.nz, b.nz);
        auto gather = [&](auto plain_depths) {
            constexpr bool kPlain = decltype(plain_depths)::value;
            for (int s = -R; s <= R + 1; ++s) {
                const Guide* g = g0 + s * T.gw;
                const int o = o0 + s * T.cw;
                const float2* ws = s_ws + (s + R) * (2 * R + 1) + R;
                if (s > -R && s <= R)
                    gather_row<K, kPlain, false>(g, ss + o, sc + o, cplane, R, s, ws, z, nx, ny, nz, acc);
                else gather_row<K, kPlain, true>(g, ss + o, sc + o, cplane, R, s, ws, z, nx, ny, nz, acc);
            }
        };
        if (plain) gather(std::true_type{});
        else gather(std::false_type{});
    }
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
        if (y + i >= H) break;
        const size_t p = (size_t)(y + i) * W + x;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const size_t o = (size_t)(view + k * N) * plane + p;
            float4 v = g_out[o];  // uncovered: pass through
            if (cov[i])
                v = i == 0 ? make_float4(acc[k][0].x, acc[k][1].x, acc[k][2].x, 0.0f)
                           : make_float4(acc[k][0].y, acc[k][1].y, acc[k][2].y, 0.0f);
            g_in[o] = make_float4(v.x, v.y, v.z, 0.0f);
        }
    }
}

template <int K>
cudaError_t launch_bwd(const float4* pos, const float4* nrm, const mcdi_camera* cams, int N, int H, int W,
                       const float* wsum, const float4* g_out, float inv2s2, int R, float4* g_in, cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    constexpr int kFew = kMaxWarps / 2;
    const long long few = (long long)((W + kTileW - 1) / kTileW) * ((H + kRows * kFew - 1) / (kRows * kFew)) * N;
    if (R <= kNearRadius && few <= (long long)kNearTiles * sms) {
        const dim3 grid((W + kTile - 1) / kTile, (H + kTile - 1) / kTile, N);
        launch_k(bilateral_bwd_near_kernel, grid, kTile * kTile, bilateral_smem(R, K), s, pos, nrm, cams, N, H, W, K,
                 wsum, g_out, inv2s2, R, g_in);
        return cudaGetLastError();
    }
    const int warps = R < kWideRadius || few <= sms ? kFew : kMaxWarps;
    const Tile T(R, warps);
    const size_t smem = (size_t)T.gw * T.gh * sizeof(Guide) + (size_t)T.cw * T.ch * (K * sizeof(float4) + sizeof(float2)) +
                        (size_t)(2 * R + 2) * (2 * R + 1) * sizeof(float2);
    e = allow_smem((const void*)bilateral_bwd_kernel<K>, smem);
    if (e != cudaSuccess) return e;
    const dim3 grid(((W + kTileW - 1) / kTileW) * ((H + kRows * warps - 1) / (kRows * warps)), 1, N);
    launch_k(bilateral_bwd_kernel<K>, grid, 32 * warps, smem, s, pos, nrm, cams, N, H, W, wsum, g_out, inv2s2, R, g_in);
    return cudaGetLastError();
}

}  // namespace

int bilateral_max_images_per_view() { return kMaxImgPerView; }

cudaError_t launch_bilateral(bool backward, const float* gb_pos, const float* gb_nrm, const mcdi_camera* cams, int N,
                             int H, int W, int n_img, const float* in, float sigma, int R, const float* wsum_in,
                             float* out, float* wsum_out, cudaStream_t s) {
    const int K = n_img / N;
    const float inv2s2 = 1.0f / (2.0f * sigma * sigma);
    const auto* pos = reinterpret_cast<const float4*>(gb_pos);
    const auto* nrm = reinterpret_cast<const float4*>(gb_nrm);
    const auto* src = reinterpret_cast<const float4*>(in);
    auto* dst = reinterpret_cast<float4*>(out);
    if (backward) {
        switch (K) {
            case 1: return launch_bwd<1>(pos, nrm, cams, N, H, W, wsum_in, src, inv2s2, R, dst, s);
            case 2: return launch_bwd<2>(pos, nrm, cams, N, H, W, wsum_in, src, inv2s2, R, dst, s);
            case 3: return launch_bwd<3>(pos, nrm, cams, N, H, W, wsum_in, src, inv2s2, R, dst, s);
            default: return launch_bwd<4>(pos, nrm, cams, N, H, W, wsum_in, src, inv2s2, R, dst, s);
        }
    }
    const size_t smem = bilateral_smem(R, K);
    const cudaError_t e = allow_smem((const void*)bilateral_fwd_kernel, smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((W + kTile - 1) / kTile, (H + kTile - 1) / kTile, N);
    launch_k(bilateral_fwd_kernel, grid, kTile * kTile, smem, s, pos, nrm, cams, N, H, W, K, src, inv2s2, R, dst,
             wsum_out);
    return cudaGetLastError();
}

}  // namespace mcdi
