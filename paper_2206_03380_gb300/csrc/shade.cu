// Shading kernels: the G-buffer ray cast, the forward MIS estimator and its
// hand-written adjoint (Sec. 3.1, Sec. 4.1, Sec. 4.2).  The ray cast walks the
// tree with a pair of lanes per pixel; forward and adjoint shade 32 consecutive
// pixels per CTA, their samples split over its four warps.  G-buffer planes are
// read and outputs written as float4.
#include "common.cuh"
#include "internal.h"
#include "shading.cuh"
#include "trace.cuh"

namespace mcdi {
namespace {

constexpr int kShadeThreads = 128;

__device__ __forceinline__ Probe make_probe(const ShadeArgs& a) {
    Probe P;
    P.env = a.env;
    P.cond = a.cond;
    P.marg = a.marg;
    P.W = a.Wp;
    P.H = a.Hp;
    P.on = *a.total > 0.0;
    return P;
}

__device__ __forceinline__ f3 cam_origin(const mcdi_camera* cams, int view) {
    return mk(cams[view].origin[0], cams[view].origin[1], cams[view].origin[2]);
}

// ---------------------------------------------------------------- G-buffer
// A warp casts 4 x 4 pixels (or 16 x 1, 8 x 2, .. 1 x 16 where a narrow image
// would leave lanes out), so that its rays visit the same nodes; a CTA's four
// warps lie 2 x 2 (or in a row or a column).  A view whose camera is too far for
// the four-wide nodes is cast with a ray per lane: in small images both lanes of a
// pair cast the same one (the rays' latency is all that counts), in large ones every
// other CTA takes two tiles.  Measured, camera 12 m away (this way / the other; the
// former kernel of 32 consecutive pixels a warp): 320 x 320: 148 / 199 us (154), 400 x
// 300: 139 / 146 (132), 512 x 512: 167 / 181 (160).
constexpr int kCastJoin = 20;  // CTAs per SM from which the image counts as large
struct CastTiles {
    int log_w, log_wx;  // log2 of the warp tile's width and of the warps side by side
    int nx, ny;         // CTAs per view
    bool join;          // whether a CTA whose view is cast with a ray per lane takes two tiles
};
CastTiles cast_tiles(int N, int H, int W, int sms) {
    CastTiles T{2, 1, 0, 0, false};
    while (T.log_w < 4 && (8 >> T.log_w) >= H) ++T.log_w;
    while (T.log_w > 0 && (1 << (T.log_w - 1)) >= W) --T.log_w;
    if ((1 << T.log_w) >= W) T.log_wx = 0;
    else if ((16 >> T.log_w) >= H) T.log_wx = 2;
    T.nx = ((W - 1) >> (T.log_w + T.log_wx)) + 1;
    T.ny = ((H - 1) >> (6 - T.log_w - T.log_wx)) + 1;
    T.join = (long long)N * T.nx * T.ny > (long long)kCastJoin * sms;
    return T;
}

__global__ void __launch_bounds__(kShadeThreads) primary_cast_kernel(
    const BvhNode* __restrict__ nodes, const TriRecord* __restrict__ tris, int n_tris, const float* __restrict__ verts,
    const float* __restrict__ vnrm, const int* __restrict__ tri_idx, int n_verts, const mcdi_camera* __restrict__ cams,
    int N, int H, int W, const CastTiles T, const float4* __restrict__ tex_kd, const float4* __restrict__ tex_korm, int S,
    float uv_ox, float uv_oz, float uv_s, float4* __restrict__ gb_pos, float4* __restrict__ gb_nrm,
    float4* __restrict__ gb_kd, float4* __restrict__ gb_korm) {
    pdl_prologue();
    __shared__ float2 stack[(kCastStack + 1) * kShadeThreads / 2];
    const int per_view = T.nx * T.ny;
    const int view = blockIdx.x / per_view;
    int tile = blockIdx.x - view * per_view, warp = threadIdx.x >> 5, ray_of_warp = (threadIdx.x & 31) >> 1;
    const mcdi_camera& C = cams[view];
    const f3 o = mk(C.origin[0], C.origin[1], C.origin[2]);
    const bool pairs = largest(o) <= wide_reach(nodes, n_tris);  // the same for the whole CTA: one view
    const bool joined = !pairs && T.join;
    if (joined) {  // a ray per lane: every other CTA takes two tiles, half a warp a warp's tile
        if (tile & 1) return;
        tile += threadIdx.x >> 6;
        warp = (threadIdx.x >> 4) & 3;
        ray_of_warp = threadIdx.x & 15;
    }
    const int ty = tile / T.nx, tx = tile - ty * T.nx;
    const int wx = warp & ((1 << T.log_wx) - 1), wy = warp >> T.log_wx;
    const int x = (((tx << T.log_wx) + wx) << T.log_w) + (ray_of_warp & ((1 << T.log_w) - 1));
    const int y = (((ty << (2 - T.log_wx)) + wy) << (4 - T.log_w)) + (ray_of_warp >> T.log_w);
    const bool inside = tile < per_view && x < W && y < H;
    const long long idx = ((long long)view * H + y) * W + x;
    const f3 d = camera_dir(C, x, y, W, H);
    // a degenerate camera's NaN passes every box test (minimum and maximum drop it) and no triangle's: a miss
    const bool live = inside && finite_ray(o, d);
    const RayInv ray = make_ray(o, d);
    float t, u = 0.f, v = 0.f;
    int leaf = kWideOverflow;
    if (pairs)
        leaf = closest_hit_wide(wide_nodes(nodes, n_tris), tris, n_tris, ray, live ? 0 : -1,
                                stack + (threadIdx.x >> 1) * (kCastStack + 1), &t, &u, &v);
    if (!inside) return;
    if (leaf == kWideOverflow) leaf = live ? closest_hit(nodes, tris, n_tris, ray, &t, &u, &v) : -1;
    float4 P = make_float4(0.f, 0.f, 0.f, 0.f), Nn = P, KD = P, KORM = P;
    if (leaf >= 0)
        gbuffer_hit(__float_as_int(__ldg(&tris[leaf].v0.w)), u, v, verts, vnrm, tri_idx, n_verts,
                    reinterpret_cast<const float*>(tex_kd), reinterpret_cast<const float*>(tex_korm), S, uv_ox, uv_oz,
                    uv_s, &P, &Nn, &KD, &KORM);
    // a pair's lanes computed the same: each writes two of the four
    const bool odd = threadIdx.x & 1;
    (odd ? gb_nrm : gb_pos)[idx] = odd ? Nn : P;
    (odd ? gb_korm : gb_kd)[idx] = odd ? KORM : KD;
    if (!joined) return;
    (odd ? gb_pos : gb_nrm)[idx] = odd ? P : Nn;
    (odd ? gb_kd : gb_korm)[idx] = odd ? KD : KORM;
}

// ---------------------------------------------------------------- forward
// Without scratch memory: a CTA covers 32 consecutive pixels with four warps
// and works through their samples in chunks of kFwdChunk, all in shared
// memory: the warps draw the chunk's samples (warp q the samples j = q mod 4),
// keep each one's unshadowed contribution and append its shadow ray; all
// lanes trace the chunk's rays (trace_rays); warp 0 adds each pixel's samples
// in order.  What bounds it is the traversal, as in the wavefront; a chunk's
// 512 rays give the CTA's 128 lanes four each, so that few idle at its end.
// Measured at 3 x 155 x 203 pixels, 11 samples, 113k triangles: 233 us
// (one thread per pixel, each lane waiting for its warp's longest ray: 669).
constexpr int kQuarters = kShadeThreads / 32;
constexpr int kFwdChunk = 16;
static_assert(kShadeThreads == kTraceThreads, "the tracer's columns are one per thread");

struct FwdShared {
    BlockRays<kFwdChunk> rays;
    float4 cd[kFwdChunk * 32];  // w: 1 where the sample has a shadow ray
    float4 cs[kFwdChunk * 32];
};

__global__ void __launch_bounds__(kShadeThreads) shade_fwd_kernel(ShadeArgs a, float4* __restrict__ c_d,
                                                                  float4* __restrict__ kd_out,
                                                                  float4* __restrict__ c_s,
                                                                  uint32_t* __restrict__ vis_mask) {
    pdl_prologue();
    extern __shared__ float4 s_fwd[];
    FwdShared& S = *reinterpret_cast<FwdShared*>(s_fwd);
    Probe Pr = make_probe(a);
    stage_marginal(Pr, reinterpret_cast<float*>(&S + 1));
    const int lane = threadIdx.x & 31, quarter = threadIdx.x >> 5;
    const long long idx = (long long)blockIdx.x * 32 + lane;
    const long long P = (long long)a.N * a.H * a.W;
    const bool in_range = idx < P;
    const int view = in_range ? (int)(idx / ((long long)a.H * a.W)) : 0;
    const uint32_t pix = (uint32_t)(idx - (long long)view * a.H * a.W);
    const int spp = a.n_light + a.n_cos + a.n_ggx;
    const int nwords = (spp + 31) >> 5;
    Pixel px{};
    const bool covered = in_range && load_pixel(a.gb_pos[idx], a.gb_nrm[idx], a.gb_kd[idx], a.gb_korm[idx],
                                                cam_origin(a.cams, view), &px);
    if (quarter == 0) {
        const f3 o = covered ? fma_rn(px.n, a.ray_eps, px.p) : mk(0.f, 0.f, 0.f);
        S.rays.origin[lane] = make_float4(o.x, o.y, o.z, 0.f);
    }
    f3 cd = mk(0.f, 0.f, 0.f), cs = cd;
    uint32_t word = 0;
    const float reach = wide_reach(a.nodes, a.n_tris);
    for (int j0 = 0; j0 < spp; j0 += kFwdChunk) {
        const int n = min(kFwdChunk, spp - j0);
        S.rays.clear();
        __syncthreads();
        for (int jj = quarter; jj < n; jj += kQuarters) {
            const int j = j0 + jj;
            f3 wi = mk(0.f, 0.f, 0.f);
            float4 dd = make_float4(0.f, 0.f, 0.f, 0.f), ds = dd;
            bool active = false;
            if (covered) {
                int t;
                float ci, inv_denom;
                const float2 u = sample_uniforms(a.seed, pix, (uint32_t)view, (uint32_t)j, a.stream_word);
                if (draw_sample(Pr, px, a.n_light, a.n_cos, a.n_ggx, j, u, &wi, &t, &ci, &inv_denom)) {
                    active = true;
                    const float4 L = __ldg(Pr.env + t);
                    const float wd = ci * MCDI_INV_PI * inv_denom;
                    dd = make_float4(L.x * wd, L.y * wd, L.z * wd, 1.f);
                    if (px.spec_on) {
                        const f3 h = half_vector(wi, px.wo);
                        const float D = ggx_D(dot_rn(px.n, h), sin2_between(px.n, h), px.a2);
                        const float G2 = 1.0f / (1.0f + ggx_lambda(ci, px.a2) + ggx_lambda(px.co, px.a2));
                        const float q = schlick_weight(dot_rn(px.wo, h));
                        const float ws = D * G2 / (4.0f * px.co) * inv_denom;
                        const f3 c = spec_colour(L, px.F0, q, ws);
                        ds = make_float4(c.x, c.y, c.z, 0.f);
                    }
                }
            }
            S.rays.append(active, jj, wi);
            S.cd[jj * 32 + lane] = dd;
            S.cs[jj * 32 + lane] = ds;
        }
        __syncthreads();
        trace_rays(a.nodes, static_cast<const TriRecord*>(a.tris), a.n_tris, reach, S.rays.stacks, S.rays);
        __syncthreads();
        if (quarter == 0) {
            for (int jj = 0; jj < n; ++jj) {
                const int j = j0 + jj;
                const bool hit = (S.rays.hit[jj] >> lane) & 1u;
                const float4 dd = S.cd[jj * 32 + lane], ds = S.cs[jj * 32 + lane];
                const float Hv = hit ? 1.0f - a.tau : 1.0f;
                if (hit) word |= 1u << (j & 31);
                if (dd.w > 0.f) {
                    cd = cd + mk(dd.x, dd.y, dd.z) * Hv;
                    cs = cs + mk(ds.x, ds.y, ds.z) * Hv;
                }
                if (in_range && vis_mask && ((j & 31) == 31 || j == spp - 1)) {
                    vis_mask[(size_t)idx * nwords + (j >> 5)] = word;
                    word = 0;
                }
            }
        }
        __syncthreads();  // the next chunk overwrites what warp 0 reads
    }
    if (quarter != 0 || !in_range) return;
    c_d[idx] = make_float4(cd.x, cd.y, cd.z, 0.f);
    c_s[idx] = make_float4(cs.x, cs.y, cs.z, 0.f);
    kd_out[idx] = covered ? make_float4(px.kd.x * (1.f - px.m), px.kd.y * (1.f - px.m), px.kd.z * (1.f - px.m), 0.f)
                          : make_float4(0.f, 0.f, 0.f, 0.f);
}

// ---------------------------------------------------------------- adjoint
// A CTA covers 32 consecutive pixels with kBwdQuarters warps; warp q handles
// the samples j = q, q + 4, ... of its lane's pixel (in increasing j) and the
// per-pixel partial sums of the four warps are added in order q = 0..3, so
// every pixel's gradient has one fixed summation order.
// Without the forward's visibility (or with samples of its own) it traces the
// shadow rays first, in chunks of kBwdChunk samples: the warps draw the
// chunk's samples and append their rays in shared memory, all lanes trace them
// (trace_rays), and the samples are drawn again for the gradients.  Measured
// at 3 x 155 x 203 pixels, 11 samples, 113k triangles: 275 us (each lane
// walking its own ray stacklessly inside the gradient loop: 453).
constexpr int kBwdQuarters = kQuarters;
constexpr int kBwdChunk = 16;
constexpr int kBwdPartials = 8;  // g_n (3), g_F0 (3), g_co, g_alpha

template <bool kRetrace>
__global__ void __launch_bounds__(kShadeThreads, 6) shade_bwd_kernel(ShadeArgs a, const float4* __restrict__ g_cd,
                                                                  const float4* __restrict__ g_kdout,
                                                                  const float4* __restrict__ g_cs,
                                                                  const uint32_t* __restrict__ vis_mask,
                                                                  float4* __restrict__ g_kd,
                                                                  float4* __restrict__ g_korm,
                                                                  float4* __restrict__ g_nrm,
                                                                  float4* __restrict__ g_env, long long first,
                                                                  long long end) {
    pdl_prologue();
    extern __shared__ float s_marg[];  // marginal CDF, then [kBwdQuarters][kBwdPartials][32] partial sums
    Probe Pr = make_probe(a);
    stage_marginal(Pr, s_marg);
    float* s_part = s_marg + ((a.Hp + 1 + 3) & ~3);
    const int lane = threadIdx.x & 31, quarter = threadIdx.x >> 5;
    const long long idx = first + (long long)blockIdx.x * 32 + lane;  // pixels [first, end) of [N][H][W]
    const bool in_range = idx < end;
    const int view = in_range ? (int)(idx / ((long long)a.H * a.W)) : 0;
    const uint32_t pix = (uint32_t)(idx - (long long)view * a.H * a.W);
    const int spp = a.n_light + a.n_cos + a.n_ggx;
    const int nwords = (spp + 31) >> 5;
    Pixel px{};
    const bool covered = in_range && load_pixel(a.gb_pos[idx], a.gb_nrm[idx], a.gb_kd[idx], a.gb_korm[idx],
                                                cam_origin(a.cams, view), &px);
    f3 gn = mk(0.f, 0.f, 0.f), gF0 = gn;
    float g_co = 0.f, g_alpha = 0.f;
    f3 gd = gn, gk = gn, gs = gn;
    if (covered) {
        gd = xyz(g_cd[idx]);
        gk = xyz(g_kdout[idx]);
        gs = xyz(g_cs[idx]);
    }
    const float a2 = px.a2;
    // the specular terms of the pixel alone: out of the sample loop, with the square root and the divisions that
    // a sample's terms share, 3967 us instead of 4132 for 8 x 800 x 800 pixels of 32 samples
    const float co4 = 4.0f * px.co, ico2 = 1.0f / (px.co * px.co), two_alpha = 2.0f / px.alpha;
    const float so = sqrtf(fmaf(a2, ico2 - 1.0f, 1.0f)), lo = 0.5f * (so - 1.0f);
    const float dlo_dco = (-2.0f * a2 * ico2 / px.co) / (4.0f * so), dlo_da = 2.0f * px.alpha * (ico2 - 1.0f) / (4.0f * so);
    BlockRays<kBwdChunk>* rays = nullptr;
    float reach = 0.0f;
    if constexpr (kRetrace) {
        reach = wide_reach(a.nodes, a.n_tris);
        rays = reinterpret_cast<BlockRays<kBwdChunk>*>(s_part + kBwdQuarters * kBwdPartials * 32);
        const f3 o = covered ? fma_rn(px.n, a.ray_eps, px.p) : mk(0.f, 0.f, 0.f);
        if (quarter == 0) rays->origin[lane] = make_float4(o.x, o.y, o.z, 0.f);
    }
    // one pass over all samples, or with kRetrace one per chunk
    for (int j0 = 0; j0 < spp; j0 += kRetrace ? kBwdChunk : spp) {
    const int j1 = kRetrace ? min(j0 + kBwdChunk, spp) : spp;
    if constexpr (kRetrace) {
        __syncthreads();  // the chunk before is done with the rays
        rays->clear();
        __syncthreads();
        for (int j = j0 + quarter; j < j1; j += kBwdQuarters) {
            f3 wi = mk(0.f, 0.f, 0.f);
            int t;
            float ci, inv_denom;
            const float2 u = sample_uniforms(a.seed, pix, (uint32_t)view, (uint32_t)j, a.stream_word);
            const bool active =
                covered && draw_sample<true>(Pr, px, a.n_light, a.n_cos, a.n_ggx, j, u, &wi, &t, &ci, &inv_denom);
            rays->append(active, j - j0, wi);
        }
        __syncthreads();
        trace_rays(a.nodes, static_cast<const TriRecord*>(a.tris), a.n_tris, reach, rays->stacks, *rays);
        __syncthreads();
    }
    for (int j = covered ? j0 + quarter : j1; j < j1; j += kBwdQuarters) {
        const uint32_t word = kRetrace ? 0u : vis_mask[(size_t)idx * nwords + (j >> 5)];
        f3 wi;
        int t;
        float ci, inv_denom;
        const float2 u = sample_uniforms(a.seed, pix, (uint32_t)view, (uint32_t)j, a.stream_word);
        if (!draw_sample<true>(Pr, px, a.n_light, a.n_cos, a.n_ggx, j, u, &wi, &t, &ci, &inv_denom)) continue;
        bool hit;
        if constexpr (kRetrace) hit = (rays->hit[j - j0] >> lane) & 1u;
        else hit = (word >> (j & 31)) & 1u;
        const float A = (hit ? 1.0f - a.tau : 1.0f) * inv_denom;
        const float4 L4 = __ldg(Pr.env + t);
        const f3 L = xyz(L4);
        // diffuse: c_d = A L ci / pi
        f3 ge = gd * (A * ci * MCDI_INV_PI);
        float g_ci = A * dot(gd, L) * MCDI_INV_PI;
        if (px.spec_on) {
            const f3 h = half_vector(wi, px.wo);
            const float nh = dot_rn(px.n, h), vh = dot_rn(px.wo, h);
            const float s2 = sin2_between(px.n, h);
            const float D = ggx_D(nh, s2, a2);
            const float ici2 = 1.0f / (ci * ci);
            const float si = sqrtf(fmaf(a2, ici2 - 1.0f, 1.0f)), li = 0.5f * (si - 1.0f);
            const float G2 = 1.0f / (1.0f + li + lo);
            const float S = D * G2 / co4, dS_dD = G2 / co4, dS_dLam = -D * G2 * G2 / co4;
            const float q = schlick_weight(vh);
            const f3 F = mk(px.F0.x + (1.f - px.F0.x) * q, px.F0.y + (1.f - px.F0.y) * q,
                            px.F0.z + (1.f - px.F0.z) * q);
            ge = ge + mk(gs.x * F.x, gs.y * F.y, gs.z * F.z) * (A * S);
            const float gS = A * (gs.x * L.x * F.x + gs.y * L.y * F.y + gs.z * L.z * F.z);
            gF0 = gF0 + mk(gs.x * L.x, gs.y * L.y, gs.z * L.z) * (A * S * (1.0f - q));
            float dD_dnh = 0.f, dD_dalpha = 0.f;
            if (nh > 0.0f) {
                const float dd = ggx_D_denom(nh, s2, a2);
                dD_dnh = -4.0f * D * nh * (a2 - 1.0f) / dd;
                dD_dalpha = D * (two_alpha - 4.0f * px.alpha * nh * nh / dd);
            }
            const float dli_dci = (-2.0f * a2 * ici2 / ci) / (4.0f * si);
            const float dli_da = 2.0f * px.alpha * (ici2 - 1.0f) / (4.0f * si);
            const float g_nh = gS * dS_dD * dD_dnh;
            g_alpha += gS * (dS_dD * dD_dalpha + dS_dLam * (dli_da + dlo_da));
            g_ci += gS * dS_dLam * dli_dci;
            g_co += gS * (dS_dLam * dlo_dco - S / px.co);
            gn = gn + h * g_nh;
        }
        gn = gn + wi * g_ci;
        // Warp-aggregated scatter: lanes whose samples landed on the same texel
        // (light samples crowd onto the bright lobes) sum their contributions
        // in lane order and the lowest lane issues one atomic for the group.
        const unsigned peers = __match_any_sync(__activemask(), t);
        if (__popc(peers) > 1) {
            f3 sum = mk(0.f, 0.f, 0.f);
            for (unsigned rest = peers; rest; rest &= rest - 1u) {
                const int q = __ffs(rest) - 1;
                sum = sum + mk(__shfl_sync(peers, ge.x, q), __shfl_sync(peers, ge.y, q), __shfl_sync(peers, ge.z, q));
            }
            ge = sum;
        }
        if (lane == __ffs(peers) - 1) atomicAdd(g_env + t, make_float4(ge.x, ge.y, ge.z, 0.f));
    }
    }
    // the four warps' partial sums of each pixel, added in warp order by warp 0
    const float part[kBwdPartials] = {gn.x, gn.y, gn.z, gF0.x, gF0.y, gF0.z, g_co, g_alpha};
#pragma unroll
    for (int k = 0; k < kBwdPartials; ++k) s_part[(quarter * kBwdPartials + k) * 32 + lane] = part[k];
    __syncthreads();
    if (quarter != 0 || !in_range) return;
    if (!covered) {
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        g_kd[idx] = z;
        g_korm[idx] = z;
        g_nrm[idx] = z;
        return;
    }
    float sum[kBwdPartials];
#pragma unroll
    for (int k = 0; k < kBwdPartials; ++k) {
        sum[k] = s_part[k * 32 + lane];
        for (int q = 1; q < kBwdQuarters; ++q) sum[k] += s_part[(q * kBwdPartials + k) * 32 + lane];
    }
    gn = mk(sum[0], sum[1], sum[2]);
    gF0 = mk(sum[3], sum[4], sum[5]);
    g_co = sum[6];
    g_alpha = sum[7];
    gn = gn + px.wo * g_co;
    const float ng = dot(px.n, gn);
    const f3 gN = (gn - px.n * ng) * (1.0f / px.lN);
    const float om = 1.0f - px.m;
    g_kd[idx] = make_float4(gk.x * om + gF0.x * px.m, gk.y * om + gF0.y * px.m, gk.z * om + gF0.z * px.m, 0.f);
    const float g_m = -(gk.x * px.kd.x + gk.y * px.kd.y + gk.z * px.kd.z) + gF0.x * (px.kd.x - 0.04f) +
                      gF0.y * (px.kd.y - 0.04f) + gF0.z * (px.kd.z - 0.04f);
    const float g_r = (px.r * px.r > 1e-4f) ? g_alpha * 2.0f * px.r : 0.0f;
    g_korm[idx] = make_float4(0.f, g_r, g_m, 0.f);
    g_nrm[idx] = make_float4(gN.x, gN.y, gN.z, 0.f);
}

inline int grid_for(long long n, int threads) { return (int)((n + threads - 1) / threads); }

}  // namespace

cudaError_t launch_primary_cast(const void* nodes, const void* tris, int n_tris, const float* verts,
                                const float* vnrm, const int* tri_idx, int n_verts, const mcdi_camera* cams, int N,
                                int H, int W, const float* tex_kd, const float* tex_korm, int tex_size, float uv_ox,
                                float uv_oz, float uv_s, float* gb_pos, float* gb_nrm, float* gb_kd, float* gb_korm,
                                cudaStream_t stream) {
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const CastTiles T = cast_tiles(N, H, W, sms);
    launch_k(primary_cast_kernel, (unsigned)T.nx * (unsigned)T.ny * (unsigned)N, kShadeThreads, 0, stream,
             static_cast<const BvhNode*>(nodes), static_cast<const TriRecord*>(tris), n_tris, verts, vnrm, tri_idx,
             n_verts, cams, N, H, W, T, reinterpret_cast<const float4*>(tex_kd), reinterpret_cast<const float4*>(tex_korm),
             tex_size, uv_ox, uv_oz, uv_s, reinterpret_cast<float4*>(gb_pos), reinterpret_cast<float4*>(gb_nrm),
             reinterpret_cast<float4*>(gb_kd), reinterpret_cast<float4*>(gb_korm));
    return cudaGetLastError();
}

cudaError_t launch_shade_fwd(const ShadeArgs& a, float4* c_d, float4* kd_out, float4* c_s, uint32_t* vis_mask,
                             cudaStream_t stream) {
    const long long P = (long long)a.N * a.H * a.W;
    const size_t smem = sizeof(FwdShared) + (size_t)(a.Hp + 1) * sizeof(float);
    const cudaError_t e = allow_smem((const void*)shade_fwd_kernel, smem);
    if (e != cudaSuccess) return e;
    launch_k(shade_fwd_kernel, grid_for(P, 32), kShadeThreads, smem, stream, a, c_d, kd_out, c_s, vis_mask);
    return cudaGetLastError();
}

cudaError_t launch_shade_bwd(const ShadeArgs& a, const float4* g_cd, const float4* g_kdout, const float4* g_cs,
                             const uint32_t* vis_mask, float4* g_kd, float4* g_korm, float4* g_nrm, float4* g_env,
                             cudaStream_t stream, long long first, long long count) {
    const long long P = (long long)a.N * a.H * a.W;
    if (count < 0) count = P - first;
    if (count <= 0) return cudaSuccess;
    const size_t smem = (size_t)(((a.Hp + 1 + 3) & ~3) + kBwdQuarters * kBwdPartials * 32) * sizeof(float);
    if (vis_mask) {
        launch_k(shade_bwd_kernel<false>, grid_for(count, 32), kShadeThreads, smem, stream, a, g_cd, g_kdout, g_cs,
                 vis_mask, g_kd, g_korm, g_nrm, g_env, first, first + count);
        return cudaGetLastError();
    }
    const size_t smem_rt = smem + sizeof(BlockRays<kBwdChunk>);
    const cudaError_t e = allow_smem((const void*)shade_bwd_kernel<true>, smem_rt);
    if (e != cudaSuccess) return e;
    launch_k(shade_bwd_kernel<true>, grid_for(count, 32), kShadeThreads, smem_rt, stream, a, g_cd, g_kdout, g_cs,
             vis_mask, g_kd, g_korm, g_nrm, g_env, first, first + count);
    return cudaGetLastError();
}

}  // namespace mcdi
