// tcgen05 implicit-GEMM 3x3 convolution (see tc_conv.cuh): the row-tile form for
// images at least 48 pixels wide, the halo-tile form for narrower ones, and for
// layers neither can hold in shared memory the general form below.
//
// General form: one CTA computes a tile of 128 output pixels (tw x th) for all output
// channels: D[128 x cout_pad] (FP32, in tensor memory) = sum over the 9 taps
// and over input-channel chunks of 16 of
//   A[128 pixels x 16 ch] (the input shifted by the tap, zero outside the
//   image: TMA out-of-bounds fill) x B[cout_pad x 16 ch]^T (weights).
// Every chunk is one tcgen05.mma (M = 128, N = cout_pad, K = 16, BF16 inputs,
// FP32 accumulation).  Operands are staged by TMA through a ring of kStages
// shared-memory buffers guarded by mbarriers: the A tile as two 8-channel
// planes of 16-byte rows (no swizzle; activations live in 8-channel planes in
// global memory, so each plane's box is a run of contiguous rows), the weight
// slice with the 32-byte swizzle:
//   warp 0 lane 0  issues the TMA loads      (waits "empty", arms "full"),
//   warp 1 lane 0  issues the MMAs           (waits "full", commits to "empty"),
//   all 4 warps    run the epilogue: tcgen05.ld of their 32 TMEM lanes, bias,
//                  ReLU, BF16 stores (kStore only: the denoiser's own layers all
//                  fit one of the other forms).
// Every wait is bounded (2 s of %globaltimer); on a timeout the kernel sets
// *err, stops issuing work, drains its own copies in flight and frees TMEM.
#include <stdio.h>

#include <mutex>

#include <cudaTypedefs.h>

#include "common.cuh"
#include "tc_conv.cuh"
#include "tcgen05.cuh"

namespace mcdi {
namespace {

constexpr int kStages = 6;
constexpr int kConvThreads = 128;

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5}], [%6];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            int c4, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5, %6}], [%7];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar)
        : "memory");
}

// coordinates (2 x, y, plane) of a plane-row map (8-byte elements, two per pixel)
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2,
                                            uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
        "[%4];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
        : "memory");
}

// Shared-memory matrix descriptor of a K-major operand whose rows are 32 bytes
// (16 BF16 channels) with the 32-byte swizzle: 8-row atoms of 256 bytes
// stacked along M/N (stride 256 B); the K extent of one MMA is one row.
__device__ __forceinline__ uint64_t sw32_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);     // start address
    d |= (uint64_t)(16u >> 4) << 16;              // leading byte offset (unused with a one-row K extent)
    d |= (uint64_t)(256u >> 4) << 32;             // stride byte offset: next 8-row atom
    d |= (uint64_t)1 << 46;                       // descriptor version
    d |= (uint64_t)6 << 61;                       // swizzle: 32 bytes
    return d;
}

// K-major operand without swizzle: core matrices of 8 rows x 16 bytes with
// rows 16 bytes apart, 8-row groups 128 bytes apart (stride byte offset) and
// the second 8-channel half of K one plane further (leading byte offset).
__device__ __forceinline__ uint64_t noswz_desc(uint32_t saddr, uint32_t lbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)(128u >> 4) << 32;
    d |= (uint64_t)1 << 46;  // descriptor version; swizzle mode 0 (none)
    return d;
}

// The same with 8-row groups `sbo` bytes apart.
__device__ __forceinline__ uint64_t rows_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// Instruction descriptor of kind::f8f6f4 with E4M3 A and B (format code 0),
// K-major, FP32 D, M x N.
__host__ __device__ constexpr uint32_t e4m3_idesc(int M, int N) {
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

#define MCDI_MMA(KIND)                                                                         \
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"                             \
                 "tcgen05.mma.cta_group::1.kind::" KIND " [%0], %1, %2, %3, p;\n\t}" ::"r"(d), \
                 "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum)                                \
                 : "memory")

template <bool FP8>
__device__ __forceinline__ void mma_issue(uint32_t d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accum) {
    if constexpr (FP8) MCDI_MMA("f8f6f4");
    else MCDI_MMA("f16");
}
#undef MCDI_MMA

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* v) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void store8_bf16(__nv_bfloat16* dst, const float* f) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
        w[i] = *reinterpret_cast<uint32_t*>(&h);
    }
    *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
}

// Element offset of pixel (x, y) of image img in 8-channel group g of a
// tensor with G groups at H x W (layout [img][g][y][x][8]).
__device__ __forceinline__ size_t plane_off(int img, int G, int g, int H, int W, int y, int x) {
    return ((((size_t)img * G + g) * H + y) * W + x) * 8;
}

// bias / activation and store of 16 output channels (two 8-channel groups) of one
// pixel, in the general form
__device__ __forceinline__ void store_act16(const ConvParams& p, const uint32_t* v, int c0, int img, int x, int y,
                                            const float* bias16, float dq) {
    float f[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        f[i] = __fadd_rn(__fmul_rn(__uint_as_float(v[i]), dq), bias16 ? bias16[i] : 0.0f);
        if (p.relu) f[i] = fmaxf(f[i], 0.0f);
    }
    __nv_bfloat16* o = p.out + plane_off(img, p.out_ctotal >> 3, (p.out_coff + c0) >> 3, p.H, p.W, y, x);
    store8_bf16(o, f);
    store8_bf16(o + (size_t)p.H * p.W * 8, f + 8);
}

// accumulator scale: 1 for BF16; (amax_x / 448) (amax_w / 448) for E4M3
// operands quantised as round(v 448 / amax)
__device__ __forceinline__ float dequant_factor(const ConvParams& p) {
    if (!p.fp8) return 1.0f;
    return (__ldg(p.x_amax) * (1.0f / 448.0f)) * (__ldg(p.w_amax) * (1.0f / 448.0f));
}

template <bool FP8>
__global__ void __launch_bounds__(kConvThreads) conv_tc_kernel(const __grid_constant__ CUtensorMap tmap_x,
                                                               const __grid_constant__ CUtensorMap tmap_w,
                                                               const ConvParams p) {
    pdl_wait();
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kStages], empty_bar[kStages], acc_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ int failed;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // 1024-byte aligned staging ring
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    const uint32_t a_bytes = 128u * 32u, b_bytes = (uint32_t)p.cout_pad * 32u;
    const uint32_t stage_bytes = (a_bytes + b_bytes + 1023u) & ~1023u;
    const uint32_t ncols = p.cout_pad <= 32 ? 32u : (p.cout_pad <= 64 ? 64u : (p.cout_pad <= 128 ? 128u : 256u));

    int tile = blockIdx.x;
    const int tx = tile % p.tiles_x;
    tile /= p.tiles_x;
    const int ty = tile % p.tiles_y;
    const int img = tile / p.tiles_y;
    const int x0 = tx * p.tw, y0 = ty * p.th;
    const int cpt = p.cin_bytes >> 5;  // 32-byte channel chunks (one MMA K-step) per tap
    const int n_chunks = 9 * cpt;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(smem_u32(&full_bar[s]), 1);
            mbar_init(smem_u32(&empty_bar[s]), 1);
        }
        mbar_init(smem_u32(&acc_bar), 1);
        failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    pdl_allow_dependents();  // every CTA holds its tensor memory by then

    int issued = 0;
    if (warp == 0 && lane == 0) {
        // ---- TMA producer
        for (int k = 0; k < n_chunks; ++k) {
            const int s = k % kStages;
            const uint32_t ph = (uint32_t)(k / kStages) & 1u;
            if (!mbar_wait(smem_u32(&empty_bar[s]), ph ^ 1u)) {
                failed = 1;
                break;
            }
            const uint32_t a_dst = base + (uint32_t)s * stage_bytes;
            const uint32_t fb = smem_u32(&full_bar[s]);
            mbar_expect_tx(fb, a_bytes + b_bytes);
            const int tap = k / cpt, cc = k - tap * cpt;
            const int dy = tap / 3, dx = tap - 3 * (tap / 3);
            const int plane = img * (p.cin_bytes >> 4) + 2 * cc;
            tma_load_4d(a_dst, &tmap_x, 0, x0 + dx - 1, y0 + dy - 1, plane, fb);
            tma_load_4d(a_dst + a_bytes / 2, &tmap_x, 0, x0 + dx - 1, y0 + dy - 1, plane + 1, fb);
            tma_load_2d(a_dst + a_bytes, &tmap_w, tap * p.cin_bytes + cc * 32, 0, fb);
            issued = k + 1;
        }
    } else if (warp == 1 && lane == 0) {
        // ---- MMA issuer
        const uint32_t idesc = FP8 ? e4m3_idesc(128, p.cout_pad) : bf16_idesc(128, p.cout_pad);
        int k = 0;
        for (; k < n_chunks; ++k) {
            const int s = k % kStages;
            const uint32_t ph = (uint32_t)(k / kStages) & 1u;
            if (!mbar_wait(smem_u32(&full_bar[s]), ph)) {
                failed = 1;
                break;
            }
            tc_fence_after();
            const uint32_t a_src = base + (uint32_t)s * stage_bytes;
            const uint64_t adesc = noswz_desc(a_src, a_bytes / 2), bdesc = sw32_desc(a_src + a_bytes);
            mma_issue<FP8>(tmem, adesc, bdesc, idesc, k > 0 ? 1u : 0u);
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_u32(&empty_bar[s]))
                         : "memory");
        }
        if (k == n_chunks)
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_u32(&acc_bar))
                         : "memory");
    }
    __syncwarp();

    // ---- epilogue: every thread owns one accumulator row (one pixel)
    const bool acc_ok = mbar_wait(smem_u32(&acc_bar), 0u);
    if (!acc_ok) failed = 1;
    __syncwarp();
    tc_fence_after();
    const int m = warp * 32 + lane;
    const int xx = m % p.tw, yy = m / p.tw;
    const int x = x0 + xx, y = y0 + yy;
    const bool valid = acc_ok && x < p.W && y < p.H;
    const float dq = dequant_factor(p);
    for (int c0 = 0; c0 < p.cout_pad; c0 += 16) {
        uint32_t v[16];
        // collective load of 16 accumulator columns of this warp's 32 lanes
        tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
        if (valid && c0 < p.cout_valid)
            store_act16(p, v, c0, img, x, y, p.bias ? p.bias + c0 : nullptr, dq);
        __syncwarp();
    }

    // ---- teardown
    tc_fence_before();
    __syncthreads();
    if (failed) {
        if (threadIdx.x == 0) atomicExch(p.err, 1u);
        // wait (bounded) for this CTA's own TMA copies still in flight
        if (warp == 0 && lane == 0) {
            for (int k = 0; k < issued; ++k) {
                const int s = k % kStages;
                if (!mbar_wait(smem_u32(&full_bar[s]), (uint32_t)(k / kStages) & 1u)) break;
            }
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
    }
}

// ---------------------------------------------------------------------------
// Row-tile form, for images at least 48 pixels wide (128-pixel row tiles).
// A persistent CTA keeps a slice of Nc output channels of the layer's weights
// resident in shared memory for its whole life ([chunk][dx][dy][Nc][16 ch],
// 32-byte swizzle, one TMA load per chunk) and loops over tiles of R output
// rows x 128 pixels.  Per 16-channel input chunk the tile's halo, R + 2 rows x
// 130 pixels of two 8-channel planes, arrives once: each halo row is one
// contiguous run in the planar activation layout, copied with one bulk copy
// (large requests instead of one per 16-byte pixel), as are the zeros of the
// rows and columns beside the image.  Rows are 16 bytes per pixel and
// unswizzled, so any row starts a valid 8-row core matrix: the A operand of
// output row r and tap (dy, dx) is the window starting at halo row
// (r + dy) * 130 + dx, and MMAs (M = 128, N = up to 3 Nc, K = 16) over
// (R + 2) / R input rows per output row do the chunk (issue_chunk).
//   warp 0          weight TMA (lane 0), halo row copies (one lane per row),
//   warp 1          MMA issue (one elected lane); accumulators of tile i in
//                   TMEM buffer i & 1,
//   warps 2..9      epilogue: TMEM lane quarter warp % 4, and the two warps of
//                   a quarter take alternate 16-column chunks of each row.
// Compiled per rows R, operand type and epilogue (RowMode), so that each
// epilogue holds only its own registers: with all in one kernel chosen at run
// time they spilled, and the spills' write-through was most of the L2 writes.
// Measured, sixteen 800 x 800 images: forward 3.64 -> 2.58 ms, input gradient
// 4.45 -> 3.70 ms; two 512 x 512: 289 -> 231 and 334 -> 278 us.  At the full
// resolution the layers move 3.7 to 6.1 TB/s (four 800 x 800 images).
constexpr int kRowThreads = 320;
constexpr int kEpiWarps = kRowThreads / 32 - 2;
constexpr int kEpiSplit = kEpiWarps / 4;  // epilogue warps per TMEM lane quarter
constexpr int kRowMaxStages = 6;
constexpr int kHaloW = 130;
constexpr int kMaxRows = 4;

__device__ __align__(16) uint8_t g_zeros[kHaloW * 16];  // source of the halo's zeros


// ---- epilogue of the row-tile form: 16 accumulator columns of one pixel, as
// packed BF16 pairs (rounding before the ReLU or the mask gives what rounding
// after it would).
enum RowMode {  // what the kernel is compiled for: a ConvEpilogue, or kStore that also writes the 2x2 max-pool
    kRowStore = kStore, kRowUp2 = kStoreUp2, kRowF32 = kStoreF32, kRowMask = kDgradMask, kRowPlain = kDgradPlain,
    kRowPoolBwd = kDgradPoolBwd, kRowPool = 6
};

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ __nv_bfloat162 as_bf162(uint32_t w) { return *reinterpret_cast<const __nv_bfloat162*>(&w); }
__device__ __forceinline__ uint32_t max_bf16(uint32_t a, uint32_t b) {
    const __nv_bfloat162 m = __hmax2(as_bf162(a), as_bf162(b));
    return *reinterpret_cast<const uint32_t*>(&m);
}
// accumulators (times dq for E4M3 operands) plus bias, rounded to BF16
template <bool FP8>
__device__ __forceinline__ void bias_pack16(const uint32_t* v, float dq, const float* bias, uint32_t* h) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4 b = *reinterpret_cast<const float4*>(bias + 4 * i);
        const float x0 = __uint_as_float(v[4 * i]), x1 = __uint_as_float(v[4 * i + 1]);
        const float x2 = __uint_as_float(v[4 * i + 2]), x3 = __uint_as_float(v[4 * i + 3]);
        if constexpr (FP8) {
            h[2 * i] = pack_bf16(__fadd_rn(__fmul_rn(x0, dq), b.x), __fadd_rn(__fmul_rn(x1, dq), b.y));
            h[2 * i + 1] = pack_bf16(__fadd_rn(__fmul_rn(x2, dq), b.z), __fadd_rn(__fmul_rn(x3, dq), b.w));
        } else {
            const float2 s = add2({x0, x1}, {b.x, b.y}), t = add2({x2, x3}, {b.z, b.w});
            h[2 * i] = pack_bf16(s.x, s.y);
            h[2 * i + 1] = pack_bf16(t.x, t.y);
        }
    }
}
template <bool FP8>
__device__ __forceinline__ void scale_pack16(const uint32_t* v, float dq, uint32_t* h) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float a = __uint_as_float(v[2 * i]), b = __uint_as_float(v[2 * i + 1]);
        h[i] = FP8 ? pack_bf16(a * dq, b * dq) : pack_bf16(a, b);
    }
}
// running max |value| of stored BF16 pairs
__device__ __forceinline__ void fold_amax(uint32_t& am, const uint32_t* h, int n) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if (i < n) am = max_bf16(am, h[i] & 0x7fff7fffu);
}
__device__ __forceinline__ void publish_amax2(unsigned* out_amax, uint32_t am) {
    if (out_amax == nullptr) return;
    const unsigned hi = am & 0xffff0000u, lo = am << 16;  // the two halves as floats' bits (non-negative)
    const unsigned w = __reduce_max_sync(0xffffffffu, hi > lo ? hi : lo);
    if ((threadIdx.x & 31) == 0 && w > *(volatile const unsigned*)out_amax) atomicMax(out_amax, w);
}
// 32 bytes (two neighbouring pixels of an 8-channel plane) in one access: whole sectors, half the instructions
struct Words8 {
    uint32_t w[8];
};
__device__ __forceinline__ void store32(__nv_bfloat16* o, const Words8& v) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(o), "r"(v.w[0]), "r"(v.w[1]),
                 "r"(v.w[2]), "r"(v.w[3]), "r"(v.w[4]), "r"(v.w[5]), "r"(v.w[6]), "r"(v.w[7])
                 : "memory");
}
__device__ __forceinline__ Words8 load32(const __nv_bfloat16* a) {
    Words8 v;
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(v.w[0]), "=r"(v.w[1]), "=r"(v.w[2]), "=r"(v.w[3]), "=r"(v.w[4]), "=r"(v.w[5]), "=r"(v.w[6]), "=r"(v.w[7])
        : "l"(a));
    return v;
}
// two 8-channel groups of one pixel, `hw` pixels apart
__device__ __forceinline__ void store16(__nv_bfloat16* o, size_t hw, const uint32_t* h) {
    *reinterpret_cast<uint4*>(o) = make_uint4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<uint4*>(o + hw * 8) = make_uint4(h[4], h[5], h[6], h[7]);
}
// h where the mask words' values are positive, +0 elsewhere
__device__ __forceinline__ void apply_mask(uint32_t* h, uint4 a, uint4 b) {
    const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    const __nv_bfloat162 zero = as_bf162(0u);
#pragma unroll
    for (int i = 0; i < 8; ++i) h[i] &= __hgt2_mask(as_bf162(w[i]), zero);
}

// kRowPoolBwd: the gradient gp (packed pairs of 16 channels) at a pooled pixel, routed to the first maximum of
// the pooled tensor's 2x2 window `e`, plus the skip gradient `gs`, masked by E > 0, into the window of `o`
// (all three at the window's first pixel and first 8-channel group; W2, hw2: the full-size row and plane)
template <bool FP8>
__device__ __forceinline__ void pool_bwd16(const uint32_t* gp, const __nv_bfloat16* e, const __nv_bfloat16* gs,
                                           __nv_bfloat16* o, int W2, size_t hw2, uint32_t& am) {
    auto half = [](uint32_t w, int hi) { return __uint_as_float(hi ? (w & 0xffff0000u) : (w << 16)); };
#pragma unroll
    for (int gg = 0; gg < 2; ++gg) {
        const size_t g0 = gg * hw2 * 8, row = (size_t)W2 * 8;
        // window pixel k of channel pair j: word 4 (k & 1) + j of row k >> 1
        const Words8 e0 = load32(e + g0), e1 = load32(e + g0 + row);
        const Words8 s0 = load32(gs + g0), s1 = load32(gs + g0 + row);
        Words8 o0, o1;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t ew[4] = {e0.w[j], e0.w[4 + j], e1.w[j], e1.w[4 + j]};
            const uint32_t sw[4] = {s0.w[j], s0.w[4 + j], s1.w[j], s1.w[4 + j]};
            float x[4][2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                float best = half(ew[0], q);
                int arg = 0;  // the window's first maximum, in window order
#pragma unroll
                for (int k = 1; k < 4; ++k) {
                    const float v = half(ew[k], q);
                    if (v > best) best = v, arg = k;
                }
                const float g = half(gp[4 * gg + j], q);
#pragma unroll
                for (int k = 0; k < 4; ++k) x[k][q] = half(sw[k], q) + (arg == k ? g : 0.0f);
            }
            uint32_t h[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) h[k] = pack_bf16(x[k][0], x[k][1]) & __hgt2_mask(as_bf162(ew[k]), as_bf162(0u));
            o0.w[j] = h[0], o0.w[4 + j] = h[1], o1.w[j] = h[2], o1.w[4 + j] = h[3];
        }
        store32(o + g0, o0);
        store32(o + g0 + row, o1);
        if constexpr (FP8) {
            fold_amax(am, o0.w, 8);
            fold_amax(am, o1.w, 8);
        }
    }
}

// The rest of 16 accumulator columns of one pixel, except for kRowF32: packed (left in w), activated or masked
// (m0, m1: the mask words), folded into amax and stored at `out` (this pixel in the first of the two planes;
// kRowUp2, kRowPoolBwd: its 2x2 block at twice the size; Ws, hws: row and plane of the output).
template <int MODE, bool FP8>
__device__ __forceinline__ void finish16(const ConvParams& p, const uint32_t* acc, float dq, const float* bias16,
                                         uint4 m0, uint4 m1, const __nv_bfloat16* pooled, const __nv_bfloat16* skip,
                                         __nv_bfloat16* out, int Ws, size_t hws, uint32_t* w, uint32_t& amax) {
    if constexpr (MODE == kRowPoolBwd) {
        scale_pack16<FP8>(acc, dq, w);
        pool_bwd16<FP8>(w, pooled, skip, out, Ws, hws, amax);
    } else {
        if constexpr (MODE == kRowMask || MODE == kRowPlain) {
            scale_pack16<FP8>(acc, dq, w);
        } else {
            bias_pack16<FP8>(acc, dq, bias16, w);
            if (p.relu) {
#pragma unroll
                for (int j = 0; j < 8; ++j) w[j] = max_bf16(w[j], 0u);
            }
        }
        if constexpr (MODE == kRowMask) apply_mask(w, m0, m1);
        if constexpr (FP8) fold_amax(amax, w, 8);
        if constexpr (MODE == kRowUp2) {
#pragma unroll
            for (int gg = 0; gg < 2; ++gg) {
                const uint32_t* u = w + 4 * gg;
                const Words8 two_px = {{u[0], u[1], u[2], u[3], u[0], u[1], u[2], u[3]}};
                store32(out + gg * hws * 8, two_px);
                store32(out + gg * hws * 8 + (size_t)Ws * 8, two_px);
            }
        } else {
            store16(out, hws, w);
        }
    }
}
// kRowF32: channels 0..2 of one pixel
__device__ __forceinline__ void finish_f32(const ConvParams& p, const uint32_t* acc, float dq, const float* bias,
                                           size_t px) {
    float f[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        f[j] = __fadd_rn(__fmul_rn(__uint_as_float(acc[j]), dq), bias[j]);
        if (p.relu) f[j] = fmaxf(f[j], 0.0f);
    }
    p.out_f32[px] = make_float4(f[0], f[1], f[2], 0.0f);
}
__device__ __forceinline__ void load_mask_words(const __nv_bfloat16* at, size_t hw, uint4* w) {
    w[0] = __ldg(reinterpret_cast<const uint4*>(at));
    w[1] = __ldg(reinterpret_cast<const uint4*>(at + hw * 8));
}

// The MMAs of one 16-channel chunk (32-byte K-step) of a tile.  Halo row hr at
// column shift dx is the A window of output rows r = hr - dy for every tap row
// dy with 0 <= r < R.  Their accumulators lie in descending row order, so those
// of dy, dy + 1, ... are adjacent columns, and the weights of one dx lie in dy
// order ([dx][dy][Nc]), so one MMA with up to kStack tap rows stacked on N
// (kStack Nc <= 256) does them: at M = 128 an MMA costs 32 cycles for reading
// its A window plus N / 4 for its weights (N / 2 of math above N = 128), so
// three rows at Nc = 32 take 56 cycles instead of 120.  A tile's first MMA
// into accumulator r (chunk 0, hr = r, dx = 0, dy = 0) overwrites it and is
// issued by itself.  Every accumulator adds its taps in the order chunk, dy, dx.
template <int R, int kStack, bool FP8>
__device__ __forceinline__ void issue_chunk(uint32_t d0, uint64_t a0, uint64_t b0, int Nc, bool first) {
    const uint32_t step = (uint32_t)Nc * 2u;  // Nc x 32 bytes per tap, in 16-byte units
#pragma unroll
    for (int hr = 0; hr < R + 2; ++hr) {
        const int lo = hr - R + 1 > 0 ? hr - R + 1 : 0, hi = hr < 2 ? hr : 2;
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
            const uint64_t a = a0 + (uint64_t)(hr * kHaloW + dx);
#pragma unroll
            for (int dy = lo; dy <= hi; dy += kStack) {  // tap rows dy ... dy + n - 1
                const int n = hi - dy + 1 < kStack ? hi - dy + 1 : kStack;
                const uint32_t d = d0 + (uint32_t)((R - 1 - hr + dy) * Nc);
                const uint64_t b = b0 + (uint64_t)((uint32_t)(dx * 3 + dy) * step);
                const uint32_t idesc = FP8 ? e4m3_idesc(128, n * Nc) : bf16_idesc(128, n * Nc);
                if (dx == 0 && dy == 0 && hr < R) {
                    if (n == 1) {
                        mma_issue<FP8>(d, a, b, idesc, first ? 0u : 1u);
                    } else if (first) {
                        mma_issue<FP8>(d, a, b, FP8 ? e4m3_idesc(128, Nc) : bf16_idesc(128, Nc), 0u);
                        mma_issue<FP8>(d + (uint32_t)Nc, a, b + step,
                                       FP8 ? e4m3_idesc(128, (n - 1) * Nc) : bf16_idesc(128, (n - 1) * Nc), 1u);
                    } else {
                        mma_issue<FP8>(d, a, b, idesc, 1u);
                    }
                } else {
                    mma_issue<FP8>(d, a, b, idesc, 1u);
                }
            }
        }
    }
}

template <int R, bool FP8, int MODE>
__global__ void __launch_bounds__(kRowThreads, 2) conv_tc_rows_kernel(const __grid_constant__ CUtensorMap tmap_wh,
                                                                   const ConvParams p, const RowPlan rp) {
    // The setup that reads nothing the preceding kernel writes (barriers, bias, tensor memory and the
    // weight load: the weights and biases are packed once) runs before the wait on that kernel, so it
    // overlaps the preceding kernel's tail when the launch is programmatically dependent.  The next kernel may
    // launch once every CTA holds its tensor memory: its CTAs' allocations then wait for this kernel's and never
    // the other way round.
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(16) float s_bias[256];
    __shared__ __align__(8) uint64_t full_bar[kRowMaxStages], empty_bar[kRowMaxStages], accf_bar[2], acce_bar[2],
        w_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int failed;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t wbase = base + (uint32_t)rp.stages * rp.stage_bytes;
    const int S = rp.stages, Nc = rp.nc;
    const int n_chunks = p.cin_bytes >> 5;
    const uint32_t w_chunk = 9u * (uint32_t)Nc * 32u;  // bytes of one chunk's weights, all taps
    const int slice = blockIdx.x % rp.n_slices;
    const int n0 = slice * Nc;
    const int first = blockIdx.x / rp.n_slices, step = gridDim.x / rp.n_slices;
    const bool has_work = first < rp.n_tiles;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(smem_u32(&full_bar[s]), 1);
            mbar_init(smem_u32(&empty_bar[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&accf_bar[b]), 1);
            mbar_init(smem_u32(&acce_bar[b]), kEpiWarps);
        }
        mbar_init(smem_u32(&w_bar), 1);
        failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int c = threadIdx.x; c < Nc; c += blockDim.x) s_bias[c] = p.bias ? p.bias[n0 + c] : 0.0f;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(rp.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    pdl_allow_dependents();  // every CTA holds its tensor memory by then

    auto tile_origin = [&](int t, int* img, int* x0, int* y0) {
        const int tx = t % p.tiles_x;
        t /= p.tiles_x;
        *y0 = (t % p.tiles_y) * R;
        *img = t / p.tiles_y;
        *x0 = tx * 128;
    };

    int issued = 0;
    bool w_issued = false;
    if (warp == 0 && has_work && lane == 0) {
        const uint32_t wb = smem_u32(&w_bar);
        mbar_expect_tx(wb, (uint32_t)n_chunks * w_chunk);
        for (int c = 0; c < n_chunks; ++c) tma_load_5d(wbase + (uint32_t)c * w_chunk, &tmap_wh, 0, n0, 0, 0, c, wb);
        w_issued = true;
    }
    pdl_wait();  // activations, masks and outputs: after the preceding kernel has completed
    if (warp == 0) {
        if (has_work) {
            // Halo rows by plain bulk copies: lane l < 2 (R + 2) owns row l % (R + 2)
            // of plane l / (R + 2).  What lies outside the image is copied from a run
            // of zeros: a whole row above or below it, or the column beside its first
            // or last pixel (further columns reach only outputs outside the image).
            const int rows = R + 2;
            const bool mine = lane < 2 * rows;
            const int q = lane / rows, hr = lane - q * rows;
            const size_t plane_bytes = (size_t)p.H * p.W * 16;
            const uint8_t* x_bytes = reinterpret_cast<const uint8_t*>(p.x);
            auto copy = [&](uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
                asm volatile(
                    "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                    "l"(src), "r"(bytes), "r"(bar)
                    : "memory");
            };
            int g = 0;
            for (int t = first; t < rp.n_tiles; t += step) {
                int img, x0, y0;
                tile_origin(t, &img, &x0, &y0);
                const int y = y0 - 1 + hr;
                const bool row_in = mine && y >= 0 && y < p.H;
                const int xa = x0 > 0 ? x0 - 1 : 0, xb = x0 + 129 > p.W ? p.W : x0 + 129;  // columns in the image
                const bool left = x0 == 0, right = xb < x0 + 129;                          // columns -1 and W
                const uint32_t n_bytes = row_in ? (uint32_t)(xb - xa) * 16u : (mine ? (uint32_t)kHaloW * 16u : 0u);
                const uint32_t edge = row_in ? ((left ? 16u : 0u) + (right ? 16u : 0u)) : 0u;
                const uint32_t total = __reduce_add_sync(0xffffffffu, n_bytes + edge);
                const uint8_t* src0 = x_bytes + (size_t)(img * (p.cin_bytes >> 4) + q) * plane_bytes + ((size_t)y * p.W + xa) * 16;
                const uint32_t row0 = base + (uint32_t)q * rp.plane_bytes + (uint32_t)hr * (uint32_t)kHaloW * 16u;
                int c = 0;
                for (; c < n_chunks; ++c, ++g) {
                    const int s = g % S;
                    if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&empty_bar[s]), ((uint32_t)(g / S) & 1u) ^ 1u))) {
                        failed = 1;
                        break;
                    }
                    const uint32_t row_smem = row0 + (uint32_t)s * rp.stage_bytes;
                    const uint32_t fb = smem_u32(&full_bar[s]);
                    if (lane == 0) mbar_expect_tx(fb, total);
                    __syncwarp();
                    if (row_in) {
                        copy(row_smem + (left ? 16u : 0u), src0 + (size_t)(2 * c) * plane_bytes, n_bytes, fb);
                        if (left) copy(row_smem, g_zeros, 16u, fb);
                        if (right) copy(row_smem + (uint32_t)(xb - x0 + 1) * 16u, g_zeros, 16u, fb);
                    } else if (mine) {
                        copy(row_smem, g_zeros, n_bytes, fb);
                    }
                    issued = g + 1;
                }
                if (c < n_chunks || failed) break;
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (has_work) {  // the whole warp runs the loop, one elected lane issues (elect_one)
            const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
            const int stack = R == 1 ? 1 : (3 * Nc <= 256 ? 3 : (2 * Nc <= 256 ? 2 : 1));
            bool ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&w_bar), 0u));
            if (!ok) failed = 1;
            int g = 0, i = 0;
            for (int t = first; ok && t < rp.n_tiles; t += step, ++i) {
                const int b = i & 1;
                if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&acce_bar[b]), ((uint32_t)(i >> 1) & 1u) ^ 1u))) {
                    failed = 1;
                    break;
                }
                tc_fence_after();
                const uint32_t d0 = tm + (uint32_t)(b * R * Nc);
                int c = 0;
                for (; c < n_chunks; ++c, ++g) {
                    const int s = g % S;
                    if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&full_bar[s]), (uint32_t)(g / S) & 1u))) {
                        failed = 1;
                        break;
                    }
                    tc_fence_after();
                    // descriptors of the stage's halo and the chunk's weights; each MMA adds an
                    // offset (in 16-byte units) to the start-address field, which stays below 2^14
                    // for any shared-memory address
                    const uint64_t a0 = noswz_desc(base + (uint32_t)s * rp.stage_bytes, rp.plane_bytes);
                    const uint64_t b0 = sw32_desc(wbase + (uint32_t)c * w_chunk);
                    if (elect_one()) {
                        if (stack == 3) issue_chunk<R, 3, FP8>(d0, a0, b0, Nc, c == 0);
                        else if (stack == 2) issue_chunk<R, 2, FP8>(d0, a0, b0, Nc, c == 0);
                        else issue_chunk<R, 1, FP8>(d0, a0, b0, Nc, c == 0);
                        asm volatile(
                            "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                smem_u32(&empty_bar[s]))
                            : "memory");
                        if (c + 1 == n_chunks)
                            asm volatile(
                                "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                    smem_u32(&accf_bar[b]))
                                : "memory");
                    }
                    __syncwarp();
                }
                if (c < n_chunks) break;
            }
        }
        __syncwarp();
    } else {
        const int q = warp & 3, h = (warp - 2) >> 2;
        const int m = q * 32 + lane;
        uint32_t amax = 0, pool_amax = 0;
        // this warp's 16-column chunks of a row: 16 h, 16 (h + kEpiSplit), ...,
        // drained two per TMEM-load wait
        const int cfirst = 16 * h, cstep = 16 * kEpiSplit;
        const size_t hw = (size_t)p.H * p.W;
        const size_t pair = (size_t)(cstep >> 3) * hw * 8;  // elements from a chunk's planes to the next one's
        // ReLU-masked input gradients: the mask words of the tile's rows are loaded before its accumulator wait,
        // so their latency does not stall the epilogue (chunk cfirst; with at most two rows also the one after)
        constexpr int kMaskChunks = R <= 2 ? 2 : 1;
        uint4 mk[MODE == kRowMask ? R : 1][MODE == kRowMask ? kMaskChunks : 1][2];
        const __nv_bfloat16* mask_px = nullptr;
        int i = 0;
        for (int t = first; t < rp.n_tiles; t += step, ++i) {
            const int b = i & 1;
            int img, x0, y0;
            tile_origin(t, &img, &x0, &y0);
            const int x = x0 + m;
            const bool x_in = x < p.W;
            // this pixel of the tile's first row in the output's, mask's and skip gradient's first plane
            // (kRowUp2, kRowPoolBwd: at twice the size)
            constexpr int sc = MODE == kRowUp2 || MODE == kRowPoolBwd ? 2 : 1;
            const int Ws = p.W * sc;
            const size_t hws = hw * (sc * sc);
            auto first_px = [&](int ctotal, int coff) {
                return ((((size_t)img * (ctotal >> 3) + ((coff + n0 + cfirst) >> 3)) * (p.H * sc) + y0 * sc) * Ws + x * sc) * 8;
            };
            __nv_bfloat16* out_px = MODE == kRowF32 ? nullptr : p.out + first_px(p.out_ctotal, p.out_coff);
            const __nv_bfloat16* skip_px = nullptr;
            if (MODE == kRowMask || MODE == kRowPoolBwd) {
                const size_t at = first_px(p.mask_ctotal, p.mask_coff);
                mask_px = p.mask + at;
                if (MODE == kRowPoolBwd) skip_px = p.gskip + at;
            }
            const size_t pairs = (size_t)(cstep >> 3) * hws * 8;
            if constexpr (MODE == kRowMask) {
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int k = 0; k < kMaskChunks; ++k)
                        if (x_in && y0 + r < p.H && cfirst + k * cstep < Nc && n0 + cfirst + k * cstep < p.cout_valid)
                            load_mask_words(mask_px + (size_t)k * pair + (size_t)r * p.W * 8, hw, mk[r][k]);
            }
            const bool ok = mbar_wait(smem_u32(&accf_bar[b]), (uint32_t)(i >> 1) & 1u);
            __syncwarp();
            if (!__all_sync(0xffffffffu, ok)) {
                failed = 1;
                break;
            }
            tc_fence_after();
            const float dq = FP8 ? dequant_factor(p) : 1.0f;
            uint32_t ha[8], hb[8];  // kRowPool: the even row's stored values of the two chunks
            constexpr int kRowUnroll = MODE == kRowPoolBwd ? 1 : R;  // (unrolled it spills)
#pragma unroll kRowUnroll
            for (int r = 0; r < R; ++r) {
                const bool valid = x_in && y0 + r < p.H;
                const uint32_t tr = tmem + (uint32_t)((b * R + R - 1 - r) * Nc) + ((uint32_t)(q * 32) << 16);
                constexpr int kPer = MODE == kRowPoolBwd || MODE == kRowMask ? 1 : 2;  // chunks per TMEM-load wait
                for (int c0 = cfirst, k = 0; c0 < Nc; c0 += kPer * cstep, k += kPer) {
                    uint32_t v[16 * kPer];
                    const int c1 = c0 + cstep;
                    const bool two = kPer == 2 && c1 < Nc;
                    tmem_ld16_async(tr + (uint32_t)c0, v);
                    if constexpr (kPer == 2) {
                        if (two) tmem_ld16_async(tr + (uint32_t)c1, v + 16);
                    }
                    tmem_wait_ld();
                    const bool va = valid && n0 + c0 < p.cout_valid, vb = two && valid && n0 + c1 < p.cout_valid;
                    uint32_t ka[8], kb[8];
                    auto chunk = [&](const uint32_t* acc, int c, int kk, uint32_t* w) {
                        if constexpr (MODE == kRowF32) {
                            finish_f32(p, acc, dq, s_bias + c, ((size_t)img * p.H + y0 + r) * p.W + x);
                        } else {
                            uint4 mw[2] = {};
                            if constexpr (MODE == kRowMask) {
                                if (kk == 0) mw[0] = mk[r][0][0], mw[1] = mk[r][0][1];
                                else if (kMaskChunks == 2 && kk == 1)
                                    mw[0] = mk[r][kMaskChunks - 1][0], mw[1] = mk[r][kMaskChunks - 1][1];
                                else load_mask_words(mask_px + (size_t)kk * pair + (size_t)r * p.W * 8, hw, mw);
                            }
                            const size_t at = (size_t)kk * pairs + (size_t)(r * sc) * Ws * 8;
                            finish16<MODE, FP8>(p, acc, dq, s_bias + c, mw[0], mw[1], mask_px + at, skip_px + at,
                                                out_px + at, Ws, hws, w, amax);
                        }
                    };
                    if (va) chunk(v, c0, k, ka);
                    if constexpr (kPer == 2) {
                        if (vb) chunk(v + 16, c1, k + 1, kb);
                    }
                    if constexpr (MODE == kRowPool && R % 2 == 0) {
                        // 2x2 max-pool of the stored values: a window's two pixels are neighbouring lanes, its two
                        // rows consecutive rows of this thread (R even, tiles start on even rows and columns)
                        if ((r & 1) == 0) {
#pragma unroll
                            for (int j = 0; j < 8; ++j) ha[j] = ka[j], hb[j] = kb[j];
                        } else {
                            const int Hp = p.H >> 1, Wp = p.W >> 1;
                            auto pool_store = [&](const uint32_t* e, const uint32_t* o, int c, bool in) {
                                uint32_t w[8];
#pragma unroll
                                for (int j = 0; j < 8; ++j) {
                                    const uint32_t u = max_bf16(e[j], o[j]);
                                    w[j] = max_bf16(u, __shfl_xor_sync(0xffffffffu, u, 1));
                                }
                                if ((lane & 1) == 0 && in) {
                                    store16(p.pool_out + plane_off(img, p.pool_ctotal >> 3, c >> 3, Hp, Wp, (y0 + r) >> 1, x >> 1),
                                            (size_t)Hp * Wp, w);
                                    if constexpr (FP8) fold_amax(pool_amax, w, 8);
                                }
                            };
                            pool_store(ha, ka, n0 + c0, va);
                            if (two) pool_store(hb, kb, n0 + c1, vb);
                        }
                    }
                    __syncwarp();
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&acce_bar[b]));
        }
        if constexpr (FP8) {
            publish_amax2(p.out_amax, amax);
            if (MODE == kRowPool) publish_amax2(p.pool_amax, pool_amax);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (failed) {
        if (threadIdx.x == 0) atomicExch(p.err, 1u);
        if (warp == 0 && lane == 0) {  // let this CTA's copies in flight land before it exits
            if (w_issued) mbar_wait(smem_u32(&w_bar), 0u);
            for (int g = 0; g < issued; ++g)
                if (!mbar_wait(smem_u32(&full_bar[g % S]), (uint32_t)(g / S) & 1u)) break;
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(rp.tmem_cols)
                     : "memory");
    }
}

// ---------------------------------------------------------------------------
// Halo-tile form, for narrower images: a CTA computes 8 x 16 output pixels of a
// slice of Nc output channels with its whole working set in shared memory at
// once.  One TMA box brings the halo, 18 rows x 10 pixels of every input plane
// (planes as rows of 8-byte elements, zeros outside the image), and one box per
// tap its weights of all channel chunks ([tap][chunk][Nc][16 ch], 32-byte
// swizzle), so the MMAs start when the halo and the first tap's weights are
// there and wait for nothing but the next tap's.  The A operand of a tap is the
// halo from pixel (dy, dx) on: a tile row's 8 pixels are one core matrix, tile
// rows 160 bytes apart.  Accumulators add their products in the order tap,
// chunk.  What bounds it is the latency of this chain (launch, halo, MMAs at
// 32 + Nc / 4 cycles, epilogue), so the output channels are spread over as many
// CTAs as there are SMs.  Measured, the network's forward at 2 x 128 x 128 (six
// of its layers are this narrow) in a graph: 184 -> 92 us (before: one TMA round
// trip per tap and chunk, 14 to 33 us a layer).
constexpr int kHaloThreads = 128;
constexpr int kHaloTw = 8, kHaloTh = 16;                         // output pixels
constexpr int kHaloPx = kHaloTw + 2, kHaloRows = kHaloTh + 2;    // input pixels
constexpr uint32_t kHaloPlane = kHaloPx * kHaloRows * 16;        // bytes of one input plane

template <bool FP8, int MODE>
__global__ void __launch_bounds__(kHaloThreads) conv_tc_halo_kernel(const __grid_constant__ CUtensorMap tmap_x8,
                                                                    const __grid_constant__ CUtensorMap tmap_wt,
                                                                    const ConvParams p, const HaloPlan hp) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(16) float s_bias[256];
    __shared__ __align__(8) uint64_t a_bar, w_bar[9], acc_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int failed;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t wbase = base + hp.a_bytes;
    const int Nc = hp.nc, n_chunks = p.cin_bytes >> 5;
    const uint32_t w_tap = (uint32_t)(n_chunks * Nc) * 32u;
    int tile = blockIdx.x;
    const int n0 = (tile % hp.n_slices) * Nc;
    tile /= hp.n_slices;
    const int x0 = (tile % hp.tiles_x) * kHaloTw;
    tile /= hp.tiles_x;
    const int y0 = (tile % hp.tiles_y) * kHaloTh, img = tile / hp.tiles_y;

    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&a_bar), 1);
        for (int t = 0; t < 9; ++t) mbar_init(smem_u32(&w_bar[t]), 1);
        mbar_init(smem_u32(&acc_bar), 1);
        failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int c = threadIdx.x; c < Nc; c += blockDim.x) s_bias[c] = p.bias ? p.bias[n0 + c] : 0.0f;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(hp.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    pdl_allow_dependents();  // every CTA holds its tensor memory by then
    if (warp == 0 && lane == 0) {  // the weights were packed once: they need not wait for the preceding kernel
        for (int t = 0; t < 9; ++t) {
            mbar_expect_tx(smem_u32(&w_bar[t]), w_tap);
            tma_load_4d(wbase + (uint32_t)t * w_tap, &tmap_wt, 0, n0, 0, t, smem_u32(&w_bar[t]));
        }
    }
    pdl_wait();  // activations, masks and outputs: after the preceding kernel has completed
    if (warp == 0) {
        if (lane == 0) {
            const int planes = 2 * n_chunks;
            mbar_expect_tx(smem_u32(&a_bar), (uint32_t)planes * kHaloPlane);
            tma_load_3d(base, &tmap_x8, 2 * (x0 - 1), y0 - 1, img * planes, smem_u32(&a_bar));
        }
        __syncwarp();
    } else if (warp == 1) {
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
        const uint32_t idesc = FP8 ? e4m3_idesc(128, Nc) : bf16_idesc(128, Nc);
        const bool leader = elect_one();
        bool ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&a_bar), 0u));
        for (int t = 0; ok && t < 9; ++t) {
            ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&w_bar[t]), 0u));
            if (!ok) break;
            tc_fence_after();
            const uint64_t a0 = rows_desc(base + (uint32_t)((t / 3) * kHaloPx + t % 3) * 16u, kHaloPlane, kHaloPx * 16u);
            const uint64_t b0 = sw32_desc(wbase + (uint32_t)t * w_tap);
            for (int c = 0; c < n_chunks; ++c) {
                const uint64_t ad = a0 + (uint64_t)((uint32_t)c * (2u * kHaloPlane >> 4));
                const uint64_t bd = b0 + (uint64_t)((uint32_t)(c * Nc) * 2u);
                const uint32_t acc = t > 0 || c > 0 ? 1u : 0u;
                if (leader) mma_issue<FP8>(tm, ad, bd, idesc, acc);
                __syncwarp();
            }
        }
        if (ok && leader)
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_u32(&acc_bar))
                         : "memory");
        __syncwarp();
        if (!ok) failed = 1;
    }
    __syncwarp();

    // ---- epilogue: every thread owns one accumulator row (one pixel)
    const int m = warp * 32 + lane;
    const int x = x0 + m % kHaloTw, y = y0 + m / kHaloTw;
    const bool in = x < p.W && y < p.H;
    constexpr int sc = MODE == kRowUp2 || MODE == kRowPoolBwd ? 2 : 1;
    const int Ws = p.W * sc;
    const size_t hw = (size_t)p.H * p.W, hws = hw * (sc * sc);
    auto first_px = [&](int ctotal, int coff) {
        return ((((size_t)img * (ctotal >> 3) + ((coff + n0) >> 3)) * (p.H * sc) + y * sc) * Ws + x * sc) * 8;
    };
    __nv_bfloat16* out_px = MODE == kRowF32 ? nullptr : p.out + first_px(p.out_ctotal, p.out_coff);
    const __nv_bfloat16 *mask_px = nullptr, *skip_px = nullptr;
    if (MODE == kRowMask || MODE == kRowPoolBwd) {
        mask_px = p.mask + first_px(p.mask_ctotal, p.mask_coff);
        if (MODE == kRowPoolBwd) skip_px = p.gskip + first_px(p.mask_ctotal, p.mask_coff);
    }
    uint4 first_mask[2] = {};
    if (MODE == kRowMask && in && n0 < p.cout_valid) load_mask_words(mask_px, hw, first_mask);
    const float dq = FP8 ? dequant_factor(p) : 1.0f;
    const bool acc_ok = mbar_wait(smem_u32(&acc_bar), 0u);
    if (!acc_ok) failed = 1;
    __syncwarp();
    tc_fence_after();
    uint32_t amax = 0, pool_amax = 0;
    for (int c0 = 0, k = 0; c0 < Nc; c0 += 16, ++k) {
        uint32_t v[16], w[8];
        tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
        const bool valid = acc_ok && in && n0 + c0 < p.cout_valid;
        if (valid) {
            if constexpr (MODE == kRowF32) {
                finish_f32(p, v, dq, s_bias + c0, ((size_t)img * p.H + y) * p.W + x);
            } else {
                uint4 mw[2] = {first_mask[0], first_mask[1]};
                if (MODE == kRowMask && k > 0) load_mask_words(mask_px + (size_t)(2 * k) * hw * 8, hw, mw);
                const size_t at = (size_t)(2 * k) * hws * 8;
                finish16<MODE, FP8>(p, v, dq, s_bias + c0, mw[0], mw[1], mask_px + at, skip_px + at, out_px + at, Ws, hws,
                                    w, amax);
            }
        }
        if constexpr (MODE == kRowPool) {  // a window is four lanes of the warp: x in bit 0, y in bit 3
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                w[j] = max_bf16(w[j], __shfl_xor_sync(0xffffffffu, w[j], 1));
                w[j] = max_bf16(w[j], __shfl_xor_sync(0xffffffffu, w[j], 8));
            }
            if (valid && (lane & 9) == 0) {
                const int Hp = p.H >> 1, Wp = p.W >> 1;
                store16(p.pool_out + plane_off(img, p.pool_ctotal >> 3, (n0 + c0) >> 3, Hp, Wp, y >> 1, x >> 1),
                        (size_t)Hp * Wp, w);
                if constexpr (FP8) fold_amax(pool_amax, w, 8);
            }
        }
        __syncwarp();
    }
    if constexpr (FP8) {
        publish_amax2(p.out_amax, amax);
        if (MODE == kRowPool) publish_amax2(p.pool_amax, pool_amax);
    }

    // ---- teardown
    tc_fence_before();
    __syncthreads();
    if (failed) {
        if (threadIdx.x == 0) {
            atomicExch(p.err, 1u);
            // wait (bounded) for this CTA's own TMA copies still in flight
            for (int t = 0; t < 9; ++t)
                if (!mbar_wait(smem_u32(&w_bar[t]), 0u)) break;
            mbar_wait(smem_u32(&a_bar), 0u);
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(hp.tmem_cols) : "memory");
    }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn(const char** why) {
    static std::once_flag once;
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    if (!fn) *why = "cuTensorMapEncodeTiled is not available from the driver";
    return fn;
}

// The driver's encoder.  It wants a context that is current in the calling thread,
// which the runtime binds only with a thread's first call that needs one: a thread
// that starts with a convolution binds it here and encodes again.
struct Encoder {
    PFN_cuTensorMapEncodeTiled_v12000 fn;
    explicit operator bool() const { return fn != nullptr; }
    template <typename... Args>
    CUresult operator()(Args... args) const {
        const CUresult r = fn(args...);
        if (r != CUDA_ERROR_INVALID_CONTEXT && r != CUDA_ERROR_NOT_INITIALIZED) return r;
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaSetDevice(dev) != cudaSuccess) return r;
        return fn(args...);
    }
};

struct DeviceLimits {
    int sms = 0;
    uint32_t rows_smem_max = 0;  // dynamic shared memory one row-tile CTA may request
    uint32_t rows_smem_two = 0;  // dynamic shared memory per CTA with two CTAs on an SM
};

const DeviceLimits& device_limits() {
    static std::once_flag once;
    static DeviceLimits L;
    std::call_once(once, [] {
        int dev = 0, optin = 0, per_sm = 0, reserved = 0;
        cudaFuncAttributes fa{};
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&L.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess ||
            cudaFuncGetAttributes(&fa, conv_tc_rows_kernel<4, false, kRowStore>) != cudaSuccess ||
            optin <= (int)fa.sharedSizeBytes) {
            L.sms = 0;
            return;
        }
        L.rows_smem_max = (uint32_t)(optin - (int)fa.sharedSizeBytes);
        const int two = per_sm / 2 - (int)fa.sharedSizeBytes - reserved;
        L.rows_smem_two = two > 0 ? (uint32_t)two : 0u;
    });
    return L;
}

uint32_t pow2_at_least(uint32_t v) {
    uint32_t c = 32;
    while (c < v) c <<= 1;
    return c;
}

// Row-tile plan: the fewest channel slices whose resident weights leave room
// for two halo stages; per slice the most rows per tile (up to kMaxRows) that
// fit tensor memory (two buffers of R accumulators) and still give 1.5 tiles
// per SM; two CTAs per SM where both fit in shared memory and tensor memory.
bool plan_rows(const ConvParams& p, RowPlan* out) {
    if (p.tw != 128 || p.th != 1) return false;
    const DeviceLimits& lim = device_limits();
    const int sms = lim.sms;
    if (sms <= 0) return false;
    const uint32_t kSmemMax = lim.rows_smem_max, kAlign = 1024u;
    const int n_chunks = p.cin_bytes / 32;
    for (int n_slices = 1; 16 * n_slices <= p.cout_pad; ++n_slices) {
        if (p.cout_pad % (16 * n_slices) != 0) continue;
        const int nc = p.cout_pad / n_slices;
        const uint32_t w_bytes = (uint32_t)n_chunks * 9u * (uint32_t)nc * 32u;
        // the largest R that fits, except that a plan of two CTAs per SM is
        // preferred to one of a single CTA with a larger R
        RowPlan single{};
        bool have_single = false;
        for (int R = kMaxRows; R >= 1; R >>= 1) {
            const uint32_t tmem_cols = pow2_at_least(2u * (uint32_t)(R * nc));
            if (tmem_cols > 512u) continue;
            RowPlan rp{};
            rp.rows = R;
            rp.nc = nc;
            rp.n_slices = n_slices;
            rp.plane_bytes = ((uint32_t)(R + 2) * kHaloW * 16u + 127u) & ~127u;
            rp.stage_bytes = (2u * rp.plane_bytes + 1023u) & ~1023u;
            rp.tmem_cols = tmem_cols;
            if (w_bytes + 2u * rp.stage_bytes + kAlign > kSmemMax) continue;
            rp.n_tiles = p.n_img * ((p.H + R - 1) / R) * p.tiles_x;
            if (R > 1 && 2 * n_slices * rp.n_tiles < 3 * sms) continue;
            // two CTAs per SM (their MMA streams interleave on the tensor core) as
            // soon as each fits a two-stage halo ring beside its weights
            const bool two = w_bytes + 2u * rp.stage_bytes + kAlign <= lim.rows_smem_two && 2u * tmem_cols <= 512u;
            const uint32_t budget = two ? lim.rows_smem_two : kSmemMax;
            int S = (int)((budget - kAlign - w_bytes) / rp.stage_bytes);
            rp.stages = S > kRowMaxStages ? kRowMaxStages : S;
            rp.smem_bytes = (uint32_t)rp.stages * rp.stage_bytes + w_bytes + kAlign;
            const int per_slice = (two ? 2 : 1) * sms / n_slices;
            rp.grid = n_slices * (per_slice < rp.n_tiles ? per_slice : rp.n_tiles);
            if (two || R == 1) {
                *out = have_single && !two ? single : rp;
                return true;
            }
            if (!have_single) {
                single = rp;
                have_single = true;
            }
        }
        if (have_single) {
            *out = single;
            return true;
        }
    }
    return false;
}

size_t conv_smem_bytes(int cout_pad) {
    const size_t stage = ((size_t)128 * 32 + (size_t)cout_pad * 32 + 1023) & ~(size_t)1023;
    return kStages * stage + 1024;
}

}  // namespace

bool encode_plane_rows_map(CUtensorMap* map, const void* base, int W, int H, long long n_planes, int box_px,
                           int box_rows, int box_planes, const char** why) {
    const Encoder enc{encode_fn(why)};
    if (!enc) return false;
    // BF16 8-channel planes [plane][H][W][16 B] as rows of 8-byte elements (two per pixel), so that a box
    // row of box_px pixels is one contiguous run for the copy engine
    const cuuint64_t dims[3] = {(cuuint64_t)W * 2, (cuuint64_t)H, (cuuint64_t)n_planes};
    const cuuint64_t str[2] = {(cuuint64_t)W * 16, (cuuint64_t)H * W * 16};
    const cuuint32_t box[3] = {(cuuint32_t)box_px * 2, (cuuint32_t)box_rows, (cuuint32_t)box_planes};
    const cuuint32_t ones[3] = {1, 1, 1};
    const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_INT64, 3, const_cast<void*>(base), dims, str, box, ones,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        *why = "plane-row tensor map rejected by the driver";
        return false;
    }
    return true;
}

// 128-pixel row tiles from 48 pixels up (narrower rows would leave most of each
// tile's MMA rows empty); below that the smallest power of two covering W
int conv_pick_tile_w(int W) {
    if (W >= 48) return 128;
    int tw = 64;
    while (tw > 8 && tw / 2 >= W) tw /= 2;
    return tw;
}

// Halo-tile plan: the tile's halo of every plane and a slice's weights fit in
// shared memory at once; the fewest channels per slice that still leave no SM
// with a second CTA, so that the chain of one is as short as it gets.
static bool plan_halo(const ConvParams& p, HaloPlan* out) {
    const DeviceLimits& lim = device_limits();
    if (lim.sms <= 0 || p.W >= kHaloMaxW) return false;
    const int n_chunks = p.cin_bytes / 32;
    HaloPlan hp{};
    hp.tiles_x = (p.W + kHaloTw - 1) / kHaloTw;
    hp.tiles_y = (p.H + kHaloTh - 1) / kHaloTh;
    const long long tiles = (long long)p.n_img * hp.tiles_x * hp.tiles_y;
    const size_t a_bytes = ((size_t)(2 * n_chunks) * kHaloPlane + 1023) & ~(size_t)1023;
    if (2 * n_chunks > 256 || a_bytes > lim.rows_smem_max) return false;
    hp.a_bytes = (uint32_t)a_bytes;
    bool found = false;
    for (int n = 1; 16 * n <= p.cout_pad; ++n) {
        if (p.cout_pad % (16 * n) != 0) continue;
        const int nc = p.cout_pad / n;
        const size_t smem = a_bytes + (size_t)9 * n_chunks * nc * 32 + 1024;
        if (smem > lim.rows_smem_max) continue;
        if (found && tiles * n > lim.sms) break;
        hp.nc = nc;
        hp.n_slices = n;
        hp.tmem_cols = pow2_at_least((uint32_t)nc);
        hp.smem_bytes = (uint32_t)smem;
        hp.grid = (int)(tiles * n);
        found = true;
    }
    if (!found || tiles * hp.n_slices > 0x7fffffffll) return false;
    *out = hp;
    return true;
}

bool conv_make_desc(ConvDesc* d, const void* x, const void* w, const char** why) {
    const Encoder enc{encode_fn(why)};
    if (!enc) return false;
    const ConvParams& p = d->p;
    d->p.x = x;
    d->halo_form = plan_halo(p, &d->hp);
    if (d->halo_form) {
        if (!encode_plane_rows_map(&d->tmap_x, x, p.W, p.H, (long long)p.n_img * (p.cin_bytes / 16), kHaloPx, kHaloRows,
                                   2 * (p.cin_bytes / 32), why))
            return false;
        const cuuint64_t tdims[4] = {32, (cuuint64_t)p.cout_pad, (cuuint64_t)(p.cin_bytes / 32), 9};
        const cuuint64_t tstr[3] = {(cuuint64_t)9 * p.cin_bytes, 32, (cuuint64_t)p.cin_bytes};
        const cuuint32_t tbox[4] = {32, (cuuint32_t)d->hp.nc, (cuuint32_t)(p.cin_bytes / 32), 1};
        const cuuint32_t ones4[4] = {1, 1, 1, 1};
        if (enc(&d->tmap_w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void*>(w), tdims, tstr, tbox, ones4,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
            *why = "tap weight tensor map rejected by the driver";
            return false;
        }
        return true;
    }
    // The maps move bytes: activations are planes of 16-byte pixel rows
    // ([img * cin_bytes / 16 + plane][H][W][16 B]), weights are K-major rows
    // of 9 * cin_bytes bytes, BF16 or E4M3 alike.
    const cuuint64_t xdims[4] = {16, (cuuint64_t)p.W, (cuuint64_t)p.H, (cuuint64_t)p.n_img * (p.cin_bytes / 16)};
    const cuuint64_t xstr[3] = {16, (cuuint64_t)p.W * 16, (cuuint64_t)p.H * p.W * 16};
    const cuuint32_t xbox[4] = {16, (cuuint32_t)p.tw, (cuuint32_t)p.th, 1};
    const cuuint32_t ones[4] = {1, 1, 1, 1};
    CUresult r = enc(&d->tmap_x, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void*>(x), xdims, xstr, xbox, ones,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        *why = "activation tensor map rejected by the driver";
        return false;
    }
    const cuuint64_t wdims[2] = {(cuuint64_t)9 * p.cin_bytes, (cuuint64_t)p.cout_pad};
    const cuuint64_t wstr[1] = {(cuuint64_t)9 * p.cin_bytes};
    const cuuint32_t wbox[2] = {32, (cuuint32_t)p.cout_pad};
    r = enc(&d->tmap_w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(w), wdims, wstr, wbox, ones,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        *why = "weight tensor map rejected by the driver";
        return false;
    }
    d->rows_form = plan_rows(d->p, &d->rp);
    if (!d->rows_form && (p.mode != kStore || p.out_amax != nullptr)) {  // what the general form can do
        *why = "layer outside the row-tile and halo-tile forms";
        return false;
    }
    if (d->rows_form) {
        const RowPlan& rp = d->rp;
        d->p.tiles_y = (p.H + rp.rows - 1) / rp.rows;
        // The same K-major weights [cout][tap][cin] viewed as (32 bytes of
        // channels, cout, tap row dy, tap column dx, chunk): one box lands in
        // shared memory as [dx][dy][nc][32 B].
        const cuuint64_t tap = (cuuint64_t)p.cin_bytes;
        const cuuint64_t hdims[5] = {32, (cuuint64_t)p.cout_pad, 3, 3, (cuuint64_t)(p.cin_bytes / 32)};
        const cuuint64_t hstr[4] = {9 * tap, 3 * tap, tap, 32};
        const cuuint32_t hwbox[5] = {32, (cuuint32_t)rp.nc, 3, 3, 1};
        const cuuint32_t ones5[5] = {1, 1, 1, 1, 1};
        r = enc(&d->tmap_wh, CU_TENSOR_MAP_DATA_TYPE_UINT8, 5, const_cast<void*>(w), hdims, hstr, hwbox, ones5,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) {
            *why = "halo weight tensor map rejected by the driver";
            return false;
        }
    }
    return true;
}

template <bool FP8>
static const void* halo_kernel(int mode) {
    switch (mode) {
        case kRowUp2: return (const void*)conv_tc_halo_kernel<FP8, kRowUp2>;
        case kRowF32: return (const void*)conv_tc_halo_kernel<FP8, kRowF32>;
        case kRowMask: return (const void*)conv_tc_halo_kernel<FP8, kRowMask>;
        case kRowPlain: return (const void*)conv_tc_halo_kernel<FP8, kRowPlain>;
        case kRowPoolBwd: return (const void*)conv_tc_halo_kernel<FP8, kRowPoolBwd>;
        case kRowPool: return (const void*)conv_tc_halo_kernel<FP8, kRowPool>;
        default: return (const void*)conv_tc_halo_kernel<FP8, kRowStore>;
    }
}
static const void* halo_kernel(bool fp8, int mode) { return fp8 ? halo_kernel<true>(mode) : halo_kernel<false>(mode); }

template <int R, bool FP8>
static const void* rows_kernel(int mode) {
    switch (mode) {
        case kRowUp2: return (const void*)conv_tc_rows_kernel<R, FP8, kRowUp2>;
        case kRowF32: return (const void*)conv_tc_rows_kernel<R, FP8, kRowF32>;
        case kRowMask: return (const void*)conv_tc_rows_kernel<R, FP8, kRowMask>;
        case kRowPlain: return (const void*)conv_tc_rows_kernel<R, FP8, kRowPlain>;
        case kRowPoolBwd: return (const void*)conv_tc_rows_kernel<R, FP8, kRowPoolBwd>;
        case kRowPool: return (const void*)conv_tc_rows_kernel<(R > 1 ? R : 2), FP8, kRowPool>;  // planned for even R only
        default: return (const void*)conv_tc_rows_kernel<R, FP8, kRowStore>;
    }
}

static const void* rows_kernel(int rows, bool fp8, int mode) {
    if (rows == 4) return fp8 ? rows_kernel<4, true>(mode) : rows_kernel<4, false>(mode);
    if (rows == 2) return fp8 ? rows_kernel<2, true>(mode) : rows_kernel<2, false>(mode);
    return fp8 ? rows_kernel<1, true>(mode) : rows_kernel<1, false>(mode);
}

bool conv_mask_prefetch(const ConvDesc& d) { return d.rows_form && d.p.mode == kDgradMask && d.rp.nc <= 64; }

cudaError_t conv_launch(const ConvDesc& d, cudaStream_t stream) {
    static std::once_flag once;
    static cudaError_t attr_err = cudaSuccess;
    std::call_once(once, [] {
        const int lim = (int)device_limits().rows_smem_max;
        const int tile = (int)conv_smem_bytes(256);
        const void* generic[2] = {(const void*)conv_tc_kernel<false>, (const void*)conv_tc_kernel<true>};
        for (const void* f : generic)
            if (attr_err == cudaSuccess)
                attr_err = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, tile);
        for (int mode = 0; mode <= kRowPool; ++mode)
            for (bool fp8 : {false, true})
                if (attr_err == cudaSuccess)
                    attr_err = cudaFuncSetAttribute(halo_kernel(fp8, mode), cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
        for (int rows : {1, 2, 4})
            for (int mode = 0; mode <= kRowPool; ++mode)
                for (bool fp8 : {false, true})
                    if (attr_err == cudaSuccess)
                        attr_err = cudaFuncSetAttribute(rows_kernel(rows, fp8, mode),
                                                        cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    });
    if (attr_err != cudaSuccess) return attr_err;
    if (d.halo_form) {
        const int mode = d.p.pool_out != nullptr ? (int)kRowPool : d.p.mode;
        using Kernel = void(const CUtensorMap, const CUtensorMap, const ConvParams, const HaloPlan);
        auto* kernel = reinterpret_cast<Kernel*>(const_cast<void*>(halo_kernel(d.p.fp8 != 0, mode)));
        launch_k_dependent(kernel, dim3(d.hp.grid), dim3(kHaloThreads), d.hp.smem_bytes, stream, d.tmap_x, d.tmap_w, d.p, d.hp);
        return cudaGetLastError();
    }
    if (d.rows_form) {
        const int mode = d.p.pool_out != nullptr ? (int)kRowPool : d.p.mode;  // run_conv pools only where the plan can
        using Kernel = void(const CUtensorMap, const ConvParams, const RowPlan);
        auto* kernel = reinterpret_cast<Kernel*>(const_cast<void*>(rows_kernel(d.rp.rows, d.p.fp8 != 0, mode)));
        launch_k_dependent(kernel, dim3(d.rp.grid), dim3(kRowThreads), d.rp.smem_bytes, stream, d.tmap_wh, d.p, d.rp);
        return cudaGetLastError();
    }
    const int n_tiles = d.p.n_img * d.p.tiles_y * d.p.tiles_x;
    const size_t smem = conv_smem_bytes(d.p.cout_pad);
    if (d.p.fp8) launch_k(conv_tc_kernel<true>, n_tiles, kConvThreads, smem, stream, d.tmap_x, d.tmap_w, d.p);
    else launch_k(conv_tc_kernel<false>, n_tiles, kConvThreads, smem, stream, d.tmap_x, d.tmap_w, d.p);
    return cudaGetLastError();
}

}  // namespace mcdi
