// Device functions of the Monte Carlo direct-illumination estimator (Sec. 3.1,
// Sec. 4.1): BVH traversal, probe / cosine / GGX sampling and densities, the
// GGX lobe, and the per-sample MIS weight.  Everything is FP32.
#pragma once

#include <float.h>

#include "common.cuh"

namespace mcdi {

// ---------------------------------------------------------------- fixed roundings
// What decides a sample (its direction, its probe texel, whether a triangle
// blocks its ray) is written with every rounding spelled out, so that the kernels
// that draw a sample or trace its ray decide it alike whatever is compiled around
// it: a sum of products as one fused multiply-add per product after the first, a +
// b (p q) as one.  One difference is kept: the adjoint's GGX samples (sample_ggx).
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float dot_rn(f3 a, f3 b) {
    return fma_rn(a.z, b.z, fma_rn(a.x, b.x, mul_rn(a.y, b.y)));
}
// the same sum with the first two products the other way round
__device__ __forceinline__ float dot_xy_rn(f3 a, f3 b) {
    return fma_rn(a.z, b.z, fma_rn(a.y, b.y, mul_rn(a.x, b.x)));
}
__device__ __forceinline__ f3 cross_rn(f3 a, f3 b) {
    return {fma_rn(a.y, b.z, -mul_rn(a.z, b.y)), fma_rn(a.z, b.x, -mul_rn(a.x, b.z)),
            fma_rn(a.x, b.y, -mul_rn(a.y, b.x))};
}
__device__ __forceinline__ f3 scale_rn(f3 a, float s) { return {mul_rn(a.x, s), mul_rn(a.y, s), mul_rn(a.z, s)}; }
__device__ __forceinline__ f3 add_rn(f3 a, f3 b) { return {add_rn(a.x, b.x), add_rn(a.y, b.y), add_rn(a.z, b.z)}; }
__device__ __forceinline__ f3 normalize_rn(f3 a) { return scale_rn(a, rsqrtf(dot_rn(a, a))); }
__device__ __forceinline__ f3 normalize_xy_rn(f3 a) { return scale_rn(a, rsqrtf(dot_xy_rn(a, a))); }
// a x + b y + c z
__device__ __forceinline__ f3 combine_rn(f3 a, float x, f3 b, float y, f3 c, float z) {
    return {fma_rn(c.x, z, fma_rn(a.x, x, mul_rn(b.x, y))), fma_rn(c.y, z, fma_rn(a.y, x, mul_rn(b.y, y))),
            fma_rn(c.z, z, fma_rn(a.z, x, mul_rn(b.z, y)))};
}
// a s + b
__device__ __forceinline__ f3 fma_rn(f3 a, float s, f3 b) {
    return {fma_rn(a.x, s, b.x), fma_rn(a.y, s, b.y), fma_rn(a.z, s, b.z)};
}

// ---------------------------------------------------------------- traversal
struct RayInv {
    f3 o, d, inv;
};

__device__ __forceinline__ RayInv make_ray(f3 o, f3 d) {
    // direction components are kept away from zero so that slab distances stay finite
    auto safe = [](float x) { return fabsf(x) < 1e-20f ? copysignf(1e-20f, x) : x; };
    RayInv r;
    r.o = o;
    r.d = d;
    r.inv = mk(1.0f / safe(d.x), 1.0f / safe(d.y), 1.0f / safe(d.z));
    return r;
}

// whether neither the ray's origin nor its direction has a NaN or an infinity
__device__ __forceinline__ bool finite_ray(f3 o, f3 d) {
    const float big = 3.402823466e38f;
    return fabsf(o.x) <= big && fabsf(o.y) <= big && fabsf(o.z) <= big && fabsf(d.x) <= big && fabsf(d.y) <= big &&
           fabsf(d.z) <= big;
}

// slab test of one box given as (lo.x, hi.x, lo.y, hi.y) + (lo.z, hi.z);
// returns the entry distance or +inf on a miss.  The exit distance is scaled by
// 1 + 2 gamma_3 so that rounding never drops a box the ray touches (Ize 2013).
__device__ __forceinline__ float slab(const RayInv& r, float4 xy, float2 z, float tmax) {
    const float tx0 = (xy.x - r.o.x) * r.inv.x, tx1 = (xy.y - r.o.x) * r.inv.x;
    const float ty0 = (xy.z - r.o.y) * r.inv.y, ty1 = (xy.w - r.o.y) * r.inv.y;
    const float tz0 = (z.x - r.o.z) * r.inv.z, tz1 = (z.y - r.o.z) * r.inv.z;
    const float t0 = fmaxf(fmaxf(fminf(tx0, tx1), fminf(ty0, ty1)), fmaxf(fminf(tz0, tz1), 0.0f));
    const float t1 = fminf(fminf(fmaxf(tx0, tx1), fmaxf(ty0, ty1)), fminf(fmaxf(tz0, tz1), tmax)) * 1.00000036f;
    return t0 <= t1 ? t0 : FLT_MAX;
}

// Moller-Trumbore, two-sided, edges inclusive, for the triangle v0 + u e1 + v e2;
// returns t (> 0) or +inf
__device__ __forceinline__ float tri_hit_v(const RayInv& r, f3 v0, f3 e1, f3 e2, float* bu, float* bv) {
    const f3 p = cross(r.d, e2);
    const float det = dot(e1, p);
    if (det == 0.0f) return FLT_MAX;
    const float inv = 1.0f / det;
    const f3 s = r.o - v0;
    const float u = dot(s, p) * inv;
    if (u < 0.0f || u > 1.0f) return FLT_MAX;
    const f3 q = cross(s, e1);
    const float v = dot(r.d, q) * inv;
    if (v < 0.0f || u + v > 1.0f) return FLT_MAX;
    const float t = dot(e2, q) * inv;
    if (!(t > 0.0f)) return FLT_MAX;
    if (bu) {
        *bu = u;
        *bv = v;
    }
    return t;
}

// the same test against triangle record k
__device__ __forceinline__ float tri_hit(const RayInv& r, const TriRecord* __restrict__ tris, int k, float* bu,
                                         float* bv) {
    const float4 v0 = __ldg(&tris[k].v0), e1 = __ldg(&tris[k].e1), e2 = __ldg(&tris[k].e2);
    return tri_hit_v(r, xyz(v0), xyz(e1), xyz(e2), bu, bv);
}

// Triangle record k in two loads: records are 48 bytes apart on 16-byte
// boundaries, so either their first 32 bytes or their last 32 start on a
// 32-byte boundary.  (Each load of a lane is one L1 wavefront when lanes read
// different records; three 16-byte loads made the tracer 3% slower.)
__device__ __forceinline__ void load_record(const TriRecord* __restrict__ tris, int k, f3& v0, f3& e1, f3& e2) {
    const char* a = reinterpret_cast<const char*>(tris + k);
    const bool odd = (reinterpret_cast<uintptr_t>(a) & 16) != 0;
    float4 x, y;
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w), "=f"(y.x), "=f"(y.y), "=f"(y.z), "=f"(y.w)
        : "l"(a + (odd ? 16 : 0)));
    const float4 z = __ldg(reinterpret_cast<const float4*>(a + (odd ? 0 : 32)));
    v0 = odd ? xyz(z) : xyz(x);
    e1 = odd ? xyz(x) : xyz(y);
    e2 = odd ? xyz(y) : xyz(z);
}

// The same test of a shadow ray (hit or not) with every rounding written out
// (the products of tri_hit_v as the compiler contracts them).
__device__ __forceinline__ bool tri_blocks(f3 o, f3 d, const TriRecord* __restrict__ tris, int k) {
    f3 v0, e1, e2;
    load_record(tris, k, v0, e1, e2);
    const f3 p = cross_rn(d, e2);
    const float det = dot_rn(e1, p);
    if (det == 0.0f) return false;
    const float inv = 1.0f / det;
    const f3 s = {__fsub_rn(o.x, v0.x), __fsub_rn(o.y, v0.y), __fsub_rn(o.z, v0.z)};
    const float u = __fmul_rn(dot_rn(s, p), inv);
    if (u < 0.0f || u > 1.0f) return false;
    const f3 q = cross_rn(s, e1);
    const float v = __fmul_rn(dot_rn(d, q), inv);
    if (v < 0.0f || __fadd_rn(u, v) > 1.0f) return false;
    return __fmul_rn(dot_rn(e2, q), inv) > 0.0f;
}

// slab test of a box given by its corners (xyz of lo and hi); same rounding
// rule as slab()
__device__ __forceinline__ bool slab_hit(const RayInv& r, float4 lo, float4 hi) {
    const float tx0 = (lo.x - r.o.x) * r.inv.x, tx1 = (hi.x - r.o.x) * r.inv.x;
    const float ty0 = (lo.y - r.o.y) * r.inv.y, ty1 = (hi.y - r.o.y) * r.inv.y;
    const float tz0 = (lo.z - r.o.z) * r.inv.z, tz1 = (hi.z - r.o.z) * r.inv.z;
    const float t0 = fmaxf(fmaxf(fminf(tx0, tx1), fminf(ty0, ty1)), fmaxf(fminf(tz0, tz1), 0.0f));
    const float t1 = fminf(fminf(fmaxf(tx0, tx1), fmaxf(ty0, ty1)), fmaxf(tz0, tz1)) * 1.00000036f;
    return t0 <= t1;
}

// One step of stackless any-hit traversal at node i of the depth-first
// layout: returns the next node index (> i), or -1 when the ray is blocked.
// kCount adds the triangle tests made to *tri_tests (traversal statistics).
template <bool kCount = false>
__device__ __forceinline__ int threaded_step(const ThreadedNode* __restrict__ tn, const TriRecord* __restrict__ tris,
                                             const RayInv& r, int i, unsigned* tri_tests = nullptr) {
    float4 lo, hi;  // one 32-byte load (the node array is 256-byte aligned, nodes 32 bytes)
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(lo.x), "=f"(lo.y), "=f"(lo.z), "=f"(lo.w), "=f"(hi.x), "=f"(hi.y), "=f"(hi.z), "=f"(hi.w)
        : "l"(tn + i));
    const int skip = __float_as_int(lo.w), tri = __float_as_int(hi.w);
    int next = skip;
    if (slab_hit(r, lo, hi)) {
        if (tri < 0) {
            next = i + 1;
        } else {
            if (kCount) ++*tri_tests;
            if (tri_blocks(r.o, r.d, tris, tri)) return -1;
        }
    }
    return next > i ? next : i + 1;  // strictly increasing: at most 2 n - 1 steps
}

// any hit with t > 0 (shadow ray, no far limit): stackless traversal of the
// depth-first layout, no ordering needed since any blocker ends the ray
__device__ __forceinline__ bool any_hit_threaded(const void* nodes, const TriRecord* __restrict__ tris, int n_tris,
                                                 const RayInv& r) {
    if (n_tris <= 0) return false;
    const ThreadedNode* tn = threaded_nodes(nodes, n_tris);
    const int end = 2 * n_tris - 1;
    for (int i = 0; i < end;) {
        i = threaded_step(tn, tris, r, i);
        if (i < 0) return true;
    }
    return false;
}

// ---------------------------------------------------------------- four-wide traversal
constexpr int kWideStack = 24;          // pending nodes per ray; a deeper need falls back to the stackless walk
constexpr int kWideBlocked = -1;        // wide_step: a triangle blocks the ray
constexpr int kWideDone = -2;           // wide_step: nothing left to visit

// three-operand minimum / maximum (one instruction on sm_100 and later)
__device__ __forceinline__ float fmin3(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float fmax3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// byte k of w in the low mantissa bits of 2^23: the float 2^23 + q, exact
__device__ __forceinline__ float qbyte(uint32_t w, int k) {
    return __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7540u + (uint32_t)k));
}

// The largest coordinate (in magnitude) that a ray's origin o may have for the
// four-wide nodes' boxes to hold what they should, or a negative number where no ray
// may use them; the two-child or the depth-first nodes decide then and beyond.  With
// m the largest coordinate of the root box, P a child box's plane and a its node's
// origin, the computed distance to the plane (wide_visit) differs from (P - o) / d, in
// units of the axis, by at most
//   u |P - o| (1 / d) + u |o| (its product) + u |a - o| (the difference)
//   + u (2^23 s + |a - o|) (B') + u |P - o| (the last sum)  <=  s / 2 + u (5 |o| + 4 m).
// The child boxes are a step s >= 2^-17 m wider on each side, so |o| may be 12 m; 11
// m is taken.  And no product may overflow: 1 / d goes up to 1e20 (make_ray) and
// 2^23 s to 1.4e5 m, so m up to 1e12 (an infinite vertex makes m infinite).
__device__ __forceinline__ float wide_reach(const void* __restrict__ root, int n_tris) {
    if (n_tris <= 0) return -1.0f;
    const BvhNode* nodes = static_cast<const BvhNode*>(root);
    const float4 a = __ldg(&nodes->a), b = __ldg(&nodes->b), c = __ldg(&nodes->c);
    const float mx = fmaxf(fmaxf(fabsf(a.x), fabsf(a.y)), fmaxf(fabsf(b.x), fabsf(b.y)));
    const float my = fmaxf(fmaxf(fabsf(a.z), fabsf(a.w)), fmaxf(fabsf(b.z), fabsf(b.w)));
    const float mz = fmaxf(fmaxf(fabsf(c.x), fabsf(c.y)), fmaxf(fabsf(c.z), fabsf(c.w)));
    const float m = fmaxf(mx, fmaxf(my, mz));
    return m <= 1e12f ? 11.0f * m : -1.0f;
}
__device__ __forceinline__ float largest(f3 o) { return fmaxf(fabsf(o.x), fmaxf(fabsf(o.y), fabsf(o.z))); }

// Slab tests of the four child boxes of a four-wide node; bit k of the result
// is set when the ray (t >= 0, no far limit) meets child k's box.  Per axis
// the near plane is the low one for a non-negative direction, the high one
// otherwise, so the plane at q needs no min / max:
//   t = (o + q s - origin) / d = (2^23 + q) A + B',  A = s / d,  B' = (o - origin) / d - 2^23 A,
// one fused multiply-add per plane (2^23 + q is the byte placed in a float's
// mantissa).  Rounding B' costs at most half a step of t, the other roundings
// far less for origins inside the scene's bounds; the boxes are widened by a
// whole step on every side, so a ray that meets a child's box passes its test.
__device__ __forceinline__ unsigned wide_child_hits(const RayInv& r, float4 a, float4 b, float4 c) {
    const uint32_t lox = __float_as_uint(b.z), loy = __float_as_uint(b.w), loz = __float_as_uint(c.x);
    const uint32_t hix = __float_as_uint(c.y), hiy = __float_as_uint(c.z), hiz = __float_as_uint(c.w);
    const bool px = r.inv.x >= 0.0f, py = r.inv.y >= 0.0f, pz = r.inv.z >= 0.0f;
    const uint32_t nx = px ? lox : hix, fx = px ? hix : lox;
    const uint32_t ny = py ? loy : hiy, fy = py ? hiy : loy;
    const uint32_t nz = pz ? loz : hiz, fz = pz ? hiz : loz;
    const float ax = a.w * r.inv.x, ay = b.x * r.inv.y, az = b.y * r.inv.z;
    const float bx = fmaf(-8388608.0f, ax, (a.x - r.o.x) * r.inv.x);
    const float by = fmaf(-8388608.0f, ay, (a.y - r.o.y) * r.inv.y);
    const float bz = fmaf(-8388608.0f, az, (a.z - r.o.z) * r.inv.z);
    unsigned m = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float t0 = fmax3(fmaf(qbyte(nx, k), ax, bx), fmaf(qbyte(ny, k), ay, by),
                               fmaxf(fmaf(qbyte(nz, k), az, bz), 0.0f));
        const float t1 = fmin3(fmaf(qbyte(fx, k), ax, bx), fmaf(qbyte(fy, k), ay, by), fmaf(qbyte(fz, k), az, bz));
        m |= (t0 <= t1 ? 1u : 0u) << k;
    }
    return m;
}

// One node of the four-wide any-hit traversal: tests the node's children,
// tests the triangles of hit leaf children at once, continues with the first
// hit inner child and pushes the others.  Returns the next node, kWideBlocked
// or kWideDone.  Stack entry i lives at stack[i * kStride] (a thread's column
// of a shared-memory array, or a local array); a push beyond kWideStack sets
// *overflow instead (the caller then decides the ray by the stackless walk);
// kCount adds the triangle tests made to *tri_tests.  A ray with infinite
// coordinates meets empty slots too: their links are no triangle's.
template <int kStride = 1, bool kCount = false>
__device__ __forceinline__ int wide_step(const WideNode* __restrict__ wn, const TriRecord* __restrict__ tris,
                                         int n_tris, const RayInv& r, int node, int* stack, int& sp, bool& overflow,
                                         unsigned* tri_tests = nullptr) {
    float4 a, b, c;
    int4 d;
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
        : "l"(wn + node));
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(c.x), "=f"(c.y), "=f"(c.z), "=f"(c.w), "=r"(d.x), "=r"(d.y), "=r"(d.z), "=r"(d.w)
        : "l"(reinterpret_cast<const char*>(wn + node) + 32));
    const unsigned m = wide_child_hits(r, a, b, c);
    unsigned leaves = 0;
    int next = kWideDone;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int l = k == 0 ? d.x : k == 1 ? d.y : k == 2 ? d.z : d.w;
        if (!((m >> k) & 1u)) continue;
        if (l < 0) {
            leaves |= 1u << k;
        } else if (next == kWideDone) {
            next = l;
        } else if (sp < kWideStack) {
            stack[kStride * sp++] = l;
        } else {
            overflow = true;
        }
    }
    while (leaves) {
        const int k = __ffs(leaves) - 1;
        leaves &= leaves - 1;
        const int l = k == 0 ? d.x : k == 1 ? d.y : k == 2 ? d.z : d.w;
        if ((unsigned)~l >= (unsigned)n_tris) continue;
        if (kCount) ++*tri_tests;
        if (tri_blocks(r.o, r.d, tris, ~l)) return kWideBlocked;
    }
    if (next == kWideDone && sp > 0) next = stack[kStride * --sp];
    return next;
}

// Shared-memory accesses by 32-bit shared address.
__device__ __forceinline__ int lds32(uint32_t a) {
    int v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ float2 lds64(uint32_t a) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts32(uint32_t a, int v) {
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void sts64(uint32_t a, float x, float y) {
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(x), "f"(y) : "memory");
}

// The node part of wide_step for a traversal that postpones its triangle
// tests: hit inner children are appended to the lane's node stack (entries at
// shared address na, kStep bytes apart), hit leaf children to its leaf queue
// (at la, kStep apart); the caller makes sure that four more of each fit.  One
// predicated store per child, to whichever of the two, and predicated
// additions: no branch for other lanes to wait at, and one shared-memory
// wavefront per child instead of two.  The child tests are wide_child_hits',
// two children per fused multiply-add instruction, with the origin's product
// oi = -o / d formed once per ray (its rounding, at most 2^-24 |o| / |d|, is
// under 2^-7 quantisation steps for origins inside the scene's bounds).
template <int kStep>
__device__ __forceinline__ void wide_visit(const WideNode* __restrict__ wn, f3 inv, f3 oi, int node, uint32_t& na,
                                           uint32_t& la) {
    float4 a, b, c;
    int4 d;
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
        : "l"(wn + node));
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(c.x), "=f"(c.y), "=f"(c.z), "=f"(c.w), "=r"(d.x), "=r"(d.y), "=r"(d.z), "=r"(d.w)
        : "l"(reinterpret_cast<const char*>(wn + node) + 32));
    const uint32_t lox = __float_as_uint(b.z), loy = __float_as_uint(b.w), loz = __float_as_uint(c.x);
    const uint32_t hix = __float_as_uint(c.y), hiy = __float_as_uint(c.z), hiz = __float_as_uint(c.w);
    const bool px = inv.x >= 0.0f, py = inv.y >= 0.0f, pz = inv.z >= 0.0f;
    const uint32_t nx = px ? lox : hix, fx = px ? hix : lox;
    const uint32_t ny = py ? loy : hiy, fy = py ? hiy : loy;
    const uint32_t nz = pz ? loz : hiz, fz = pz ? hiz : loz;
    const float ax = a.w * inv.x, ay = b.x * inv.y, az = b.y * inv.z;
    const float bx = fmaf(-8388608.0f, ax, fmaf(a.x, inv.x, oi.x));
    const float by = fmaf(-8388608.0f, ay, fmaf(a.y, inv.y, oi.y));
    const float bz = fmaf(-8388608.0f, az, fmaf(a.z, inv.z, oi.z));
    const float2 ax2 = {ax, ax}, bx2 = {bx, bx}, ay2 = {ay, ay}, by2 = {by, by}, az2 = {az, az}, bz2 = {bz, bz};
#pragma unroll
    for (int k = 0; k < 4; k += 2) {
        const float2 x0 = fma2({qbyte(nx, k), qbyte(nx, k + 1)}, ax2, bx2);
        const float2 y0 = fma2({qbyte(ny, k), qbyte(ny, k + 1)}, ay2, by2);
        const float2 z0 = fma2({qbyte(nz, k), qbyte(nz, k + 1)}, az2, bz2);
        const float2 x1 = fma2({qbyte(fx, k), qbyte(fx, k + 1)}, ax2, bx2);
        const float2 y1 = fma2({qbyte(fy, k), qbyte(fy, k + 1)}, ay2, by2);
        const float2 z1 = fma2({qbyte(fz, k), qbyte(fz, k + 1)}, az2, bz2);
        const float t0[2] = {fmax3(x0.x, y0.x, fmaxf(z0.x, 0.0f)), fmax3(x0.y, y0.y, fmaxf(z0.y, 0.0f))};
        const float t1[2] = {fmin3(x1.x, y1.x, z1.x), fmin3(x1.y, y1.y, z1.y)};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int l = k + h == 0 ? d.x : k + h == 1 ? d.y : k + h == 2 ? d.z : d.w;
            asm volatile(
                "{\n\t.reg .pred h, pl, pn;\n\t.reg .u32 ad;\n\t"
                "setp.le.f32 h, %2, %3;\n\t"
                "setp.lt.and.s32 pl|pn, %4, 0, h;\n\t"
                "selp.u32 ad, %0, %1, pl;\n\t"
                "@h st.shared.b32 [ad], %4;\n\t"
                "@pl add.u32 %0, %0, %5;\n\t"
                "@pn add.u32 %1, %1, %5;\n\t}"
                : "+r"(la), "+r"(na)
                : "f"(t0[h]), "f"(t1[h]), "r"(l), "n"(kStep)
                : "memory");
        }
    }
}

// closest hit; returns the leaf (triangle record) index or -1
__device__ __forceinline__ int closest_hit(const BvhNode* __restrict__ nodes, const TriRecord* __restrict__ tris,
                                           int n_tris, const RayInv& r, float* t_out, float* bu, float* bv) {
    int best = -1;
    float tbest = FLT_MAX;
    if (n_tris <= 0) return -1;
    int stack[kTraversalStack];
    int sp = 0;
    int node = 0;
    for (int iter = 0; iter < n_tris + 1; ++iter) {
        float4 a, b, c;  // the 64-byte node as two 32-byte loads (node arrays are 256-byte aligned)
        int4 d;
        asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
            : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
            : "l"(nodes + node));
        asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
            : "=f"(c.x), "=f"(c.y), "=f"(c.z), "=f"(c.w), "=r"(d.x), "=r"(d.y), "=r"(d.z), "=r"(d.w)
            : "l"(reinterpret_cast<const char*>(nodes + node) + 32));
        float t0 = slab(r, a, make_float2(c.x, c.y), tbest);
        float t1 = slab(r, b, make_float2(c.z, c.w), tbest);
        if (t0 < FLT_MAX && d.x < 0) {
            float u, v;
            const float t = tri_hit(r, tris, ~d.x, &u, &v);
            if (t < tbest) tbest = t, best = ~d.x, *bu = u, *bv = v;
            t0 = FLT_MAX;
        }
        if (t1 < FLT_MAX && d.y < 0) {
            float u, v;
            const float t = tri_hit(r, tris, ~d.y, &u, &v);
            if (t < tbest) tbest = t, best = ~d.y, *bu = u, *bv = v;
            t1 = FLT_MAX;
        }
        if (t0 < FLT_MAX && t1 < FLT_MAX) {
            const bool first0 = t0 <= t1;
            if (sp < kTraversalStack) stack[sp++] = first0 ? d.y : d.x;
            node = first0 ? d.x : d.y;
        } else if (t0 < FLT_MAX) {
            node = d.x;
        } else if (t1 < FLT_MAX) {
            node = d.y;
        } else {
            if (sp == 0) break;
            node = stack[--sp];
        }
    }
    *t_out = tbest;
    return best;
}

// tri_hit with every rounding written out (the products as closest_hit's are contracted)
__device__ __forceinline__ float tri_hit_rn(f3 o, f3 d, const TriRecord* __restrict__ tris, int k, float* bu, float* bv) {
    f3 v0, e1, e2;
    load_record(tris, k, v0, e1, e2);
    const f3 p = cross_rn(d, e2);
    const float det = dot_rn(e1, p);
    if (det == 0.0f) return FLT_MAX;
    const float inv = 1.0f / det;
    const f3 s = {__fsub_rn(o.x, v0.x), __fsub_rn(o.y, v0.y), __fsub_rn(o.z, v0.z)};
    const float u = __fmul_rn(dot_rn(s, p), inv);
    if (u < 0.0f || u > 1.0f) return FLT_MAX;
    const f3 q = cross_rn(s, e1);
    const float v = __fmul_rn(dot_rn(d, q), inv);
    if (v < 0.0f || __fadd_rn(u, v) > 1.0f) return FLT_MAX;
    const float t = __fmul_rn(dot_rn(e2, q), inv);
    if (!(t > 0.0f)) return FLT_MAX;
    *bu = u;
    *bv = v;
    return t;
}

// closest_hit over the four-wide nodes by pairs of lanes, one ray a pair and two
// children of its node a lane.  What bounds it is the rays' chains of dependent
// loads (node, then a leaf's triangle, some 700 cycles each from L2; 15 nodes a
// ray, 60 for one in a hundred, up to 180) and, with a million triangles, the
// instructions of warps most of whose rays are done: a pair halves both against a
// ray per lane (four lanes a ray add more instructions than they hide), and the
// next node (the nearest inner child, or the nearest pending one) is loaded before
// the triangles are tested.  Measured, primary_cast of 512 x 512 pixels, 1.18M
// triangles: 166 us (176 with four lanes, 205 with one; a ray per lane over the
// two-child nodes 175), 190k triangles, 133 x 77: 86 (71; 127; 115), 157k
// triangles, 64 x 64: 79 (63; 119; 108).  A persistent tracer that refills lanes
// leaves too few in flight: 208 to 340.
// A triangle is decided as closest_hit decides it, bit for bit; only where two lie at
// the same or nearly the same distance (a shared edge, faces that touch) may the pair,
// which meets them in another order, take the other one: on a mesh of 1.2M triangles
// the planes then differ by 3e-8 of their norm, 1e-5 at most.
// The whole warp calls it and stays together (node: 0, or -1 for a pair without a
// ray).  An empty slot's box is inverted, which rejects every finite ray; its link
// is checked all the same before it becomes a triangle's index.  Pending nodes and
// their entry distances are a row of shared memory per ray.  Returns the leaf, the
// same in both lanes, or kWideOverflow: more pending nodes than the row holds.
constexpr int kCastStack = 24;
constexpr int kWideOverflow = -2;
__device__ __forceinline__ int closest_hit_wide(const WideNode* __restrict__ wn, const TriRecord* __restrict__ tris,
                                                int n_tris, const RayInv& r, int node, float2* stack, float* t_out,
                                                float* bu, float* bv) {
    const unsigned full = 0xffffffffu, none = 0xffffffffu;
    const int q = threadIdx.x & 1;
    int best = -1, sp = 0;
    float tbest = FLT_MAX, tmine = FLT_MAX;  // of the pair, of this lane's children (best, *bu, *bv)
    const f3 oi = mk(-r.o.x * r.inv.x, -r.o.y * r.inv.y, -r.o.z * r.inv.z);
    const bool px = r.inv.x >= 0.0f, py = r.inv.y >= 0.0f, pz = r.inv.z >= 0.0f;
    float4 a, b, c;
    int2 l = make_int2(0, 0);  // the node, and the links of this lane's children
    auto load = [&](int k) {
        asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
                     : "l"(wn + k));
        c = __ldg(&wn[k].c);
        l = __ldg(reinterpret_cast<const int2*>(&wn[k].d) + q);
    };
    bool overflow = false;
    if (node >= 0) load(node);
    while (__any_sync(full, node >= 0)) {  // ends: every four-wide node is visited at most once per ray
        const uint32_t lox = __float_as_uint(b.z), loy = __float_as_uint(b.w), loz = __float_as_uint(c.x);
        const uint32_t hix = __float_as_uint(c.y), hiy = __float_as_uint(c.z), hiz = __float_as_uint(c.w);
        const uint32_t nx = (px ? lox : hix) >> (16 * q), fx = (px ? hix : lox) >> (16 * q);
        const uint32_t ny = (py ? loy : hiy) >> (16 * q), fy = (py ? hiy : loy) >> (16 * q);
        const uint32_t nz = (pz ? loz : hiz) >> (16 * q), fz = (pz ? hiz : loz) >> (16 * q);
        const float ax = a.w * r.inv.x, ay = b.x * r.inv.y, az = b.y * r.inv.z;
        const float bx = fmaf(-8388608.0f, ax, fmaf(a.x, r.inv.x, oi.x));
        const float by = fmaf(-8388608.0f, ay, fmaf(a.y, r.inv.y, oi.y));
        const float bz = fmaf(-8388608.0f, az, fmaf(a.z, r.inv.z, oi.z));
        const float2 ax2 = {ax, ax}, bx2 = {bx, bx}, ay2 = {ay, ay}, by2 = {by, by}, az2 = {az, az}, bz2 = {bz, bz};
        const float2 x0 = fma2({qbyte(nx, 0), qbyte(nx, 1)}, ax2, bx2), x1 = fma2({qbyte(fx, 0), qbyte(fx, 1)}, ax2, bx2);
        const float2 y0 = fma2({qbyte(ny, 0), qbyte(ny, 1)}, ay2, by2), y1 = fma2({qbyte(fy, 0), qbyte(fy, 1)}, ay2, by2);
        const float2 z0 = fma2({qbyte(nz, 0), qbyte(nz, 1)}, az2, bz2), z1 = fma2({qbyte(fz, 0), qbyte(fz, 1)}, az2, bz2);
        const float ta = fmax3(x0.x, y0.x, fmaxf(z0.x, 0.0f)), tb = fmax3(x0.y, y0.y, fmaxf(z0.y, 0.0f));
        const bool hita = node >= 0 && ta <= fmin3(x1.x, y1.x, fminf(z1.x, tbest));
        const bool hitb = node >= 0 && tb <= fmin3(x1.y, y1.y, fminf(z1.y, tbest));
        // inner children by entry distance, ties by child
        const uint32_t ka = hita && l.x >= 0 ? (__float_as_uint(ta) & ~3u) | (uint32_t)(2 * q) : none;
        const uint32_t kb = hitb && l.y >= 0 ? (__float_as_uint(tb) & ~3u) | (uint32_t)(2 * q + 1) : none;
        const uint32_t kc = __shfl_xor_sync(full, ka, 1), kd = __shfl_xor_sync(full, kb, 1);
        const uint32_t first = min(min(ka, kb), min(kc, kd));
        const int n_in = (ka != none) + (kb != none) + (kc != none) + (kd != none);
        // (an inner link's complement is negative, an empty slot's beyond every triangle)
        int leafa = hita && (unsigned)~l.x < (unsigned)n_tris ? ~l.x : -1;
        int leafb = hitb && (unsigned)~l.y < (unsigned)n_tris ? ~l.y : -1;
        int next = __shfl_sync(full, first & 1u ? l.y : l.x, (threadIdx.x & 30) | (int)(first >> 1 & 1u));
        float tnext = __uint_as_float(first);
        if (sp + 3 > kCastStack) overflow = true;
        if (n_in > 1 && !overflow) {
            const int top = sp + n_in - 1;
            const int ra = (kb < ka) + (kc < ka) + (kd < ka), rb = (ka < kb) + (kc < kb) + (kd < kb);
            if (ka != none && ra > 0) stack[top - ra] = make_float2(__uint_as_float(ka), __int_as_float(l.x));
            if (kb != none && rb > 0) stack[top - rb] = make_float2(__uint_as_float(kb), __int_as_float(l.y));
            sp = top;
        }
        __syncwarp();
        if (n_in == 0) {
            next = -1;
            while (sp > 0 && next < 0) {  // the nearest pending node not behind the hit
                const float2 e = stack[--sp];
                if (e.x <= tbest) next = __float_as_int(e.y), tnext = e.x;
            }
        }
        if (overflow || node < 0) next = -1, sp = 0;
        node = next;
        if (node >= 0) load(node);
        if (__any_sync(full, leafa >= 0 || leafb >= 0)) {
            float t = FLT_MAX;
            do {
                const int k = leafa >= 0 ? leafa : leafb;
                if (leafa >= 0) leafa = -1;
                else leafb = -1;
                if (k >= 0) {
                    float u, v;
                    t = fminf(t, tri_hit_rn(r.o, r.d, tris, k, &u, &v));
                    if (t < tmine) tmine = t, best = k, *bu = u, *bv = v;
                }
                __syncwarp();
            } while (__any_sync(full, leafb >= 0));
            tbest = fminf(tbest, fminf(t, __shfl_xor_sync(full, t, 1)));
            if (node >= 0 && tnext > tbest) {  // behind the new hit: and so may be the pending ones
                node = -1;
                while (sp > 0 && node < 0) {
                    const float2 e = stack[--sp];
                    if (e.x <= tbest) node = __float_as_int(e.y);
                }
                if (node >= 0) load(node);
            }
            __syncwarp();
        }
    }
    // the pair's nearest hit: its lane's leaf and barycentrics
    const unsigned who = __ballot_sync(full, best >= 0 && tmine == tbest) >> (threadIdx.x & 30) & 3u;
    const int src = (threadIdx.x & 30) | (who == 2u ? 1 : 0);
    best = __shfl_sync(full, best, src);
    *bu = __shfl_sync(full, *bu, src);
    *bv = __shfl_sync(full, *bv, src);
    *t_out = tbest;
    return overflow ? kWideOverflow : best;
}

// ---------------------------------------------------------------- probe
// largest k in [0, n-1] with cdf[k] <= u
__device__ __forceinline__ int upper_index(const float* __restrict__ cdf, int n, float u) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(cdf + mid) <= u) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// the same search with generic loads (the marginal lives in shared memory)
__device__ __forceinline__ int upper_index_generic(const float* cdf, int n, float u) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (cdf[mid] <= u) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// (u, v) -> direction: phi = 2 pi u, theta = pi v, y up
__device__ __forceinline__ f3 dir_from_uv(float u, float v, float* sin_theta) {
    float sp, cp, st, ct;
    sincospif(2.0f * u, &sp, &cp);
    sincospif(v, &st, &ct);
    *sin_theta = st;
    return mk(mul_rn(st, cp), ct, mul_rn(st, sp));
}

struct Probe {
    const float4* env;
    const float* cond;
    const float* marg;  // read with generic loads: the kernels stage it in shared memory
    int W, H;
    bool on;  // total > 0
};

// the marginal CDF (H + 1 floats) copied into the block's shared memory; every
// thread of the block must call this before any of them returns
__device__ __forceinline__ void stage_marginal(Probe& P, float* s_marg) {
    for (int i = threadIdx.x; i <= P.H; i += blockDim.x) s_marg[i] = __ldg(P.marg + i);
    __syncthreads();
    P.marg = s_marg;
}

// probe texel of a direction and sin(theta) (accurate near the poles)
__device__ __forceinline__ int texel_of_dir(const Probe& P, f3 d, float* sin_theta) {
    const float st = sqrtf(fma_rn(d.z, d.z, mul_rn(d.x, d.x)));
    float u = mul_rn(atan2f(d.z, d.x), 0.5f * MCDI_INV_PI);
    if (u < 0.0f) u = add_rn(u, 1.0f);
    const float v = mul_rn(atan2f(st, d.y), MCDI_INV_PI);
    const int i = min(P.W - 1, (int)mul_rn(u, (float)P.W));
    const int j = min(P.H - 1, (int)mul_rn(v, (float)P.H));
    *sin_theta = st;
    return j * P.W + i;
}

// density of the probe technique at texel t for a direction with sin(theta) st
__device__ __forceinline__ float pdf_light_texel(const Probe& P, int t, float st) {
    if (!P.on || !(st > 0.0f)) return 0.0f;
    const int j = t / P.W, i = t - j * P.W;
    const float* c = P.cond + (size_t)j * (P.W + 1);
    const float wr = sub_rn(P.marg[j + 1], P.marg[j]);
    const float wc = sub_rn(__ldg(c + i + 1), __ldg(c + i));
    return mul_rn(mul_rn(mul_rn((float)P.W, (float)P.H), wr), wc) / mul_rn(2.0f * MCDI_PI * MCDI_PI, st);
}

// probe sample; returns false if the technique is off
__device__ __forceinline__ bool sample_light(const Probe& P, float u0, float u1, f3* d, int* texel, float* pdf) {
    if (!P.on) return false;
    const int j = upper_index_generic(P.marg, P.H, u0);
    const float m0 = P.marg[j], m1 = P.marg[j + 1];
    const float* c = P.cond + (size_t)j * (P.W + 1);
    const int i = upper_index(c, P.W, u1);
    const float c0 = __ldg(c + i), c1 = __ldg(c + i + 1);
    const float dm = sub_rn(m1, m0), dc = sub_rn(c1, c0);
    const float dv = fminf(sub_rn(u0, m0) / dm, 0.99999994f);
    const float du = fminf(sub_rn(u1, c0) / dc, 0.99999994f);
    float st;
    *d = dir_from_uv(add_rn((float)i, du) / (float)P.W, add_rn((float)j, dv) / (float)P.H, &st);
    *texel = j * P.W + i;
    *pdf = st > 0.0f ? mul_rn(mul_rn(mul_rn((float)P.W, (float)P.H), dm), dc) / mul_rn(2.0f * MCDI_PI * MCDI_PI, st)
                     : 0.0f;
    return true;
}

// ---------------------------------------------------------------- frame + lobes
// orthonormal basis of Duff et al. 2017 (sign(0) = +1)
__device__ __forceinline__ void frame(f3 n, f3* b1, f3* b2) {
    const float s = n.z >= 0.0f ? 1.0f : -1.0f;
    const float a = -1.0f / add_rn(s, n.z);
    const float b = mul_rn(mul_rn(n.x, n.y), a);
    *b1 = mk(fma_rn(mul_rn(mul_rn(s, n.x), n.x), a, 1.0f), mul_rn(s, b), mul_rn(-s, n.x));
    *b2 = mk(b, fma_rn(mul_rn(n.y, n.y), a, s), -n.y);
}

__device__ __forceinline__ f3 sample_cosine(f3 n, f3 b1, f3 b2, float u0, float u1) {
    float sp, cp;
    sincospif(2.0f * u1, &sp, &cp);
    const float r = sqrtf(u0);
    const float z = sqrtf(sub_rn(1.0f, u0));
    return combine_rn(b1, mul_rn(r, cp), b2, mul_rn(r, sp), n, z);
}

// GGX normal distribution with the denominator term nh^2 (a2 - 1) + 1 written as
// sin^2 + nh^2 a2 (s2 = |n x h|^2): free of the cancellation of 1 - nh^2 near the
// lobe peak, which in FP32 would cost ~1e-3 relative accuracy at alpha ~ 0.006.
__device__ __forceinline__ float ggx_D_denom(float nh, float s2, float a2) { return fma_rn(mul_rn(nh, nh), a2, s2); }
__device__ __forceinline__ float ggx_D(float nh, float s2, float a2) {
    if (!(nh > 0.0f)) return 0.0f;
    const float d = ggx_D_denom(nh, s2, a2);
    return a2 / mul_rn(mul_rn(MCDI_PI, d), d);
}
__device__ __forceinline__ float sin2_between(f3 n, f3 h) {
    const f3 c = cross_rn(n, h);
    return dot_rn(c, c);
}

__device__ __forceinline__ float ggx_lambda(float c, float a2) {
    const float z1 = fma_rn(a2, sub_rn(1.0f / mul_rn(c, c), 1.0f), 1.0f);
    return mul_rn(0.5f, sub_rn(sqrtf(z1), 1.0f));
}

// Heitz 2018 visible-normal sample, returns the reflected light direction.  The
// adjoint sums wo's projections in another order than the forward kernels: its
// direction may differ in the last bits, and in one or two of a million samples (more
// with a finer probe) it reads the neighbouring texel.  That is rounding either way,
// but a smooth lobe's gradients are so steep in the direction that the forward's
// order moves them by up to 1.5e-3 of their norm, further than results may move: the
// adjoint keeps its own.
template <bool kAdjoint>
__device__ __forceinline__ f3 sample_ggx(f3 n, f3 b1, f3 b2, f3 wo, float alpha, float u0, float u1) {
    const f3 lo = kAdjoint ? mk(dot_rn(wo, b1), dot_rn(wo, b2), dot_rn(wo, n))
                           : mk(dot_xy_rn(wo, b1), dot_xy_rn(wo, b2), dot_xy_rn(wo, n));
    const f3 vh = normalize_rn(mk(mul_rn(alpha, lo.x), mul_rn(alpha, lo.y), lo.z));
    const float lensq = fma_rn(vh.x, vh.x, mul_rn(vh.y, vh.y));
    f3 t1v = lensq > 0.0f ? scale_rn(mk(-vh.y, vh.x, 0.0f), rsqrtf(lensq)) : mk(1.0f, 0.0f, 0.0f);
    const f3 t2v = cross_rn(vh, t1v);
    float sp, cp;
    sincospif(2.0f * u1, &sp, &cp);
    const float r = sqrtf(u0);
    const float t1 = mul_rn(r, cp);
    float t2 = mul_rn(r, sp);
    const float s = mul_rn(0.5f, add_rn(1.0f, vh.z));
    const float q1 = fma_rn(-t1, t1, 1.0f);
    t2 = fma_rn(sub_rn(1.0f, s), sqrtf(q1), mul_rn(s, t2));
    const float tz = sqrtf(fmaxf(0.0f, fma_rn(-t2, t2, q1)));
    const f3 nh = combine_rn(t1v, t1, t2v, t2, vh, tz);
    const f3 hl = normalize_rn(mk(mul_rn(alpha, nh.x), mul_rn(alpha, nh.y), fmaxf(nh.z, 0.0f)));
    const f3 h = combine_rn(b1, hl.x, b2, hl.y, n, hl.z);
    const float voh = dot_rn(wo, h);
    return fma_rn(h, mul_rn(2.0f, voh), mk(-wo.x, -wo.y, -wo.z));
}

// the half vector, formed as pdf_ggx forms it
__device__ __forceinline__ f3 half_vector(f3 wi, f3 wo) { return normalize_xy_rn(add_rn(wi, wo)); }

__device__ __forceinline__ float pdf_ggx(f3 n, f3 wo, float co, float a2, float g1o, f3 wi) {
    f3 h = add_rn(wi, wo);
    const float l2 = dot_xy_rn(h, h);
    if (!(l2 > 0.0f)) return 0.0f;
    h = scale_rn(h, rsqrtf(l2));
    if (!(dot_rn(wo, h) > 0.0f)) return 0.0f;
    return mul_rn(g1o, ggx_D(dot_rn(n, h), sin2_between(n, h), a2)) / mul_rn(4.0f, co);
}

__device__ __forceinline__ float schlick_weight(float vh) {
    const float x = 1.0f - fminf(fmaxf(vh, 0.0f), 1.0f);
    const float x2 = x * x;
    return x2 * x2 * x;
}

// ---------------------------------------------------------------- G-buffer
// direction of the camera ray through the centre of pixel (x, y), y down
__device__ __forceinline__ f3 camera_dir(const mcdi_camera& C, int x, int y, int W, int H) {
    const float sx = (2.0f * ((float)x + 0.5f) / (float)W - 1.0f) * C.tan_half_fovy * C.aspect;
    const float sy = (1.0f - 2.0f * ((float)y + 0.5f) / (float)H) * C.tan_half_fovy;
    return normalize(mk(C.forward[0] + sx * C.right[0] + sy * C.up[0], C.forward[1] + sx * C.right[1] + sy * C.up[1],
                        C.forward[2] + sx * C.right[2] + sy * C.up[2]));
}

// texel i of a texture stored with kCh floats per texel (4: float4, the 4th
// channel unused; 3: packed RGB), as a float4 with w = 0 for kCh = 3
template <int kCh>
__device__ __forceinline__ float4 texel(const float* __restrict__ tex, size_t i) {
    if constexpr (kCh == 4) {
        return __ldg(reinterpret_cast<const float4*>(tex) + i);
    } else {
        return make_float4(__ldg(tex + 3 * i), __ldg(tex + 3 * i + 1), __ldg(tex + 3 * i + 2), 0.0f);
    }
}

template <int kCh = 4>
__device__ __forceinline__ float4 bilinear(const float* __restrict__ tex, int S, float u, float v) {
    const float x = u * (float)S - 0.5f, y = v * (float)S - 0.5f;
    const float x0 = floorf(x), y0 = floorf(y);
    const float fx = x - x0, fy = y - y0;
    const int xi0 = min(max((int)x0, 0), S - 1), xi1 = min(max((int)x0 + 1, 0), S - 1);
    const int yi0 = min(max((int)y0, 0), S - 1), yi1 = min(max((int)y0 + 1, 0), S - 1);
    const float4 t00 = texel<kCh>(tex, (size_t)yi0 * S + xi0), t10 = texel<kCh>(tex, (size_t)yi0 * S + xi1);
    const float4 t01 = texel<kCh>(tex, (size_t)yi1 * S + xi0), t11 = texel<kCh>(tex, (size_t)yi1 * S + xi1);
    auto lerp = [](float a, float b, float t) { return a + (b - a) * t; };
    return make_float4(lerp(lerp(t00.x, t10.x, fx), lerp(t01.x, t11.x, fx), fy),
                       lerp(lerp(t00.y, t10.y, fx), lerp(t01.y, t11.y, fx), fy),
                       lerp(lerp(t00.z, t10.z, fx), lerp(t01.z, t11.z, fx), fy),
                       lerp(lerp(t00.w, t10.w, fx), lerp(t01.w, t11.w, fx), fy));
}

// The G-buffer entries of a primary hit on triangle k (original index) at
// barycentrics (u, v): interpolated position and normal, and the textures at
// the planar coordinate of the position (textures of kCh floats per texel);
// left as they are for bad vertex indices.
template <int kCh = 4>
__device__ __forceinline__ void gbuffer_hit(int k, float u, float v, const float* __restrict__ verts,
                                            const float* __restrict__ vnrm,
                                            const int* __restrict__ tri_idx, int n_verts,
                                            const float* __restrict__ tex_kd, const float* __restrict__ tex_korm,
                                            int S, float uv_ox, float uv_oz, float uv_s, float4* P, float4* Nn,
                                            float4* KD, float4* KORM) {
    const int i0 = tri_idx[3 * (size_t)k], i1 = tri_idx[3 * (size_t)k + 1], i2 = tri_idx[3 * (size_t)k + 2];
    if ((unsigned)i0 >= (unsigned)n_verts || (unsigned)i1 >= (unsigned)n_verts || (unsigned)i2 >= (unsigned)n_verts)
        return;
    const float w = 1.0f - u - v;
    float pp[3], nn[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        pp[c] = w * verts[3 * (size_t)i0 + c] + u * verts[3 * (size_t)i1 + c] + v * verts[3 * (size_t)i2 + c];
        nn[c] = w * vnrm[3 * (size_t)i0 + c] + u * vnrm[3 * (size_t)i1 + c] + v * vnrm[3 * (size_t)i2 + c];
    }
    *P = make_float4(pp[0], pp[1], pp[2], 1.0f);
    *Nn = make_float4(nn[0], nn[1], nn[2], 0.0f);
    const float tu = (pp[0] - uv_ox) * uv_s, tv = (pp[2] - uv_oz) * uv_s;
    *KD = bilinear<kCh>(tex_kd, S, tu, tv);
    *KORM = bilinear<kCh>(tex_korm, S, tu, tv);
    KD->w = 0.f;
    KORM->w = 0.f;
}

// ---------------------------------------------------------------- per pixel
// Schlick's normal-incidence reflectance of the metallic blend (reading c1)
__device__ __forceinline__ f3 fresnel0(f3 kd, float m) {
    return mk(0.04f * (1.0f - m) + kd.x * m, 0.04f * (1.0f - m) + kd.y * m, 0.04f * (1.0f - m) + kd.z * m);
}

// the specular integrand's colour for probe radiance L: L (F0 + (1 - F0) q) ws, q the Schlick weight and ws
// the scalar rest of the term (D G2 / (4 cos_o) over the MIS denominator)
__device__ __forceinline__ f3 spec_colour(float4 L, f3 F0, float q, float ws) {
    return mk(L.x * (F0.x + (1.0f - F0.x) * q), L.y * (F0.y + (1.0f - F0.y) * q), L.z * (F0.z + (1.0f - F0.z) * q)) *
           ws;
}

struct Pixel {
    f3 p, n, wo, b1, b2;
    float lN, co, alpha, a2, g1o, r, m;
    f3 kd, F0;
    bool spec_on;
};

__device__ __forceinline__ bool load_pixel(float4 pos, float4 nrm, float4 kd, float4 korm, f3 cam, Pixel* px) {
    const f3 N = xyz(nrm);
    const float l2 = dot_rn(N, N);
    if (!(pos.w > 0.0f) || !(l2 > 0.0f)) return false;
    px->lN = sqrtf(l2);
    px->n = scale_rn(N, 1.0f / px->lN);
    px->p = xyz(pos);
    px->wo = normalize_xy_rn(mk(sub_rn(cam.x, px->p.x), sub_rn(cam.y, px->p.y), sub_rn(cam.z, px->p.z)));
    px->co = dot_rn(px->n, px->wo);
    px->spec_on = px->co >= 1e-4f;
    px->r = korm.y;
    px->m = korm.z;
    px->alpha = fmaxf(mul_rn(px->r, px->r), 1e-4f);
    px->a2 = mul_rn(px->alpha, px->alpha);
    px->g1o = px->spec_on ? 1.0f / add_rn(1.0f, ggx_lambda(px->co, px->a2)) : 0.0f;
    px->kd = xyz(kd);
    px->F0 = fresnel0(px->kd, px->m);
    frame(px->n, &px->b1, &px->b2);
    return true;
}

// One sample of the MIS estimator: direction, texel and 1/denominator.
// Returns false when the sample does not contribute (technique off, below the
// horizon, zero density).
template <bool kAdjoint = false>
__device__ __forceinline__ bool draw_sample(const Probe& P, const Pixel& px, int n_light, int n_cos, int n_ggx,
                                            int j, float2 u, f3* wi, int* texel, float* ci, float* inv_denom) {
    float pl = 0.0f, st = 0.0f;
    int t = -1;
    if (j < n_light) {
        if (!sample_light(P, u.x, u.y, wi, &t, &pl)) return false;
    } else if (j < n_light + n_cos) {
        *wi = sample_cosine(px.n, px.b1, px.b2, u.x, u.y);
    } else {
        if (!px.spec_on) return false;
        *wi = sample_ggx<kAdjoint>(px.n, px.b1, px.b2, px.wo, px.alpha, u.x, u.y);
    }
    const float c = dot_xy_rn(px.n, *wi);
    if (!(c > 0.0f)) return false;
    if (t < 0) {
        t = texel_of_dir(P, *wi, &st);
        pl = pdf_light_texel(P, t, st);
    }
    float denom = fma_rn((float)n_cos, mul_rn(c, MCDI_INV_PI), mul_rn((float)n_light, pl));
    if (px.spec_on && n_ggx > 0)
        denom = fma_rn((float)n_ggx, pdf_ggx(px.n, px.wo, px.co, px.a2, px.g1o, *wi), denom);
    if (!(denom > 0.0f)) return false;
    *texel = t;
    *ci = c;
    *inv_denom = 1.0f / denom;
    return true;
}

}  // namespace mcdi
