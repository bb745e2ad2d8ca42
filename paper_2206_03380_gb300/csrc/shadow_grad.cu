// Shadow-visibility gradients (the ablation of the paper's appendix
// "Visibility gradients from shadows"; Sec. 3.1 "Shadow gradients"): the
// boundary term of the blocked set of each pixel's shadow rays, estimated by
// edge sampling, scattered to the mesh's vertex positions.
//
// With H = 1 - tau B (B: the shadow ray from o = p + eps n is blocked), the
// pixel's integral of g(w) H(w) moves with the mesh only through the boundary
// of the blocked set, made of silhouette edges seen from o.  For an edge (a, b)
// and x(s) = a + s (b - a), w = (x - o) / r:
//   d/d(a, b) = -tau int_0^1 g(w) V+(s) n_out ((1 - s), s) |w x (b - a)| / r^2 ds,
// n_out the unit normal of the plane (o, a, b) away from the edge's faces and
// V+ whether the ray just outside the edge (w + eta n_out) reaches the probe.
// g is the forward integrand weighted by the upstream gradients of c_d, c_s.
// Each pixel draws M edges uniformly (e = floor(u0 E) in integer arithmetic)
// and s = u1; a sample weighs E / M.
//
// The edge table lists each undirected edge once, in the order of its first
// half-edge h = 3 t + i, as (a, b, c1, c2): the owner half-edge's endpoints,
// the opposite vertex of its face and that of the next face on the edge (-1
// on a boundary).  It is built with a hash table (first and second half-edge
// of each key by atomicMin), then an ordered compaction.
#include <limits.h>

#include <algorithm>

#include "common.cuh"
#include "internal.h"
#include "shading.cuh"
#include "trace.cuh"

namespace mcdi {
namespace {

constexpr unsigned long long kEmptyKey = ~0ull;
constexpr int kEdgeThreads = 256;
constexpr int kEdgeItems = 8;  // half-edges per thread in the ordered compaction
constexpr int kEdgeTile = kEdgeThreads * kEdgeItems;
constexpr int kGradThreads = 128;

__device__ __forceinline__ unsigned long long edge_key(int a, int b) {
    const unsigned lo = (unsigned)min(a, b), hi = (unsigned)max(a, b);
    return ((unsigned long long)lo << 32) | hi;
}

// 64-bit finaliser of MurmurHash3 (Appleby), spreading keys over the table
__device__ __forceinline__ unsigned long long mix64(unsigned long long k) {
    k ^= k >> 33;
    k *= 0xff51afd7ed558ccdull;
    k ^= k >> 33;
    k *= 0xc4ceb9fe1a85ec53ull;
    k ^= k >> 33;
    return k;
}

__device__ __forceinline__ int tri_vertex(const int* __restrict__ tris, int h, int step) {
    const int t = h / 3, i = h - 3 * t;
    return __ldg(tris + 3 * t + (i + step) % 3);
}

__global__ void __launch_bounds__(kEdgeThreads) edge_clear_kernel(unsigned long long* keys, int* first, int* second,
                                                                  long long cap) {
    pdl_prologue();
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < cap; k += (long long)gridDim.x * blockDim.x) {
        keys[k] = kEmptyKey;
        first[k] = INT_MAX;
        second[k] = INT_MAX;
    }
}

// insert every half-edge's key (linear probing, at most `cap` probes) and keep
// the smallest half-edge index per key
__global__ void __launch_bounds__(kEdgeThreads) edge_insert_kernel(const int* __restrict__ tris, int n_half,
                                                                   unsigned long long* keys, int* first, int* slot_of,
                                                                   long long cap, unsigned* err) {
    pdl_prologue();
    const int h = blockIdx.x * blockDim.x + threadIdx.x;
    if (h >= n_half) return;
    const unsigned long long key = edge_key(tri_vertex(tris, h, 0), tri_vertex(tris, h, 1));
    long long slot = (long long)(mix64(key) & (unsigned long long)(cap - 1));
    for (long long probe = 0; probe < cap; ++probe) {
        const unsigned long long old = atomicCAS(keys + slot, kEmptyKey, key);
        if (old == kEmptyKey || old == key) {
            atomicMin(first + slot, h);
            slot_of[h] = (int)slot;
            return;
        }
        slot = (slot + 1) & (cap - 1);
    }
    slot_of[h] = -1;
    atomicOr(err, 1u);
}

// the smallest half-edge index after the first, per key
__global__ void __launch_bounds__(kEdgeThreads) edge_second_kernel(int n_half, const int* __restrict__ slot_of,
                                                                   const int* __restrict__ first, int* second) {
    pdl_prologue();
    const int h = blockIdx.x * blockDim.x + threadIdx.x;
    if (h >= n_half) return;
    const int s = slot_of[h];
    if (s >= 0 && first[s] != h) atomicMin(second + s, h);
}

__device__ __forceinline__ bool owns_edge(const int* __restrict__ slot_of, const int* __restrict__ first, int h) {
    const int s = slot_of[h];
    return s >= 0 && first[s] == h;
}

// edges owned by each tile of kEdgeTile half-edges
__global__ void __launch_bounds__(kEdgeThreads) edge_count_kernel(int n_half, const int* __restrict__ slot_of,
                                                                  const int* __restrict__ first, int* tile_count) {
    pdl_prologue();
    __shared__ int s_warp[kEdgeThreads / 32];
    const int base = blockIdx.x * kEdgeTile + threadIdx.x * kEdgeItems;
    int c = 0;
#pragma unroll
    for (int k = 0; k < kEdgeItems; ++k) c += (base + k < n_half && owns_edge(slot_of, first, base + k)) ? 1 : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < kEdgeThreads / 32; ++w) t += s_warp[w];
        tile_count[blockIdx.x] = t;
    }
}

// exclusive scan of the tile counts (one block); the total is the edge count,
// or -1 if a key found no slot
__global__ void __launch_bounds__(1024) edge_offsets_kernel(int n_tiles, const int* __restrict__ tile_count,
                                                            int* tile_off, int* n_edges, const unsigned* err) {
    pdl_prologue();
    __shared__ int s_warp[32];
    __shared__ int s_carry;
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int base = 0; base < n_tiles; base += 1024) {
        const int i = base + threadIdx.x;
        const int v = i < n_tiles ? tile_count[i] : 0;
        int x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_warp[warp] = x;
        __syncthreads();
        if (warp == 0) {
            int w = s_warp[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += y;
            }
            s_warp[lane] = w;
        }
        __syncthreads();
        const int incl = x + (warp > 0 ? s_warp[warp - 1] : 0);
        if (i < n_tiles) tile_off[i] = s_carry + incl - v;
        __syncthreads();
        if (threadIdx.x == 1023) s_carry += incl;
        __syncthreads();
    }
    if (threadIdx.x == 0) *n_edges = *err ? -1 : s_carry;
}

// write each owned edge at its rank in half-edge order
__global__ void __launch_bounds__(kEdgeThreads) edge_write_kernel(const int* __restrict__ tris, int n_half,
                                                                  const int* __restrict__ slot_of,
                                                                  const int* __restrict__ first,
                                                                  const int* __restrict__ second,
                                                                  const int* __restrict__ tile_off, int4* edges) {
    pdl_prologue();
    __shared__ int s_warp[kEdgeThreads / 32];
    const int base = blockIdx.x * kEdgeTile + threadIdx.x * kEdgeItems;
    unsigned own = 0;
#pragma unroll
    for (int k = 0; k < kEdgeItems; ++k)
        if (base + k < n_half && owns_edge(slot_of, first, base + k)) own |= 1u << k;
    const int c = __popc(own), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    int before = 0;
    for (int w = 0; w < warp; ++w) before += s_warp[w];
    int rank = tile_off[blockIdx.x] + before + x - c;
    for (; own; own &= own - 1u) {
        const int h = base + __ffs(own) - 1;
        const int s2 = second[slot_of[h]];
        edges[rank++] = make_int4(tri_vertex(tris, h, 0), tri_vertex(tris, h, 1), tri_vertex(tris, h, 2),
                                  s2 == INT_MAX ? -1 : tri_vertex(tris, s2, 2));
    }
}

// vertex i: an 8-byte load of its aligned pair and one of the third component
// (the edge samples' random gathers cost one L1 wavefront per lane and load);
// `pairs`: whether the array is 8-byte aligned, the same for the whole grid
__device__ __forceinline__ f3 load_vert(const float* __restrict__ v, int i, bool pairs) {
    const float* p = v + 3 * (size_t)i;
    if (!pairs) return mk(__ldg(p), __ldg(p + 1), __ldg(p + 2));
    const int odd = i & 1;
    const float2 q = __ldg(reinterpret_cast<const float2*>(p + odd));
    const float t = __ldg(p + (odd ? 0 : 2));
    return odd ? mk(t, q.x, q.y) : mk(q.x, q.y, t);
}

__device__ __forceinline__ void scatter3(float* g, int i, f3 d) {
    atomicAdd(g + 3 * (size_t)i, d.x);
    atomicAdd(g + 3 * (size_t)i + 1, d.y);
    atomicAdd(g + 3 * (size_t)i + 2, d.z);
}

// The outer rays of a CTA's candidate samples, in shared memory, traced by
// trace_rays.  They graze surfaces and visit many nodes, so a list too short to
// keep the CTA's 128 lanes busy is traced in up to 16 parts per ray, by as many
// lanes, that start at the nodes two levels below the root (a node with a leaf
// or empty child stands for itself).  Parts find a hit twice and visit what a
// ray's end would have spared: lists of up to 32 rays are split.  Measured
// (grad kernel, no lists split / up to 32 / all): 171 / 160 / 166 us with 4
// candidates per 2048 samples, 339 / 319 / 431 us with 100.
struct OuterRays {
    static constexpr int kParts = 16;
    static constexpr unsigned kSplit = 32;  // the longest list whose rays are traced in parts
    static constexpr int kCap = 256;
    float4 dir[kCap];     // w: the sample (offset in the CTA's run, int bits)
    float4 origin[kCap];
    unsigned hit[kCap / 32];
    int part[kParts];  // start nodes, kWideDone beyond the last
    unsigned n, head;
    TraceStacks stacks;

    __device__ __forceinline__ void find_parts(const void* nodes, int n_tris) {  // one thread
        int list[kParts];
        int k = 1;
        list[0] = 0;
        if (n_tris > 0) {
            const WideNode* wn = wide_nodes(nodes, n_tris);
            for (int level = 0; level < 2; ++level) {
                int next[kParts], m = 0;
                for (int i = 0; i < k; ++i) {
                    const int4 d = __ldg(&wn[list[i]].d);
                    if (d.x < 0 || d.y < 0 || d.z < 0 || d.w < 0) {
                        next[m++] = list[i];
                    } else {
                        next[m] = d.x, next[m + 1] = d.y, next[m + 2] = d.z, next[m + 3] = d.w;
                        m += 4;
                    }
                }
                k = m;
                for (int i = 0; i < k; ++i) list[i] = next[i];
            }
        }
        for (int i = 0; i < kParts; ++i) part[i] = i < k ? list[i] : kWideDone;
    }
    __device__ __forceinline__ unsigned pending() const { return *(volatile const unsigned*)&n; }
    // parts a ray is traced in: while a round's rays in parts would be few per lane
    __device__ __forceinline__ int parts() const { return pending() <= kSplit ? kParts : 1; }
    __device__ __forceinline__ unsigned count() const { return pending() * parts(); }
    __device__ __forceinline__ unsigned take(unsigned k) { return atomicAdd(&head, k); }
    __device__ __forceinline__ void load(int id, f3& o, f3& d) const {
        o = xyz(origin[id]);
        d = xyz(dir[id]);
    }
    __device__ __forceinline__ int start(unsigned i, int, f3& o, f3& d, int& node) const {
        const bool split = pending() <= kSplit;
        const int id = (int)(split ? i / kParts : i);
        load(id, o, d);
        const unsigned done = ((volatile const unsigned*)hit)[id >> 5] >> (id & 31);  // by another part
        node = done & 1u ? kWideDone : split ? part[i % kParts] : 0;
        return id;
    }
    __device__ __forceinline__ void blocked(int id) { atomicOr(&hit[id >> 5], 1u << (id & 31)); }
};

// What an edge sample is up to its outer ray.
struct EdgeSample {
    int4 ed;
    f3 o, w, nout, ab;
    float s, r2, ci;
};

// Sample j of a pixel (position and normal only; the shading setup waits for
// the few samples whose outer ray is open): false unless its edge is a
// silhouette seen from the pixel, above the horizon.
__device__ __forceinline__ bool draw_edge_sample(const ShadeArgs& a, const float* __restrict__ verts, int n_verts,
                                                 const int4* __restrict__ edges, int E, long long idx, int view,
                                                 uint32_t pix, int j, EdgeSample* S) {
    const float4 pos = a.gb_pos[idx];
    const f3 N = xyz(a.gb_nrm[idx]);
    const float l2 = dot(N, N);
    if (!(pos.w > 0.0f) || !(l2 > 0.0f) || E <= 0) return false;
    const f3 nrm = N * (1.0f / sqrtf(l2));  // as load_pixel forms it
    const uint4 x = philox4x32_10(make_uint4(pix, (uint32_t)view, (uint32_t)j, a.stream_word),
                                  make_uint2((uint32_t)(a.seed & 0xffffffffull), (uint32_t)(a.seed >> 32)));
    const int e = (int)(((unsigned long long)(x.x >> 8) * (unsigned)E) >> 24);
    S->s = (float)(x.y >> 8) * 5.9604644775390625e-8f;
    const int4 ed = __ldg(edges + e);
    S->ed = ed;
    if ((unsigned)ed.x >= (unsigned)n_verts || (unsigned)ed.y >= (unsigned)n_verts ||
        (unsigned)ed.z >= (unsigned)n_verts || ed.w >= n_verts)
        return false;
    const f3 o = xyz(pos) + nrm * a.ray_eps;
    const bool pairs = ((size_t)verts & 7) == 0;
    const f3 va = load_vert(verts, ed.x, pairs), vb = load_vert(verts, ed.y, pairs);
    // the horizon first: it needs two of the four vertices
    S->ab = vb - va;
    const f3 d = va + S->ab * S->s - o;
    S->r2 = dot(d, d);
    S->w = d * (1.0f / sqrtf(S->r2));
    S->ci = dot(nrm, S->w);
    if (!(S->ci > 0.0f)) return false;
    const f3 m = cross(va - o, vb - o);
    const float lm = sqrtf(dot(m, m));
    if (!(lm > 0.0f)) return false;
    const f3 vc = load_vert(verts, ed.z, pairs);
    const float s1 = dot(m, vc - o);
    const float s2 = ed.w >= 0 ? dot(m, load_vert(verts, ed.w, pairs) - o) : s1;
    if (!(s1 * s2 > 0.0f)) return false;  // both faces on one side of the plane (o, a, b): silhouette
    S->nout = m * ((s1 > 0.0f ? -1.0f : 1.0f) / lm);
    S->o = o;
    return true;
}

// A CTA owns a run of rounds * kGradThreads (pixel, edge sample) pairs.  Its
// threads draw them, a round of one each at a time; the few that are candidates
// (silhouette, above the horizon: 0.2% of the samples of the mesh below) append
// their outer ray in shared memory, and when a round might overflow the list,
// or after the last, all lanes trace the list (trace_rays) and the samples whose
// ray is open are drawn again and scattered.  What bounds it is the latency of
// the samples' gathers (60%), then of the grazing outer rays' node chains.  Runs
// are as long as 32 rounds where that still gives each SM its 7 CTAs (their ends
// are then few), down to one round where the samples are few: of 300 x 400 x 9
// samples in 8 rounds 82 us, of 200 x 150 x 2 in one 61 (the whole warp walking
// one outer ray at a time over the depth-first nodes, a sample per thread: 153
// and 91).  Measured, 4.2M samples (512 x 512, 16 each) of 297k edges: 157 us
// (243).
constexpr int kMaxRounds = 32, kGradBlocksPerSM = 7;

__global__ void __launch_bounds__(kGradThreads) shadow_edge_grad_kernel(
    ShadeArgs a, const float* __restrict__ verts, int n_verts, const int4* __restrict__ edges,
    const int* __restrict__ n_edges_dev, int max_edges, int M, float eta, const float4* __restrict__ g_cd,
    const float4* __restrict__ g_cs, float* g_verts, float* sample_w, int rounds) {
    pdl_prologue();
    __shared__ OuterRays rays;
    const long long P = (long long)a.N * a.H * a.W, total = P * M;
    const long long run0 = (long long)blockIdx.x * (rounds * kGradThreads);
    const int lane = threadIdx.x & 31;
    const int E = min(max(*n_edges_dev, 0), max_edges);
    // pixel, view and sample of the run's pair k, by 32-bit divisions from the run's first
    __shared__ long long s_idx;
    __shared__ unsigned s_first[3];  // sample, pixel, view
    const unsigned HW = (unsigned)a.H * (unsigned)a.W;
    auto locate = [&](unsigned k, long long* idx, int* view, uint32_t* pix, int* j) {
        const unsigned t = s_first[0] + k, q = t / (unsigned)M, p = s_first[1] + q, v = p / HW;
        *j = (int)(t - q * (unsigned)M);
        *idx = s_idx + q;
        *view = (int)(s_first[2] + v);
        *pix = p - v * HW;
    };
    auto flush = [&]() {  // whole CTA, after a barrier
        if (rays.pending() == 0u) return;
        if (rays.pending() <= OuterRays::kSplit) {
            if (threadIdx.x == 0) rays.find_parts(a.nodes, a.n_tris);
            __syncthreads();
        }
        trace_rays(a.nodes, static_cast<const TriRecord*>(a.tris), a.n_tris, wide_reach(a.nodes, a.n_tris), rays.stacks,
                   rays);
        __syncthreads();
        const unsigned n = rays.n;
        for (unsigned i = threadIdx.x; i < n; i += kGradThreads) {
            if ((rays.hit[i >> 5] >> (i & 31)) & 1u) continue;
            const int k = __float_as_int(rays.dir[i].w);
            long long idx;
            int view, j;
            uint32_t pix;
            locate(k, &idx, &view, &pix, &j);
            EdgeSample S;
            if (!draw_edge_sample(a, verts, n_verts, edges, E, idx, view, pix, j, &S)) continue;  // (it was one)
            Pixel px{};
            load_pixel(a.gb_pos[idx], a.gb_nrm[idx], a.gb_kd[idx], a.gb_korm[idx],
                       mk(a.cams[view].origin[0], a.cams[view].origin[1], a.cams[view].origin[2]), &px);
            Probe Pr;
            Pr.W = a.Wp;
            Pr.H = a.Hp;
            float st;
            const int t = texel_of_dir(Pr, S.w, &st);
            const f3 L = xyz(__ldg(a.env + t));
            const f3 gd = xyz(g_cd[idx]);
            float gw = (L.x * gd.x + L.y * gd.y + L.z * gd.z) * S.ci * MCDI_INV_PI;
            if (px.spec_on) {
                const f3 gs = xyz(g_cs[idx]);
                const f3 h = normalize(S.w + px.wo);
                const float nh = dot(px.n, h), vh = dot(px.wo, h);
                const float D = ggx_D(nh, sin2_between(px.n, h), px.a2);
                const float G2 = 1.0f / (1.0f + ggx_lambda(S.ci, px.a2) + ggx_lambda(px.co, px.a2));
                const float q = schlick_weight(vh);
                const f3 F = mk(px.F0.x + (1.f - px.F0.x) * q, px.F0.y + (1.f - px.F0.y) * q,
                                px.F0.z + (1.f - px.F0.z) * q);
                gw += (L.x * gs.x * F.x + L.y * gs.y * F.y + L.z * gs.z * F.z) * D * G2 / (4.0f * px.co);
            }
            const f3 c = cross(S.w, S.ab);
            const float J = sqrtf(dot(c, c)) / S.r2;
            const float wt = -a.tau * gw * J * ((float)E / (float)M);
            if (wt != 0.0f) {
                scatter3(g_verts, S.ed.x, S.nout * (wt * (1.0f - S.s)));
                scatter3(g_verts, S.ed.y, S.nout * (wt * S.s));
            }
            if (sample_w) sample_w[run0 + k] = wt;
        }
    };
    auto clear = [&]() {  // whole CTA, between barriers
        if (threadIdx.x == 0) rays.n = rays.head = 0u;
        if (threadIdx.x < OuterRays::kCap / 32) rays.hit[threadIdx.x] = 0u;
    };
    clear();
    if (threadIdx.x == 0) {
        s_idx = run0 / M;
        const long long view = s_idx / HW;
        s_first[0] = (unsigned)(run0 - s_idx * M);
        s_first[1] = (unsigned)(s_idx - view * HW);
        s_first[2] = (unsigned)view;
    }
    __syncthreads();
    for (int r = 0; r < rounds; ++r) {
        const int k = r * kGradThreads + threadIdx.x;
        const long long tid = run0 + k;
        EdgeSample S;
        bool cand = false;
        if (tid < total) {
            long long idx;
            int view, j;
            uint32_t pix;
            locate(k, &idx, &view, &pix, &j);
            cand = draw_edge_sample(a, verts, n_verts, edges, E, idx, view, pix, j, &S);
            if (sample_w) sample_w[tid] = 0.0f;
        }
        const unsigned mask = __ballot_sync(0xffffffffu, cand);
        if (mask) {
            unsigned base = 0;
            if (lane == 0) base = atomicAdd(&rays.n, (unsigned)__popc(mask));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (cand) {
                const unsigned i = base + __popc(mask & ((1u << lane) - 1u));
                const f3 dir = normalize(S.w + S.nout * eta);
                rays.dir[i] = make_float4(dir.x, dir.y, dir.z, __int_as_float(k));
                rays.origin[i] = make_float4(S.o.x, S.o.y, S.o.z, 0.f);
            }
        }
        __syncthreads();
        const bool full = rays.pending() > OuterRays::kCap - kGradThreads;
        if (full || r == rounds - 1) {
            flush();
            __syncthreads();
            if (r == rounds - 1) break;
            clear();
        }
        __syncthreads();  // every thread has read the count before the next round adds to it
    }
}

inline size_t edge_table_cap(int n_tris) {
    size_t cap = 1;
    while (cap < (size_t)6 * (size_t)(n_tris > 0 ? n_tris : 1)) cap <<= 1;  // >= 2 x the half-edges
    return cap;
}

}  // namespace

EdgeScratch edge_scratch_layout(int n_tris) {
    EdgeScratch L{};
    const size_t nh = (size_t)3 * (n_tris > 0 ? n_tris : 1);
    L.cap = edge_table_cap(n_tris);
    L.n_tiles = (int)((nh + kEdgeTile - 1) / kEdgeTile);
    size_t o = 0;
    L.keys = o; o = align256(o + L.cap * sizeof(unsigned long long));
    L.first = o; o = align256(o + L.cap * sizeof(int));
    L.second = o; o = align256(o + L.cap * sizeof(int));
    L.slot_of = o; o = align256(o + nh * sizeof(int));
    L.tile_count = o; o = align256(o + (size_t)L.n_tiles * sizeof(int));
    L.tile_off = o; o = align256(o + (size_t)L.n_tiles * sizeof(int));
    L.err = o; o = align256(o + sizeof(unsigned));
    L.total = o;
    return L;
}

cudaError_t launch_build_edge_table(const int* tris, int n_tris, int4* edges, int* n_edges, void* scratch,
                                    const EdgeScratch& L, cudaStream_t stream) {
    char* ws = static_cast<char*>(scratch);
    auto* keys = reinterpret_cast<unsigned long long*>(ws + L.keys);
    int* first = reinterpret_cast<int*>(ws + L.first);
    int* second = reinterpret_cast<int*>(ws + L.second);
    int* slot_of = reinterpret_cast<int*>(ws + L.slot_of);
    int* tile_count = reinterpret_cast<int*>(ws + L.tile_count);
    int* tile_off = reinterpret_cast<int*>(ws + L.tile_off);
    unsigned* err = reinterpret_cast<unsigned*>(ws + L.err);
    const int n_half = 3 * n_tris;
    cudaError_t e = cudaMemsetAsync(err, 0, sizeof(unsigned), stream);
    if (e != cudaSuccess) return e;
    const long long cap = (long long)L.cap;
    const int clear_blocks = (int)((cap + kEdgeThreads - 1) / kEdgeThreads < 4096 ? (cap + kEdgeThreads - 1) / kEdgeThreads
                                                                                   : 4096);
    launch_k(edge_clear_kernel, clear_blocks, kEdgeThreads, 0, stream, keys, first, second, cap);
    const int hb = (n_half + kEdgeThreads - 1) / kEdgeThreads;
    launch_k(edge_insert_kernel, hb, kEdgeThreads, 0, stream, tris, n_half, keys, first, slot_of, cap, err);
    launch_k(edge_second_kernel, hb, kEdgeThreads, 0, stream, n_half, (const int*)slot_of, (const int*)first, second);
    launch_k(edge_count_kernel, L.n_tiles, kEdgeThreads, 0, stream, n_half, (const int*)slot_of, (const int*)first,
             tile_count);
    launch_k(edge_offsets_kernel, 1, 1024, 0, stream, L.n_tiles, (const int*)tile_count, tile_off, n_edges,
             (const unsigned*)err);
    launch_k(edge_write_kernel, L.n_tiles, kEdgeThreads, 0, stream, tris, n_half, (const int*)slot_of,
             (const int*)first, (const int*)second, (const int*)tile_off, edges);
    return cudaGetLastError();
}

cudaError_t launch_shadow_edge_grad(const ShadeArgs& a, const float* verts, int n_verts, const int4* edges,
                                    const int* n_edges, int max_edges, int n_samples, float eta, const float4* g_cd,
                                    const float4* g_cs, float* g_verts, float* sample_w, cudaStream_t stream) {
    const long long n = (long long)a.N * a.H * a.W * n_samples;
    if (n <= 0) return cudaGetLastError();
    // the longest runs that still give every SM its CTAs
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const long long resident = (long long)sms * kGradBlocksPerSM * kGradThreads;
    const int rounds = (int)std::min<long long>(std::max<long long>(n / resident, 1), kMaxRounds);
    const long long run = (long long)rounds * kGradThreads;
    launch_k(shadow_edge_grad_kernel, (int)((n + run - 1) / run), kGradThreads, 0, stream, a, verts,
             n_verts, edges, n_edges, max_edges, n_samples, eta, g_cd, g_cs, g_verts, sample_w, rounds);
    return cudaGetLastError();
}

}  // namespace mcdi
