// Any-hit traversal of many shadow rays by the warps of a CTA (Sec. 3.1, App.
// A): the loop shared by the wavefront's persistent tracer and by the kernels
// that trace the rays of their own pixels.
#pragma once

#include "shading.cuh"

namespace mcdi {

constexpr int kTraceThreads = 128;       // threads per CTA that traces
constexpr int kTraceStepsPerRefill = 8;  // 4: 6% slower, 12 and 16: within 1%
constexpr int kTraceNodes = 20;          // pending nodes per lane (a visit needs four free)
constexpr int kTraceLeaves = 8;          // postponed triangle tests per lane (a visit needs four free)
constexpr int kLeafBatch = 16;           // lanes holding one that start a triangle round (12 to 22: within 1%)

struct TraceStacks {  // a CTA's columns: one thread's entries in one bank
    int node[kTraceNodes * kTraceThreads];
    int leaf[kTraceLeaves * kTraceThreads];
};

// Every lane of every warp of the CTA calls it.  A lane holds a ray, the
// four-wide node it visits next, a stack of pending nodes and a queue of leaf
// triangles whose boxes its ray hit; every kTraceStepsPerRefill steps the warp
// gives the lanes that are out of nodes the next rays of the list.
//
// A step visits one node per lane.  Triangle tests are postponed and run as
// warp-wide rounds, one triangle per lane that holds one, once kLeafBatch
// lanes do or a lane's queue is full.  A lane whose nodes are done takes its
// next ray at once, although triangles of the last one may still be queued:
// queue entries below lmark belong to the previous ray, whose origin and
// direction stay at hand (R.load), and the lane only waits for a round when
// those are still there as the next ray ends too.  (Waiting for the tests
// instead, with rounds forced by waiting lanes, takes a round at nearly every
// step with a quarter of its lanes, or leaves lanes idle.)
//
// A ray whose pending nodes outgrow the stack, or whose origin lies beyond `reach`
// (wide_reach), is decided by the stackless walk of the depth-first copy instead.
//
// R supplies the rays: R.count() of them, the same for all warps; R.take(n)
// (lane 0) reserves the next n and returns the first; R.start(i, id, o, d,
// node) loads ray i, sets the node it starts at (0, the root, or kWideDone for
// none) and returns the lane's handle for it (id: the handle of its ray
// before); R.load(id, o, d) gives a ray again by handle (the current ray's or
// the one before); R.blocked(id) records a hit.
template <class R>
__device__ __forceinline__ void trace_rays(const void* __restrict__ nodes, const TriRecord* __restrict__ tris,
                                           int n_tris, float reach, TraceStacks& st, R& rays) {
    constexpr int kStep = 4 * kTraceThreads;
    if (n_tris <= 0) return;  // nothing can block a ray
    const unsigned n_rays = rays.count();
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const WideNode* wn = wide_nodes(nodes, n_tris);
    const uint32_t nbase = (uint32_t)__cvta_generic_to_shared(st.node + threadIdx.x);
    const uint32_t lbase = (uint32_t)__cvta_generic_to_shared(st.leaf + threadIdx.x);
    const uint32_t nroom = nbase + (kTraceNodes - 4) * kStep, lroom = lbase + (kTraceLeaves - 4) * kStep;
    uint32_t na = nbase, la = lbase;  // first free entries
    uint32_t lmark = lbase;           // leaf entries below it belong to the lane's previous ray
    int cur = 0, last = 0;            // handles of the current and the previous ray
    int node = kWideDone;             // a lane out of nodes has node < 0
    f3 inv = mk(0.f, 0.f, 0.f), oi = inv;
    bool more = true;  // rays left in the list (the same for the whole warp)
    while (true) {
        const bool free_lane = node < 0 && lmark == lbase;
        const unsigned idle = __ballot_sync(full, free_lane);
        if (more && idle) {
            unsigned base = 0;
            if (lane == 0) base = rays.take((unsigned)__popc(idle));
            base = __shfl_sync(full, base, 0);
            const unsigned my = base + __popc(idle & lt);
            if (free_lane && my < n_rays) {
                f3 o, d;
                last = cur;
                cur = rays.start(my, cur, o, d, node);
                inv = make_ray(o, d).inv;
                oi = mk(-o.x * inv.x, -o.y * inv.y, -o.z * inv.z);
                lmark = la;
                if (!(largest(o) <= reach)) na = nroom + kStep;  // as if its pending nodes had outgrown the stack
            }
            more = base + (unsigned)__popc(idle) < n_rays;
        } else if (!__any_sync(full, node >= 0 || la != lbase)) {
            break;
        }
        // every node is visited at most once, so a ray ends within n - 1 visits and as many rounds
        for (int step = 0; step < kTraceStepsPerRefill; ++step) {
            if (node >= 0 && la <= lroom && na <= nroom) {
                wide_visit<kStep>(wn, inv, oi, node, na, la);
                node = kWideDone;
                if (na != nbase) {
                    na -= kStep;
                    node = lds32(na);
                }
            }
            const unsigned pend = __ballot_sync(full, la != lbase);
            // a lane that cannot go on without a round: its queue is full, or its next ray waits for the previous one
            const bool must = la > lroom || (node < 0 && lmark != lbase);
            if (__popc(pend) >= kLeafBatch || __any_sync(full, must) || !__any_sync(full, node >= 0)) {
                if (la != lbase) {
                    la -= kStep;
                    const int k = ~lds32(la);
                    const bool prev = la < lmark;
                    if (prev) lmark = la;
                    f3 o, d;
                    rays.load(prev ? last : cur, o, d);
                    // (an empty slot's link can only come from a ray with infinite coordinates)
                    if ((unsigned)k < (unsigned)n_tris && tri_blocks(o, d, tris, k)) {
                        rays.blocked(prev ? last : cur);
                        if (prev) {
                            la = lmark = lbase;  // nothing of the current ray is queued above it
                        } else {
                            la = lmark;
                            node = kWideDone;
                            na = nbase;
                        }
                    }
                }
            }
            if (node >= 0 && na > nroom) {  // more pending nodes than the stack holds, or not for these nodes
                f3 o, d;
                rays.load(cur, o, d);
                if (any_hit_threaded(nodes, tris, n_tris, make_ray(o, d))) rays.blocked(cur);
                node = kWideDone;
                na = nbase;
            }
        }
    }
}

// The shadow rays of a CTA's 32 pixels for kChunk consecutive samples, in
// shared memory: appended by the warps that draw the samples, then traced by
// trace_rays.  hit[j] has bit p set when the ray of the chunk's sample j of
// pixel p is blocked.
template <int kChunk>
struct BlockRays {
    static constexpr int kRays = 32 * kChunk;
    float4 dir[kRays];  // w: pixel | sample << 5 (int bits)
    float4 origin[32];
    unsigned hit[kChunk];
    unsigned n, head;
    TraceStacks stacks;

    // every thread, before the chunk's rays are appended (a barrier must follow)
    __device__ __forceinline__ void clear() {
        if (threadIdx.x == 0) n = head = 0u;
        if (threadIdx.x < kChunk) hit[threadIdx.x] = 0u;
    }
    // whole warps: lane p's ray for the chunk's sample j
    __device__ __forceinline__ void append(bool active, int j, f3 d) {
        const int lane = threadIdx.x & 31;
        const unsigned act = __ballot_sync(0xffffffffu, active);
        if (act == 0u) return;
        unsigned base = 0;
        if (lane == 0) base = atomicAdd(&n, (unsigned)__popc(act));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (active) dir[base + __popc(act & ((1u << lane) - 1u))] = make_float4(d.x, d.y, d.z, __int_as_float(lane | j << 5));
    }
    __device__ __forceinline__ unsigned count() const { return *(volatile const unsigned*)&n; }
    __device__ __forceinline__ unsigned take(unsigned k) { return atomicAdd(&head, k); }
    __device__ __forceinline__ void load(int id, f3& o, f3& d) const {
        const float4 v = dir[id];
        d = xyz(v);
        o = xyz(origin[__float_as_int(v.w) & 31]);
    }
    __device__ __forceinline__ int start(unsigned i, int, f3& o, f3& d, int& node) const {
        load((int)i, o, d);
        node = 0;
        return (int)i;
    }
    __device__ __forceinline__ void blocked(int id) {
        const int w = __float_as_int(dir[id].w);
        atomicOr(&hit[w >> 5], 1u << (w & 31));
    }
};

}  // namespace mcdi
