// The culling traversal kernels (device code only); hrr_cull.cu instantiates and launches them.
//
// Hierarchical Russian-roulette culling with blue-noise dithered QMC sequences (Sec. 1).
//
// For eye j with shift r_j (tile entry at its pixel), the traversal starts at the root and,
// at every visited node, tests the node's children from one record:
//   * a child with leaf range [a, b) survives unless the range minimum
//     v(a, b) = min_{i in [a,b)} (brev(i) + r_j) mod 2^32 passes the conservative cull test
//     (v is at least the threshold of every light below; then none can be accepted);
//   * a surviving internal child is descended; a surviving leaf child i (whose box is the
//     light's position and whose minimum is its own value) is accepted iff
//     brev(i) + r_j < ceil(p_ij 2^32) (exact float32 p).
// The accepted set therefore equals flat Russian roulette over all pairs.
//
// Node width. The hierarchy is binary; a traversal reads it either with binary nodes
// (64-byte records: both children) or with nodes of width four (128-byte records: the four
// grandchildren, or a leaf child in place of its two slots), visiting only even-depth nodes.
// The cull test is monotone (a smaller box, a smaller maximum intensity and a range minimum
// over a sub-range never turn a cull into a visit), so both widths accept the same pairs;
// width four pops half as many nodes, with half the stack traffic and loop overhead per
// child tested, for one extra range minimum per visit.
//
// Execution: a persistent grid (a whole number of resident blocks per SM) in which each
// warp traverses one eye at a time. The newest of the warp's pending nodes are kept in shared
// memory (binary records: a linear stack; width four: a ring); every step pops up to 32 nodes,
// one per lane, and the lanes push the children that survive their tests back as one compacted
// run (ballot + popc). All lanes of a step execute the same test on the same eye, leaf children
// included, so the warp stays converged. A leaf child that survives (about one in a hundred
// visits, nearly all of them accepted) is queued in shared memory, and the exact pair test runs
// on 32 queued leaves at a time, and on the rest when the eye is done. Testing leaves in the step
// itself took a divergent branch with one or two lanes in two of three steps. When the shared
// entries would overflow, the oldest move to a per-warp area in global memory, and they come
// back when few are left. The stack never exceeds
// (w - 1) * 32 * L + 32 entries for node width w and L depth levels of pushed nodes (each
// remainder of a pushed run below the top holds at most (w - 1) * 32 entries, and the
// shallowest depth of those runs grows from the bottom of the stack to its top), and the
// spill area is sized by that bound.
//
// Memory: the kernel is bound by the L1 data pipe (one scattered record per lane per
// step), so each record is fetched with 256-bit loads that do not allocate in L1. A node's
// range minimum is attained at one index, which lies in exactly one child; carrying the
// minimum with each stack entry (its index is brev(v - r)) means only the other children's
// minima have to be computed. The accepted pairs of one batch of queued leaves are appended
// to the output with one atomic and neighbouring 8-byte stores.
//
// The head (forms with top levels, binary records): each eye starts by evaluating the 62
// nodes below the root of the top HRR_TOP_LEVELS levels, one per lane in two passes,
// instead of walking those levels one per step with 1, 2, 4, 8 and 16 lanes busy. A
// single-frame launch stages the top slots in shared memory once per block; in a batched
// launch, whose warps move between frames, each eye reads its frame's slots (3 KB, cached
// in L1 and L2) directly. The cull test is
// monotone: a child's box lies inside its parent's, its maximum intensity is at most the
// parent's and its range minimum at least the parent's, and the test culls at least as
// much for each, so a node below the root is visited iff its own test passes, whatever its
// ancestors' results. The head counts the root and the visited nodes above the deepest top
// level as visits, tests the top's leaves, and pushes the visited nodes of the deepest top
// level (with their range minima) as the stack the walk starts from: the same visited set, visit
// count and accepted set as a walk from the root.
//
// One launch may cover many frames (a batch): the eye cursor then runs over the eyes of all
// frames, each warp finds its eye's frame by binary search over the frames' cursor offsets,
// and the frames' descriptors are read through the constant cache. Frames of different
// sizes share the launch without any per-frame tail.
#pragma once

#include <algorithm>

#include "hrr_internal.cuh"

namespace {

constexpr uint32_t kMaxFrames = HRR_CULL_MAX_FRAMES;  // frames of one batched launch

// Resident threads per SM each instantiation is compiled for (the register budget):
// 48 registers for binary records (5 blocks of 256 threads), 64 for width four. With 40
// registers and 6 blocks the binary form spills, and the frame takes 4% longer.
template <int W>
constexpr int min_blocks(int threads) {
    return (W == 2 ? 1280 : 1024) / threads;
}

using Frame = hrr_cull_frame_t;
static_assert(sizeof(Frame) == 144, "frame descriptor layout");

struct Launch {
    uint32_t n_frames;
    uint32_t spill_cap;             // stack entries per warp in the spill area
    unsigned long long total;       // eyes of this launch over all frames
    unsigned long long *cursor;     // global eye cursor (starts at 0)
    unsigned long long *flags;      // HRR_FLAG_* bits
    uint2 *spill;                   // grid warps x spill_cap stack entries
    unsigned long long *host;       // pinned host words for the frame's counts and flags, or null
};

// The end of a launch that reports to the host by itself (Lc.host set, a frame of its own): the
// last block to finish writes accepted pairs, visits and flags to the host words and clears the
// five words at fr.counts (with the cursor and the blocks done) for the context's next launch.
// A small call is bound by what surrounds its kernel: with this instead of a clearing and a copy
// on the stream (and connection weights that report their flag likewise) a 32x32-eye probe of
// 4,096 lights takes 70 us, cull and weights, instead of 81.
__device__ __forceinline__ void report(const Launch &Lc, unsigned long long *counts) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(&counts[4], 1ull) + 1ull == gridDim.x) {
        __threadfence();
        for (int k = 0; k < 3; ++k) __stcs(&Lc.host[k], __ldcg(&counts[k]));
        for (int k = 0; k < 5; ++k) __stcg(&counts[k], 0ull);
        __threadfence_system();
    }
}

// The launch's frame descriptors travel as a kernel parameter, so the traversal reads them
// through the constant cache (and may re-read them instead of holding them in registers).
template <uint32_t N>
struct FrameArray {
    Frame f[N];
};

// Frame f of the launch (always the only one for a single frame).
template <bool BATCH>
__device__ __forceinline__ const Frame &frame_at(const Frame *F, uint32_t f) {
    if constexpr (!BATCH) return F[0];
    else return F[f];
}

// 32 bytes (two float4, or four pairs of floats) as one 256-bit read-only load that does not
// allocate in L1: the records are scattered and rarely reused from L1, and filling it with
// them would take L1 data-pipe cycles (they come from L2 either way).
__device__ __forceinline__ void load32(const float4 *p, float4 &a, float4 &b) {
    asm("ld.global.nc.L1::no_allocate.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
        : "l"(p));
}
__device__ __forceinline__ void load32(const float4 *p, hrr_f2 &a, hrr_f2 &b, hrr_f2 &c, hrr_f2 &d) {
    asm("ld.global.nc.L1::no_allocate.v4.b64 {%0,%1,%2,%3}, [%4];" : "=l"(a), "=l"(b), "=l"(c), "=l"(d) : "l"(p));
}

// Range minimum of (brev(i) + r) over the L >= 1 indices from a; c = brev(2^32 - r).
template <int VARIANT>
__device__ __forceinline__ uint32_t range_min(uint32_t a, uint32_t L, uint32_t r, uint32_t c) {
    if (VARIANT == 0) return hrr_range_min_value(a, L, r, 0u - r, c);
    uint32_t k;
    return hrr_rangemin_closed(a, a + L, r, &k);
}

// The index at which brev(i) + r is v.
__device__ __forceinline__ uint32_t index_of(uint32_t v, uint32_t r) { return __brev(v - r); }

// The eye a traversal works on.
struct Eye {
    float x, y, z, tau;
    float scale;    // the node test's scale, hrr_node_scale(tau)
    uint32_t r, c;  // shift and brev(2^32 - r)
};

// What one lane's visit produces: up to W children to push (node, range minimum) and up to W
// surviving leaves.
template <int W>
struct Visit {
    bool go[W], leaf[W];
    uint32_t node[W], vmin[W], light[W];  // node: the child's record (slot of pairs, index of wide)
};

// Test one child slot: it survives unless its range minimum v culls it; the box is (lo, imax,
// hi), for a leaf the light itself, which fails this test only if the pair is rejected.
__device__ __forceinline__ bool survives(const Eye &E, const float4 &lo, const float4 &hi, uint32_t v) {
    float den, rhs;
    hrr_node_bound(E.scale, lo.x, lo.y, lo.z, hi.x, hi.y, hi.z, lo.w, E.x, E.y, E.z, den, rhs);
    return !hrr_node_culls(v, den, rhs);
}

// A visit of node g read with width four: its 128-byte record holds the four grandchild
// slots [first, s0], [s0 + 1, split], [split + 1, s1], [s1 + 1, last] (a leaf child fills its
// first slot and leaves the second empty). The parent's minimum is attained in one child; one
// more range minimum gives the other child's, and one more per internal child splits it
// between that child's two slots.
template <int VARIANT>
__device__ __forceinline__ void visit(const float4 *wide, uint32_t n_lights, uint32_t g, uint32_t vmin,
                                      const Eye &E, unsigned long long *flags, Visit<4> &V) {
    float4 q[8];
    load32(&wide[8 * (size_t)g], q[0], q[1]);
    load32(&wide[8 * (size_t)g + 2], q[2], q[3]);
    load32(&wide[8 * (size_t)g + 4], q[4], q[5]);
    load32(&wide[8 * (size_t)g + 6], q[6], q[7]);
    const uint32_t s0 = __float_as_uint(q[1].w), split = __float_as_uint(q[3].w);
    const uint32_t s1 = __float_as_uint(q[5].w), other = __float_as_uint(q[7].w);
    const uint32_t first = min(g, other), last = max(g, other);
    const bool c0int = first != split, c1int = split + 1u != last;
    // first <= s0 <= split < last, split < s1 <= last, and an internal child's split inside it
    // (so every internal slot is a node below g, with a record)
    if (last >= n_lights || s0 - first > split - first || split - first >= last - first ||
        s1 - split - 1u > last - split - 1u || (c0int && s0 == split) || (c1int && s1 == last)) {
        atomicOr(flags, HRR_FLAG_TOPOLOGY);  // corrupt record
        return;
    }
    const bool in0 = index_of(vmin, E.r) <= split;
    const uint32_t vc = range_min<VARIANT>(in0 ? split + 1u : first, in0 ? last - split : split - first + 1u, E.r, E.c);
    const uint32_t vA = in0 ? vmin : vc, vB = in0 ? vc : vmin;  // range minima of children 0 and 1
    uint32_t v[4] = {vA, vA, vB, vB};
    if (c0int) {
        const bool at0 = index_of(vA, E.r) <= s0;
        const uint32_t vx = range_min<VARIANT>(at0 ? s0 + 1u : first, at0 ? split - s0 : s0 - first + 1u, E.r, E.c);
        v[0] = at0 ? vA : vx;
        v[1] = at0 ? vx : vA;
    }
    if (c1int) {
        const bool at2 = index_of(vB, E.r) <= s1;
        const uint32_t vy = range_min<VARIANT>(at2 ? s1 + 1u : split + 1u, at2 ? last - s1 : s1 - split, E.r, E.c);
        v[2] = at2 ? vB : vy;
        v[3] = at2 ? vy : vB;
    }
    const uint32_t a[4] = {first, s0 + 1u, split + 1u, s1 + 1u};
    const uint32_t b[4] = {s0, split, s1, last};  // inclusive; a > b: an empty slot
    V.node[0] = s0;
    V.node[1] = s0 + 1u;
    V.node[2] = s1;
    V.node[3] = s1 + 1u;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        V.vmin[t] = v[t];
        const bool s = a[t] <= b[t] && survives(E, q[2 * t], q[2 * t + 1], v[t]);
        V.go[t] = s && a[t] < b[t];
        V.leaf[t] = s && a[t] == b[t];
        V.light[t] = a[t];
    }
}

// The exact test of one light per lane (`has`: the lane has one, at position (x, y, z) of
// intensity w and sorted index i) for eye j, and the accepted pairs appended to the frame's
// output: one atomic, neighbouring stores (warp-collective). The pairs are written once and
// never read by the kernel, so they are stored with the streaming (evict-first) hint: the
// output stream then does not push the node records out of L2.
__device__ __forceinline__ void take(const Frame &fr, const Eye &E, uint32_t j, int lane, bool has, const float4 &l,
                                     uint32_t i) {
    const bool acc = has && hrr_pair_accepts(__brev(i) + E.r, E.tau, l.x, l.y, l.z, l.w, E.x, E.y, E.z);
    const unsigned bal = __ballot_sync(0xFFFFFFFFu, acc);
    if (bal == 0u) return;
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(&fr.counts[0], (unsigned long long)__popc(bal));
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    const unsigned long long o = base + __popc(bal & ((1u << lane) - 1u));
    if (acc && o < fr.cap) __stcs(&fr.pairs[o], make_uint2(j, __ldg(&fr.perm[i])));
}

// A queued leaf: the record that holds it, its place t there and its sorted index, with the
// bits of t in the words' top bits (lights and width-four records number less than 2^31;
// binary records need only the low bit of t).
template <int W>
__device__ __forceinline__ uint2 queued(uint32_t node, uint32_t t, uint32_t light) {
    return make_uint2(W == 2 ? node : node | (t >> 1 << 31), light | (t << 31));
}

// The light (position, intensity) at place t of a record.
template <int W, bool PAIRED>
__device__ __forceinline__ float4 light_of(const float4 *records, uint32_t node, uint32_t t) {
    if constexpr (W == 2 && !PAIRED) {
        return __ldg(&records[4 * (size_t)hrr_slot_node(node) + 2u * t]);
    } else if constexpr (W == 2) {
        const float *p = reinterpret_cast<const float *>(records + 4 * (size_t)node) + t;
        return make_float4(-__ldg(p), -__ldg(p + 2), -__ldg(p + 4), __ldg(p + 12));
    } else {
        return __ldg(&records[8 * (size_t)node + 2u * t]);
    }
}

// Take the n <= 32 newest of the warp's queued leaves.
template <int W, bool PAIRED>
__device__ __forceinline__ void take_queued(const Frame &fr, const Eye &E, uint32_t j, int lane, const uint2 *q,
                                            uint32_t n) {
    const bool has = (uint32_t)lane < n;
    float4 l = make_float4(0.f, 0.f, 0.f, 0.f);
    uint32_t i = 0;
    if (has) {
        const uint2 e = q[lane];
        const uint32_t t = (W == 2 ? 0u : e.x >> 31 << 1) | (e.y >> 31);
        i = e.y & 0x7FFFFFFFu;
        l = light_of<W, PAIRED>(fr.nodes, W == 2 ? e.x : e.x & 0x7FFFFFFFu, t);
    }
    __syncwarp();
    take(fr, E, j, lane, has, l, i);
}

// The head of eye j's traversal over the top slots `top` (shared memory for a single frame,
// global memory for a batch): takes the top's surviving leaves, pushes the visited nodes of
// the deepest top level onto the empty ring, and returns the visits it accounts for (the
// root and the visited nodes above that level).
template <int VARIANT, bool BATCH>
__device__ __forceinline__ uint32_t head(const float4 *top, const Eye &E, const Frame &fr, int lane, uint32_t j,
                                         uint2 *ring, uint32_t &pushed) {
    constexpr uint32_t kDeep = HRR_TOP_SLOTS / 2;  // first slot of the deepest top level
    const unsigned lt = (1u << lane) - 1u;
    uint32_t visits = 1, n = 0;  // the root
#pragma unroll
    for (uint32_t p = 0; p < (HRR_TOP_SLOTS + 31) / 32; ++p) {
        const uint32_t s = 1u + (uint32_t)lane + 32u * p;  // slots 1 .. HRR_TOP_SLOTS - 1
        bool vis = false, leaf = false;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        uint32_t node = 0, vmin = 0, light = 0;
        if (s < HRR_TOP_SLOTS) {
            float4 h, x;
            if constexpr (BATCH) {
                a = __ldg(&top[3 * s]);
                h = __ldg(&top[3 * s + 1]);
                x = __ldg(&top[3 * s + 2]);
            } else {
                a = top[3 * s];
                h = top[3 * s + 1];
                x = top[3 * s + 2];
            }
            const uint32_t kind = __float_as_uint(x.z);
            const uint32_t first = __float_as_uint(h.w), last = __float_as_uint(x.x);
            if (kind != HRR_TOP_EMPTY) {
                vmin = range_min<VARIANT>(first, last - first + 1u, E.r, E.c);
                const bool alive = survives(E, a, h, vmin);
                vis = alive && kind == HRR_TOP_INTERNAL;
                leaf = alive && kind == HRR_TOP_LEAF;
                node = 2u * __float_as_uint(x.y) - (s & 1u ? 0u : 1u);  // odd heap slots are child 0
                light = first;
            }
        }
        const bool deep = s >= kDeep;
        visits += __popc(__ballot_sync(0xFFFFFFFFu, vis && !deep));
        const unsigned bp = __ballot_sync(0xFFFFFFFFu, vis && deep);
        if (vis && deep) ring[n + __popc(bp & lt)] = make_uint2(node, vmin);
        n += __popc(bp);
        if (__any_sync(0xFFFFFFFFu, leaf)) take(fr, E, j, lane, leaf, a, light);
    }
    __syncwarp();
    pushed = n;
    return visits;
}

// Range minimum over leaves [a, z].
template <int VARIANT>
__device__ __forceinline__ uint32_t range_min_leaves(uint32_t a, uint32_t z, const Eye &E) {
    if (VARIANT == 0) return hrr_range_min_leaves(a, z, E.r, 0u - E.r, E.c);
    uint32_t k;
    return hrr_rangemin_closed(a, z + 1u, E.r, &k);
}

// The walk over binary records for eye j, from the R entries that `stack` holds (shared memory,
// kRing entries, oldest first); returns the visits it makes, the sum with those before it at
// most n_lights - 1. Each step visits up to 32 nodes, one per lane. Everything rare shares a
// test with something else that is rare: fewer than 32 entries or visits left; surviving leaves
// or a corrupt record. That and the clamped range minimum took a step from 180 to 134 warp
// instructions, the issue slots from 81% to 65%, and left the L1 data pipe as the limit (94 to 96% on
// 480x270 eyes and 2^20 lights: 42 wavefronts a step for the records, 8 for the stack). PAIRED is
// false for a tree without paired records: the same walk over its binary ones (5.58 ms instead of
// 5.12 on those eyes and lights, 24.2 instead of 20.6 on 960x540).
template <int VARIANT, uint32_t kRing, bool PAIRED>
__device__ __forceinline__ uint32_t walk_pairs(const Frame &fr, const Eye &E, uint32_t j, int lane, uint2 *stack,
                                               uint2 *queue, uint32_t R, uint32_t before, uint2 *spill,
                                               uint32_t spill_cap, unsigned long long *flags) {
    const unsigned lt = (1u << lane) - 1u;
    const uint32_t n_lights = fr.n_lights;
    const float4 *records = fr.nodes;
    const hrr_f2 ex = hrr_pack2(E.x, E.x), ey = hrr_pack2(E.y, E.y), ez = hrr_pack2(E.z, E.z);
    uint32_t P = 0;         // older entries, in the spill area
    uint32_t queued_n = 0;  // surviving leaves still to be taken
    int left = (int)(n_lights - before);  // each internal node is visited at most once per eye
    for (;;) {
        if (min((int)R, left) < 32) {
            if (P && R < 32u) {  // bring spilled entries back under the others
                const uint32_t fc = min(P, kRing / 2 - R);
                uint2 up = make_uint2(0u, 0u);
                if ((uint32_t)lane < R) up = stack[lane];
                __syncwarp();
                if ((uint32_t)lane < R) stack[fc + lane] = up;
                for (uint32_t k = lane; k < fc; k += 32) stack[k] = spill[P - fc + k];
                P -= fc;
                R += fc;
                __syncwarp();
            }
            if (R == 0u) break;
            if (left <= 0) {
                if (lane == 0) atomicOr(flags, HRR_FLAG_TOPOLOGY);
                break;
            }
        }
        const uint32_t m = min(32u, R);
        const bool active = (uint32_t)lane < m;
        // Idle lanes take the last lane's entry, whose line the load touches anyway. (Any one record
        // for all idle lanes, the root's say, becomes the line that every SM asks one L2 slice for:
        // 8.2 ms instead of 7.3 for 960x540 eyes and 50,021 lights.)
        const uint2 e = stack[R - m + min((uint32_t)lane, m - 1u)];
        R -= m;
        left -= (int)m;
        __syncwarp();

        hrr_f2 nlox, nloy, nloz, nhix, nhiy, nhiz, imax, links;
        const uint32_t node = hrr_slot_node(e.x);
        if constexpr (PAIRED) {
            load32(&records[4 * (size_t)e.x], nlox, nloy, nloz, nhix);
            load32(&records[4 * (size_t)e.x + 2], nhiy, nhiz, imax, links);
        } else {
            hrr_load_binary(&records[4 * (size_t)node], nlox, nloy, nloz, nhix, nhiy, nhiz, imax, links);
        }
        const uint32_t split = (uint32_t)links, other = (uint32_t)(links >> 32);
        const uint32_t first = min(node, other), last = max(node, other);
        // needs first <= split < last < n
        const bool ok = active && last < n_lights && split - first < last - first;
        const bool in0 = index_of(e.y, E.r) <= split;
        // the other child's minimum (of a leaf: its own value)
        const uint32_t vnew = range_min_leaves<VARIANT>(in0 ? split + 1u : first, in0 ? last : split, E);
        const uint32_t v0 = in0 ? e.y : vnew, v1 = in0 ? vnew : e.y;
        hrr_f2 den, rhs;
        hrr_bound2(nlox, nloy, nloz, nhix, nhiy, nhiz, imax, ex, ey, ez, E.scale, den, rhs);
        bool s0, s1;
        hrr_survive2(den, rhs, v0, v1, ok, s0, s1);
        const bool go0 = s0 && first != split, go1 = s1 && split + 1u != last;
        const unsigned b0 = __ballot_sync(0xFFFFFFFFu, go0), b1 = __ballot_sync(0xFFFFFFFFu, go1);
        const uint32_t n = __popc(b0) + __popc(b1);
        if (R + n > kRing) {  // move the oldest entries to the spill area and the others down
            const uint32_t s = (R + n - kRing + 31u) & ~31u;
            if (P + s > spill_cap) {  // cannot happen: the area holds the bound
                if (lane == 0) atomicOr(flags, HRR_FLAG_STACK);
                break;
            }
            for (uint32_t k = lane; k < s; k += 32) spill[P + k] = stack[k];
            P += s;
            R -= s;
            for (uint32_t k = 0; k < R; k += 32) {
                __syncwarp();
                uint2 down = make_uint2(0u, 0u);
                if (k + lane < R) down = stack[s + k + lane];
                __syncwarp();
                if (k + lane < R) stack[k + lane] = down;
            }
            __syncwarp();
        }
        // Lane by lane, each lane's survivors side by side: siblings (whose records share a
        // line) are popped together by neighbouring lanes.
        uint2 *at = stack + R + __popc(b0 & lt) + __popc(b1 & lt);
        if (go0) *at++ = make_uint2(2u * split, v0);
        if (go1) *at = make_uint2(2u * split + 1u, v1);
        R += n;
        __syncwarp();
        const bool leaf0 = s0 && !go0, leaf1 = s1 && !go1;
        if (__any_sync(0xFFFFFFFFu, leaf0 || leaf1 || active != ok)) {
            if (active && !ok) atomicOr(flags, HRR_FLAG_TOPOLOGY);
            const unsigned q0 = __ballot_sync(0xFFFFFFFFu, leaf0), q1 = __ballot_sync(0xFFFFFFFFu, leaf1);
            if (leaf0) queue[queued_n + __popc(q0 & lt)] = queued<2>(e.x, 0u, split);
            queued_n += __popc(q0);
            if (leaf1) queue[queued_n + __popc(q1 & lt)] = queued<2>(e.x, 1u, last);
            queued_n += __popc(q1);
            __syncwarp();
            while (queued_n >= 32u) {
                queued_n -= 32u;
                take_queued<2, PAIRED>(fr, E, j, lane, queue + queued_n, 32u);
            }
        }
    }
    if (queued_n) take_queued<2, PAIRED>(fr, E, j, lane, queue, queued_n);
    return n_lights - before - (uint32_t)left;
}

// The traversal over the frames F (F[0] alone for a single frame); TOP levels of the
// hierarchy evaluated by the head (0: none, the walk starts at the root). PAIRED: the records of
// width two are paired ones, for every frame of the launch.
template <int VARIANT, bool BATCH, int W, int RING, int THREADS, int TOP, bool PAIRED>
__device__ __forceinline__ void traverse(const Launch &Lc, const Frame *F) {
    constexpr int kWarps = THREADS / 32;
    constexpr uint32_t kRing = RING;
    constexpr uint32_t kRingMask = kRing - 1;
    // a step pushes at most 32 W entries; making room for them must only move entries that
    // are resident (see the spill below), which needs kRing >= 32 W + 31
    static_assert((kRing & kRingMask) == 0 && kRing >= 32 * W + 32, "ring size");
    constexpr uint32_t kQueue = 32 * W + 32;  // a step queues at most 32 W leaves onto fewer than 32
    // the head reads the frames' binary records and pushes at most 32 entries
    static_assert(TOP == 0 || (TOP == (int)HRR_TOP_LEVELS && W == 2 && kRing >= 32), "top levels");
    __shared__ uint2 queue_all[kWarps][kQueue];  // surviving leaves of the eye (see queued)
    __shared__ uint2 ring_all[kWarps][kRing];  // (node, its range minimum)
    constexpr bool kTopShared = TOP > 0 && !BATCH;
    __shared__ float4 top_s[kTopShared ? 3 * HRR_TOP_SLOTS : 1];
    if constexpr (kTopShared) {
        if (F[0].n_lights > 1) {
            const float4 *src = F[0].top;
            for (uint32_t k = threadIdx.x; k < 3 * HRR_TOP_SLOTS; k += THREADS) top_s[k] = __ldg(&src[k]);
        }
        __syncthreads();
    }

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    uint2 *queue = queue_all[warp];
    uint2 *ring = ring_all[warp];
    // This warp's spill area (formed where it is used, so that it holds no registers).
#define HRR_WARP_SPILL (Lc.spill + ((size_t)blockIdx.x * kWarps + warp) * Lc.spill_cap)
    uint32_t f = 0;
    unsigned long long visit_acc = 0;  // visits of finished eyes of frame f, not yet published

    for (;;) {
        // The warp's next eye (warp-uniform from here on).
        unsigned long long gcur = 0;
        if (lane == 0) gcur = atomicAdd(Lc.cursor, 1ull);
        gcur = __shfl_sync(0xFFFFFFFFu, gcur, 0);
        if (gcur >= Lc.total) break;
        if constexpr (BATCH) {  // last frame whose cursor offset is <= gcur
            uint32_t lo = 0, hi = Lc.n_frames - 1;
            while (lo < hi) {
                const uint32_t mid = (lo + hi + 1) >> 1;
                if (frame_at<BATCH>(F, mid).cursor_begin <= gcur) lo = mid;
                else hi = mid - 1;
            }
            if (lo != f && visit_acc) {
                if (lane == 0) atomicAdd(&frame_at<BATCH>(F, f).counts[1], visit_acc);
                visit_acc = 0;
            }
            f = lo;
        }
        const Frame &fr = frame_at<BATCH>(F, f);
        const float4 *nodes = fr.nodes;
        const uint32_t n_lights = fr.n_lights;
        const uint32_t j = fr.eye_begin + (uint32_t)(gcur - fr.cursor_begin);
        Eye E;
        E.x = fr.ex[j];
        E.y = fr.ey[j];
        E.z = fr.ez[j];
        E.tau = fr.tau;
        E.scale = hrr_node_scale(fr.tau);
        const uint32_t tx = fr.px[j] % fr.tile_w, ty = fr.py[j] % fr.tile_h;
        E.r = fr.tile[ty * fr.tile_w + tx] + fr.shift_offset;
        if (n_lights == 1) {  // the root is a leaf (record 0, slot 0, in either layout)
            if (lane == 0 && fr.eye_visits) fr.eye_visits[j] = 0;
            take(fr, E, j, lane, lane == 0, light_of<W, PAIRED>(nodes, 0u, 0u), 0u);
            continue;
        }
        E.c = __brev(0u - E.r);
        // Stack: logical entries [0, S); the newest R of them are in the ring at index & mask,
        // the others in the spill area at their logical index.
        uint32_t S = 1, R = 1, visits = 0;
        uint32_t queued_n = 0;  // surviving leaves of this eye still to be taken
        if constexpr (TOP > 0) {
            const float4 *top = kTopShared ? top_s : fr.top;
            visits = head<VARIANT, BATCH>(top, E, fr, lane, j, ring, S);
            R = S;
        } else {
            if (lane == 0) ring[0] = make_uint2(0u, range_min<VARIANT>(0u, n_lights, E.r, E.c));
            __syncwarp();
        }
        if constexpr (W == 2) {
            visits += walk_pairs<VARIANT, kRing, PAIRED>(fr, E, j, lane, ring, queue, S, visits, HRR_WARP_SPILL,
                                                         Lc.spill_cap, Lc.flags);
        } else {
            while (S > 0) {
                if (visits >= n_lights) {  // each internal node is visited at most once per eye
                    if (lane == 0) atomicOr(Lc.flags, HRR_FLAG_TOPOLOGY);
                    break;
                }
                const uint32_t m = min(32u, S);
                if (R < m) {  // bring spilled entries back into the ring
                    const uint32_t fc = min(S - R, kRing / 2 - R);
                    const uint32_t base = S - R - fc;
                    const uint2 *spill = HRR_WARP_SPILL;
                    for (uint32_t k = lane; k < fc; k += 32) ring[(base + k) & kRingMask] = spill[base + k];
                    R += fc;
                    __syncwarp();
                }
                const bool active = (uint32_t)lane < m;
                uint2 e = make_uint2(0u, 0u);
                if (active) e = ring[(S - m + lane) & kRingMask];
                S -= m;
                R -= m;
                visits += m;
                __syncwarp();

                Visit<W> V;
    #pragma unroll
                for (int t = 0; t < W; ++t) {
                    V.go[t] = V.leaf[t] = false;
                    V.node[t] = V.vmin[t] = V.light[t] = 0;
                }
                if (active) visit<VARIANT>(nodes, n_lights, e.x, e.y, E, Lc.flags, V);
                // Push the surviving children as one compacted run.
                unsigned bal[W];
                uint32_t n = 0;
    #pragma unroll
                for (int t = 0; t < W; ++t) {
                    bal[t] = __ballot_sync(0xFFFFFFFFu, V.go[t]);
                    n += __popc(bal[t]);
                }
                if (n) {
                    if (R + n > kRing) {  // move the oldest resident entries to the spill area
                        const uint32_t s = (R + n - kRing + 31u) & ~31u;
                        const uint32_t base = S - R;
                        if (base + s > Lc.spill_cap) {  // cannot happen: the area holds the bound
                            if (lane == 0) atomicOr(Lc.flags, HRR_FLAG_STACK);
                            break;
                        }
                        uint2 *spill = HRR_WARP_SPILL;
                        for (uint32_t k = lane; k < s; k += 32) spill[base + k] = ring[(base + k) & kRingMask];
                        R -= s;
                        __syncwarp();
                    }
                    // Lane by lane, each lane's survivors side by side: siblings (whose records
                    // are neighbours in memory) are popped together by neighbouring lanes.
                    uint32_t pos = S;
    #pragma unroll
                    for (int t = 0; t < W; ++t) pos += __popc(bal[t] & lt);
    #pragma unroll
                    for (int t = 0; t < W; ++t) {
                        if (V.go[t]) ring[pos & kRingMask] = make_uint2(V.node[t], V.vmin[t]);
                        pos += V.go[t] ? 1u : 0u;
                    }
                    S += n;
                    R += n;
                    __syncwarp();
                }
                bool any_leaf = false;
    #pragma unroll
                for (int t = 0; t < W; ++t) any_leaf |= V.leaf[t];
                if (__any_sync(0xFFFFFFFFu, any_leaf)) {
    #pragma unroll
                    for (int t = 0; t < W; ++t) {
                        const unsigned b = __ballot_sync(0xFFFFFFFFu, V.leaf[t]);
                        if (V.leaf[t]) queue[queued_n + __popc(b & lt)] = queued<W>(e.x, (uint32_t)t, V.light[t]);
                        queued_n += __popc(b);
                    }
                    __syncwarp();
                    while (queued_n >= 32u) {
                        queued_n -= 32u;
                        take_queued<W, false>(fr, E, j, lane, queue + queued_n, 32u);
                    }
                }
            }
            if (queued_n) take_queued<W, false>(fr, E, j, lane, queue, queued_n);
        }
        if (lane == 0) {
            uint32_t *ev = frame_at<BATCH>(F, f).eye_visits;
            if (ev) ev[j] = visits;
        }
        visit_acc += visits;
    }
    if (lane == 0 && visit_acc) {
        if constexpr (BATCH) atomicAdd(&frame_at<BATCH>(F, f).counts[1], visit_acc);
        else atomicAdd(&F[0].counts[1], visit_acc);
    }
    if constexpr (!BATCH) {
        if (Lc.host) report(Lc, F[0].counts);
    }
#undef HRR_WARP_SPILL
}

// A single frame travels as a plain kernel parameter; a batch's frames as a grid-constant
// array (indexed by the frame a warp is on).
template <int VARIANT, int W, int RING, int THREADS, int TOP, bool PAIRED>
__global__ void __launch_bounds__(THREADS, min_blocks<W>(THREADS))
cull_single_kernel(const Launch Lc, const Frame fr) {
    traverse<VARIANT, false, W, RING, THREADS, TOP, PAIRED>(Lc, &fr);
}

template <int VARIANT, int W, int RING, int THREADS, int TOP, bool PAIRED>
__global__ void __launch_bounds__(THREADS, min_blocks<W>(THREADS))
cull_batch_kernel(const __grid_constant__ Launch Lc, const __grid_constant__ FrameArray<kMaxFrames> FA) {
    traverse<VARIANT, true, W, RING, THREADS, TOP, PAIRED>(Lc, FA.f);
}

}  // namespace
