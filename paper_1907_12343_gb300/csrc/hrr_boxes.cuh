// The box pass: bounding boxes, maximum intensities and height of a hierarchy whose topology
// (split, other end and parent links) is known, written into its 64-byte records and, for
// light hierarchies, into the records derived from them. Device code and its launches; the
// light builder and the triangle scenes instantiate it with their own leaves.
//
// Nodes are contiguous leaf ranges, so a box can be had two ways, and each is used where it is
// short. A block owns kBoxBlock leaves in a row and the nodes of the same numbers; a node whose
// whole range lies inside one block (all but a few in a hundred) is finished there, in shared
// memory: a thread per leaf climbs, leaving the box it carries in its parent's shared entry, and
// the second child to arrive goes on with the parent. A node that spans blocks is listed, and
// a second kernel computes its children's boxes straight from their ranges, one warp per node:
// the leaves at the range's two ends and, between them, aggregates of 32, 32^2, ... leaves that
// the first kernel leaves behind (at most 64 loads a level, all of a level in flight at once).
// Nothing waits for anything: with every node climbed to through global memory (a fence, an
// atomic and a dependent load per level) the pass was a chain of some thirty L2 round trips,
// 206 us for 2^20 lights and 67 us more for the derived records; the two kernels take 90 and
// 27 us with the derived records (refit of 2^20 lights: 640 -> 485 us; the rest is allocation).
// The first is bound by latency at 24 to 48 resident warps per SM (three blocks measured 90 us
// against 97 us for two) and by its stores, the second by its dependent loads.
#pragma once

#include <algorithm>

#include "hrr_internal.cuh"

namespace {

constexpr uint32_t kBoxBlock = 512;  // leaves, and threads, of a block
constexpr int kBoxLevels = 7;        // 32^7 > 2^31 leaves
constexpr int kSpanThreads = 256;

constexpr size_t pad256(size_t b) { return (b + 255) & ~size_t(255); }

template <typename T>
T *carve(char *&p, size_t count) {
    T *r = reinterpret_cast<T *>(p);
    p += (sizeof(T) * count + 255) & ~size_t(255);
    return r;
}

// Groups of 32^level leaves.
__host__ __device__ constexpr uint32_t box_groups(uint32_t n, int level) {
    return (uint32_t)(((uint64_t)n + (1ull << (5 * level)) - 1) >> (5 * level));
}
// Whether the groups of a level are kept: until a level has at most 64.
__host__ __device__ constexpr bool box_level(uint32_t n, int level) { return level < kBoxLevels && box_groups(n, level - 1) > 64u; }
__host__ __device__ constexpr uint32_t box_groups_total(uint32_t n) {
    uint32_t k = 0;
    for (int l = 1; box_level(n, l); ++l) k += box_groups(n, l);
    return k;
}

// What the pass works with besides the records; box_reset clears what must start cleared.
struct BoxScratch {
    uint32_t *leaf_parent, *int_parent;  // n each: parent node << 1 | which child; all ones: none
    uint32_t *child_height;              // 2n: heights of the spanning nodes' children inside blocks
    uint32_t *span;                      // n: the nodes that span blocks ...
    uint32_t *span_count;                // ... and their number
    uint32_t *root_height;
    float4 *groups;                      // 2 per group, level by level: (low, imax), (high, 0)
    uint32_t *arrived;                   // per group: parts of it that are done
};

// child_height false: the caller has 8 bytes a leaf for those itself.
constexpr size_t box_scratch_bytes(uint32_t n, bool child_height = true) {
    const size_t un = n, g = box_groups_total(n) + 1;
    return 3 * pad256(sizeof(uint32_t) * un) + (child_height ? pad256(sizeof(uint32_t) * 2 * un) : 0) + 2 * pad256(sizeof(uint32_t)) +
           pad256(2 * sizeof(float4) * g) + pad256(sizeof(uint32_t) * g);
}
inline BoxScratch carve_boxes(char *&p, uint32_t n, bool child_height = true) {
    const size_t un = n, g = box_groups_total(n) + 1;
    BoxScratch s;
    s.leaf_parent = carve<uint32_t>(p, un);
    s.int_parent = carve<uint32_t>(p, un);
    s.span = carve<uint32_t>(p, un);
    s.child_height = child_height ? carve<uint32_t>(p, 2 * un) : nullptr;
    s.span_count = carve<uint32_t>(p, 1);
    s.root_height = carve<uint32_t>(p, 1);
    s.groups = carve<float4>(p, 2 * g);
    s.arrived = carve<uint32_t>(p, g);
    return s;
}

// Leaf i's share of what must start cleared (i < n; n > number of groups), without and with the
// parent links.
__device__ __forceinline__ void box_reset_counts(const BoxScratch &s, uint32_t i, uint32_t n) {
    if (i < box_groups_total(n)) s.arrived[i] = 0u;
    if (i == 0) *s.span_count = *s.root_height = 0u;
}
__device__ __forceinline__ void box_reset(const BoxScratch &s, uint32_t i, uint32_t n) {
    s.leaf_parent[i] = s.int_parent[i] = 0xFFFFFFFFu;
    box_reset_counts(s, i, n);
}

struct Box {
    float lo[3], hi[3], m;  // corners, maximum intensity
};
__device__ __forceinline__ Box box_empty() {
    const float inf = __int_as_float(0x7f800000);
    return {{inf, inf, inf}, {-inf, -inf, -inf}, -inf};
}
__device__ __forceinline__ Box box_of(float4 a, float4 b) { return {{a.x, a.y, a.z}, {b.x, b.y, b.z}, a.w}; }
__device__ __forceinline__ void box_join(Box &x, const Box &y) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        x.lo[c] = fminf(x.lo[c], y.lo[c]);
        x.hi[c] = fmaxf(x.hi[c], y.hi[c]);
    }
    x.m = fmaxf(x.m, y.m);
}
__device__ __forceinline__ float4 box_a(const Box &b) { return make_float4(b.lo[0], b.lo[1], b.lo[2], b.m); }
__device__ __forceinline__ float4 box_b(const Box &b, uint32_t w) {
    return make_float4(b.hi[0], b.hi[1], b.hi[2], __uint_as_float(w));
}
// Floats as unsigned integers of the same order, for the warp-wide integer reductions.
__device__ __forceinline__ uint32_t ordered(float f) {
    const uint32_t u = __float_as_uint(f);
    return u ^ ((uint32_t)((int32_t)u >> 31) | 0x80000000u);
}
__device__ __forceinline__ float unordered(uint32_t u) {
    return __uint_as_float(u ^ ((uint32_t)((int32_t)~u >> 31) | 0x80000000u));
}
// The union over the warp, in every lane.
__device__ __forceinline__ Box warp_box(const Box &x) {
    Box r;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        r.lo[c] = unordered(__reduce_min_sync(0xFFFFFFFFu, ordered(x.lo[c])));
        r.hi[c] = unordered(__reduce_max_sync(0xFFFFFFFFu, ordered(x.hi[c])));
    }
    r.m = unordered(__reduce_max_sync(0xFFFFFFFFu, ordered(x.m)));
    return r;
}

// Leaves that are lights: position and intensity.
struct PointLeaves {
    static constexpr bool kOwnNodes = false;  // without derived records the nodes are a caller's array
    const float4 *pos;
    __device__ __forceinline__ Box operator()(uint32_t i) const {
        const float4 p = pos[i];
        return {{p.x, p.y, p.z}, {p.x, p.y, p.z}, p.w};
    }
};

// The groups above the blocks' own: after a block's groups of 32 are written, the last part of
// each larger group to finish reduces it (warp 0 of the block).
__device__ __forceinline__ void box_finish_groups(const BoxScratch &s, uint32_t base, uint32_t n) {
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t below = 0;  // first group of the level below
    for (int l = 2; box_level(n, l); ++l) {
        const uint32_t have = box_groups(n, l - 1), at = below + have, g = base >> (5 * l);
        uint32_t parts;
        if (l == 2) parts = min(1024u / kBoxBlock, (n - (g << 10) + kBoxBlock - 1) / kBoxBlock);
        else parts = min(32u, have - 32u * g);
        uint32_t old = 0;
        if (lane == 0) {
            __threadfence();
            old = atomicAdd(&s.arrived[at + g], 1u);
        }
        if (__shfl_sync(0xFFFFFFFFu, old, 0) + 1u != parts) return;
        __threadfence();
        Box x = box_empty();
        const uint32_t c = 32u * g + lane;
        if (c < have) x = box_of(__ldcg(&s.groups[2 * (size_t)(below + c)]), __ldcg(&s.groups[2 * (size_t)(below + c) + 1]));
        x = warp_box(x);
        if (lane == 0) {
            s.groups[2 * (size_t)(at + g)] = box_a(x);
            s.groups[2 * (size_t)(at + g) + 1] = box_b(x, 0u);
        }
        below = at;
    }
}

// The groups of 32 leaves (a warp each: `mine` is leaf g's box, empty past the last leaf).
__device__ __forceinline__ void box_groups_of_32(const BoxScratch &s, const Box &mine, uint32_t g, uint32_t n) {
    if (!box_level(n, 1)) return;
    const Box w = warp_box(mine);
    if ((g & 31u) == 0 && g < n) {
        s.groups[2 * (size_t)(g >> 5)] = box_a(w);
        s.groups[2 * (size_t)(g >> 5) + 1] = box_b(w, 0u);
        __threadfence();
    }
}

// All groups on their own, for what needs ranges' boxes before the topology is there.
template <typename LEAVES>
__global__ void __launch_bounds__(kBoxBlock) groups_kernel(LEAVES leaf, uint32_t n, BoxScratch s) {
    chain_begin();
    const uint32_t base = blockIdx.x * kBoxBlock, g = base + threadIdx.x;
    box_groups_of_32(s, g < n ? leaf(g) : box_empty(), g, n);
    __syncthreads();
    if (threadIdx.x < 32u) box_finish_groups(s, base, n);
}
template <typename LEAVES>
cudaError_t groups_enqueue(const LEAVES &leaf, uint32_t n, const BoxScratch &s, cudaStream_t st) {
    return launch_chained(groups_kernel<LEAVES>, (n + kBoxBlock - 1) / kBoxBlock, kBoxBlock, st, leaf, n, s);
}

// The union of leaves [a, b] (a <= b), by a whole warp.
template <typename LEAVES>
__device__ __forceinline__ Box box_range(const LEAVES &leaf, const BoxScratch &s, uint32_t n, uint32_t a, uint32_t b) {
    const uint32_t lane = threadIdx.x & 31u;
    Box x = box_empty();
    uint32_t lo = a, hi = b + 1u, at = 0;  // entries [lo, hi) of the level, whose first group is `at`
    for (int l = 0;; ++l) {
        const bool done = hi - lo <= 64u;
        const uint32_t lup = done ? lo + 32u : (lo + 31u) & ~31u, hdn = done ? lo + 32u : hi & ~31u;
        const uint32_t i = lo + lane, j = hdn + lane;
        const bool left = i < min(lup, hi), right = j < hi;
        if (l == 0) {
            if (left) box_join(x, leaf(i));
            if (right) box_join(x, leaf(j));
        } else {
            if (left) box_join(x, box_of(s.groups[2 * (size_t)(at + i)], s.groups[2 * (size_t)(at + i) + 1]));
            if (right) box_join(x, box_of(s.groups[2 * (size_t)(at + j)], s.groups[2 * (size_t)(at + j) + 1]));
            at += box_groups(n, l);
        }
        if (done) break;
        lo = lup >> 5;
        hi = hdn >> 5;
        if (lo >= hi) break;
    }
    return warp_box(x);
}

// 32 bytes as one 256-bit store: the records' threads are 64 or 128 bytes apart, and each store
// instruction costs a line per lane.
__device__ __forceinline__ void store32(float4 *p, const float4 &a, const float4 &b) {
    asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 :
                 : "l"(p), "f"(a.x), "f"(a.y), "f"(a.z), "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w)
                 : "memory");
}

// The four slots of a width-four record (hrr_tree::wide) from the boxes of its grandchildren
// (q[0], q[1] the children of child 0, or child 0 itself in q[0] when it is a leaf; q[2], q[3]
// of child 1) and the children's splits.
__device__ __forceinline__ void store_wide(float4 *w, const float4 (&a)[4], const float4 (&b)[4], bool leaf0, bool leaf1,
                                           uint32_t split0, uint32_t split, uint32_t split1, uint32_t other) {
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 a1 = leaf0 ? zero : a[1], b1 = leaf0 ? zero : b[1], a3 = leaf1 ? zero : a[3], b3 = leaf1 ? zero : b[3];
    store32(w, a[0], make_float4(b[0].x, b[0].y, b[0].z, __uint_as_float(split0)));
    store32(w + 2, a1, make_float4(b1.x, b1.y, b1.z, __uint_as_float(split)));
    store32(w + 4, a[2], make_float4(b[2].x, b[2].y, b[2].z, __uint_as_float(split1)));
    store32(w + 6, a3, make_float4(b3.x, b3.y, b3.z, __uint_as_float(other)));
}
// A node's record from its children's boxes. OWN: an array of the library's, which is aligned. A
// caller's array (a build without allocation) need not be aligned to more than a word: it takes
// the 256-bit stores where its address allows them, else one word at a time.
template <bool OWN>
__device__ __forceinline__ void store_record(float4 *r, float4 a0, float4 b0, float4 a1, float4 b1, uint32_t split,
                                             uint32_t other) {
    if (!OWN && ((uintptr_t)r & 31u) != 0) {
        const float v[16] = {a0.x, a0.y, a0.z, a0.w, b0.x, b0.y, b0.z, __uint_as_float(split),
                             a1.x, a1.y, a1.z, a1.w, b1.x, b1.y, b1.z, __uint_as_float(other)};
        volatile float *f = reinterpret_cast<volatile float *>(r);  // word by word: no wider store may be made of these
#pragma unroll
        for (int k = 0; k < 16; ++k) f[k] = v[k];
        return;
    }
    store32(r, a0, make_float4(b0.x, b0.y, b0.z, __uint_as_float(split)));
    store32(r + 2, a1, make_float4(b1.x, b1.y, b1.z, __uint_as_float(other)));
}

// A node's paired record (hrr_tree::pairs).
__device__ __forceinline__ void store_pairs(float4 *r, float4 a0, float4 b0, float4 a1, float4 b1, uint32_t split,
                                            uint32_t other) {
    store32(r, make_float4(-a0.x, -a1.x, -a0.y, -a1.y), make_float4(-a0.z, -a1.z, -b0.x, -b1.x));
    store32(r + 2, make_float4(-b0.y, -b1.y, -b0.z, -b1.z),
            make_float4(a0.w, a1.w, __uint_as_float(split), __uint_as_float(other)));
}

// The records derived from the binary ones, or none (scenes, builds into caller's arrays); pairs
// alone may be missing. DERIVED below: 0 none, 1 the top slots and the width-four records, 2 all.
struct Derived {
    float4 *pairs, *wide;
};

// The nodes inside blocks, the groups, the list of spanning nodes.
template <int DERIVED, typename LEAVES>
__global__ void __launch_bounds__(kBoxBlock, 3) box_kernel(LEAVES leaf, uint32_t n, hrr_node *nodes, Derived der,
                                                        BoxScratch s, bool have_groups, unsigned long long *flags) {
    __shared__ float4 sa[2][kBoxBlock], sb[2][kBoxBlock];  // child: (low, imax), (high, height)
    __shared__ uint32_t arrived[kBoxBlock], up[kBoxBlock], cut[kBoxBlock];
    __shared__ bool inside[kBoxBlock];
    chain_begin();
    if (*(volatile unsigned long long *)flags & (HRR_FLAG_NONFINITE | HRR_FLAG_UNSORTED)) return;  // set before the launch
    const uint32_t t = threadIdx.x, base = blockIdx.x * kBoxBlock, g = base + t;
    uint32_t split = 0, other = 0, first = 0, last = 0;
    bool whole = false;  // node g exists and lies inside the block
    if (g < n - 1) {
        split = nodes[g].split;
        other = nodes[g].other_end;
        first = min(g, other);
        last = max(g, other);
        if (last >= n || split < first || split >= last) atomicOr(flags, HRR_FLAG_TOPOLOGY);
        else if (first >= base && last - base < kBoxBlock) whole = true;
        else s.span[atomicAdd(s.span_count, 1u)] = g;
    }
    arrived[t] = 0;
    inside[t] = whole;
    cut[t] = split;
    up[t] = whole ? s.int_parent[g] : 0xFFFFFFFFu;
    const Box mine = g < n ? leaf(g) : box_empty();
    if (!have_groups) box_groups_of_32(s, mine, g, n);
    __syncthreads();
    if (!have_groups && t < 32u) box_finish_groups(s, base, n);

    if (g < n) {
        Box x = mine;
        uint32_t h = 0, code = s.leaf_parent[g];
        for (;;) {
            const uint32_t node = code >> 1, c = code & 1u, k = node - base;
            if (code == 0xFFFFFFFFu || node >= n - 1) {  // every link is set by the topology
                atomicOr(flags, HRR_FLAG_TOPOLOGY);
                break;
            }
            if (k >= kBoxBlock || !inside[k]) {  // the parent spans blocks
                s.child_height[2 * (size_t)node + c] = h;
                break;
            }
            sa[c][k] = box_a(x);
            sb[c][k] = box_b(x, h);
            __threadfence_block();
            if (atomicAdd(&arrived[k], 1u) != 1u) break;  // the sibling finishes the node
            __threadfence_block();
            x = box_of(sa[0][k], sb[0][k]);
            box_join(x, box_of(sa[1][k], sb[1][k]));
            h = 1u + max(__float_as_uint(sb[0][k].w), __float_as_uint(sb[1][k].w));
            if (node == 0) {
                *s.root_height = h;
                break;
            }
            code = up[k];
        }
    }
    __syncthreads();
    if (whole && arrived[t] == 2u) {
        const float4 a0 = sa[0][t], b0 = sb[0][t], a1 = sa[1][t], b1 = sb[1][t];
        store_record<(DERIVED > 0 || LEAVES::kOwnNodes)>(reinterpret_cast<float4 *>(nodes) + 4 * (size_t)g, a0, b0, a1, b1, split, other);
        if (DERIVED) {  // the children's entries are in the block too
            const bool leaf0 = first == split, leaf1 = split + 1u == last;
            const uint32_t k0 = leaf0 ? t : split - base, k1 = leaf1 ? t : split + 1u - base;
            const float4 a[4] = {sa[0][k0], sa[1][k0], leaf1 ? a1 : sa[0][k1], sa[1][k1]};
            const float4 b[4] = {sb[0][k0], sb[1][k0], leaf1 ? b1 : sb[0][k1], sb[1][k1]};
            if (DERIVED > 1) store_pairs(der.pairs + 4 * (size_t)hrr_node_slot(g, other), a0, b0, a1, b1, split, other);
            store_wide(der.wide + 8 * (size_t)g, a, b, leaf0, leaf1, leaf0 ? split : cut[k0], split, leaf1 ? last : cut[k1],
                       other);
        }
    }
}

// Node and range at heap slot s of the top (the bits of s + 1 below its leading one, high to
// low: 0 = child 0, 1 = child 1). A slot below a leaf is empty; a record whose split is outside
// its node's range (not produced by the builder) empties the slots below it.
__device__ __forceinline__ uint32_t top_walk(uint32_t s, const hrr_node *nodes, uint32_t n, uint32_t &first,
                                             uint32_t &last, uint32_t &node) {
    first = last = node = 0;
    if (n <= 1) return HRR_TOP_EMPTY;
    const uint32_t path = s + 1u;
    uint32_t kind = HRR_TOP_INTERNAL;
    last = n - 1u;
    for (int b = 30 - __clz(path); b >= 0; --b) {
        const uint32_t split = kind == HRR_TOP_INTERNAL ? nodes[node].split : 0u;
        if (kind != HRR_TOP_INTERNAL || split < first || split >= last) {
            first = last = node = 0;
            return HRR_TOP_EMPTY;
        }
        if (((path >> b) & 1u) == 0u) last = node = split;
        else first = node = split + 1u;
        kind = first == last ? HRR_TOP_LEAF : HRR_TOP_INTERNAL;
    }
    return kind;
}

// The nodes that span blocks (a warp each), the top slots (a warp each), and the height (a
// thread per spanning node: its depth by the parent links, plus the heights of its children
// inside blocks). Blocks [0, box_blocks) do the first two, the others the last.
template <int DERIVED, typename LEAVES>
__global__ void __launch_bounds__(kSpanThreads) span_kernel(LEAVES leaf, uint32_t n, hrr_node *nodes, Derived der,
                                                            BoxScratch s, uint32_t box_blocks,
                                                            unsigned long long *flags) {
    chain_begin();
    if (*(volatile unsigned long long *)flags & (HRR_FLAG_NONFINITE | HRR_FLAG_UNSORTED)) return;
    const uint32_t count = *s.span_count;
    if (blockIdx.x >= box_blocks) {
        uint32_t h = 0;
        for (uint32_t k = (blockIdx.x - box_blocks) * kSpanThreads + threadIdx.x; k < count;
             k += (gridDim.x - box_blocks) * kSpanThreads) {
            const uint32_t g = s.span[k], split = nodes[g].split, other = nodes[g].other_end;
            const uint32_t first = min(g, other), last = max(g, other);
            uint32_t below = 0;
            const bool in0 = first / kBoxBlock == split / kBoxBlock, in1 = (split + 1u) / kBoxBlock == last / kBoxBlock;
            if (in0) below = s.child_height[2 * (size_t)g];
            if (in1) below = max(below, s.child_height[2 * (size_t)g + 1]);
            if (!in0 && !in1) continue;
            uint32_t depth = 1, up = g;
            while (up != 0u && depth < 4096u) {  // no hierarchy is that deep
                up = s.int_parent[up] >> 1;
                ++depth;
                if (up >= n - 1) break;
            }
            if (up != 0u) atomicOr(flags, HRR_FLAG_TOPOLOGY);
            h = max(h, depth + below);
        }
        h = __reduce_max_sync(0xFFFFFFFFu, h);
        if ((threadIdx.x & 31) == 0 && h) atomicMax(s.root_height, h);
        return;
    }
    const uint32_t lane = threadIdx.x & 31u, warps = box_blocks * (kSpanThreads / 32);
    const uint32_t tops = DERIVED ? HRR_TOP_SLOTS : 0u;
    float4 *top = reinterpret_cast<float4 *>(nodes) + 4 * (size_t)(n > 1 ? n - 1 : 1);
    for (uint32_t k = blockIdx.x * (kSpanThreads / 32) + (threadIdx.x >> 5); k < count + tops; k += warps) {
        if (DERIVED && k < tops) {  // box, range, node number and kind; the root's box is not stored
            uint32_t first, last, node;
            const uint32_t kind = top_walk(k, nodes, n, first, last, node);
            Box x = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, 0.f};
            if (kind != HRR_TOP_EMPTY && k > 0) x = box_range(leaf, s, n, first, last);
            if (lane == 0) {
                top[3 * k] = box_a(x);
                top[3 * k + 1] = box_b(x, first);
                top[3 * k + 2] = make_float4(__uint_as_float(last), __uint_as_float(node), __uint_as_float(kind), 0.f);
            }
            continue;
        }
        const uint32_t g = s.span[k - tops], split = nodes[g].split, other = nodes[g].other_end;
        const uint32_t first = min(g, other), last = max(g, other);
        if (!DERIVED) {
            const Box x0 = box_range(leaf, s, n, first, split), x1 = box_range(leaf, s, n, split + 1u, last);
            if (lane == 0)
                store_record<LEAVES::kOwnNodes>(reinterpret_cast<float4 *>(nodes) + 4 * (size_t)g, box_a(x0), box_b(x0, 0u),
                                                box_a(x1), box_b(x1, 0u), split, other);
            continue;
        }
        // the grandchildren's boxes; the children's are their unions
        const bool leaf0 = first == split, leaf1 = split + 1u == last;
        const uint32_t split0 = leaf0 ? split : nodes[split].split, split1 = leaf1 ? last : nodes[split + 1u].split;
        if (split0 < first || split0 > split || split1 < split + 1u || split1 > last) {
            if (lane == 0) atomicOr(flags, HRR_FLAG_TOPOLOGY);
            continue;
        }
        Box q[4] = {box_range(leaf, s, n, first, split0), box_empty(), box_range(leaf, s, n, split + 1u, split1), box_empty()};
        if (split0 < split) q[1] = box_range(leaf, s, n, split0 + 1u, split);
        if (split1 < last) q[3] = box_range(leaf, s, n, split1 + 1u, last);
        if (lane == 0) {
            Box x0 = q[0], x1 = q[2];
            box_join(x0, q[1]);
            box_join(x1, q[3]);
            store_record<true>(reinterpret_cast<float4 *>(nodes) + 4 * (size_t)g, box_a(x0), box_b(x0, 0u), box_a(x1),
                               box_b(x1, 0u), split, other);
            const float4 a[4] = {box_a(q[0]), box_a(q[1]), box_a(q[2]), box_a(q[3])};
            const float4 b[4] = {box_b(q[0], 0u), box_b(q[1], 0u), box_b(q[2], 0u), box_b(q[3], 0u)};
            if (DERIVED > 1)
                store_pairs(der.pairs + 4 * (size_t)hrr_node_slot(g, other), box_a(x0), box_b(x0, 0u), box_a(x1),
                            box_b(x1, 0u), split, other);
            store_wide(der.wide + 8 * (size_t)g, a, b, leaf0, leaf1, split0, split, split1, other);
        }
    }
}

// Both kernels, for n >= 2 leaves: the records of `nodes` and, unless `der` is empty, the derived
// records (the top slots after the records, the paired and width-four records); *s.root_height gets the height.
// have_groups: groups_enqueue has run on the same leaves.
template <typename LEAVES>
cudaError_t boxes_enqueue(const LEAVES &leaf, uint32_t n, hrr_node *nodes, const Derived &der, const BoxScratch &s,
                          unsigned long long *flags, cudaStream_t st, bool have_groups = false) {
    const unsigned blocks = (n + kBoxBlock - 1) / kBoxBlock;
    const unsigned bb = std::min(608u, 8u + blocks), hb = std::min(152u, 1u + blocks / 16u);
    const auto run = [&](auto box, auto span) {
        launch_chained(box, blocks, kBoxBlock, st, leaf, n, nodes, der, s, have_groups, flags);
        launch_chained(span, bb + hb, kSpanThreads, st, leaf, n, nodes, der, s, bb, flags);
    };
    if (der.pairs) run(box_kernel<2, LEAVES>, span_kernel<2, LEAVES>);
    else if (der.wide) run(box_kernel<1, LEAVES>, span_kernel<1, LEAVES>);
    else run(box_kernel<0, LEAVES>, span_kernel<0, LEAVES>);
    return cudaGetLastError();
}

}  // namespace
