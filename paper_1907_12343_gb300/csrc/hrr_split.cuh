// Cost-driven topology over the Morton order.
//
// A top-down build: every range [f, l] splits at the k
// (children [f, k], [k+1, l]) that minimises C(k) = w(L) + w(R) over every k in [f, l),
//     w(X) = u^2 ((A + 0.1 P) + 1e-4) c sqrt(c),
// with c the child's light count, u its maximum intensity (clamped at 0) times the
// reciprocal of the range's, A = dx dy + dy dz + dz dx and P = dx + dy + dz of its box; in
// float with every operation rounded separately (no contraction; sqrt and the reciprocal
// correctly rounded). A non-finite C never wins; ties go to the least |c_L - c_R|, then
// the least k. Ranges deeper than the cost depth (root = 1)
// take the radix split, which bounds the height. Node numbering and parent links are those
// of topology_kernel, so the box pass finishes the hierarchy unchanged.
//
// Boxes and maxima are min / max reductions, exact in any order, so parallel scans give
// the same prefix and suffix aggregates at every k as a serial sweep, and the same costs
// bit for bit. Three kinds of ranges:
//   * more than 1024 lights: one kernel per level, tiles of 1024 lights, a block per tile and a
//     run of 4 lights per thread. What lies before and after a tile in its range comes from the
//     aggregates of 32^k lights (box_range), so no pass collects tile totals first; the last tile
//     of a range to finish picks its split. Ranges and tiles are counted on the device, so the
//     levels are launched one behind the other, a batch between two looks at the counts.
//   * 33 to 1024 lights: one block builds the whole subtree from shared memory; a split of more
//     than 256 lights takes the block, of more than 32 a warp (runs of 2, 4 or 8 lights per lane),
//     and the rest are subtrees of a warp each.
//   * up to 32 lights: one warp builds the whole subtree, a light per lane.
// With one level of every size per pass, four kernels and a host round trip each, the build of
// 2^20 lights took 1843 us, now 980 to 1000 us (a whole call; its device time is 0.93 ms). What is left is instructions (the subtrees of 33 to 1024
// lights and below: 212 and 132 us) and the latency of about twenty levels (8 to 20 us each).
#pragma once

#include <algorithm>

#include "hrr_boxes.cuh"
#include "hrr_internal.cuh"
#include "hrr_order.cuh"

namespace {

constexpr int kSplitThreads = 256;  // block size of the level and subtree kernels
constexpr int kTileRun = 4;         // lights per thread in a tile
constexpr uint32_t kSegTile = kSplitThreads * kTileRun;
constexpr int kMidRun = 8;          // lights per lane for ranges of 33..256 lights, per thread above
constexpr uint32_t kSmallMax = 32, kMidMax = 32 * kMidRun;
constexpr int kSubThreads = 128;    // block size of the kernel for 33..kSubMax lights
constexpr uint32_t kSubMax = kSubThreads * kMidRun;
static_assert(kSubMax == kSegTile, "a tiled range has two tiles or more");
constexpr uint32_t kNoSplit = 0xFFFFFFFFu;

struct Seg {
    uint32_t node, f, l, depth;
};

using Agg = Box;  // box and maximum intensity of a set of lights

struct Best {  // a candidate split, ordered by (c, d, k)
    float c;
    uint32_t d, k;
};

// Where splits are recorded and the ranges they leave are listed: those of more than kSubMax
// lights for the next level, the others for the kernels that finish them (they are disjoint,
// so the lists hold n / 2 ranges of two lights or more, n / 33 of more than 32).
struct SplitOut {
    hrr_node *nodes;
    uint32_t *leaf_parent, *int_parent;
    uint32_t cost_depth;
    Seg *small, *sub, *radix;        // up to 32, up to kSubMax, below the cost depth
    uint32_t *counts;                // [0] small, [1] sub, [2] radix
    Seg *big;                        // the next level's
    uint32_t *big_t0;                // first tile of each (increasing)
    unsigned long long *big_count;   // (ranges << 32) | tiles
};

__device__ __forceinline__ Agg agg_empty() { return box_empty(); }
__device__ __forceinline__ Agg agg_of(float4 p) { return {{p.x, p.y, p.z}, {p.x, p.y, p.z}, p.w}; }
__device__ __forceinline__ Agg agg_join(const Agg &a, const Agg &b) {
    Agg r = a;
    box_join(r, b);
    return r;
}
__device__ __forceinline__ Agg agg_shfl(const Agg &a, int delta, bool up) {
    Agg r;
    for (int c = 0; c < 3; ++c) {
        r.lo[c] = up ? __shfl_up_sync(0xFFFFFFFFu, a.lo[c], delta) : __shfl_down_sync(0xFFFFFFFFu, a.lo[c], delta);
        r.hi[c] = up ? __shfl_up_sync(0xFFFFFFFFu, a.hi[c], delta) : __shfl_down_sync(0xFFFFFFFFu, a.hi[c], delta);
    }
    r.m = up ? __shfl_up_sync(0xFFFFFFFFu, a.m, delta) : __shfl_down_sync(0xFFFFFFFFu, a.m, delta);
    return r;
}
// w(X) of a child of c lights, given the reciprocal of the range's maximum intensity
__device__ __forceinline__ float child_cost(const Agg &x, float inv, uint32_t c) {
    const float u = __fmul_rn(fmaxf(x.m, 0.f), inv);
    const float dx = __fsub_rn(x.hi[0], x.lo[0]), dy = __fsub_rn(x.hi[1], x.lo[1]), dz = __fsub_rn(x.hi[2], x.lo[2]);
    const float a = __fadd_rn(__fadd_rn(__fmul_rn(dx, dy), __fmul_rn(dy, dz)), __fmul_rn(dz, dx));
    const float p = __fadd_rn(__fadd_rn(dx, dy), dz);
    const float g = __fadd_rn(__fadd_rn(a, __fmul_rn(0.1f, p)), 1e-4f);
    const float cf = __uint2float_rn(c);
    return __fmul_rn(__fmul_rn(__fmul_rn(u, u), g), __fmul_rn(cf, __fsqrt_rn(cf)));
}

// Reciprocal of a range's maximum intensity m: 0 for a dark range, and a maximum below the
// smallest normal float counts as that float.
__device__ __forceinline__ float range_inv(float m) {
    const float mx = fmaxf(m, 0.f);
    return mx > 0.f ? __fdiv_rn(1.f, fmaxf(mx, __int_as_float(0x00800000))) : 0.f;
}

// C(k) for children of cl and cr lights, given range_inv of the range's maximum (the larger
// of the children's)
__device__ __forceinline__ float split_cost(const Agg &L, const Agg &R, uint32_t cl, uint32_t cr, float inv) {
    return __fadd_rn(child_cost(L, inv, cl), child_cost(R, inv, cr));
}

__device__ __forceinline__ Best best_none() { return {__int_as_float(0x7f800000), kNoSplit, kNoSplit}; }
// o < b in (cost, |c_L - c_R|, k) order; a NaN cost never wins
__device__ __forceinline__ void best_take(Best &b, const Best &o) {
    if (o.c < b.c || (o.c == b.c && (o.d < b.d || (o.d == b.d && o.k < b.k)))) b = o;
}
__device__ __forceinline__ Best warp_best(Best b) {  // the warp's best, in lane 0
    for (int d = 16; d > 0; d >>= 1) {
        const Best o = {__shfl_down_sync(0xFFFFFFFFu, b.c, d), __shfl_down_sync(0xFFFFFFFFu, b.d, d),
                        __shfl_down_sync(0xFFFFFFFFu, b.k, d)};
        best_take(b, o);
    }
    return b;
}
// The block's best, in thread 0; sh holds one entry per warp.
template <int THREADS>
__device__ __forceinline__ Best block_best(Best b, Best *sh) {
    b = warp_best(b);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = b;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < THREADS / 32; ++w) best_take(b, sh[w]);
    __syncthreads();
    return b;
}

// Exclusive scans over the lanes of a warp: the aggregates of lanes [0, lane) and (lane, 31].
__device__ __forceinline__ void warp_scans(const Agg &x, Agg &before, Agg &after) {
    const int lane = threadIdx.x & 31;
    Agg pre = x, suf = x;
    for (int d = 1; d < 32; d <<= 1) {
        const Agg u = agg_shfl(pre, d, true), v = agg_shfl(suf, d, false);
        if (lane >= d) pre = agg_join(pre, u);
        if (lane + d < 32) suf = agg_join(suf, v);
    }
    before = agg_shfl(pre, 1, true);
    after = agg_shfl(suf, 1, false);
    if (lane == 0) before = agg_empty();
    if (lane == 31) after = agg_empty();
}

// Exclusive scans over the threads of a block; sh holds one entry per warp.
template <int THREADS>
__device__ __forceinline__ void block_scans(const Agg &x, Agg &before, Agg &after, Agg *sh) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    Agg wb, wa;
    warp_scans(x, wb, wa);
    if (lane == 31) sh[w] = agg_join(wb, x);
    __syncthreads();
    Agg bb = agg_empty(), ba = agg_empty();
    for (int v = 0; v < THREADS / 32; ++v) {
        const Agg s = sh[v];
        if (v < w) bb = agg_join(bb, s);
        if (v > w) ba = agg_join(ba, s);
    }
    before = agg_join(bb, wb);
    after = agg_join(wa, ba);
    __syncthreads();
}

// The lights [a, min(a + R, end)) of a thread's run; returns their count.
template <int R>
__device__ __forceinline__ uint32_t load_run(const float4 *spos, uint32_t a, uint32_t end, float4 (&p)[R]) {
    const uint32_t cnt = a < end ? min((uint32_t)R, end - a) : 0u;
#pragma unroll
    for (int i = 0; i < R; ++i) p[i] = (uint32_t)i < cnt ? spos[a + i] : make_float4(0.f, 0.f, 0.f, 0.f);
    return cnt;
}
template <int R>
__device__ __forceinline__ Agg run_agg(const float4 (&p)[R], uint32_t cnt) {
    Agg x = agg_empty();
#pragma unroll
    for (int i = 0; i < R; ++i)
        if ((uint32_t)i < cnt) x = agg_join(x, agg_of(p[i]));
    return x;
}
// Every split k = a + i (k < l) of a run, given the aggregates of [f, a) and of the lights
// of [f, l] after the run.
template <int R>
__device__ __forceinline__ void run_best(const float4 (&p)[R], uint32_t cnt, uint32_t a, const Agg &before,
                                         const Agg &after, uint32_t f, uint32_t l, Best &b) {
    Agg suf[R + 1];  // suf[i]: lights a + i .. of the run, then the rest of the range
    suf[R] = after;
#pragma unroll
    for (int i = R - 1; i >= 0; --i) suf[i] = (uint32_t)i < cnt ? agg_join(agg_of(p[i]), suf[i + 1]) : suf[i + 1];
    const float inv = range_inv(fmaxf(before.m, suf[0].m));  // the same for every split of the range
    Agg pre = before;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        if ((uint32_t)i < cnt) {
            pre = agg_join(pre, agg_of(p[i]));
            const uint32_t k = a + i;
            if (k < l) {
                const uint32_t cl = k - f + 1, cr = l - k;
                best_take(b, {split_cost(pre, suf[i + 1], cl, cr, inv), cl > cr ? cl - cr : cr - cl, k});
            }
        }
    }
}

// The best split in runs of R lights per lane of a warp (or thread of a block, SCAN giving the
// aggregates before and after each run): `lights` holds the range's, in shared memory. Runs of
// more than 4 are taken 4 at a time, with the other lights of the run joined to what lies before
// and after, so that few suffix aggregates are held at once.
template <int R, typename SCAN>
__device__ __forceinline__ Best runs_best(const Seg &g, const float4 *lights, uint32_t lane, const SCAN &scan) {
    constexpr int C = R < 4 ? R : 4, N = R / C;  // chunks of C lights
    const uint32_t a = lane * R, m = g.l - g.f + 1;
    Agg part[N], all = agg_empty();
#pragma unroll
    for (int k = 0; k < N; ++k) {
        float4 p[C];
        const uint32_t cnt = load_run<C>(lights, a + k * C, m, p);
        part[k] = run_agg<C>(p, cnt);
        all = agg_join(all, part[k]);
    }
    Agg before, after;
    scan(all, before, after);
    Best b = best_none();
#pragma unroll
    for (int k = 0; k < N; ++k) {
        Agg left = before, right = after;
#pragma unroll
        for (int j = 0; j < N; ++j) {
            if (j < k) left = agg_join(left, part[j]);
            if (j > k) right = agg_join(right, part[j]);
        }
        float4 p[C];
        const uint32_t cnt = load_run<C>(lights, a + k * C, m, p);
        run_best<C>(p, cnt, g.f + a + k * C, left, right, g.f, g.l, b);
    }
    return b;
}

// Radix split of [f, l]: the last k whose ordering key (Morton key, position) has a 0 at
// the highest bit where the keys of f and l differ (binary search; the digit is sorted).
__device__ uint32_t radix_split(const uint64_t *__restrict__ keys, uint32_t f, uint32_t l) {
    const uint64_t kf = keys[f], kl = keys[l];
    uint32_t lo = f, hi = l;  // digit(lo) = 0, digit(hi) = 1
    if (kf != kl) {
        const int bit = 63 - __clzll((long long)(kf ^ kl));
        while (hi - lo > 1) {
            const uint32_t mid = lo + (hi - lo) / 2;
            if ((keys[mid] >> bit) & 1ull) hi = mid; else lo = mid;
        }
    } else {
        const int bit = 31 - __clz(f ^ l);
        while (hi - lo > 1) {
            const uint32_t mid = lo + (hi - lo) / 2;
            if ((mid >> bit) & 1u) hi = mid; else lo = mid;
        }
    }
    return lo;
}

// Record the split s of range g: the node's record and its children's parent links.
__device__ __forceinline__ void record_split(const Seg &g, uint32_t s, const SplitOut &o) {
    o.nodes[g.node].split = s;
    o.nodes[g.node].other_end = g.node == g.f ? g.l : g.f;
    const uint32_t code = g.node << 1;
    if (s == g.f) o.leaf_parent[s] = code; else o.int_parent[s] = code;
    if (s + 1 == g.l) o.leaf_parent[s + 1] = code | 1u; else o.int_parent[s + 1] = code | 1u;
}

// Record the split s of range g and list its internal children.
__device__ void commit_split(const Seg &g, uint32_t s, const SplitOut &o) {
    if (s == kNoSplit) s = g.f;  // no finite cost: non-finite lights, which fail the build
    record_split(g, s, o);
    const Seg kids[2] = {{s, g.f, s, g.depth + 1}, {s + 1, s + 1, g.l, g.depth + 1}};
    for (int c = 0; c < 2; ++c) {
        const Seg &k = kids[c];
        if (k.f == k.l) continue;
        const uint32_t m = k.l - k.f + 1;
        if (k.depth > o.cost_depth) {
            o.radix[atomicAdd(&o.counts[2], 1u)] = k;
        } else if (m <= kSmallMax) {
            o.small[atomicAdd(&o.counts[0], 1u)] = k;
        } else if (m <= kSubMax) {
            o.sub[atomicAdd(&o.counts[1], 1u)] = k;
        } else {
            const unsigned long long old = atomicAdd(o.big_count, (1ull << 32) | ((m + kSegTile - 1) / kSegTile));
            const uint32_t i = (uint32_t)(old >> 32);
            o.big[i] = k;
            o.big_t0[i] = (uint32_t)old;
        }
    }
}

// Ranges below the cost depth: the radix tree over each range's own keys, every node of it on
// its own as in topology_kernel (node i's range starts or ends at i; the range's root has the
// number that its parent gave it). Blocks are dealt out evenly over the ranges.
// Nothing is done on keys that are not sorted (the build starts over, or fails), whose prefix
// lengths can give a split outside its range; the kernels of the cost splits read no keys but in
// searches that end inside a range.
__global__ void __launch_bounds__(kSplitThreads) radix_subtrees_kernel(const uint64_t *__restrict__ keys, SplitOut o,
                                                                       const unsigned long long *flags) {
    chain_begin();
    const uint32_t count = o.counts[2];
    if (count == 0 || (*flags & HRR_FLAG_UNSORTED)) return;
    const uint32_t per = max(1u, gridDim.x / count);  // blocks per range
    for (uint32_t w = blockIdx.x; w < per * count; w += gridDim.x) {
        const Seg g = o.radix[w / per];
        for (uint32_t i = g.f + (w % per) * kSplitThreads + threadIdx.x; i < g.l; i += per * kSplitThreads) {
            uint32_t first, last, split;
            radix_node(keys, g.f, g.l, i, first, last, split);
            const uint32_t node = i == g.f ? g.node : i;
            record_split({node, first, last, 0u}, split, o);
        }
    }
}

// Ranges of up to 32 lights: one warp builds the whole subtree, one level of it per
// iteration. Lane j holds light f0 + j and the range of the level that holds it; scans and
// the reduction to the range's first lane are segmented by those ranges.
__device__ __forceinline__ void subtree_warp(const Seg &g0, const float4 *lights /* of the range */,
                                             const uint64_t *__restrict__ keys, const SplitOut &o) {
    const int lane = threadIdx.x & 31;
    const uint32_t i = g0.f + (uint32_t)lane;
    const bool valid = i <= g0.l;
    const Agg self = valid ? agg_of(lights[lane]) : agg_empty();
    Seg g = valid ? g0 : Seg{i, i, i, 0u};  // lanes past the range: a closed range of their own
    // a range of at most 32 lights is at most 31 levels deep
    for (int level = 0; level < 32 && __any_sync(0xFFFFFFFFu, g.l > g.f); ++level) {
        const int lf = (int)(g.f - g0.f), ll = (int)(g.l - g0.f);  // this lane's range, as lanes
        const int most = (int)__reduce_max_sync(0xFFFFFFFFu, (unsigned)(ll - lf));  // scans reach no further
        Agg pre = self, suf = self;  // inclusive scans within the range
        for (int d = 1; d <= most; d <<= 1) {
            const Agg u = agg_shfl(pre, d, true), v = agg_shfl(suf, d, false);
            if (lane - d >= lf) pre = agg_join(pre, u);
            if (lane + d <= ll) suf = agg_join(suf, v);
        }
        const Agg right = agg_shfl(suf, 1, false);  // [i + 1, l] for i < l
        Best b = best_none();
        if (lane < ll) {
            const uint32_t cl = i - g.f + 1, cr = g.l - i;
            b = {split_cost(pre, right, cl, cr, range_inv(fmaxf(pre.m, right.m))), cl > cr ? cl - cr : cr - cl, i};
        }
        for (int d = 1; d <= most; d <<= 1) {  // the range's best split, in its first lane
            const Best ob = {__shfl_down_sync(0xFFFFFFFFu, b.c, d), __shfl_down_sync(0xFFFFFFFFu, b.d, d),
                             __shfl_down_sync(0xFFFFFFFFu, b.k, d)};
            if (lane + d <= ll) best_take(b, ob);
        }
        uint32_t s = 0;
        if (lane == lf && ll > lf) {
            s = g.depth <= o.cost_depth ? (b.k == kNoSplit ? g.f : b.k) : radix_split(keys, g.f, g.l);
            record_split(g, s, o);
        }
        s = __shfl_sync(0xFFFFFFFFu, s, lf);
        if (ll > lf) g = i <= s ? Seg{s, g.f, s, g.depth + 1} : Seg{s + 1, s + 1, g.l, g.depth + 1};
    }
}

__global__ void __launch_bounds__(kSplitThreads, 5) subtree_kernel(const float4 *__restrict__ spos,
                                                                const uint64_t *__restrict__ keys, SplitOut o) {
    chain_begin();
    const uint32_t count = o.counts[0];
    for (uint32_t w = (blockIdx.x * kSplitThreads + threadIdx.x) >> 5; w < count; w += gridDim.x * (kSplitThreads / 32)) {
        const Seg g = o.small[w];
        subtree_warp(g, spos + g.f, keys, o);
    }
}

// Ranges of 33 to kSubMax lights: a block each, the lights in shared memory. What it leaves of up
// to 32 lights goes to subtree_kernel's list.
__global__ void __launch_bounds__(kSubThreads, 7) sub_kernel(const float4 *__restrict__ spos,
                                                          SplitOut o) {
    constexpr uint32_t kWarps = kSubThreads / 32;
    __shared__ float4 pos[kSubMax];
    __shared__ Seg wide[2][4], mid[2][kSubMax / (kSmallMax + 1) + 1], small[kSubMax / 2];
    __shared__ uint32_t n_wide[2], n_mid[2], n_small, small_at;
    __shared__ Agg sh[kWarps];
    __shared__ Best shb[kWarps];
    const uint32_t t = threadIdx.x, warp = t >> 5, lane = t & 31u;
    chain_begin();
    const uint32_t count = o.counts[1];
    // list a range of this block's (or below the cost depth) after its parent's split is known
    auto split_done = [&](const Seg &g, uint32_t s, uint32_t q) {
        if (s == kNoSplit) s = g.f;
        record_split(g, s, o);
        const Seg kids[2] = {{s, g.f, s, g.depth + 1}, {s + 1, s + 1, g.l, g.depth + 1}};
        for (int c = 0; c < 2; ++c) {
            const Seg &k = kids[c];
            const uint32_t m = k.l - k.f + 1;
            if (m == 1) continue;
            if (k.depth > o.cost_depth) o.radix[atomicAdd(&o.counts[2], 1u)] = k;
            else if (m <= kSmallMax) small[atomicAdd(&n_small, 1u)] = k;
            else if (m <= kMidMax) mid[q][atomicAdd(&n_mid[q], 1u)] = k;
            else wide[q][atomicAdd(&n_wide[q], 1u)] = k;
        }
    };
    for (uint32_t r = blockIdx.x; r < count; r += gridDim.x) {
        const Seg root = o.sub[r];
        const uint32_t m = root.l - root.f + 1;
        for (uint32_t i = t; i < m; i += kSubThreads) pos[i] = spos[root.f + i];
        if (t == 0) {
            n_wide[0] = m > kMidMax;
            n_mid[0] = m <= kMidMax;
            n_wide[1] = n_mid[1] = n_small = 0;
            if (m > kMidMax) wide[0][0] = root;
            else mid[0][0] = root;
        }
        __syncthreads();
        uint32_t q = 0;  // list in use; the other one is filled
        while (n_wide[q] | n_mid[q]) {
            const uint32_t nw = n_wide[q], nm = n_mid[q];
            for (uint32_t k = 0; k < nw; ++k) {  // the block, 8 lights per thread
                const Seg g = wide[q][k];
                Best b = runs_best<kMidRun>(g, pos + (g.f - root.f), t, [&](const Agg &x, Agg &before, Agg &after) {
                    block_scans<kSubThreads>(x, before, after, sh);
                });
                b = block_best<kSubThreads>(b, shb);
                if (t == 0) split_done(g, b.k, q ^ 1u);
            }
            for (uint32_t k = warp; k < nm; k += kWarps) {  // a warp each, as few lights per lane as hold it
                const Seg g = mid[q][k];
                const uint32_t size = g.l - g.f + 1;
                const float4 *lights = pos + (g.f - root.f);
                const auto scan = [](const Agg &x, Agg &before, Agg &after) { warp_scans(x, before, after); };
                Best b = size <= 64 ? runs_best<2>(g, lights, lane, scan)
                                    : size <= 128 ? runs_best<4>(g, lights, lane, scan)
                                                  : runs_best<kMidRun>(g, lights, lane, scan);
                b = warp_best(b);
                if (lane == 0) split_done(g, b.k, q ^ 1u);
            }
            __syncthreads();
            if (t == 0) n_wide[q] = n_mid[q] = 0;
            q ^= 1u;
            __syncthreads();
        }
        if (t == 0 && n_small) small_at = atomicAdd(&o.counts[0], n_small);
        __syncthreads();
        for (uint32_t k = t; k < n_small; k += kSubThreads) o.small[small_at + k] = small[k];
        __syncthreads();  // before the lists and lights are refilled
    }
}

// The big range holding tile t: the last i with big_t0[i] <= t.
__device__ __forceinline__ uint32_t range_of_tile(const uint32_t *big_t0, uint32_t n_big, uint32_t t) {
    uint32_t lo = 0, hi = n_big;
    while (hi - lo > 1) {
        const uint32_t mid = lo + (hi - lo) / 2;
        if (big_t0[mid] <= t) lo = mid; else hi = mid;
    }
    return lo;
}

// The root's place in the lists.
__global__ void root_kernel(Seg root, uint32_t tiles, Seg *small, Seg *sub, Seg *big, uint32_t *big_t0, uint32_t *counts,
                            unsigned long long *big_count) {
    chain_begin();
    const uint32_t m = root.l - root.f + 1;
    if (m <= kSmallMax) {
        small[0] = root;
        counts[0] = 1;
    } else if (m <= kSubMax) {
        sub[0] = root;
        counts[1] = 1;
    } else {
        big[0] = root;
        big_t0[0] = 0;
        *big_count = (1ull << 32) | tiles;
    }
}

// One level of the ranges of more than kSubMax lights: every split in a tile; the last tile of
// a range to finish reduces the tiles' best splits and records the range's.
__global__ void __launch_bounds__(kSplitThreads, 4) split_level_kernel(
    const Seg *big, const uint32_t *big_t0, const unsigned long long *big_count,
    const float4 *__restrict__ spos, uint32_t n, BoxScratch boxes, Best *tile_best, uint32_t *done, SplitOut o) {
    __shared__ Agg sh[kSplitThreads / 32], edge[2];
    __shared__ Best shb[kSplitThreads / 32];
    __shared__ uint32_t s_i;
    __shared__ int s_last;
    chain_begin();
    const unsigned long long have = *big_count;
    if (blockIdx.x >= (uint32_t)have) return;
    if (threadIdx.x == 0) s_i = range_of_tile(big_t0, (uint32_t)(have >> 32), blockIdx.x);
    __syncthreads();
    const uint32_t ri = s_i, t0 = big_t0[ri];
    const Seg g = big[ri];
    const uint32_t nt = (g.l - g.f + 1 + kSegTile - 1) / kSegTile;
    const uint32_t start = g.f + (blockIdx.x - t0) * kSegTile;
    const uint32_t end = g.l + 1 - start > kSegTile ? start + kSegTile : g.l + 1;  // lights [start, end)
    const uint32_t a = start + threadIdx.x * kTileRun;
    float4 p[kTileRun];
    const uint32_t cnt = load_run<kTileRun>(spos, a, end, p);
    if (threadIdx.x < 64) {  // the range before the tile (warp 0) and after it (warp 1)
        const bool first = threadIdx.x < 32;
        Agg x = agg_empty();
        if (first ? start > g.f : end <= g.l)
            x = box_range(PointLeaves{spos}, boxes, n, first ? g.f : end, first ? start - 1u : g.l);
        if ((threadIdx.x & 31) == 0) edge[first ? 0 : 1] = x;
    }
    Agg before, after;
    block_scans<kSplitThreads>(run_agg<kTileRun>(p, cnt), before, after, sh);
    before = agg_join(edge[0], before);
    after = agg_join(after, edge[1]);
    Best b = best_none();
    run_best<kTileRun>(p, cnt, a, before, after, g.f, g.l, b);
    b = block_best<kSplitThreads>(b, shb);
    if (threadIdx.x == 0) {
        tile_best[blockIdx.x] = b;
        __threadfence();
        s_last = atomicAdd(&done[ri], 1u) == nt - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    Best r = best_none();
    for (uint32_t j = threadIdx.x; j < nt; j += kSplitThreads) {
        const Best *q = &tile_best[t0 + j];
        best_take(r, {__ldcg(&q->c), __ldcg(&q->d), __ldcg(&q->k)});
    }
    r = block_best<kSplitThreads>(r, shb);
    if (threadIdx.x == 0) {
        done[ri] = 0;
        commit_split(g, r.k, o);
    }
}

// The cost-driven topology for n >= 2 sorted lights: writes split / other_end of every
// record and the parent links. The groups of `boxes` must be there (groups_enqueue).
int cost_topology(hrr_ctx *ctx, const float4 *spos, const uint64_t *keys, uint32_t n, uint32_t cost_depth,
                  hrr_node *nodes, const BoxScratch &boxes, const unsigned long long *flags, cudaStream_t st) {
    const size_t un = n, cap_b = un / (kSubMax + 1) + 1;  // ranges of more than kSubMax lights in a level
    const size_t cap_t = un / kSegTile + cap_b + 1;       // tiles of those
    constexpr uint32_t kLevels = 68;                      // they are at most as deep as the cost depth (64)
    const size_t words = 4 + 2 * (kLevels + 1) + cap_b;   // counts, levels' counts, done
    const size_t bytes = 2 * pad256(sizeof(Seg) * (un / 2 + 1)) + pad256(sizeof(Seg) * (un / 33 + 1)) +
                         2 * (pad256(sizeof(Seg) * cap_b) + pad256(sizeof(uint32_t) * cap_b)) +
                         pad256(sizeof(Best) * cap_t) + pad256(sizeof(uint32_t) * words);
    char *scratch = nullptr;
    cudaError_t e = hrr_alloc(ctx, &scratch, bytes);
    if (e != cudaSuccess) return hrr_cuda_fail(ctx, e, "topology scratch");
    char *p = scratch;
    SplitOut o{};
    o.nodes = nodes;
    o.leaf_parent = boxes.leaf_parent;
    o.int_parent = boxes.int_parent;
    o.cost_depth = cost_depth;
    o.small = carve<Seg>(p, un / 2 + 1);
    o.radix = carve<Seg>(p, un / 2 + 1);
    o.sub = carve<Seg>(p, un / 33 + 1);
    Seg *big[2];
    uint32_t *t0[2];
    for (int k = 0; k < 2; ++k) {
        big[k] = carve<Seg>(p, cap_b);
        t0[k] = carve<uint32_t>(p, cap_b);
    }
    Best *tile_best = carve<Best>(p, cap_t);
    uint32_t *w = carve<uint32_t>(p, words);
    o.counts = w;
    unsigned long long *level_count = reinterpret_cast<unsigned long long *>(w + 4);  // ranges and tiles per level
    uint32_t *done = w + 4 + 2 * (kLevels + 1);

    // The root goes to its list; its count, on the device, tells the kernels that it is there.
    const Seg root{0u, 0u, n - 1, 1u};
    const uint32_t root_tiles = (uint32_t)((un + kSegTile - 1) / kSegTile);
    e = cudaMemsetAsync(w, 0, sizeof(uint32_t) * words, st);
    if (e == cudaSuccess) {
        root_kernel<<<1, 1, 0, st>>>(root, root_tiles, o.small, o.sub, big[0], t0[0], o.counts, level_count);
        ++ctx->launches;
    }
    uint64_t left = n > kSubMax;  // ranges of more than kSubMax lights still to split
    uint32_t level = 0;
    // two levels per halving and one (21 for 2^20 lights, the last few of which seldom have any such
    // range left), then a few at a time
    uint32_t batch = 2;
    for (size_t m = un / kSubMax; m > 1; m >>= 1) batch += batch & 1 ? 2 : 1;
    int rc = HRR_OK;
    while (e == cudaSuccess && left) {
        for (uint32_t k = 0; k < batch && level < kLevels; ++k, ++level) {
            o.big = big[(level + 1) & 1];
            o.big_t0 = t0[(level + 1) & 1];
            o.big_count = level_count + level + 1;
            const unsigned grid = level == 0 ? root_tiles : (unsigned)cap_t;
            launch_chained(split_level_kernel, grid, kSplitThreads, st, big[level & 1], t0[level & 1], level_count + level,
                           spos, n, boxes, tile_best, done, o);
            ++ctx->launches;
        }
        unsigned long long *host = &ctx->host_counters[5];
        if ((e = cudaGetLastError()) != cudaSuccess) break;
        if ((e = cudaMemcpyAsync(host, level_count + level, sizeof(*host), cudaMemcpyDeviceToHost, st)) != cudaSuccess) break;
        if ((e = cudaMemcpyAsync(&ctx->host_counters[2], flags, sizeof(*flags), cudaMemcpyDeviceToHost, st)) != cudaSuccess) break;
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess) break;
        if (ctx->host_counters[2] & (HRR_FLAG_UNSORTED | HRR_FLAG_NONFINITE)) break;  // the build starts over, or fails
        left = *host;
        if (left && level >= kLevels) {  // the radix split bounds the height
            rc = hrr_fail(ctx, HRR_ERR_DEVICE, "topology build did not terminate");
            break;
        }
        batch = 4;
    }
    if (e == cudaSuccess && rc == HRR_OK) {
        const unsigned sub_grid = (unsigned)std::min<size_t>(un / 33 + 1, (size_t)ctx->sm_count * 16);
        const unsigned small_grid = (unsigned)std::min<size_t>(un / 16 + 1, (size_t)ctx->sm_count * 5);
        launch_chained(sub_kernel, sub_grid, kSubThreads, st, spos, o);
        launch_chained(subtree_kernel, small_grid, kSplitThreads, st, spos, keys, o);
        launch_chained(radix_subtrees_kernel, (unsigned)ctx->sm_count * 4u, kSplitThreads, st, keys, o, flags);
        ctx->launches += 3;
        e = cudaGetLastError();
    }
    cudaFreeAsync(scratch, st);
    if (e != cudaSuccess) return hrr_cuda_fail(ctx, e, "topology build");
    return rc;
}

}  // namespace
