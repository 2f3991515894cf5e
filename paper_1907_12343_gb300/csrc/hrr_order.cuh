// Leaf order and radix topology: Morton keys of points, their sort, and the binary radix tree over
// (key, sorted position). The light builder and the triangle scenes (by their centroids) share it.
#pragma once

#include <algorithm>

#include "hrr_boxes.cuh"
#include "hrr_internal.cuh"
#include "hrr_sort.cuh"

namespace {

constexpr int kOrderThreads = 256;

// Spread the low 21 bits of v so that bit k moves to bit 3k.
__device__ __forceinline__ uint64_t spread3(uint64_t v) {
    v &= 0x1FFFFFull;
    v = (v | (v << 32)) & 0x1F00000000FFFFull;
    v = (v | (v << 16)) & 0x1F0000FF0000FFull;
    v = (v | (v << 8)) & 0x100F00F00F00F00Full;
    v = (v | (v << 4)) & 0x10C30C30C30C30C3ull;
    v = (v | (v << 2)) & 0x1249249249249249ull;
    return v;
}

// floor(x * 2^21) clamped to [0, 2^21 - 1]; x * 2^21 is exact in float.
__device__ __forceinline__ uint32_t grid_cell(float x) {
    const float s = __fmul_rn(x, 2097152.0f);
    if (!(s >= 0.0f)) return 0u;
    const float f = floorf(s);
    return f >= 2097151.0f ? 2097151u : (uint32_t)f;
}

// Keys, finiteness checks, and the digit counts of the sort's passes. Blocks stride over the
// lights, so that few add their counts to the totals.
__global__ void __launch_bounds__(kOrderThreads) morton_kernel(const float *__restrict__ x,
                                                          const float *__restrict__ y,
                                                          const float *__restrict__ z,
                                                          const float *__restrict__ inten,
                                                          uint32_t n, uint64_t *__restrict__ keys,
                                                          int shift, int passes, uint32_t *hist,
                                                          unsigned long long *flags) {
    __shared__ uint32_t cnt[kSortPasses * 256];
    chain_begin();
    for (int k = threadIdx.x; k < 256 * passes; k += kOrderThreads) cnt[k] = 0;
    __syncthreads();
    for (uint32_t i = blockIdx.x * kOrderThreads + threadIdx.x; i < n; i += gridDim.x * kOrderThreads) {
        const float px = x[i], py = y[i], pz = z[i], w = inten[i];
        if (!isfinite(px) || !isfinite(py) || !isfinite(pz) || !isfinite(w))
            atomicOr(flags, HRR_FLAG_NONFINITE);
        const uint64_t key = (spread3(grid_cell(px)) << 2) | (spread3(grid_cell(py)) << 1) | spread3(grid_cell(pz));
        keys[i] = key;
        count_digits(cnt, key, shift, passes);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < 256 * passes; k += kOrderThreads)
        if (cnt[k]) atomicAdd(&hist[k], cnt[k]);
}
inline unsigned morton_grid(uint32_t n) { return std::min(608u, (n + 4 * kOrderThreads - 1) / (4 * kOrderThreads)); }

// After the sort: sorted keys, permutation and lights, and the box pass's scratch reset. With
// RUNS the keys are sorted by their upper halves only, and light i's place among the lights that
// share its upper half is counted from their lower ones (ties by the order they are in); a run
// of more than kRunMax lights raises HRR_FLAG_RUNS and stays as it is. After a sort that gave up
// nothing is done: its values index the lights.
template <bool RUNS>
__global__ void __launch_bounds__(kOrderThreads) gather_sorted_kernel(const float *__restrict__ x,
                                                                 const float *__restrict__ y,
                                                                 const float *__restrict__ z,
                                                                 const float *__restrict__ inten,
                                                                 const uint64_t *keys_in, const uint32_t *vals_in, uint32_t n,
                                                                 uint64_t *__restrict__ keys, uint32_t *__restrict__ perm,
                                                                 float4 *__restrict__ spos, BoxScratch s,
                                                                 unsigned long long *flags) {
    chain_begin();
    const uint32_t i = blockIdx.x * kOrderThreads + threadIdx.x;
    if (i >= n) return;
    const uint32_t v = vals_in[i];
    const uint64_t key = keys_in[i];
    if (*(volatile unsigned long long *)flags & HRR_FLAG_WAIT) return;  // read beside v and the key, not before them
    const float4 p = make_float4(x[v], y[v], z[v], inten[v]);
    uint32_t to = i;
    if (RUNS) {
        uint32_t left = 0, right = 0, ahead = 0;  // neighbours of the run, and those that move ahead of i
        while (left <= kRunMax && left < i) {
            const uint64_t o = keys_in[i - left - 1u];
            if ((o ^ key) >> kTopShift) break;
            ahead += o <= key;
            ++left;
        }
        while (right <= kRunMax && i + right + 1u < n) {
            const uint64_t o = keys_in[i + right + 1u];
            if ((o ^ key) >> kTopShift) break;
            ahead += o < key;
            ++right;
        }
        if (left + right + 1u > kRunMax) atomicOr(flags, HRR_FLAG_RUNS);
        else to = i - left + ahead;
    }
    keys[to] = key;
    perm[to] = v;
    spos[to] = p;
    box_reset(s, i, n);
}

// Common-prefix length of the ordering keys (Morton key, sorted position) of leaves i, j; -1
// outside [f, l].
__device__ __forceinline__ int prefix_len(const uint64_t *__restrict__ keys, int64_t f, int64_t l, int64_t i, int64_t j) {
    if (j < f || j > l) return -1;
    const uint64_t ki = keys[i], kj = keys[j];
    if (ki != kj) return __clzll((long long)(ki ^ kj));
    return 64 + __clz((uint32_t)(i ^ j));
}

// Range and split of node i of the binary radix tree over the leaves [f, l] (f <= i < l): each
// node finds them from its neighbours' common-prefix lengths (Karras, HPG 2012).
__device__ __forceinline__ void radix_node(const uint64_t *__restrict__ keys, uint32_t f32, uint32_t l32, uint32_t i32,
                                           uint32_t &first, uint32_t &last, uint32_t &split) {
    const int64_t f = f32, l = l32, i = i32;
    const int d = (prefix_len(keys, f, l, i, i + 1) - prefix_len(keys, f, l, i, i - 1)) >= 0 ? 1 : -1;
    const int dmin = prefix_len(keys, f, l, i, i - d);
    int64_t most = 2;
    while (prefix_len(keys, f, l, i, i + most * d) > dmin) most <<= 1;
    int64_t len = 0;
    for (int64_t t = most >> 1; t >= 1; t >>= 1)
        if (prefix_len(keys, f, l, i, i + (len + t) * d) > dmin) len += t;
    const int64_t j = i + len * d;
    const int dnode = prefix_len(keys, f, l, i, j);
    int64_t s = 0, t = len;
    do {
        t = (t + 1) >> 1;
        if (prefix_len(keys, f, l, i, i + (s + t) * d) > dnode) s += t;
    } while (t > 1);
    split = (uint32_t)(i + s * d + (d < 0 ? -1 : 0));
    first = (uint32_t)(i < j ? i : j);
    last = (uint32_t)(i < j ? j : i);
}

__global__ void __launch_bounds__(kOrderThreads) topology_kernel(const uint64_t *keys,
                                                            uint32_t n, hrr_node *__restrict__ nodes,
                                                            uint32_t *__restrict__ leaf_parent,
                                                            uint32_t *__restrict__ int_parent,
                                                            const unsigned long long *flags) {
    chain_begin();
    const uint32_t i = blockIdx.x * kOrderThreads + threadIdx.x;
    if (i >= n - 1 || (*flags & HRR_FLAG_UNSORTED)) return;
    uint32_t first, last, split;
    radix_node(keys, 0u, n - 1, i, first, last, split);
    nodes[i].split = split;
    nodes[i].other_end = i == first ? last : first;
    const uint32_t code = i << 1;
    if (first == split) leaf_parent[split] = code; else int_parent[split] = code;
    if (last == split + 1) leaf_parent[split + 1] = code | 1u; else int_parent[split + 1] = code | 1u;
}

}  // namespace
