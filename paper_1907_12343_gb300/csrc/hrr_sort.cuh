// Stable sort of (63-bit key, value) by least-significant 8-bit digits, one kernel per digit.
//
// Every digit's counts over all keys are taken once, while the keys are made (they do not
// depend on the order). A pass then reads and writes each key once: a block takes the next
// tile, ranks its keys by digit, publishes its digit counts and sums those of the tiles before
// it (decoupled look-back: the counts of a tile, or the sums up to it, whichever is there), and
// writes its keys out in runs of equal digits through shared memory. A tile waits only for
// tiles with lower tickets, whose blocks are running or done. Every wait is bounded: one that runs
// out raises HRR_FLAG_WAIT, the tile goes on with the sum it has (so that those behind it end
// too; no place past the arrays is written), and the kernels after the sort leave its result
// alone, parts of which are then not written; the call reports HRR_ERR_TIMEOUT. With a histogram,
// a scan and a scatter kernel per digit the sort was a chain of 24 launches of 3 to 29 us each
// (340 us for 2^20 keys, 290 us for 100,003).
//
// Few lights share the upper 32 bits of their keys, so a build sorts by those (four passes) and
// puts the short runs that agree in them in order afterwards (gather_sorted_kernel); keys with
// longer runs go through all eight passes (sort_bits_from).
#pragma once

#include "hrr_internal.cuh"

namespace {

constexpr uint32_t kSortThreads = 256;  // one digit value per thread
constexpr int kSortPasses = 8;          // of a full sort
constexpr int kTopShift = 31;           // the upper 32 of the 63 key bits
constexpr uint32_t kRunMax = 64;        // longest run ordered without a full sort
constexpr uint32_t kWaitPolls = 1u << 20;
// Keys per thread: small tiles while they leave SMs idle otherwise (at 2^17 keys 128 tiles of
// 1024 on 152 SMs), large ones above, where each tile costs a look-back.
constexpr int kSortSmall = 4, kSortLarge = 16;
inline int sort_items(uint32_t n) { return n <= (1u << 17) ? kSortSmall : kSortLarge; }
constexpr size_t sort_tiles(size_t n) {  // the most tiles of any n' <= n
    const size_t small = n < (1u << 17) ? n : (1u << 17);
    const size_t a = (small + kSortThreads * kSortSmall - 1) / (kSortThreads * kSortSmall);
    const size_t b = (n + kSortThreads * kSortLarge - 1) / (kSortThreads * kSortLarge);
    return a > b ? a : b;
}

// Cleared before a sort: digit counts per pass, a tile ticket per pass, and per tile and digit
// one word: (2 pass + 1) << 32 | count of the tile, or (2 pass + 2) << 32 | sum up to and with it.
struct SortScratch {
    uint32_t *hist;             // kSortPasses x 256
    uint32_t *ticket;           // kSortPasses
    unsigned long long *state;  // tiles x 256
};
constexpr size_t sort_scratch_bytes(size_t n) {
    return sizeof(uint32_t) * (kSortPasses * 256 + 64) + sizeof(unsigned long long) * 256 * sort_tiles(n);
}
inline SortScratch carve_sort(char *&p, size_t n) {
    SortScratch s;
    s.hist = reinterpret_cast<uint32_t *>(p);
    s.ticket = s.hist + kSortPasses * 256;
    s.state = reinterpret_cast<unsigned long long *>(s.ticket + 64);
    p += (sort_scratch_bytes(n) + 255) & ~size_t(255);
    return s;
}

__device__ __forceinline__ unsigned long long load_state(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void store_state(unsigned long long *p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" : : "l"(p), "l"(v) : "memory");
}

// Add a key's digits to the block's counts (cnt: passes x 256 in shared memory).
__device__ __forceinline__ void count_digits(uint32_t *cnt, uint64_t key, int shift, int passes) {
    for (int q = 0; q < passes; ++q) atomicAdd(&cnt[256 * q + ((key >> (shift + 8 * q)) & 255u)], 1u);
}

// Exclusive sums over the block's 256 threads of two values; sh: 16 words.
__device__ __forceinline__ void scan2(uint32_t a, uint32_t b, uint32_t &ea, uint32_t &eb, uint32_t *sh) {
    const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
    uint32_t x = a, y = b;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, x, o), v = __shfl_up_sync(0xFFFFFFFFu, y, o);
        if (lane >= (uint32_t)o) {
            x += u;
            y += v;
        }
    }
    if (lane == 31u) {
        sh[w] = x;
        sh[8 + w] = y;
    }
    __syncthreads();
    ea = x - a;
    eb = y - b;
    for (uint32_t k = 0; k < w; ++k) {
        ea += sh[k];
        eb += sh[8 + k];
    }
}

// One pass: digit (key >> shift) & 255. vals_in NULL: the values are the indices.
template <int ITEMS>
__global__ void __launch_bounds__(kSortThreads) sort_pass_kernel(const uint64_t *keys_in, const uint32_t *vals_in,
                                                                 uint64_t *keys_out, uint32_t *vals_out, uint32_t n, int shift,
                                                                 int pass, SortScratch s, unsigned long long *flags) {
    constexpr uint32_t kTile = kSortThreads * ITEMS, kWarps = kSortThreads / 32;
    // Tiles looked back on at once: their words are loaded together, so that many tiles ahead cost
    // few round trips. A build of 100,003 lights (98 small tiles) takes 164 us with 32 against 186 with
    // 8 or 16; large tiles have no registers for more than 16 (a cost-driven build of 2^20 lights, when
    // its launches were not chained yet: 1065 us, 1073 with 8 or 32).
    constexpr uint32_t kLook = ITEMS <= kSortSmall ? 32u : 16u;
    __shared__ uint64_t exchange[kTile];
    __shared__ uint32_t warp_cnt[kWarps][256];
    __shared__ uint32_t start[256], to[256], sums[16], s_tile;
    const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5, lt = (1u << lane) - 1u;
    chain_begin();
    if (t == 0) s_tile = atomicAdd(&s.ticket[pass], 1u);
#pragma unroll
    for (uint32_t w = 0; w < kWarps; ++w) warp_cnt[w][t] = 0;
    __syncthreads();
    const uint32_t tile = s_tile, base = tile * kTile, mine = base + warp * 32u * ITEMS + lane;
    uint64_t key[ITEMS];
    uint32_t val[ITEMS], at[ITEMS];  // at: rank among the warp's equal digits, then place in the tile
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const uint32_t i = mine + 32u * k;
        key[k] = i < n ? keys_in[i] : 0ull;
        val[k] = i >= n ? 0u : vals_in ? vals_in[i] : i;
    }
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {  // in tile order: earlier items, then earlier lanes
        const bool valid = mine + 32u * k < n;
        const uint32_t d = (uint32_t)(key[k] >> shift) & 255u;
        uint32_t peers = __ballot_sync(0xFFFFFFFFu, valid);
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const uint32_t v = __ballot_sync(0xFFFFFFFFu, (d >> b) & 1u);
            peers &= (d >> b) & 1u ? v : ~v;
        }
        uint32_t before = 0;
        if (valid) before = warp_cnt[warp][d];
        at[k] = before + __popc(peers & lt);
        __syncwarp();
        if (valid && (peers >> lane) == 1u) warp_cnt[warp][d] = before + __popc(peers);  // the last peer
        __syncwarp();
    }
    __syncthreads();
    // thread t: digit t
    uint32_t count = 0;
#pragma unroll
    for (uint32_t w = 0; w < kWarps; ++w) {
        const uint32_t c = warp_cnt[w][t];
        warp_cnt[w][t] = count;
        count += c;
    }
    const unsigned long long part = (unsigned long long)(2 * pass + 1) << 32, all = (unsigned long long)(2 * pass + 2) << 32;
    unsigned long long *mystate = s.state + 256ull * tile + t;
    store_state(mystate, (tile == 0 ? all : part) | count);
    uint32_t local, global;
    scan2(count, s.hist[256 * pass + t], local, global, sums);
    uint32_t prefix = 0;
    if (tile > 0) {
        uint32_t polls = 0;
        for (uint32_t next = tile; next > 0;) {  // sum tiles next - 1, next - 2, ...
            unsigned long long v[kLook];
            const uint32_t m = min(next, kLook);
#pragma unroll
            for (uint32_t k = 0; k < kLook; ++k) v[k] = k < m ? load_state(s.state + 256ull * (next - 1u - k) + t) : 0ull;
            uint32_t used = 0;
            bool end = false, open = true;
#pragma unroll
            for (uint32_t k = 0; k < kLook; ++k) {
                if (open && k < m && v[k] >= part) {
                    prefix += (uint32_t)v[k];
                    ++used;
                    end = v[k] >= all;
                    open = !end;
                } else {
                    open = false;
                }
            }
            if (end) break;
            next -= used;
            if (used == 0 && ++polls > kWaitPolls) {  // cannot happen: lower tiles run or are done
                atomicOr(flags, HRR_FLAG_WAIT);
                break;
            }
        }
        store_state(mystate, all | (prefix + count));
    }
    start[t] = local;
    to[t] = global + prefix - local;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const uint32_t d = (uint32_t)(key[k] >> shift) & 255u;
        at[k] += start[d] + warp_cnt[warp][d];
        if (mine + 32u * k < n) exchange[at[k]] = key[k];
    }
    __syncthreads();
    const uint32_t have = min(kTile, n - base);
    uint32_t out[ITEMS];
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const uint32_t i = kSortThreads * k + t;
        out[k] = 0xFFFFFFFFu;
        if (i < have) {
            const uint64_t x = exchange[i];
            out[k] = to[(uint32_t)(x >> shift) & 255u] + i;
            if (out[k] < n) keys_out[out[k]] = x;
        }
    }
    __syncthreads();
    uint32_t *values = reinterpret_cast<uint32_t *>(exchange);
#pragma unroll
    for (int k = 0; k < ITEMS; ++k)
        if (mine + 32u * k < n) values[at[k]] = val[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < ITEMS; ++k)
        if (out[k] < n) vals_out[out[k]] = values[kSortThreads * k + t];
}

// Passes of a sort from key bit `shift` up (a whole number, and even: the result is back in
// keys0, vals0). vals0's first contents are not read.
inline constexpr int sort_passes(int shift) { return shift ? 4 : kSortPasses; }
inline void sort_enqueue(uint64_t *keys0, uint32_t *vals0, uint64_t *keys1, uint32_t *vals1, uint32_t n, int shift,
                         const SortScratch &s, unsigned long long *flags, cudaStream_t st) {
    const int items = sort_items(n);
    const unsigned tiles = (unsigned)(((size_t)n + kSortThreads * items - 1) / (kSortThreads * items));
    for (int q = 0; q < sort_passes(shift); ++q) {
        const uint64_t *kin = q & 1 ? keys1 : keys0;
        const uint32_t *vin = q == 0 ? nullptr : q & 1 ? vals1 : vals0;
        uint64_t *kout = q & 1 ? keys0 : keys1;
        uint32_t *vout = q & 1 ? vals0 : vals1;
        if (items == kSortSmall)
            launch_chained(sort_pass_kernel<kSortSmall>, tiles, kSortThreads, st, kin, vin, kout, vout, n, shift + 8 * q, q, s, flags);
        else
            launch_chained(sort_pass_kernel<kSortLarge>, tiles, kSortThreads, st, kin, vin, kout, vout, n, shift + 8 * q, q, s, flags);
    }
}

}  // namespace
