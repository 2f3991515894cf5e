// Forced into every translation unit of a copy of the library (fake_lib.py), to make runtime calls
// fail, or clear memory in another way, where an environment variable asks for it:
//   HRR_FAKE_TICKETS  the tile tickets of a sort start at one: no block takes the first tile, and
//                     those that wait for it wait in vain
//   HRR_FAKE_MEMORY   bytes that allocations from memory pools may take together; hrr_fake_used()
//                     is what they take
#pragma once
#include <cuda_runtime.h>

#include <cstdlib>
#include <map>
#include <mutex>

inline cudaError_t fake_memset(void *p, int v, size_t bytes, cudaStream_t st) {
    static const unsigned ones[8] = {1, 1, 1, 1, 1, 1, 1, 1};
    cudaError_t e = cudaMemsetAsync(p, v, bytes, st);
    // the sort's scratch is the only larger one: counts of 8 passes x 256 digits, then the tickets
    if (e == cudaSuccess && bytes > (1u << 16) && getenv("HRR_FAKE_TICKETS"))
        e = cudaMemcpyAsync(static_cast<char *>(p) + 8 * 256 * 4, ones, sizeof ones, cudaMemcpyHostToDevice, st);
    return e;
}
#define cudaMemsetAsync fake_memset

struct FakePool {
    std::mutex mu;
    std::map<void *, size_t> live;
    size_t used = 0;
};
inline FakePool fake_pool;

inline cudaError_t fake_pool_malloc(void **p, size_t bytes, cudaMemPool_t pool, cudaStream_t st) {
    std::lock_guard<std::mutex> lock(fake_pool.mu);
    const char *most = getenv("HRR_FAKE_MEMORY");
    if (most && fake_pool.used + bytes > strtoull(most, nullptr, 10)) {
        *p = nullptr;
        return cudaErrorMemoryAllocation;
    }
    const cudaError_t e = cudaMallocFromPoolAsync(p, bytes, pool, st);
    if (e == cudaSuccess) fake_pool.used += fake_pool.live[*p] = bytes;
    return e;
}
inline cudaError_t fake_free(void *p, cudaStream_t st) {
    std::lock_guard<std::mutex> lock(fake_pool.mu);
    if (auto it = fake_pool.live.find(p); it != fake_pool.live.end()) {
        fake_pool.used -= it->second;
        fake_pool.live.erase(it);
    }
    return cudaFreeAsync(p, st);
}
extern "C" __attribute__((used, visibility("default"))) inline unsigned long long hrr_fake_used() { return fake_pool.used; }
#define cudaMallocFromPoolAsync fake_pool_malloc
#define cudaFreeAsync fake_free
