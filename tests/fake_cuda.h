// Forced into every translation unit of a copy of the library (fake_lib.py), to make runtime calls
// fail, or clear memory in another way, where an environment variable asks for it:
//   HRR_FAKE_TICKETS  the tile tickets of a sort start at one: no block takes the first tile, and
//                     those that wait for it wait in vain
#pragma once
#include <cuda_runtime.h>

#include <cstdlib>

inline cudaError_t fake_memset(void *p, int v, size_t bytes, cudaStream_t st) {
    static const unsigned ones[8] = {1, 1, 1, 1, 1, 1, 1, 1};
    cudaError_t e = cudaMemsetAsync(p, v, bytes, st);
    // the sort's scratch is the only larger one: counts of 8 passes x 256 digits, then the tickets
    if (e == cudaSuccess && bytes > (1u << 16) && getenv("HRR_FAKE_TICKETS"))
        e = cudaMemcpyAsync(static_cast<char *>(p) + 8 * 256 * 4, ones, sizeof ones, cudaMemcpyHostToDevice, st);
    return e;
}
#define cudaMemsetAsync fake_memset
