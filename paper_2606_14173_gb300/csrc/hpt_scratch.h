// Scratch of the wave-optics calls: from the context's pool, in groups of fields or maps that shrink when
// the device is nearly full.
#pragma once
#include <algorithm>

#include <cuda_runtime.h>

namespace hpt {

// the items of 'total' that go through together: as many as keep within 'most' bytes, at least one
inline int group_items(long long total, size_t item_bytes, size_t most)
{
    return (int)std::min<long long>(total, std::max<size_t>(1, most / item_bytes));
}

// get(G), an allocation for groups of G items; while it finds no memory, G is halved, down to one item
template <class GET> cudaError_t get_group(int &G, GET get)
{
    for (;;) {
        const cudaError_t e = get(G);
        if (e != cudaErrorMemoryAllocation || G == 1) return e;
        G = (G + 1) / 2;
    }
}

// an allocation from the pool; when the device is full, again after what the pool keeps was given back (a
// failed one can leave the pool larger)
inline cudaError_t pool_alloc(void **p, size_t bytes, cudaMemPool_t pool, cudaStream_t s)
{
    cudaError_t e = cudaMallocFromPoolAsync(p, bytes, pool, s);
    if (e != cudaErrorMemoryAllocation) return e;
    (void)cudaGetLastError();
    (void)cudaMemPoolTrimTo(pool, 0);
    e = cudaMallocFromPoolAsync(p, bytes, pool, s);
    if (e == cudaErrorMemoryAllocation) {
        (void)cudaGetLastError();
        (void)cudaMemPoolTrimTo(pool, 0);
    }
    return e;
}

}  // namespace hpt
