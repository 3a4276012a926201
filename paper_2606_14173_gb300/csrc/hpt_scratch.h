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

// f(first, n) for consecutive groups of up to G items
template <class F> cudaError_t for_groups(long long total, int G, F f)
{
    cudaError_t e = cudaSuccess;
    for (long long first = 0; first < total && e == cudaSuccess; first += G) e = f(first, (int)std::min<long long>(G, total - first));
    return e;
}

// Where field 'first' of a list with 'per' fields to a wavelength lies, and the wavelength of the f-th after it.
struct FieldPlace {
    int lam, field;
};
inline FieldPlace field_place(long long first, int per) { return {(int)(first / per), (int)(first % per)}; }
__host__ __device__ inline int lambda_of(FieldPlace p, int f, int per)
{
    return p.lam + (int)(((unsigned)p.field + (unsigned)f) / (unsigned)per);
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
