// rs_block.cuh -- a context's memory pool and the blocks taken from it (host code).
#pragma once

#include <cuda_runtime_api.h>

#include <atomic>

// The pool of a context's trees and halo tables.  The context and every block
// in use hold it, and the last one destroys it: a context may go before its
// trees, and destroying a pool whose blocks were in use ended in a crash.
struct RsPool {
    cudaMemPool_t mem = nullptr;
    int device = 0;
    std::atomic<int> holders{1};
};

inline void rs_pool_release(RsPool *pool)
{
    if (!pool || pool->holders.fetch_sub(1) != 1) return;
    cudaMemPoolDestroy(pool->mem);
    delete pool;
}

// The context's own hold: what the pool keeps free, and what is given back to
// it later, goes to the device.
inline void rs_pool_retire(RsPool *pool)
{
    if (!pool) return;
    unsigned long long keep = 0;
    cudaMemPoolSetAttribute(pool->mem, cudaMemPoolAttrReleaseThreshold, &keep);
    cudaMemPoolTrimTo(pool->mem, 0);
    rs_pool_release(pool);
}

// Frees a block of the pool, from any thread.  Nothing that frees such a block
// waits for the device and cudaDeviceSynchronize waits for the current one, which
// in the calling thread may be another: the block's own is made current, and the
// thread's restored.  (cudaFree gives the block back too, but the pool goes on
// counting it as used.)
inline void rs_block_give_back(void *p, RsPool *pool)
{
    if (!p) return;
    int current = pool->device;
    cudaGetDevice(&current);
    if (current != pool->device) cudaSetDevice(pool->device);
    cudaDeviceSynchronize();
    cudaFreeAsync(p, 0);
    cudaStreamSynchronize(0);
    if (current != pool->device) cudaSetDevice(current);
    rs_pool_release(pool);
}
