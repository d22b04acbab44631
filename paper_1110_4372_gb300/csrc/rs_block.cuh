// rs_block.cuh -- giving back a block of a context's memory pool (host code).
#pragma once

#include <cuda_runtime_api.h>

// Frees a pool's block of `device`, from any thread.  cudaFree does not wait
// for such a block and cudaDeviceSynchronize waits for the current device, which
// in the calling thread may be another one: the block's own is made current for
// both, and the thread's restored.
inline void rs_block_give_back(void *p, int device)
{
    if (!p) return;
    int current = device;
    cudaGetDevice(&current);
    if (current != device) cudaSetDevice(device);
    cudaDeviceSynchronize();
    cudaFree(p);
    if (current != device) cudaSetDevice(current);
}
