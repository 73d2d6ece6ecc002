// What a launch has to know about a kernel, asked of the runtime once: how many
// of its blocks are resident per SM at a shared-memory size, and the permission
// to use all of a block's shared memory (the permission is a property of the
// kernel on a device, so every thread sets the same largest value and none takes
// it away from another). The two questions cost several microseconds per launch,
// a product of a thousand rows makes a dozen launches.
//
// Kept per host thread and device, in arrays of a fixed size (no allocation that
// could throw under the C entry points); nothing depends on the data.
#pragma once

#include <cstddef>

#include <cuda_runtime.h>

#include "kernels.h"

namespace smash {

inline void allow_smem(const void *kernel) {
    struct Known {
        const void *kernel;
        int dev;
    };
    thread_local Known known[256];
    thread_local int n = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    for (int x = 0; x < n; ++x)
        if (known[x].kernel == kernel && known[x].dev == dev) return;
    cudaFuncAttributes a;
    if (cudaFuncGetAttributes(&a, kernel) != cudaSuccess) return;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             max_smem_per_block() - (int)a.sharedSizeBytes) != cudaSuccess)
        return;
    if (n == 256) n = 0;
    known[n++] = Known{kernel, dev};
}

// Resident blocks per SM of nt threads with smem bytes of dynamic shared memory
// (0: such a block cannot run).
inline int resident_per_sm(const void *kernel, int nt, size_t smem) {
    struct Known {
        const void *kernel;
        size_t smem;
        int dev, nt, blocks;
    };
    thread_local Known known[256];
    thread_local int n = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    for (int x = 0; x < n; ++x) {
        const Known &k = known[x];
        if (k.kernel == kernel && k.smem == smem && k.nt == nt && k.dev == dev) return k.blocks;
    }
    allow_smem(kernel);
    int blocks = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, kernel, nt, smem) != cudaSuccess) return 0;
    if (n == 256) n = 0;
    known[n++] = Known{kernel, smem, dev, nt, blocks};
    return blocks;
}

}  // namespace smash
