// What a launch has to know about a kernel, asked of the runtime once: how many
// of its blocks are resident per SM at a shared-memory size, and the permission
// to use all of a block's shared memory (the permission is a property of the
// kernel on a device, so every thread sets the same largest value and none takes
// it away from another). The two questions cost several microseconds per launch,
// a product of a thousand rows makes a dozen launches.
//
// Kept per host thread and device, a bounded number of them; nothing depends on
// the data.
#pragma once

#include <cstddef>
#include <vector>

#include <cuda_runtime.h>

#include "kernels.h"

namespace smash {

inline void allow_smem(const void *kernel) {
    struct Known {
        const void *kernel;
        int dev;
    };
    thread_local std::vector<Known> known;
    int dev = 0;
    cudaGetDevice(&dev);
    for (const Known &k : known)
        if (k.kernel == kernel && k.dev == dev) return;
    cudaFuncAttributes a;
    if (cudaFuncGetAttributes(&a, kernel) != cudaSuccess) return;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             max_smem_per_block() - (int)a.sharedSizeBytes) != cudaSuccess)
        return;
    known.push_back(Known{kernel, dev});
}

// Resident blocks per SM of nt threads with smem bytes of dynamic shared memory
// (0: such a block cannot run).
inline int resident_per_sm(const void *kernel, int nt, size_t smem) {
    struct Known {
        const void *kernel;
        size_t smem;
        int dev, nt, blocks;
    };
    thread_local std::vector<Known> known;
    int dev = 0;
    cudaGetDevice(&dev);
    for (const Known &k : known)
        if (k.kernel == kernel && k.smem == smem && k.nt == nt && k.dev == dev) return k.blocks;
    allow_smem(kernel);
    int blocks = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, kernel, nt, smem) != cudaSuccess) return 0;
    if (known.size() >= 256) known.clear();
    known.push_back(Known{kernel, smem, dev, nt, blocks});
    return blocks;
}

}  // namespace smash
