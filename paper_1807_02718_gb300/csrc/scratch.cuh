// Work space of one call from the device's stream-ordered allocator, returned
// on the same stream when the call's launches have been issued.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

namespace fh {

struct Scratch {
    std::vector<void *> bufs;
    cudaStream_t st;
    template <class T> T *get(size_t count) {
        void *p = nullptr;
        if (cudaMallocAsync(&p, std::max<size_t>(count, 1) * sizeof(T), st) != cudaSuccess) return nullptr;
        bufs.push_back(p);
        return static_cast<T *>(p);
    }
    ~Scratch() {
        for (void *p : bufs) cudaFreeAsync(p, st);
    }
};

}  // namespace fh
