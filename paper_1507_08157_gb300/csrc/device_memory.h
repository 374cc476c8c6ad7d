// Device allocations of the library. Contexts keep the memory of destroyed states for their next one
// (SlabPool in api.cu): an allocation that fails gives that back and is tried once more.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <new>
#include <vector>

namespace tddft {

bool release_spare_slabs();   // frees the memory that contexts keep of destroyed states; true if there was any

// n values of T (at least one), not initialised; throws std::bad_alloc
template <typename T>
T *device_alloc(size_t n) {
    void *p = nullptr;
    if (n == 0) n = 1;
    cudaError_t e = cudaMalloc(&p, n * sizeof(T));
    if (e != cudaSuccess) {
        cudaGetLastError();
        if (release_spare_slabs()) e = cudaMalloc(&p, n * sizeof(T));
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        throw std::bad_alloc();
    }
    return static_cast<T *>(p);
}

// owning list of device allocations (freed on release or destruction)
struct Mem {
    std::vector<void *> ptrs;
    template <typename T>
    T *alloc(size_t n) {
        ptrs.reserve(ptrs.size() + 1);
        T *p = device_alloc<T>(n);
        ptrs.push_back(p);
        return p;
    }
    void release() {
        for (void *p : ptrs) cudaFree(p);
        ptrs.clear();
    }
    ~Mem() { release(); }
};

// A buffer that grows on demand and is never shrunk; empty after a failed growth
struct Scratch {
    float *p = nullptr;
    size_t cap = 0;
    float *get(size_t n) {
        if (n > cap) {
            cap = 0;
            if (p) cudaFree(p);   // synchronises the device: earlier users of the buffer are done
            p = nullptr;
            p = device_alloc<float>(n);
            cap = n;
        }
        return p;
    }
};

}  // namespace tddft
