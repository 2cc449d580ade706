// Allocators of a search's device pieces.  Every one of them makes a piece a
// whole number of 256 bytes: kernels read the ends of pieces in 16-byte
// vectors (plan_kernel), past the last element asked for.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

namespace hicops {

constexpr uint64_t align256(uint64_t x) { return (x + 255) & ~uint64_t(255); }

template <class T>
constexpr uint64_t piece_bytes(uint64_t n) { return align256(sizeof(T) * (n ? n : 1)); }

// stream-ordered scratch from a pool (or the device's default one); freed on every exit path
struct Scratch {
    cudaStream_t s;
    cudaMemPool_t pool;
    std::vector<void*> ptrs;
    explicit Scratch(cudaStream_t st, cudaMemPool_t p = nullptr) : s(st), pool(p) {}
    template <class T>
    cudaError_t get(T** p, uint64_t n) {
        const uint64_t bytes = piece_bytes<T>(n);
        cudaError_t e = pool ? cudaMallocFromPoolAsync((void**)p, bytes, pool, s) : cudaMallocAsync((void**)p, bytes, s);
        if (e == cudaSuccess) ptrs.push_back(*p);
        return e;
    }
    ~Scratch() { for (void* p : ptrs) cudaFreeAsync(p, s); }
};

// persistent scratch of a plan
struct Arena {
    std::vector<void*> ptrs;
    template <class T>
    cudaError_t get(T** p, uint64_t n) {
        cudaError_t e = cudaMalloc((void**)p, piece_bytes<T>(n));
        if (e == cudaSuccess) ptrs.push_back(*p);
        return e;
    }
    ~Arena() { for (void* p : ptrs) cudaFree(p); }
};

// The same over caller memory.  Carve hands out consecutive pieces of one
// buffer and fails when they would not fit; Tally only adds up the bytes Carve
// would hand out.
struct Carve {
    unsigned char* base;
    uint64_t cap, used;
    template <class T>
    cudaError_t get(T** p, uint64_t n) {
        const uint64_t bytes = piece_bytes<T>(n);
        if (used + bytes > cap) return cudaErrorMemoryAllocation;
        *p = reinterpret_cast<T*>(base + used);
        used += bytes;
        return cudaSuccess;
    }
};

struct Tally {
    uint64_t used = 0;
    template <class T>
    cudaError_t get(T** p, uint64_t n) {
        *p = nullptr;
        used += piece_bytes<T>(n);
        return cudaSuccess;
    }
};

}  // namespace hicops
