// Host check of the search's allocators (pieces.h): the runtime's allocation
// calls are replaced by ones that note the bytes asked for, and every piece has
// to hold the 16-byte vector that its last element lies in.  Prints "ok".
#include <cstdio>

#include "pieces.h"

namespace {
unsigned char g_memory[1 << 20];
uint64_t g_bytes = 0;   // of the last allocation
cudaError_t note(void** p, size_t bytes) {
    *p = g_memory;
    g_bytes = bytes;
    return cudaSuccess;
}
}  // namespace

extern "C" {
cudaError_t cudaMalloc(void** p, size_t bytes) { return note(p, bytes); }
cudaError_t cudaMallocAsync(void** p, size_t bytes, cudaStream_t) { return note(p, bytes); }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t bytes, cudaMemPool_t, cudaStream_t) { return note(p, bytes); }
cudaError_t cudaFree(void*) { return cudaSuccess; }
cudaError_t cudaFreeAsync(void*, cudaStream_t) { return cudaSuccess; }
}

template <class T>
bool whole(const char* who, uint64_t n, uint64_t bytes) {
    const uint64_t last = n ? n - 1 : 0;
    const uint64_t need = (last * sizeof(T) / 16 + 1) * 16;   // the end of the last element's vector
    if (bytes >= need && bytes % 16 == 0) return true;
    printf("%s: %llu elements of %zu bytes in a piece of %llu\n", who, (unsigned long long)n, sizeof(T),
           (unsigned long long)bytes);
    return false;
}

template <class T>
bool check(uint64_t n) {
    T* p = nullptr;
    hicops::Arena arena;
    arena.get(&p, n);
    bool ok = whole<T>("Arena", n, g_bytes);
    for (int pool = 0; pool < 2; ++pool) {
        hicops::Scratch scratch(nullptr, pool ? reinterpret_cast<cudaMemPool_t>(g_memory) : nullptr);
        scratch.get(&p, n);
        ok = whole<T>("Scratch", n, g_bytes) && ok;
    }
    hicops::Tally tally;
    tally.get(&p, n);
    ok = whole<T>("Tally", n, tally.used) && ok;
    hicops::Carve carve{g_memory, sizeof(g_memory), 0};
    ok = carve.get(&p, n) == cudaSuccess && carve.used == tally.used && whole<T>("Carve", n, carve.used) && ok;
    return ok;
}

int main() {
    bool ok = true;
    for (uint64_t n : {0, 1, 2, 3, 4, 5, 63, 64, 65, 12345}) ok = check<uint32_t>(n) && check<uint64_t>(n) && check<uint8_t>(n) && ok;
    if (ok) puts("ok");
    return ok ? 0 : 1;
}
