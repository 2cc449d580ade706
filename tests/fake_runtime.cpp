// A CUDA runtime of two devices without kernels, to link the library's objects
// against on the host: device memory is host memory, a launch runs nothing but
// checks what a device would: more than 48 KB of dynamic shared memory is
// refused unless the function was opted in on the current device.  Runs the
// checks named on the command line and prints "ok".
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <utility>
#include <vector>

#include "hicops.h"

namespace {
struct Dim3 { unsigned x, y, z; };
const int kSms[2] = {152, 100};
int g_device = 0, g_error = 0;
std::set<std::pair<int, const void*>> g_opted;     // (device, function)
std::map<int, unsigned> g_grid;                    // largest grid of a kernel of much shared memory, by device
struct Call { Dim3 grid, block; size_t smem; void* stream; } g_call;
int give(void** p, size_t n) {
    n = (n + 256) / 256 * 256;
    *p = aligned_alloc(256, n);
    if (*p) memset(*p, 0, n);
    return *p ? 0 : 2;
}
}  // namespace

extern "C" {
int cudaGetDevice(int* d) { *d = g_device; return 0; }
int cudaSetDevice(int d) { g_device = d; return 0; }
int cudaDeviceGetAttribute(int* v, int attr, int d) { *v = attr == 16 ? kSms[d] : 0; return 0; }
int cudaFuncSetAttribute(const void* f, int attr, int) {
    if (attr == 8) g_opted.insert({g_device, f});
    return 0;
}
int cudaMalloc(void** p, size_t n) { return give(p, n); }
int cudaMallocAsync(void** p, size_t n, void*) { return give(p, n); }
int cudaMallocFromPoolAsync(void** p, size_t n, void*, void*) { return give(p, n); }
int cudaHostAlloc(void** p, size_t n, unsigned) { return give(p, n); }
int cudaFree(void* p) { free(p); return 0; }
int cudaFreeAsync(void* p, void*) { free(p); return 0; }
int cudaFreeHost(void* p) { free(p); return 0; }
int cudaMemcpy(void* d, const void* s, size_t n, int) { memmove(d, s, n); return 0; }
int cudaMemcpyAsync(void* d, const void* s, size_t n, int, void*) { memmove(d, s, n); return 0; }
int cudaMemsetAsync(void* d, int v, size_t n, void*) { memset(d, v, n); return 0; }
int cudaMemPoolCreate(void** p, const void*) { return give(p, 1); }
int cudaMemPoolDestroy(void* p) { free(p); return 0; }
int cudaMemPoolSetAttribute(void*, int, void*) { return 0; }
int cudaStreamCreateWithFlags(void** s, unsigned) { return give(s, 1); }
int cudaStreamDestroy(void* s) { free(s); return 0; }
int cudaStreamSynchronize(void*) { return 0; }
int cudaStreamBeginCapture(void*, int) { return 801; }
int cudaStreamEndCapture(void*, void**) { return 801; }
int cudaGraphInstantiate(void**, void*, unsigned long long) { return 801; }
int cudaGraphLaunch(void*, void*) { return 801; }
int cudaGraphDestroy(void*) { return 0; }
int cudaGraphExecDestroy(void*) { return 0; }
int cudaEventCreate(void** e) { return give(e, 1); }
int cudaEventCreateWithFlags(void** e, unsigned) { return give(e, 1); }
int cudaEventDestroy(void* e) { free(e); return 0; }
int cudaEventRecord(void*, void*) { return 0; }
int cudaEventSynchronize(void*) { return 0; }
int cudaEventElapsedTime(float* ms, void*, void*) { *ms = 0; return 0; }
int cudaGetSymbolAddress(void**, const void*) { return 801; }
int cudaGetDriverEntryPointByVersion(const char*, void**, unsigned, unsigned long long, int*) { return 801; }
int cudaGetLastError() { const int e = g_error; g_error = 0; return e; }
const char* cudaGetErrorString(int) { return "refused by the fake runtime"; }

unsigned __cudaPushCallConfiguration(Dim3 grid, Dim3 block, size_t smem, void* stream) {
    g_call = Call{grid, block, smem, stream};
    return 0;
}
int __cudaPopCallConfiguration(Dim3* grid, Dim3* block, size_t* smem, void** stream) {
    *grid = g_call.grid;
    *block = g_call.block;
    *smem = g_call.smem;
    *stream = g_call.stream;
    return 0;
}
int __cudaGetKernel(const void** kernel, const void* function) { *kernel = function; return 0; }
int __cudaLaunchKernel(const void* f, Dim3 grid, Dim3, void**, size_t smem, void*) {
    if (smem <= 48u * 1024u) return 0;
    if (!g_opted.count({g_device, f})) return g_error = 1;
    if (grid.x > g_grid[g_device]) g_grid[g_device] = grid.x;
    return 0;
}
struct LaunchConfig {
    Dim3 grid, block;
    size_t smem;
    void *stream, *attrs;
    unsigned n_attrs;
};
int cudaLaunchKernelExC(const LaunchConfig* c, const void* f, void** args) {
    return __cudaLaunchKernel(f, c->grid, c->block, args, c->smem, c->stream);
}
void** __cudaRegisterFatBinary(void*) { static void* handle; return &handle; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction() {}
void __cudaRegisterVar() {}
}

#define CHECK(c)                                                                              \
    do {                                                                                      \
        if (!(c)) { printf("line %d: %s (%s)\n", __LINE__, #c, hicops_last_error()); return 1; } \
    } while (0)

// An index on each device, and searches in every launch shape.
int two_devices() {
    const char seq[] = "PEPTIDEKAAAGGGKMMMSSSRTTTVVVKLLLNNNR";
    const uint64_t off[2] = {0, sizeof(seq) - 1};
    const hicops_proteins prot{1, seq, off};
    const uint32_t n = 4096;
    std::vector<uint64_t> peak(n + 1, 0);
    std::vector<double> prec(n, 500.0), tol(n, 10.0);
    std::vector<uint8_t> z(n, 2);
    const float none = 0;
    for (uint32_t min_shared : {1u, 2u, 4u})
        for (uint32_t bins : {50u, 300u, 700u}) {
            hicops_params p{};
            p.min_len = 5;
            p.max_len = 20;
            p.min_mass = 100;
            p.max_mass = 5000;
            p.frag_mz_min = 100;
            p.frag_mz_max = 2000;
            p.bin_width_da = 1.0;
            p.top_n_peaks = bins;
            p.min_shared = min_shared;
            p.top_k = 5;
            p.hist_bins = 256;
            p.intensity_scale = 100;
            std::vector<hicops_psm> psm((size_t)n * p.top_k);
            for (int device : {0, 1, 0}) {
                cudaSetDevice(device);
                hicops_index* idx = nullptr;
                CHECK(hicops_build_index(&prot, nullptr, 0, &p, &idx) == HICOPS_OK);
                for (uint32_t threads : {0u, 256u, 384u, 512u}) {
                    const hicops_search_config cfg{threads, 0, 0, 0};
                    CHECK(hicops_index_set_config(idx, &cfg) == HICOPS_OK);
                    const hicops_batch b{n, 1, peak.data(), &none, &none, prec.data(), z.data(), tol.data(), nullptr};
                    CHECK(hicops_search(idx, &b, psm.data(), nullptr, nullptr) == HICOPS_OK);
                }
                hicops_index_free(idx);
            }
        }
    for (int device : {0, 1}) CHECK(g_grid[device] == 3u * kSms[device]);   // three CTAs an SM at most
    return 0;
}

// Device bytes of a server's launch of n spectra of npk peaks before windows
// were cut by cost: a request that filled a pool then has to be taken now.
uint64_t bytes_before(uint64_t n, uint64_t npk, uint64_t k, uint64_t bins, uint64_t sms) {
    auto piece = [](uint64_t b) { return (b + 255) / 256 * 256; };
    uint64_t segs = (8 * sms + n - 1) / n, scan = 1;
    segs = segs < 1 ? 1 : segs > 64 ? 64 : segs;
    for (uint64_t m = n; m > 2048;) {
        m = (m + 2047) / 2048;
        scan += 2 * m;
    }
    uint64_t b = piece(8 * (n + 1)) + 2 * piece(npk ? 4 * npk : 1) + 2 * piece(8 * n) + piece(n) + piece(32 * n * k) +
                 piece(1024 * n) + piece(4 * n);                                             // spectra and results
    b += 2 * piece(4 * n * bins) + 4 * piece(4 * n) + piece(8 * (n + 1)) + piece(8 * scan);   // queries, windows, prefix
    b += piece(16 * n * segs * k) + piece(8) + 2 * piece(4 * n * segs) + piece(4 * 2 * 64);   // units and their order
    return b + piece(1024 * n) + piece(4 * n);
}

int server_blocks() {
    const char seq[] = "PEPTIDEKAAAGGGKMMMSSSRTTTVVVKLLLNNNR";
    const uint64_t off[2] = {0, sizeof(seq) - 1};
    const hicops_proteins prot{1, seq, off};
    for (uint32_t k : {1u, 5u, 32u})
        for (uint32_t bins : {1u, 100u, 1000u}) {
            hicops_params p{};
            p.min_len = 5;
            p.max_len = 20;
            p.min_mass = 100;
            p.max_mass = 5000;
            p.frag_mz_min = 100;
            p.frag_mz_max = 2000;
            p.bin_width_da = 1.0;
            p.top_n_peaks = bins;
            p.min_shared = 4;
            p.top_k = k;
            p.hist_bins = 256;
            p.intensity_scale = 100;
            hicops_index* idx = nullptr;
            CHECK(hicops_build_index(&prot, nullptr, 0, &p, &idx) == HICOPS_OK);
            for (uint32_t n : {1u, 2u, 5u, 19u, 64u, 65u, 512u, 1216u, 1217u, 5000u, 32768u}) {
                const uint64_t npk = n == 1 ? 512 : 100ull * n;
                hicops_server_cfg cfg{1, n, bytes_before(n, npk, k, bins, (uint64_t)kSms[0])};
                hicops_server* srv = nullptr;
                CHECK(hicops_server_create(idx, &cfg, &srv) == HICOPS_OK);
                std::vector<uint64_t> peak(n + 1);
                for (uint32_t i = 0; i <= n; ++i) peak[i] = npk * i / n;
                std::vector<float> mz(npk, 500.0f), inten(npk, 1.0f);
                std::vector<double> prec(n, 500.0), tol(n, 10.0);
                std::vector<uint8_t> z(n, 2);
                const hicops_batch b{n, 0, peak.data(), mz.data(), inten.data(), prec.data(), z.data(), tol.data(), nullptr};
                uint64_t ticket = 0;
                CHECK(hicops_server_submit(srv, &b, &ticket) == HICOPS_OK);
                std::vector<hicops_psm> psm((size_t)n * k);
                CHECK(hicops_server_poll(srv, ticket, 60000, psm.data(), nullptr, nullptr) == HICOPS_OK);
                hicops_server_destroy(srv);
            }
            hicops_index_free(idx);
        }
    return 0;
}

int main(int argc, char** argv) {
    for (int i = 1; i < argc; ++i) {
        const int bad = !strcmp(argv[i], "two_devices") ? two_devices() : !strcmp(argv[i], "server_blocks") ? server_blocks() : 1;
        if (bad) return bad;
    }
    puts("ok");
    return 0;
}
