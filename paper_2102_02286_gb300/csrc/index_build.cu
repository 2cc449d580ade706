// Device side of superstep 1 (paper: Supplementary Algorithm 1,
// model_spectrum + parallel_index): b/y model spectra for every database
// entry, integer m/z binning, and the fragment-ion index as a CSR whose
// buckets list peptide ids in ascending order.  The paper indexes with a
// CFIR-style inverted index built by a parallel sort; here the sort is a
// stable LSD radix sort by bin over (bin, pid, isY) keys emitted in pid
// order, so each bucket comes out pid-ascending without a comparison sort.
#include <algorithm>
#include <new>
#include <cmath>
#include <chrono>
#include <vector>

#include "dev_common.cuh"

namespace hicops {
namespace {

constexpr int kIonThreads = 128;
constexpr uint64_t kPoolKeep = 128ull << 20;   // 12,000 spectra of 500 peaks; no more for 64 shards than 8 GB
constexpr int kIonStage = 2048;      // ion bins a warp stages in shared memory (8 KB)

struct IonArgs {
    const uint32_t* base;        // [P] base peptide id
    const uint64_t* mask;        // [P] modified-position mask
    const uint64_t* base_off;    // [B+1]
    const char* residues;        // concatenated base sequences
    const double* mres;          // [128]
    const double* mmod;          // [128]
    double w, mz_lo, mz_hi;
    uint64_t P;
    // the same masses and limits in bins, with 32 fraction bits (fixed_ions)
    const int64_t* fix;          // [2][128]: unmodified, modified
    int64_t b_add, y_add;        // proton; water + proton
    int64_t lo, hi;
    uint32_t tol;                // most that a fixed-point value can be off, in 2^-32 bins
    int fixed;                   // the fixed-point values hold for this index
};

// Visits the distinct in-range ion bins of one peptide in ascending bin
// order; a bin reached by both a b and a y ion is reported once, as b.
// b_i = (m_1 + .. + m_i) + proton, summed left to right;
// y_i = ((m_L + m_{L-1} + .. + m_{i+1}) + H2O) + proton, summed from the C terminus.
// Collected and sorted, so a modification that takes a residue's mass below
// zero (sums that do not ascend) is indexed alike.
template <class F>
__device__ __noinline__ void each_ion_bin_fp64(const IonArgs& a, uint64_t pid, F emit) {
    const uint32_t b = a.base[pid];
    const uint64_t m = a.mask[pid];
    const char* s = a.residues + a.base_off[b];
    const int L = (int)(a.base_off[b + 1] - a.base_off[b]);
    uint32_t list[2 * kMaxLen];      // bin << 1 | isY, ascending
    int n = 0;
    auto add = [&](double mz, uint32_t isy) {
        if (mz < a.mz_lo || mz >= a.mz_hi) return;
        const uint32_t v = ((uint32_t)floor(mz / a.w) << 1) | isy;   // n_bins < 2^31 (parameter check)
        int i = n++;
        for (; i > 0 && list[i - 1] > v; --i) list[i] = list[i - 1];
        list[i] = v;
    };
    auto rm = [&](int j) -> double {
        const unsigned char c = (unsigned char)s[j];
        return ((m >> j) & 1ull) ? a.mmod[c] : a.mres[c];
    };
    double pre = 0.0, suf = 0.0;
    for (int i = 1; i < L; ++i) {
        pre = pre + rm(i - 1);
        add(pre + kProtonDa, 0u);
    }
    for (int i = L - 1; i >= 1; --i) {
        suf = suf + rm(i);
        add((suf + kWaterDa) + kProtonDa, 1u);
    }
    for (int i = 0; i < n; ++i)
        if (i == 0 || (list[i] >> 1) != (list[i - 1] >> 1)) emit(list[i] >> 1, list[i] & 1u);
}

// The same visits from fixed-point sums in units of a bin (32 fraction bits):
// the high word of a sum is the bin, so an ion costs integer additions where
// the FP64 form costs a division on a unit of 2 lanes a clock.  a.tol bounds
// the distance between the fixed-point value and the FP64 quotient, so a value
// farther than that from every bin edge and from both limits of the m/z range
// has the FP64 form's bin.  At a value nearer than that the visit ends and
// returns false: everything visited up to there is a prefix of the FP64
// form's visits, which the caller then takes from the start.
// One ion per step, from the stream with the lower bin (b at equal bins).
template <class F>
__device__ __forceinline__ bool each_ion_bin_fixed(const IonArgs& a, const int64_t* fix, uint64_t pid, F&& emit) {
    const uint32_t b = a.base[pid];
    const uint64_t m = a.mask[pid];
    const char* s = a.residues + a.base_off[b];
    const int L = (int)(a.base_off[b + 1] - a.base_off[b]);
    if (L < 2) return true;
    constexpr int64_t kDone = 0x7fffffffffffffffll;
    bool sure = true;
    auto check = [&](int64_t v) -> int64_t {
        sure = sure && (uint32_t)v + a.tol >= 2u * a.tol && llabs(v - a.lo) > (int64_t)a.tol &&
               llabs(v - a.hi) > (int64_t)a.tol;
        return v >= a.hi ? kDone : v;
    };
    auto rm = [&](int j) { return fix[((uint32_t)(m >> j) & 1u) << 7 | (unsigned char)s[j]]; };
    int ib = 0, iy = L - 1;               // residues taken next
    int64_t sb = a.b_add + rm(0), sy = a.y_add + rm(L - 1);
    int64_t vb = check(sb), vy = check(sy);
    uint32_t last = 0xffffffffu;
    while (sure && (vb != kDone || vy != kDone)) {
        const bool tb = (vb >> 32) <= (vy >> 32);
        const int64_t v = tb ? vb : vy;
        const uint32_t bin = (uint32_t)(v >> 32);
        if (v >= a.lo && bin != last) { emit(bin, tb ? 0u : 1u); last = bin; }
        const int j = tb ? ++ib : --iy;
        const bool more = tb ? j < L - 1 : j >= 1;
        int64_t nv = kDone;
        if (more) {
            const int64_t sum = (tb ? sb : sy) + rm(j);
            nv = check(sum);
            if (tb) sb = sum; else sy = sum;
        }
        if (tb) vb = nv; else vy = nv;
    }
    return sure;
}

// 2.73 -> 0.20 ms for 50 M ions of 1.6 M peptides: bound by the issue of some 30
// integer instructions an ion.
__global__ void __launch_bounds__(kIonThreads) ion_count_kernel(IonArgs a, uint32_t* __restrict__ count,
                                                                uint32_t* __restrict__ groups) {
    __shared__ int64_t fix[256];
    for (int i = threadIdx.x; i < 256; i += blockDim.x) fix[i] = a.fix[i];
    __syncthreads();
    const uint64_t pid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (pid >= a.P) return;
    uint32_t n = 0;
    if (!a.fixed || !each_ion_bin_fixed(a, fix, pid, [&](uint32_t, uint32_t) { ++n; })) {
        uint32_t m = 0;
        each_ion_bin_fp64(a, pid, [&](uint32_t, uint32_t) { ++m; });
        n = m;
    }
    count[pid] = n;
    groups[pid] = (n + 3u) >> 2;   // the forward list's length in groups of 4
}

// Keys for the sort by bin, and the forward list.  A warp's 32 lists are
// neighbours in both arrays: they are staged in shared memory, padding
// included, and written from there in whole lines; lists that do not fit
// (more than 64 ions a peptide) are written ion by ion.
// 2.74 -> 0.52 ms for 50 M ions (600 MB written).
__global__ void __launch_bounds__(kIonThreads) ion_emit_kernel(IonArgs a, const uint64_t* __restrict__ off,
                                                               uint64_t* __restrict__ keys,
                                                               const uint64_t* __restrict__ fwd_off,
                                                               uint32_t* __restrict__ fwd) {
    __shared__ int64_t fix[256];
    __shared__ __align__(16) uint32_t stage_all[kIonThreads / 32][kIonStage];
    for (int i = threadIdx.x; i < 256; i += blockDim.x) fix[i] = a.fix[i];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const uint64_t pid0 = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u);
    if (pid0 >= a.P) return;
    uint32_t* stage = stage_all[threadIdx.x >> 5];
    const uint64_t pid = pid0 + lane;
    const bool mine = pid < a.P;
    const uint64_t f0 = fwd_off[pid0], f1 = fwd_off[min(pid0 + 32, a.P)];
    const uint64_t o = mine ? off[pid] : 0, f = mine ? fwd_off[pid] : f0;
    const bool fits = (f1 - f0) * 4 <= (uint64_t)kIonStage;
    const uint32_t low = (uint32_t)(pid << 1);
    uint32_t n = 0;
    if (mine) {
        uint32_t* list = fits ? stage + 4 * (uint32_t)(f - f0) : fwd + 4 * f;
        auto put = [&](uint32_t bin, uint32_t isy) {
            list[n] = (bin << 1) | isy;   // n_bins < 2^31 (parameter check)
            if (!fits) keys[o + n] = ((uint64_t)bin << 32) | (low | isy);
            ++n;
        };
        if (!a.fixed || !each_ion_bin_fixed(a, fix, pid, put)) {
            uint32_t m = 0;
            uint32_t* to = list;
            uint64_t* key = fits ? nullptr : keys + o;
            each_ion_bin_fp64(a, pid, [&m, to, key, low](uint32_t bin, uint32_t isy) {
                to[m] = (bin << 1) | isy;
                if (key) key[m] = ((uint64_t)bin << 32) | (low | isy);
                ++m;
            });
            n = m;
        }
        for (uint32_t i = n; i & 3; ++i) list[i] = 0xffffffffu;
    }
    if (!fits) return;   // the whole warp
    __syncwarp();
    uint4* out = reinterpret_cast<uint4*>(fwd) + f0;
    const uint4* in = reinterpret_cast<const uint4*>(stage);
    for (uint32_t i = lane; i < (uint32_t)(f1 - f0); i += 32) out[i] = in[i];
    for (int l = 0; l < 32; ++l) {
        const uint32_t cnt = __shfl_sync(0xffffffffu, n, l);
        const uint64_t to = __shfl_sync(0xffffffffu, o, l);
        const uint32_t from = 4 * (uint32_t)(__shfl_sync(0xffffffffu, f, l) - f0);
        const uint32_t plow = (uint32_t)((pid0 + l) << 1);
        for (uint32_t i = lane; i < cnt; i += 32) {
            const uint32_t e = stage[from + i];
            keys[to + i] = ((uint64_t)(e >> 1) << 32) | (plow | (e & 1u));
        }
    }
}

// LS[v] = round(2^32 log10 v) of the host's libm.  The device's log10 and the
// host's each lie within 2 ulp of the true value, under 2^-14 in these units
// (log10 v < 8), so a value farther than 2^-10 from a rounding edge rounds
// alike; the others (2 in 1,000) are listed and computed by the host.
__global__ void ls_kernel(int64_t* __restrict__ ls, uint32_t n, uint32_t* __restrict__ list,
                          unsigned long long* __restrict__ listed) {
    const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n) return;
    const double x = v < 2 ? 0.0 : ldexp(log10((double)v), 32);
    const double lo = floor(x);
    ls[v] = (int64_t)floor(x + 0.5);
    if (fabs((x - lo) - 0.5) < 0x1p-10) list[atomicAdd(listed, 1ull)] = v;
}

__global__ void ls_patch_kernel(int64_t* __restrict__ ls, const uint32_t* __restrict__ list,
                                const int64_t* __restrict__ value, uint32_t n) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) ls[list[i]] = value[i];
}

// ---- stable LSD radix sort on the bin field (bits 32..) of 64-bit keys

constexpr int kRsBits = 8;
constexpr int kRsRadix = 1 << kRsBits;
constexpr int kRsWarps = 8;
constexpr int kRsRounds = 16;
constexpr int kRsTile = kRsWarps * 32 * kRsRounds;

__device__ __forceinline__ uint32_t digit_of(uint64_t k, int shift) {
    return (uint32_t)(k >> shift) & (kRsRadix - 1);
}

// counts[d * ntiles + tile] = number of keys of tile with digit d
__global__ void __launch_bounds__(kRsWarps * 32) rs_count_kernel(const uint64_t* __restrict__ keys, uint64_t n,
                                                                 int shift, uint32_t* __restrict__ counts,
                                                                 uint64_t ntiles) {
    __shared__ uint32_t h[kRsRadix];
    for (int i = threadIdx.x; i < kRsRadix; i += blockDim.x) h[i] = 0;
    __syncthreads();
    const uint64_t base = (uint64_t)blockIdx.x * kRsTile;
    for (int i = threadIdx.x; i < kRsTile; i += blockDim.x) {
        const uint64_t g = base + i;
        if (g < n) atomicAdd(&h[digit_of(keys[g], shift)], 1u);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < kRsRadix; d += blockDim.x) counts[(uint64_t)d * ntiles + blockIdx.x] = h[d];
}

// Stable scatter: warp w owns items [w*32*R, (w+1)*32*R) of the tile and
// walks them in order, 32 at a time; equal digits inside a round are ranked
// by lane.
__global__ void __launch_bounds__(kRsWarps * 32) rs_scatter_kernel(const uint64_t* __restrict__ in,
                                                                   uint64_t* __restrict__ out, uint64_t n,
                                                                   int shift, const uint64_t* __restrict__ offs,
                                                                   uint64_t ntiles) {
    __shared__ uint32_t wcount[kRsWarps][kRsRadix];
    __shared__ uint64_t tile_base[kRsRadix];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < kRsWarps * kRsRadix; i += blockDim.x) (&wcount[0][0])[i] = 0;
    for (int d = threadIdx.x; d < kRsRadix; d += blockDim.x) tile_base[d] = offs[(uint64_t)d * ntiles + blockIdx.x];
    __syncthreads();
    const uint64_t wbase = (uint64_t)blockIdx.x * kRsTile + (uint64_t)w * 32 * kRsRounds;
    const unsigned lt = (1u << lane) - 1u;
    // pass 1: per-warp digit counts
    for (int r = 0; r < kRsRounds; ++r) {
        const uint64_t g = wbase + (uint64_t)r * 32 + lane;
        const uint32_t d = g < n ? digit_of(in[g], shift) : 0xffffu;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        if (d != 0xffffu && (peers & lt) == 0) wcount[w][d] += __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // exclusive prefix over warps, per digit
    for (int d = threadIdx.x; d < kRsRadix; d += blockDim.x) {
        uint32_t run = 0;
        for (int ww = 0; ww < kRsWarps; ++ww) {
            uint32_t c = wcount[ww][d];
            wcount[ww][d] = run;
            run += c;
        }
    }
    __syncthreads();
    // pass 2: scatter
    for (int r = 0; r < kRsRounds; ++r) {
        const uint64_t g = wbase + (uint64_t)r * 32 + lane;
        uint64_t k = 0;
        uint32_t d = 0xffffu;
        if (g < n) { k = in[g]; d = digit_of(k, shift); }
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        uint32_t before = 0;
        if (d != 0xffffu) before = wcount[w][d];
        __syncwarp();
        if (d != 0xffffu) {
            out[tile_base[d] + before + __popc(peers & lt)] = k;
            if ((peers & lt) == 0) wcount[w][d] = before + __popc(peers);
        }
        __syncwarp();
    }
}

// off[b] = first position whose bin is >= b (keys sorted by bin)
__global__ void bucket_off_kernel(const uint64_t* __restrict__ keys, uint64_t n, uint32_t nbins,
                                  uint64_t* __restrict__ off) {
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i > n) return;
    const int64_t prev = i == 0 ? -1 : (int64_t)(keys[i - 1] >> 32);
    const int64_t cur = i == n ? (int64_t)nbins : (int64_t)(keys[i] >> 32);
    for (int64_t b = prev + 1; b <= cur; ++b) off[b] = i;
}

// Per bucket: its size rounded up to whole groups of 4 entries (16 bytes, so
// that every bucket starts 16-byte aligned in the entry array), whether it
// holds an entry, whether it is hot; and the largest size.
__global__ void __launch_bounds__(256) bucket_kernel(const uint64_t* __restrict__ off, uint32_t nbins, uint64_t hot_lo,
                                                     uint32_t* __restrict__ psz, uint32_t* __restrict__ some,
                                                     uint32_t* __restrict__ hot, unsigned long long* __restrict__ mx) {
    __shared__ unsigned long long block_max;
    if (threadIdx.x == 0) block_max = 0;
    __syncthreads();
    const uint32_t b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < nbins) {
        const uint64_t size = off[b + 1] - off[b];
        psz[b] = (uint32_t)((size + 3) & ~3ull);
        some[b] = size ? 1u : 0u;
        hot[b] = size >= hot_lo ? 1u : 0u;
        if (size) atomicMax(&block_max, (unsigned long long)size);
    }
    __syncthreads();
    if (threadIdx.x == 0 && block_max) atomicMax(mx, block_max);
}

// row of every flagged bin (its rank among the flagged; -1 for the others), and the bins by rank
__global__ void row_of_kernel(const uint32_t* __restrict__ flag, const uint64_t* __restrict__ scan, uint32_t nbins,
                              int32_t* __restrict__ row, uint32_t* __restrict__ bin_of) {
    const uint32_t b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nbins) return;
    row[b] = flag[b] ? (int32_t)scan[b] : -1;
    if (flag[b] && bin_of) bin_of[scan[b]] = b;
}

// The stored form of the sorted keys, one read of them:
// entry[poff[bin] + rank in bucket] = pid << 1 | isY; the up to 3 slots after
// a bucket's last entry keep the pad value 0xffffffff (pid 2^31 - 1, above
// every peptide id, so a bucket stays pid-sorted and no window contains it).
// Chunk skip table: skip[row * stride + j] = number of entries of the bucket
// with pid < j * 2^kChunkShift, for j = 0 .. stride-1 (the last column is the
// bucket size).  Every cell is written by exactly one entry.
__global__ void store_kernel(const uint64_t* __restrict__ keys, uint64_t n, const uint64_t* __restrict__ off,
                             const uint64_t* __restrict__ poff, uint32_t* __restrict__ entry,
                             const int32_t* __restrict__ row, uint32_t stride, uint32_t* __restrict__ skip) {
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint64_t key = keys[i];
    const uint32_t bin = (uint32_t)(key >> 32);
    const uint32_t ch = ((uint32_t)key >> 1) >> kChunkShift;
    const uint64_t b0 = off[bin], b1 = off[bin + 1];
    const uint32_t rel = (uint32_t)(i - b0);
    entry[poff[bin] + rel] = (uint32_t)key;
    const uint32_t jlo = (i == b0) ? 0u : (((uint32_t)keys[i - 1] >> 1) >> kChunkShift) + 1u;
    if (jlo > ch && i + 1 != b1) return;
    uint32_t* base = skip + (uint64_t)row[bin] * stride;
    for (uint32_t j = jlo; j <= ch; ++j) base[j] = rel;
    if (i + 1 == b1)
        for (uint32_t j = ch + 1; j < stride; ++j) base[j] = (uint32_t)(b1 - b0);
}

// Hot buckets as pid bitmaps: bit pid of hb[h] (b ion) or hy[h] (y ion).  One
// block makes one chunk (2^kChunkShift pids) of one bucket's two bitmaps in
// shared memory from the chunk's run of entries and writes them whole, zero
// words included; the last chunk's block also writes the row's spare words.
// 3.34 ms (a global atomic for every entry, and a memset) -> 0.02 ms for an
// index of 50 M entries.
__global__ void __launch_bounds__(256) hot_fill_kernel(const uint32_t* __restrict__ entry,
                                                       const uint64_t* __restrict__ poff,
                                                       const uint32_t* __restrict__ hot_bin,
                                                       const int32_t* __restrict__ row, uint32_t stride,
                                                       const uint32_t* __restrict__ skip, uint64_t words,
                                                       uint32_t* __restrict__ hb, uint32_t* __restrict__ hy,
                                                       uint32_t* __restrict__ hflags) {
    constexpr uint32_t kWords = kChunk / 32;
    __shared__ __align__(16) uint32_t bm[2][kWords];
    __shared__ uint32_t seen;
    const uint32_t chunks = stride - 1, h = blockIdx.x / chunks, c = blockIdx.x % chunks;
    for (uint32_t i = threadIdx.x; i < 2 * kWords; i += blockDim.x) (&bm[0][0])[i] = 0;
    if (threadIdx.x == 0) seen = 0;
    __syncthreads();
    const uint32_t bin = hot_bin[h];
    const uint32_t* sk = skip + (uint64_t)row[bin] * stride + c;
    const uint32_t* e = entry + poff[bin];
    uint32_t kinds = 0;
    for (uint32_t i = sk[0] + threadIdx.x; i < sk[1]; i += blockDim.x) {
        const uint32_t v = e[i], pid = (v >> 1) & (kChunk - 1);
        atomicOr(&bm[v & 1u][pid >> 5], 1u << (pid & 31));
        kinds |= (v & 1u) ? 2u : 1u;
    }
    kinds = __reduce_or_sync(0xffffffffu, kinds);
    if ((threadIdx.x & 31) == 0 && kinds) atomicOr(&seen, kinds);
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < 2 * kWords / 4; i += blockDim.x) {
        const uint32_t y = i >= kWords / 4, j = i - y * (kWords / 4);
        uint4* to = reinterpret_cast<uint4*>((y ? hy : hb) + h * words + (uint64_t)c * kWords);   // words % 4 == 0
        to[j] = reinterpret_cast<const uint4*>(bm[y])[j];
    }
    if (c + 1 == chunks)
        for (uint64_t i = (uint64_t)chunks * kWords + threadIdx.x; i < words; i += blockDim.x)
            hb[h * words + i] = hy[h * words + i] = 0;
    if (threadIdx.x == 0 && seen) atomicOr(&hflags[h], seen);
}

// the search's record of every bin
__global__ void bin_info_kernel(const uint64_t* __restrict__ off, const int32_t* __restrict__ row,
                                const int32_t* __restrict__ hot_id, const uint32_t* __restrict__ hflags,
                                uint32_t nbins, BinInfo* __restrict__ out) {
    const uint32_t b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nbins) return;
    const int32_t h = hot_id[b];
    const uint32_t groups = (uint32_t)((off[b + 1] - off[b]) >> 2);   // < 2^30 (bucket limit)
    out[b] = BinInfo{(uint32_t)(off[b] >> 2), row[b], h, groups << 2 | (h >= 0 ? hflags[h] : 0u)};
}

template <class T>
cudaError_t dalloc(T** p, uint64_t n, std::vector<void*>& tmp) {
    cudaError_t e = cudaMalloc((void**)p, sizeof(T) * (n ? n : 1));
    if (e == cudaSuccess) tmp.push_back(*p);
    return e;
}

// The residue masses and m/z limits in bins with 32 fraction bits, and how far
// a sum of them can lie from the FP64 quotient: a fixed-point term is off by
// half a unit and by its own division's rounding, the FP64 sum by half an ulp
// of at most the range's end plus one residue for each of its additions, the
// FP64 quotient by half an ulp.  66 terms and additions (kMaxLen and two
// constants), all doubled.  Left to FP64 altogether: masses that are not
// positive and finite, and grids so fine that a sum could leave 60 bits or the
// bound reach an eighth of a bin.
void fixed_ions(IonArgs* a, const double* mres, const double* mmod, int64_t* fix) {
    a->fixed = 0;
    double top = 0.0;
    for (int c = 0; c < 256; ++c) {
        const double m = c < 128 ? mres[c] : mmod[c - 128];
        fix[c] = 0;
        // bytes that are no residue have no mass and occur in no peptide
        if (m == 0.0) continue;
        if (!(m > 0.0) || !std::isfinite(m)) return;
        top = std::max(top, m);
    }
    const double reach = (a->mz_hi + top + kWaterDa + kProtonDa) / a->w;
    const double tol = 2.0 * (34.0 + 70.0 * 0x1p-53 * reach * 0x1p32);
    if (!(reach < 0x1p28) || !(tol < 0x1p29)) return;
    auto in_bins = [&](double m) { return (int64_t)std::llrint(std::ldexp(m / a->w, 32)); };
    for (int c = 0; c < 256; ++c) fix[c] = in_bins(c < 128 ? mres[c] : mmod[c - 128]);
    a->b_add = in_bins(kProtonDa);
    a->y_add = in_bins(kWaterDa) + in_bins(kProtonDa);
    a->lo = in_bins(a->mz_lo);
    a->hi = in_bins(a->mz_hi);
    a->tol = (uint32_t)std::ceil(tol);
    a->fixed = 1;
}

struct TmpFree {
    std::vector<void*> ptrs;
    void release(void* p) {
        ptrs.erase(std::find(ptrs.begin(), ptrs.end(), p));
        cudaFree(p);
    }
    ~TmpFree() { for (void* p : ptrs) cudaFree(p); }
};

}  // namespace

void free_device_index(hicops_index* idx) {
    DeviceIndex& d = idx->dev;
    if (d.device >= 0) {
        int cur = -1;
        cudaGetDevice(&cur);
        if (cur != d.device) cudaSetDevice(d.device);
        cudaFree(d.mass);
        cudaFree(d.off);
        cudaFree(d.entry);
        cudaFree(d.lf);
        cudaFree(d.ls);
        cudaFree(d.skip_row);
        cudaFree(d.skip);
        cudaFree(d.hot_id);
        cudaFree(d.hot_b);
        cudaFree(d.hot_y);
        cudaFree(d.hot_flags);
        cudaFree(d.bins);
        cudaFree(d.fwd_off);
        cudaFree(d.fwd);
        cudaFree(d.pid_map);
        for (void* e : d.ev) if (e) cudaEventDestroy((cudaEvent_t)e);
        if (d.pool) cudaMemPoolDestroy((cudaMemPool_t)d.pool);   // (the frees above have waited for its last call)
        if (cur >= 0 && cur != d.device) cudaSetDevice(cur);
    }
    d = DeviceIndex{};
}

hicops_status upload_index(hicops_index* idx) {
    if (idx->dev.ready) return HICOPS_OK;
    auto t0 = std::chrono::steady_clock::now();
    DeviceIndex& d = idx->dev;
    HC_CUDA(cudaGetDevice(&d.device));
    const hicops_status ready = search_setup(idx);
    if (ready != HICOPS_OK) return ready;
    const hicops_params& p = idx->p;
    const uint64_t P = idx->mass.size();
    const uint64_t B = idx->bases->base_off.size() - 1;
    TmpFree tf;   // destroyed after the stream guard has synchronised
    cudaStream_t s;
    HC_CUDA(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
    struct StreamGuard { cudaStream_t s; ~StreamGuard() { cudaStreamSynchronize(s); cudaStreamDestroy(s); } } sg{s};

    // Scratch of the searches: a pool of the index's own, which keeps up to
    // kPoolKeep bytes over a synchronisation.  The device's default pool keeps
    // none, and mapping a search's scratch anew costs it 200 us.
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = d.device;
    cudaMemPool_t pool;
    HC_CUDA(cudaMemPoolCreate(&pool, &props));
    d.pool = pool;
    uint64_t keep = kPoolKeep;
    HC_CUDA(cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep));

    // persistent parts
    HC_CUDA(cudaMalloc(&d.mass, sizeof(double) * (P ? P : 1)));
    HC_CUDA(cudaMemcpyAsync(d.mass, idx->mass.data(), sizeof(double) * P, cudaMemcpyHostToDevice, s));
    if (!idx->pid_map.empty()) {   // a subset: its rows report global pids
        HC_CUDA(cudaMalloc(&d.pid_map, sizeof(uint32_t) * P));
        HC_CUDA(cudaMemcpyAsync(d.pid_map, idx->pid_map.data(), sizeof(uint32_t) * P, cudaMemcpyHostToDevice, s));
    }
    HC_CUDA(cudaMalloc(&d.off, sizeof(uint64_t) * (idx->n_bins + 1)));
    // score tables (host libm, FP64): LF[n] = round(2^32 sum_{i<=n} log10 i), LS[s] = round(2^32 log10 s)
    std::vector<int64_t> lf(kMaxLen + 1);
    double acc = 0.0;
    lf[0] = 0;
    for (uint32_t n = 1; n <= kMaxLen; ++n) {
        if (n >= 2) acc = acc + std::log10((double)n);
        lf[n] = std::llround(std::ldexp(acc, 32));
    }
    const uint32_t n_ls = (uint32_t)idx->s_max + 1;   // s_max < 2^20 (parameter check)
    HC_CUDA(cudaMalloc(&d.lf, sizeof(int64_t) * lf.size()));
    HC_CUDA(cudaMalloc(&d.ls, sizeof(int64_t) * n_ls));
    HC_CUDA(cudaMemcpyAsync(d.lf, lf.data(), sizeof(int64_t) * lf.size(), cudaMemcpyHostToDevice, s));
    uint64_t* d_total;        // ions; LS values left to the host; largest bucket
    HC_CUDA(dalloc(&d_total, 3, tf.ptrs));
    HC_CUDA(cudaMemsetAsync(d_total, 0, 3 * sizeof(uint64_t), s));
    uint32_t* d_list;
    HC_CUDA(dalloc(&d_list, n_ls, tf.ptrs));
    ls_kernel<<<(n_ls + 255) / 256, 256, 0, s>>>(d.ls, n_ls, d_list, (unsigned long long*)d_total + 1);
    HC_CUDA(cudaGetLastError());

    // temporaries: peptide table
    uint32_t* d_base;
    uint64_t *d_mask, *d_boff;
    char* d_res;
    double *d_mres, *d_mmod;
    int64_t* d_fix;
    HC_CUDA(dalloc(&d_base, P, tf.ptrs));
    HC_CUDA(dalloc(&d_mask, P, tf.ptrs));
    HC_CUDA(dalloc(&d_boff, B + 1, tf.ptrs));
    HC_CUDA(dalloc(&d_res, idx->bases->residues.size() + 1, tf.ptrs));
    HC_CUDA(dalloc(&d_mres, 128, tf.ptrs));
    HC_CUDA(dalloc(&d_mmod, 128, tf.ptrs));
    HC_CUDA(dalloc(&d_fix, 256, tf.ptrs));
    HC_CUDA(cudaMemcpyAsync(d_base, idx->base.data(), sizeof(uint32_t) * P, cudaMemcpyHostToDevice, s));
    HC_CUDA(cudaMemcpyAsync(d_mask, idx->mask.data(), sizeof(uint64_t) * P, cudaMemcpyHostToDevice, s));
    HC_CUDA(cudaMemcpyAsync(d_boff, idx->bases->base_off.data(), sizeof(uint64_t) * (B + 1), cudaMemcpyHostToDevice, s));
    HC_CUDA(cudaMemcpyAsync(d_res, idx->bases->residues.data(), idx->bases->residues.size(), cudaMemcpyHostToDevice, s));
    HC_CUDA(cudaMemcpyAsync(d_mres, idx->mres, sizeof(double) * 128, cudaMemcpyHostToDevice, s));
    HC_CUDA(cudaMemcpyAsync(d_mmod, idx->mmod, sizeof(double) * 128, cudaMemcpyHostToDevice, s));

    IonArgs a{d_base, d_mask, d_boff, d_res, d_mres, d_mmod, p.bin_width_da, p.frag_mz_min, p.frag_mz_max, P,
              d_fix, 0, 0, 0, 0, 0, 0};
    int64_t fix[256];
    fixed_ions(&a, idx->mres, idx->mmod, fix);
    HC_CUDA(cudaMemcpyAsync(d_fix, fix, sizeof(fix), cudaMemcpyHostToDevice, s));
    uint32_t *d_cnt, *d_groups;
    uint64_t* d_ionoff;
    HC_CUDA(dalloc(&d_cnt, P, tf.ptrs));
    HC_CUDA(dalloc(&d_groups, P, tf.ptrs));
    HC_CUDA(dalloc(&d_ionoff, P, tf.ptrs));
    HC_CUDA(cudaMalloc(&d.fwd_off, sizeof(uint64_t) * (P + 1)));
    uint64_t* d_scan_tmp;
    HC_CUDA(dalloc(&d_scan_tmp, scan_tmp_words(P), tf.ptrs));
    const unsigned pgrid = (unsigned)((P + kIonThreads - 1) / kIonThreads);
    if (P) ion_count_kernel<<<pgrid, kIonThreads, 0, s>>>(a, d_cnt, d_groups);
    HC_CUDA(cudaGetLastError());
    HC_CUDA(exclusive_scan<uint32_t>(d_cnt, P, d_ionoff, d_total, d_scan_tmp, s));
    HC_CUDA(exclusive_scan<uint32_t>(d_groups, P, d.fwd_off, d.fwd_off + P, d_scan_tmp, s));
    uint64_t totals[3] = {0, 0, 0};
    HC_CUDA(cudaMemcpyAsync(&d.n_fwd, d.fwd_off + P, sizeof(uint64_t), cudaMemcpyDeviceToHost, s));
    HC_CUDA(cudaMemcpyAsync(totals, d_total, sizeof(totals), cudaMemcpyDeviceToHost, s));
    HC_CUDA(cudaStreamSynchronize(s));
    const uint64_t E = totals[0];

    std::vector<uint32_t> ls_at(totals[1]);
    std::vector<int64_t> ls_val(totals[1]);
    if (!ls_at.empty()) {
        int64_t* d_val;
        HC_CUDA(dalloc(&d_val, ls_at.size(), tf.ptrs));
        HC_CUDA(cudaMemcpyAsync(ls_at.data(), d_list, sizeof(uint32_t) * ls_at.size(), cudaMemcpyDeviceToHost, s));
        HC_CUDA(cudaStreamSynchronize(s));
        for (size_t i = 0; i < ls_at.size(); ++i)
            ls_val[i] = std::llround(std::ldexp(std::log10((double)ls_at[i]), 32));
        HC_CUDA(cudaMemcpyAsync(d_val, ls_val.data(), sizeof(int64_t) * ls_val.size(), cudaMemcpyHostToDevice, s));
        ls_patch_kernel<<<(unsigned)((ls_at.size() + 255) / 256), 256, 0, s>>>(d.ls, d_list, d_val,
                                                                              (uint32_t)ls_at.size());
        HC_CUDA(cudaGetLastError());
    }

    uint64_t *keys, *keys2;
    HC_CUDA(dalloc(&keys, E, tf.ptrs));
    HC_CUDA(dalloc(&keys2, E, tf.ptrs));
    HC_CUDA(cudaMalloc(&d.fwd, 16 * (d.n_fwd ? d.n_fwd : 1)));
    if (P) ion_emit_kernel<<<pgrid, kIonThreads, 0, s>>>(a, d_ionoff, keys, d.fwd_off, d.fwd);
    HC_CUDA(cudaGetLastError());

    // stable radix sort on the bin bits
    int bin_bits = 1;
    while ((1ull << bin_bits) < idx->n_bins) ++bin_bits;
    const uint64_t ntiles = (E + kRsTile - 1) / kRsTile;
    if (E) {
        uint32_t* counts;
        uint64_t* offs;
        HC_CUDA(dalloc(&counts, ntiles * kRsRadix, tf.ptrs));
        HC_CUDA(dalloc(&offs, ntiles * kRsRadix, tf.ptrs));
        uint64_t* stmp;
        HC_CUDA(dalloc(&stmp, scan_tmp_words(ntiles * kRsRadix), tf.ptrs));
        for (int shift = 32; shift < 32 + bin_bits; shift += kRsBits) {
            rs_count_kernel<<<(unsigned)ntiles, kRsWarps * 32, 0, s>>>(keys, E, shift, counts, ntiles);
            HC_CUDA(cudaGetLastError());
            HC_CUDA(exclusive_scan<uint32_t>(counts, ntiles * kRsRadix, offs, nullptr, stmp, s));
            rs_scatter_kernel<<<(unsigned)ntiles, kRsWarps * 32, 0, s>>>(keys, keys2, E, shift, offs, ntiles);
            HC_CUDA(cudaGetLastError());
            std::swap(keys, keys2);
        }
    }
    // bucket offsets of the sorted keys (uoff), then the stored layout: each
    // bucket padded to a multiple of 4 entries (d.off), so that the search
    // reads whole 16-byte groups
    const uint32_t nb = idx->n_bins;
    const unsigned bgrid = (nb + 255) / 256;
    const unsigned egrid = (unsigned)((E + 255) / 256);
    uint64_t* uoff;
    HC_CUDA(dalloc(&uoff, (uint64_t)nb + 1, tf.ptrs));
    bucket_off_kernel<<<(unsigned)((E + 1 + 255) / 256), 256, 0, s>>>(keys, E, nb, uoff);
    HC_CUDA(cudaGetLastError());
    const uint64_t hot_lo = std::max<uint64_t>(2, P >> kHotShift);
    uint32_t *psz, *some, *hot, *hot_bin;
    uint64_t *some_at, *hot_at, *rtotal, *btmp;
    HC_CUDA(dalloc(&psz, nb, tf.ptrs));
    HC_CUDA(dalloc(&some, nb, tf.ptrs));
    HC_CUDA(dalloc(&hot, nb, tf.ptrs));
    HC_CUDA(dalloc(&hot_bin, nb, tf.ptrs));
    HC_CUDA(dalloc(&some_at, nb, tf.ptrs));
    HC_CUDA(dalloc(&hot_at, nb, tf.ptrs));
    HC_CUDA(dalloc(&rtotal, 4, tf.ptrs));     // stored entries, skip rows, hot buckets, largest bucket
    HC_CUDA(dalloc(&btmp, scan_tmp_words(nb), tf.ptrs));
    HC_CUDA(cudaMemsetAsync(rtotal, 0, 4 * sizeof(uint64_t), s));
    HC_CUDA(cudaMalloc(&d.skip_row, sizeof(int32_t) * nb));
    HC_CUDA(cudaMalloc(&d.hot_id, sizeof(int32_t) * nb));
    bucket_kernel<<<bgrid, 256, 0, s>>>(uoff, nb, hot_lo, psz, some, hot, (unsigned long long*)rtotal + 3);
    HC_CUDA(cudaGetLastError());
    HC_CUDA(exclusive_scan<uint32_t>(psz, nb, d.off, d.off + nb, btmp, s));
    HC_CUDA(cudaMemcpyAsync(rtotal, d.off + nb, sizeof(uint64_t), cudaMemcpyDeviceToDevice, s));
    HC_CUDA(exclusive_scan<uint32_t>(some, nb, some_at, rtotal + 1, btmp, s));
    HC_CUDA(exclusive_scan<uint32_t>(hot, nb, hot_at, rtotal + 2, btmp, s));
    row_of_kernel<<<bgrid, 256, 0, s>>>(some, some_at, nb, d.skip_row, nullptr);
    HC_CUDA(cudaGetLastError());
    row_of_kernel<<<bgrid, 256, 0, s>>>(hot, hot_at, nb, d.hot_id, hot_bin);
    HC_CUDA(cudaGetLastError());
    uint64_t sizes[4];
    HC_CUDA(cudaMemcpyAsync(sizes, rtotal, sizeof(sizes), cudaMemcpyDeviceToHost, s));
    HC_CUDA(cudaStreamSynchronize(s));
    const uint64_t Ep = sizes[0], rows = sizes[1], nhot = sizes[2], mx = sizes[3];
    // the sort's other buffer goes before the stored entries come, so that the
    // build's peak stays at 20 bytes an entry (two key buffers and the forward lists)
    tf.release(keys2);
    if (mx >= (1ull << 32) - 3) {
        set_error("a bucket holds %llu entries (limit 2^32 - 4)", (unsigned long long)mx);
        return HICOPS_EOVERFLOW;
    }
    // stored entries and the chunk skip tables of every non-empty bucket
    // (positions relative to the bucket start); four spare words: the entry
    // allocation is never empty and ends 16-byte aligned
    HC_CUDA(cudaMalloc(&d.entry, sizeof(uint32_t) * (Ep + 4)));
    HC_CUDA(cudaMemsetAsync(d.entry, 0xff, sizeof(uint32_t) * (Ep + 4), s));
    d.skip_stride = (uint32_t)(((P + kChunk - 1) >> kChunkShift) + 1);
    HC_CUDA(cudaMalloc(&d.skip, sizeof(uint32_t) * (rows ? rows : 1) * d.skip_stride));
    if (E) store_kernel<<<egrid, 256, 0, s>>>(keys, E, uoff, d.off, d.entry, d.skip_row, d.skip_stride, d.skip);
    HC_CUDA(cudaGetLastError());

    // hot buckets as bitmaps
    d.n_hot = (uint32_t)nhot;
    // rows cover every pid of the last search chunk (up to 2 * kChunk past P)
    // and start 16-byte aligned
    d.hot_words = ((P + 2ull * kChunk + 31) / 32 + 3) & ~3ull;
    const uint64_t hbytes = sizeof(uint32_t) * (nhot ? nhot : 1) * d.hot_words;
    HC_CUDA(cudaMalloc(&d.hot_b, hbytes));
    HC_CUDA(cudaMalloc(&d.hot_y, hbytes));
    HC_CUDA(cudaMalloc(&d.hot_flags, sizeof(uint32_t) * (nhot ? nhot : 1)));
    HC_CUDA(cudaMemsetAsync(d.hot_flags, 0, sizeof(uint32_t) * (nhot ? nhot : 1), s));
    // a peptide has at most 126 ions, so at most 126 * 64 buckets hold 1/64 of the
    // peptides each: nhot * chunks < 2^31
    if (nhot)
        hot_fill_kernel<<<(unsigned)(nhot * (d.skip_stride - 1)), 256, 0, s>>>(
            d.entry, d.off, hot_bin, d.skip_row, d.skip_stride, d.skip, d.hot_words, d.hot_b, d.hot_y, d.hot_flags);
    HC_CUDA(cudaGetLastError());
    HC_CUDA(cudaMalloc(&d.bins, sizeof(BinInfo) * nb));
    bin_info_kernel<<<bgrid, 256, 0, s>>>(d.off, d.skip_row, d.hot_id, d.hot_flags, nb, d.bins);
    HC_CUDA(cudaGetLastError());
    HC_CUDA(cudaStreamSynchronize(s));
    cudaFree(d.skip_row);
    cudaFree(d.hot_id);
    cudaFree(d.hot_flags);
    d.skip_row = d.hot_id = nullptr;
    d.hot_flags = nullptr;

    d.n_stored = Ep;
    d.bytes = sizeof(double) * P + sizeof(uint64_t) * (idx->n_bins + 1) + sizeof(uint32_t) * (Ep + 4) +
              sizeof(int64_t) * (lf.size() + n_ls) + sizeof(BinInfo) * nb +
              sizeof(uint32_t) * rows * d.skip_stride + 2 * hbytes + sizeof(uint64_t) * (P + 1) +
              16 * (d.n_fwd ? d.n_fwd : 1);
    idx->stats.n_entries = E;
    idx->stats.max_bucket = mx;
    idx->stats.device_bytes = d.bytes;
    idx->stats.device_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    d.ready = true;
    return HICOPS_OK;
}

}  // namespace hicops

extern "C" hicops_status hicops_index_upload(hicops_index* idx) {
    if (!idx) { hicops::set_error("index is NULL"); return HICOPS_EINVAL; }
    hicops_status st = hicops::upload_index(idx);
    if (st != HICOPS_OK) hicops::free_device_index(idx);
    return st;
}

// The device keeps every bucket padded to a multiple of 4 entries; the copy
// leaves the pad slots out, so buckets are back to back as documented.
extern "C" hicops_status hicops_index_copy_csr(const hicops_index* idx, uint64_t* off, uint32_t* entries) {
    if (!idx || !idx->dev.ready) { hicops::set_error("index not uploaded"); return HICOPS_EINVAL; }
    if (!off && !entries) return HICOPS_OK;
    const uint32_t nb = idx->n_bins;
    std::vector<uint64_t> poff(nb + 1);
    std::vector<uint32_t> pent;
    try {
        pent.resize(idx->dev.n_stored);
    } catch (const std::bad_alloc&) {
        hicops::set_error("out of host memory");
        return HICOPS_ENOMEM;
    }
    HC_CUDA(cudaMemcpy(poff.data(), idx->dev.off, sizeof(uint64_t) * (nb + 1), cudaMemcpyDeviceToHost));
    if (!pent.empty())
        HC_CUDA(cudaMemcpy(pent.data(), idx->dev.entry, sizeof(uint32_t) * pent.size(), cudaMemcpyDeviceToHost));
    uint64_t o = 0;
    for (uint32_t b = 0; b < nb; ++b) {
        if (off) off[b] = o;
        for (uint64_t i = poff[b]; i < poff[b + 1] && pent[i] != 0xffffffffu; ++i) {
            if (entries) entries[o] = pent[i];
            ++o;
        }
    }
    if (off) off[nb] = o;
    return HICOPS_OK;
}
