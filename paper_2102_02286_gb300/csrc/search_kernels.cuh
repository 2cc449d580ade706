// Device kernels of the search path (included by search.cu only):
// preprocessing + precursor window, unit planning, the shared-peak search
// kernels (search_kernel.cuh, count_kernel.cuh), the top-k merge + e-value, and
// the work count.
#pragma once

#include <cfloat>
#include <cmath>

#include "dev_common.cuh"

namespace hicops {
namespace {

constexpr int kPrepThreads = 256;
constexpr int kPrepWarps = kPrepThreads / 32;   // spectra per block of prep_kernel's last blocks
constexpr int kPrepWarpPeaks = 512;        // spectra with at most this many raw peaks: one warp each
constexpr uint32_t kPrepBigBlocks = 608;   // blocks for the others, at most (4 an SM)
constexpr int kMinSegPids = (int)kChunk;  // smallest segment of a split window
constexpr int kMaxSegs = 64;              // most segments a window is split into
constexpr int kMergeWarps = 8;          // spectra per merge block

struct UnitTop {
    int64_t key;
    uint32_t pid;
    uint32_t packed;    // nb << 26 | ny << 20 | S
};

struct PrepArgs {
    const uint64_t* peak_off;
    const float* mz;
    const float* inten;
    const double* prec_mz;
    const uint8_t* charge;
    const double* tol;
    uint32_t n;
    uint32_t topn;      // peaks retained
    uint32_t stride;    // qbin / qiq words per spectrum (>= topn)
    double w;
    float mz_lo, mz_hi; // least floats not below the limits (as doubles) of the m/z range
    uint64_t inv_w;     // 1 / w = inv_w * 2^(inv_exp - 64), inv_w with its top bit set
    int inv_exp;
    uint32_t scale;
    const double* mass;
    uint64_t P;
    uint32_t* qbin;     // [n * stride]
    uint32_t* qiq;      // [n * stride]
    uint32_t* qn;       // [n]
    uint32_t* lo;       // [n]
    uint32_t* hi;       // [n]
    const BinInfo* bins;
    uint32_t n_bins, tol_bins;
    float per_peptide;  // of groups in a bucket to its hits a peptide
    uint32_t slices;    // hot peaks that are bitmap slices at most (min_shared - 2)
    float count_from;   // hits a peptide from which on the spectrum's units are counted (count_kernel.cuh)
    uint32_t* cost;     // [n] what the spectrum's window costs (Cost), and kCounted, or NULL
    uint32_t* hist;     // [n * kHistBins] set to zero here, or NULL
    uint32_t* ns;       // [n] likewise
};

// By the whole block, which it ends with a barrier.  A thread takes pairs, not
// elements of which every other one has nothing to do: the issue of the steps is
// what bounds it.  6,000 spectra of 6,000 peaks, preprocessing 5.8 -> 4.5 ms.
__device__ __forceinline__ void bitonic_sort_u64(uint64_t* s, int npow) {
    for (int k = 2; k <= npow; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int p = threadIdx.x; p < npow >> 1; p += blockDim.x) {
                const int i = 2 * p - (p & (j - 1)), ixj = i + j;      // (p without the bits below j, twice, and those)
                const uint64_t a = s[i], b = s[ixj];
                const bool up = (i & k) == 0;
                if ((a > b) == up) { s[i] = b; s[ixj] = a; }
            }
            __syncthreads();
        }
    }
}

__device__ __forceinline__ int next_pow2(int v) {
    int p = 1;
    while (p < v) p <<= 1;
    return p;
}

// floor(mz / w) of the FP64 quotient, for a finite mz in the m/z range.  The
// product of mz's 24-bit mantissa and the 64-bit 1 / w gives the quotient
// with 32 fraction bits; it and the FP64 quotient are each within 2^-52 of
// the true one, relatively, so off a bin edge by more than that both have the
// same floor, and only at an edge is the FP64 division (a unit of 2 lanes a
// clock) made.
__device__ __forceinline__ uint32_t bin_of(const PrepArgs& a, float mz) {
    const uint32_t bits = __float_as_uint(mz), e = bits >> 23;      // mz > 0
    const uint64_t m = (bits & 0x7fffffu) | 0x800000u;
    const int sh = 158 - (int)e - a.inv_exp;
    if (e != 0 && (uint32_t)sh < 64u) {
        const uint64_t v = __umul64hi(m << 40, a.inv_w) >> sh;
        const uint32_t bin = (uint32_t)(v >> 32), tol = 2u + (bin >> 19);
        if ((uint32_t)v + tol >= 2u * tol) return bin;
    }
    return (uint32_t)floor((double)mz / a.w);
}

// max(1, floor(I * scale / top)) of the FP64 form, 0 < I <= top: I * scale is
// exact in FP64 (24 + 20 bits), and a quotient that is not whole lies
// 2^-(24 + d) or more from a whole number (d: difference of the exponents)
// where half its ulp is under 2^-(33 + d), so the FP64 floor is the floor of
// the true quotient of integers, which a float estimate and one step give.
__device__ __forceinline__ uint32_t quantise(float I, float top, uint32_t scale) {
    const uint32_t bi = __float_as_uint(I), bt = __float_as_uint(top);
    const uint32_t ei = max(bi >> 23, 1u), et = max(bt >> 23, 1u), d = et - ei;
    if (d > 20u) return 1u;                     // num < 2^44 <= den
    const uint32_t mi = (bi & 0x7fffffu) | (bi >> 23 ? 0x800000u : 0u);
    const uint32_t mt = (bt & 0x7fffffu) | (bt >> 23 ? 0x800000u : 0u);
    const uint64_t num = (uint64_t)mi * scale;
    const uint64_t den = (uint64_t)mt << d;
    if (den > num) return 1u;
    uint32_t r = (uint32_t)(__uint2float_rn(mi) * __uint2float_rn(scale) / __ull2float_rn(den));
    if (r * den > num) --r;
    else if ((r + 1ull) * den <= num) ++r;
    return r;
}

// The precursor window by one warp: first index with mass >= xlo (lanes 0 to
// 15) and first with mass > xhi (the others), 16 pivots of each a step: 6
// dependent loads for ten million masses where a binary search makes 24.
__device__ __forceinline__ void warp_window(const double* __restrict__ mass, uint64_t n, double xlo, double xhi,
                                            int lane, uint32_t* lo, uint32_t* hi) {
    const bool upper = lane >= 16;
    const uint32_t sub = lane & 15u;
    const double x = upper ? xhi : xlo;
    uint32_t a = 0, b = (uint32_t)n;             // n < 2^31
    while (__any_sync(0xffffffffu, a < b)) {
        const uint32_t len = b - a;
        const bool last = len <= 16u;
        const uint32_t p = a + (last ? sub : (uint32_t)((uint64_t)len * (sub + 1u) / 17u));
        bool below = false;
        if (p < b) {
            const double v = __ldg(mass + p);
            below = upper ? v <= x : v < x;
        }
        const uint32_t c = __popc((__ballot_sync(0xffffffffu, below) >> (upper ? 16 : 0)) & 0xffffu);
        if (last) {
            a = b = a + c;
        } else {
            const uint32_t na = c ? a + (uint32_t)((uint64_t)len * c / 17u) + 1u : a;
            if (c < 16u) b = a + (uint32_t)((uint64_t)len * (c + 1u) / 17u);
            a = na;
        }
    }
    *lo = __shfl_sync(0xffffffffu, a, 0);
    *hi = __shfl_sync(0xffffffffu, a, 16);
}

// What searching a spectrum's window costs, in units of 64 entries (0 for an
// empty window), estimated from the sizes of its peaks' buckets: the entries
// to stream (a share W / P of every bucket, but for the hot peaks that become
// bitmap slices, the densest), and where there are slices enough that every
// peptide hit twice is looked at, those peptides, W lambda^2 / 2 of them at
// lambda hits a peptide and kRepeatCost entries each (a fit to the measured
// times gives 16 to 22; 40 splits the spectra whose peptides share fragments
// beyond chance a little more).  Over 5,000 spectra the estimate's correlation
// with the time is 0.90, of the entries alone 0.84.  It decides where windows
// are split and in what order the units are taken, never what is found.
// 1,111 spectra at +-500 Da: search 644 us with even pieces in their order ->
// 388 us; 5,000 at a tolerance of one bin 3.21 -> 2.46 ms; 37: 51 -> 39 us;
// 30,000: 7.95 -> 7.59 ms.
// Where a spectrum's units are counted instead (kCounted), the same entries and
// a look at every counter, which costs what kCounterCost entries do.
constexpr float kRepeatCost = 40.0f;
constexpr float kCounterCost = 1.3f;
constexpr uint32_t kCounted = 0x80000000u;

struct Cost {
    static constexpr int kEarly = 4;
    int2 early[kEarly];                    // the first peaks' hot and flags, on their way
    float ordinary = 0.0f, hot = 0.0f;     // groups of 4 entries
    float top = 0.0f, next = 0.0f;         // the densest hot peaks'
    uint32_t nhot = 0;
    static __device__ __forceinline__ int2 bucket(const PrepArgs& a, uint32_t bin) {
        return __ldg(reinterpret_cast<const int2*>(a.bins + bin) + 1);
    }
    __device__ __forceinline__ void add(int2 b) {
        const float g = (float)((uint32_t)b.y >> 2);
        if (b.x >= 0) {
            hot += g;
            ++nhot;
            next = fmaxf(next, fminf(top, g));
            top = fmaxf(top, g);
        } else {
            ordinary += g;
        }
    }
    // by a whole warp: the lanes' sums and greatest together, then the cost
    __device__ __forceinline__ uint32_t of_window(const PrepArgs& a, uint32_t W, int lane) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ordinary += __shfl_xor_sync(0xffffffffu, ordinary, o);
        nhot = __reduce_add_sync(0xffffffffu, nhot);
        float streamed = 0.0f;
        if (nhot > a.slices) {   // uniform
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) hot += __shfl_xor_sync(0xffffffffu, hot, o);
            // (floats that are not negative order as integers)
            const uint32_t t = __reduce_max_sync(0xffffffffu, __float_as_uint(top));
            const bool mine = __float_as_uint(top) == t;
            const unsigned holders = __ballot_sync(0xffffffffu, mine);
            const bool first = mine && (holders & ((1u << lane) - 1u)) == 0;
            const float t2 = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(first ? next : top)));
            if (a.slices) hot -= __uint_as_float(t) + (float)(a.slices - 1u) * t2;
            streamed = fmaxf(hot, 0.0f);
        }
        const float lambda = (ordinary + streamed) * a.per_peptide;
        const bool counted = lambda >= a.count_from;
        const float each = lambda + (counted ? kCounterCost
                                     : nhot >= a.slices ? 0.5f * kRepeatCost * lambda * lambda : 0.0f);
        return W ? (counted ? kCounted : 0u) + 1u + (uint32_t)fminf(each * (float)W * (1.0f / 64.0f), 2.0e9f) : 0u;
    }
};

// A spectrum's count, window and cost, by one whole warp.  Its keep bins are
// the keys' high words (SHIFT 32) or low words (0).
template <int SHIFT>
__device__ __forceinline__ void put_window(const PrepArgs& a, uint32_t q, const uint64_t* keys, int keep, double prec,
                                           double tol, uint32_t z, int lane) {
    uint32_t lo = 0, hi = 0;
    Cost c;
    if (keep) {   // warp-uniform
        if (a.cost) {
#pragma unroll
            for (int i = 0; i < Cost::kEarly; ++i) {
                const int t = lane + 32 * i;
                c.early[i] = t < keep ? Cost::bucket(a, (uint32_t)(keys[t] >> SHIFT)) : make_int2(-1, 0);
            }
        }
        const double Mq = __dmul_rn(__dsub_rn(prec, kProtonDa), (double)z);
        warp_window(a.mass, a.P, __dsub_rn(Mq, tol), __dadd_rn(Mq, tol), lane, &lo, &hi);
        if (a.cost) {
#pragma unroll
            for (int i = 0; i < Cost::kEarly; ++i) c.add(c.early[i]);
#pragma unroll 4
            for (int t = lane + 32 * Cost::kEarly; t < keep; t += 32) c.add(Cost::bucket(a, (uint32_t)(keys[t] >> SHIFT)));
            // the other bins within the fragment tolerance (two peaks' common ones twice)
            for (int d = 1; d <= (int)a.tol_bins; ++d) {
#pragma unroll 2
                for (int t = lane; t < keep; t += 32) {
                    const uint32_t bin = (uint32_t)(keys[t] >> SHIFT);
                    if (bin >= (uint32_t)d) c.add(Cost::bucket(a, bin - d));
                    if (bin + d < a.n_bins) c.add(Cost::bucket(a, bin + d));
                }
            }
        }
    }
    if (a.cost) {
        const uint32_t cost = c.of_window(a, hi - lo, lane);
        if (lane == 0) a.cost[q] = cost;
    }
    if (lane == 0) {
        a.qn[q] = (uint32_t)keep;
        a.lo[q] = lo;
        a.hi[q] = hi;
    }
}

// Spectra of more than kPrepWarpPeaks raw peaks, one block each, any number
// of raw peaks: the raw peaks are taken in chunks of kPrepChunk, and each
// chunk is merged with the running list of the best top_n bins so far (in
// raw form again: bin << 32 | intensity bits), sorted by bin, reduced to one
// representative per bin (its largest intensity), re-keyed by (intensity
// desc, bin asc), sorted, and cut to top_n.  A bin's value in the list only
// grows, so a bin left out at some chunk has top_n better bins from then on:
// the final list is the top_n bins of the whole spectrum by their largest
// intensity (R8), whatever the chunking.
constexpr int kPrepSort = kPrepWarps * kPrepWarpPeaks;  // keys sorted per chunk
constexpr int kPrepChunk = kPrepSort - (int)kMaxTopN;   // raw peaks per chunk

struct PrepShared {
    uint64_t keys[kPrepSort];
    uint64_t best[kMaxTopN];         // the running list, raw form
    uint32_t big[kPrepThreads];
    int nrep, nbig;
};

__device__ __noinline__ void prep_block(const PrepArgs& a, uint32_t q, PrepShared& sh) {
    uint64_t* const keys = sh.keys;
    uint64_t* const best = sh.best;
    const uint64_t p0 = a.peak_off[q], cnt = a.peak_off[q + 1] - p0;
    const double prec = a.prec_mz[q];
    const double tol = a.tol[q];
    const uint32_t z = a.charge[q];
    const bool valid = z > 0 && isfinite(prec) && isfinite(tol) && tol >= 0.0;
    int keep = 0;
    if (valid) {
        for (uint64_t base = 0; base < cnt; base += kPrepChunk) {
            const int m = (int)min((uint64_t)kPrepChunk, cnt - base);
            const int total = m + keep;
            const int npow = next_pow2(total);
            // key = bin << 32 | intensity bits (positive finite floats order as integers)
            for (int i = threadIdx.x; i < npow; i += blockDim.x) {
                uint64_t k = ~0ull;
                if (i < m) {
                    const float mz = a.mz[p0 + base + i], I = a.inten[p0 + base + i];
                    if (isfinite(mz) && isfinite(I) && I > 0.0f && mz >= a.mz_lo && mz < a.mz_hi)
                        k = ((uint64_t)bin_of(a, mz) << 32) | __float_as_uint(I);
                } else if (i < total) {
                    k = best[i - m];
                }
                keys[i] = k;
            }
            if (threadIdx.x == 0) sh.nrep = 0;
            __syncthreads();
            bitonic_sort_u64(keys, npow);
            // one representative per bin: the last (most intense) of each run
            uint64_t rep[kPrepSort / kPrepThreads];
            int nr = 0;
            for (int i = threadIdx.x; i < npow; i += blockDim.x) {
                const uint64_t k = keys[i];
                if (k == ~0ull) continue;
                const bool last = (i + 1 == npow) || ((keys[i + 1] >> 32) != (k >> 32));
                // re-key: intensity descending, then bin ascending
                if (last) rep[nr++] = ((uint64_t)(~(uint32_t)k) << 32) | (k >> 32);
            }
            __syncthreads();
            for (int r = 0; r < nr; ++r) keys[atomicAdd(&sh.nrep, 1)] = rep[r];
            __syncthreads();
            const int nrep = sh.nrep;
            const int npow2 = next_pow2(nrep > 0 ? nrep : 1);
            for (int i = nrep + threadIdx.x; i < npow2; i += blockDim.x) keys[i] = ~0ull;
            __syncthreads();
            bitonic_sort_u64(keys, npow2);
            keep = nrep < (int)a.topn ? nrep : (int)a.topn;
            // the running list back in raw form for the next chunk
            for (int t = threadIdx.x; t < keep; t += blockDim.x) {
                const uint64_t k = keys[t];
                best[t] = ((uint64_t)(uint32_t)k << 32) | (uint32_t)~(uint32_t)(k >> 32);
            }
            __syncthreads();
        }
        if (keep > 0) {
            const float top = __uint_as_float(~(uint32_t)(keys[0] >> 32));
            for (int t = threadIdx.x; t < keep; t += blockDim.x) {
                const uint64_t k = keys[t];
                a.qbin[(uint64_t)q * a.stride + t] = (uint32_t)k;
                a.qiq[(uint64_t)q * a.stride + t] = quantise(__uint_as_float(~(uint32_t)(k >> 32)), top, a.scale);
            }
        }
    }
    if (threadIdx.x < 32) put_window<0>(a, q, keys, keep, prec, tol, z, threadIdx.x);
    __syncthreads();     // the keys, before the next spectrum's
}

__device__ __noinline__ void warp_bitonic_sort_u64(uint64_t* s, int npow, int lane) {
    for (int k = 2; k <= npow; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = lane; i < npow; i += 32) {
                const int ixj = i ^ j;
                if (ixj > i) {
                    const uint64_t x = s[i], y = s[ixj];
                    const bool up = (i & k) == 0;
                    if ((x > y) == up) { s[i] = y; s[ixj] = x; }
                }
            }
            __syncwarp();
        }
    }
}

// A spectrum of at most kPrepWarpPeaks raw peaks by one warp, in a 4 KB slice
// of shared memory.  Peak lists come ascending in m/z as a rule, so the sort
// by bin is made only where the bins do not ascend, and the cut to the top_n
// most intense bins (lower bins first at equal intensities) only where there
// are more: as a search for the intensity at the cut, bit by bit, instead of a
// sort by intensity.  The retained peaks come out ascending in their bins;
// what the search makes of them does not depend on their order.
// 30,000 spectra of 100 peaks: 0.40 ms (two sorts, FP64 divisions, a binary
// search by one lane) -> 0.08 ms; one spectrum: 43 -> 11 us.
__device__ __forceinline__ void prep_warp(const PrepArgs& a, uint32_t q, uint64_t p0, int cnt, uint64_t* keys,
                                          int lane) {
    const double prec = a.prec_mz[q];
    const double tol = a.tol[q];
    const uint32_t z = a.charge[q];
    const bool valid = z > 0 && isfinite(prec) && isfinite(tol) && tol >= 0.0;
    const unsigned lt = (1u << lane) - 1u;
    int keep = 0;
    if (valid && cnt > 0) {
        // the usable peaks, in their order: bin << 32 | intensity bits
        // (positive finite floats order as integers)
        int m = 0;
        bool ascends = true;
        uint32_t before = 0;                 // the last bin of the rounds before
        for (int i0 = 0; i0 < cnt; i0 += 32) {
            const int i = i0 + lane;
            bool ok = false;
            float mz = 0.0f, I = 0.0f;
            if (i < cnt) {
                mz = __ldg(a.mz + p0 + i);
                I = __ldg(a.inten + p0 + i);
                ok = isfinite(mz) && isfinite(I) && I > 0.0f && mz >= a.mz_lo && mz < a.mz_hi;
            }
            const uint32_t bin = ok ? bin_of(a, mz) : 0u;
            const unsigned use = __ballot_sync(0xffffffffu, ok);
            if (ok) keys[m + __popc(use & lt)] = ((uint64_t)bin << 32) | __float_as_uint(I);
            // the usable lane below, or the rounds before
            const unsigned lower = use & lt;
            const uint32_t prev = __shfl_sync(0xffffffffu, bin, lower ? 31 - __clz(lower) : lane);
            if (ok && (lower ? prev : before) > bin) ascends = false;
            if (use) before = __shfl_sync(0xffffffffu, bin, 31 - __clz(use));
            m += __popc(use);
        }
        if (!__all_sync(0xffffffffu, ascends)) {
            const int npow = next_pow2(m);
            for (int i = m + lane; i < npow; i += 32) keys[i] = ~0ull;
            __syncwarp();
            warp_bitonic_sort_u64(keys, npow, lane);
        }
        __syncwarp();
        // one peak per bin, its most intense, compacted in place: a run's
        // representative is made at its last peak and written at or before
        // the run's first, so the peaks of runs that are not over stay
        int nrep = 0;
        uint32_t top = 0;
        for (int i0 = 0; i0 < m; i0 += 32) {
            const int i = i0 + lane;
            bool last = false;
            uint32_t bin = 0, val = 0;
            if (i < m) {
                const uint64_t k = keys[i];
                bin = (uint32_t)(k >> 32);
                last = i + 1 == m || (uint32_t)(keys[i + 1] >> 32) != bin;
                if (last) {
                    val = (uint32_t)k;
                    for (int j = i - 1; j >= 0 && (uint32_t)(keys[j] >> 32) == bin; --j) val = max(val, (uint32_t)keys[j]);
                }
            }
            const unsigned msk = __ballot_sync(0xffffffffu, last);
            __syncwarp();
            if (last) keys[nrep + __popc(msk & lt)] = ((uint64_t)bin << 32) | val;
            top = max(top, val);
            nrep += __popc(msk);
            __syncwarp();
        }
        top = __reduce_max_sync(0xffffffffu, top);
        keep = min(nrep, (int)a.topn);
        // the cut: the largest intensity that top_n bins reach, and how many
        // of the bins right at it are kept
        uint32_t cut = 0, ties = 0;
        if (nrep > keep) {
            for (int bit = 30; bit >= 0; --bit) {
                const uint32_t c = cut | 1u << bit;
                uint32_t got = 0;
                for (int i = lane; i < nrep; i += 32) got += (uint32_t)keys[i] >= c;
                if (__reduce_add_sync(0xffffffffu, got) >= (uint32_t)keep) cut = c;
            }
            uint32_t above = 0;
            for (int i = lane; i < nrep; i += 32) above += (uint32_t)keys[i] > cut;
            ties = (uint32_t)keep - __reduce_add_sync(0xffffffffu, above);
        }
        uint32_t out = 0;
        for (int i0 = 0; i0 < nrep; i0 += 32) {
            const int i = i0 + lane;
            const uint64_t k = i < nrep ? keys[i] : 0ull;
            const uint32_t val = (uint32_t)k;
            bool use = i < nrep;
            if (nrep > keep) {   // uniform
                const unsigned tie = __ballot_sync(0xffffffffu, use && val == cut);
                use = use && (val > cut || (val == cut && (uint32_t)__popc(tie & lt) < ties));
                ties -= min(ties, (uint32_t)__popc(tie));
            }
            const unsigned msk = __ballot_sync(0xffffffffu, use);
            if (use) {
                const uint64_t at = (uint64_t)q * a.stride + out + __popc(msk & lt);
                a.qbin[at] = (uint32_t)(k >> 32);
                a.qiq[at] = quantise(__uint_as_float(val), __uint_as_float(top), a.scale);
            }
            __syncwarp();
            if (use) keys[out + __popc(msk & lt)] = k;   // (at or before its own place)
            out += __popc(msk);
        }
        __syncwarp();
    }
    put_window<32>(a, q, keys, keep, prec, tol, z, lane);
}

// Query preprocessing (R8) and the precursor window.  The first big_blocks
// blocks take the spectra of more than kPrepWarpPeaks raw peaks, one a block,
// found by all threads at once; the others a spectrum a warp.
__global__ void __launch_bounds__(kPrepThreads) prep_kernel(const __grid_constant__ PrepArgs a, uint32_t big_blocks) {
    __shared__ PrepShared sh;
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    // a spectrum's peaks lie inside the batch's [peak_off[0], peak_off[n]),
    // else it is invalid and nothing of it is read
    const uint64_t first = a.peak_off[0], end = a.peak_off[a.n];
    auto count = [&](uint32_t q, uint64_t* p0) {
        const uint64_t p1 = a.peak_off[q + 1];
        *p0 = a.peak_off[q];
        return *p0 <= p1 && *p0 >= first && p1 <= end ? p1 - *p0 : 0ull;
    };
    uint64_t p0;
    if (blockIdx.x >= big_blocks) {
        const uint32_t q = (blockIdx.x - big_blocks) * kPrepWarps + wi;
        if (q >= a.n) return;
        if (a.hist) {
            for (uint32_t i = lane; i < kHistBins; i += 32) a.hist[(uint64_t)q * kHistBins + i] = 0;
            if (lane == 0) a.ns[q] = 0;
        }
        const uint64_t cnt = count(q, &p0);
        if (cnt <= (uint64_t)kPrepWarpPeaks) prep_warp(a, q, p0, (int)cnt, sh.keys + wi * kPrepWarpPeaks, lane);
        return;
    }
    for (uint64_t at = blockIdx.x; at < a.n; at += (uint64_t)big_blocks * kPrepThreads) {
        if (threadIdx.x == 0) sh.nbig = 0;
        __syncthreads();
        const uint64_t q = at + (uint64_t)big_blocks * threadIdx.x;
        if (q < a.n && count((uint32_t)q, &p0) > (uint64_t)kPrepWarpPeaks) sh.big[atomicAdd(&sh.nbig, 1)] = (uint32_t)q;
        __syncthreads();
        const int nbig = sh.nbig;
        for (int i = 0; i < nbig; ++i) prep_block(a, sh.big[i], sh);
        __syncthreads();
    }
}

// A work unit: {spectrum, segment [lo, hi), unit number}.  The window of
// spectrum q is split evenly into its ns units.
__device__ __forceinline__ uint4 unit_record(uint32_t q, uint32_t lo, uint32_t hi, uint32_t ns, uint32_t s,
                                             uint64_t u0) {
    const uint32_t len = (uint32_t)(((uint64_t)(hi - lo) + ns - 1) / ns);
    const uint64_t a = (uint64_t)lo + (uint64_t)s * len;
    return make_uint4(q, (uint32_t)min(a, (uint64_t)hi), (uint32_t)min(a + len, (uint64_t)hi), (uint32_t)(u0 + s));
}

// How windows are split.  seg_pids given: into pieces of that many peptides.
// Else by cost: into pieces of 1 / split of the batch's whole cost, so n
// spectra have at most n + split units, and the spectra with common fragments,
// which cost tens of the others, are in as many pieces.  No piece is under
// kMinSegPids peptides, or under kUnitCost, where a unit's own set-up
// outweighs its entries, unless the batch has less than that a CTA.
struct PlanArgs {
    const uint32_t* lo;
    const uint32_t* hi;
    const uint32_t* cost;
    uint32_t n, max_seg, seg_pids, split, ctas;
    uint64_t* seg_off;
    uint4* unit;
    unsigned long long* work;    // the unit counters of the search (0) and of the count (2), set to zero; where
                                 // the counted units start (1)
};
constexpr uint32_t kUnitCost = 128, kUnitCostMin = 16;   // 8,192 and 1,024 entries

// The planning of a batch in one block: the spectra's units, their prefix, and
// the unit records, costliest first, since the persistent CTAs take them in
// this order and the cheap ones fill the end of the launch (a counting sort
// over quarter octaves of the unit's cost), and the counted ones behind.  One block, since a grid's scan and
// sort take seven launches: bound by latency, 7 us for a few spectra, 17 us for
// 5,000 (38 us by seven launches), 58 us for 30,000 (38 us).
constexpr uint32_t kPlanThreads = 1024, kPlanFew = 128;   // up to kPlanFew spectra: as many threads
constexpr uint32_t kPlanEach = 4;          // consecutive spectra of a thread
constexpr uint32_t kPlanBuckets = 512;     // a quarter octave of cost, four times (lanes that are alike spread over them)
// COUNTS: there may be counted units.
template <bool COUNTS>
__global__ void __launch_bounds__(kPlanThreads) plan_kernel(const __grid_constant__ PlanArgs a) {
    constexpr uint32_t kBuckets = (COUNTS ? 2u : 1u) * kPlanBuckets;     // of the units, then of the counted ones
    __shared__ __align__(16) uint32_t bucket[kBuckets];
    __shared__ unsigned long long csum[kPlanThreads / 32];
    __shared__ uint32_t wsum[kPlanThreads / 32];
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const uint32_t step = blockDim.x * kPlanEach;
    uint32_t lo[kPlanEach], hi[kPlanEach], cost[kPlanEach];
    // (a piece of the workspace is a whole number of 256 bytes (pieces.h): whole vectors, whose words behind n
    // are left)
    auto fetch = [&](uint32_t q0) {
        uint4 l{}, h{}, c{};
        if (q0 < a.n) {
            l = *reinterpret_cast<const uint4*>(a.lo + q0);
            h = *reinterpret_cast<const uint4*>(a.hi + q0);
            c = *reinterpret_cast<const uint4*>(a.cost + q0);
        }
        lo[0] = l.x; lo[1] = l.y; lo[2] = l.z; lo[3] = l.w;
        hi[0] = h.x; hi[1] = h.y; hi[2] = h.z; hi[3] = h.w;
        cost[0] = c.x;
        cost[1] = q0 + 1 < a.n ? c.y : 0u;
        cost[2] = q0 + 2 < a.n ? c.z : 0u;
        cost[3] = q0 + 3 < a.n ? c.w : 0u;
    };
    // the batch's cost
    fetch(tid * kPlanEach);
    auto bare = [](uint32_t c) { return COUNTS ? c & ~kCounted : c; };
    unsigned long long sum = (unsigned long long)bare(cost[0]) + bare(cost[1]) + bare(cost[2]) + bare(cost[3]);
#pragma unroll 8
    for (uint32_t q = step + tid; q < a.n; q += blockDim.x) sum += bare(a.cost[q]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) csum[warp] = sum;
    for (uint32_t i = tid; i < kBuckets; i += blockDim.x) bucket[i] = 0;
    if (tid == 0) a.work[0] = 0ull;
    if (COUNTS && tid == 0) a.work[2] = 0ull;
    __syncthreads();
    sum = lane < nwarps ? csum[lane] : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    // (a float not above 1 / piece: 1 + floor of a cost's product with it is at
    // most 1 + cost / piece, so the units keep to n + split)
    const unsigned long long share = sum / a.split, cta = sum / a.ctas;
    const unsigned long long least = min(max(cta, (unsigned long long)kUnitCostMin), (unsigned long long)kUnitCost);
    const float per = __frcp_rd(__ull2float_ru(max(share + 1ull, least)));
    uint32_t ns[kPlanEach], at[kPlanEach];    // units, their bucket
    auto cut = [&]() {
#pragma unroll
        for (uint32_t i = 0; i < kPlanEach; ++i) {
            const uint32_t c = bare(cost[i]), W = hi[i] - lo[i];
            uint32_t k = 0;
            if (c) {
                if (a.seg_pids) k = W / a.seg_pids + (W % a.seg_pids ? 1u : 0u);
                else k = min(1u + __float2uint_rz(__fmul_rz(__uint2float_rz(c), per)),
                             (W + (kMinSegPids - 1)) / kMinSegPids);   // W < 2^31
                k = min(k, a.max_seg);
            }
            ns[i] = k;
            const int b = (int)(__float_as_uint(__fdividef((float)c, (float)max(k, 1u))) >> 21) - (int)(0x3f800000u >> 21);
            at[i] = 4u * (kPlanBuckets / 4u - 1u - (uint32_t)min(max(b, 0), (int)kPlanBuckets / 4 - 1)) + (lane & 3u);
            if (COUNTS && (cost[i] & kCounted)) at[i] += kPlanBuckets;
        }
    };
    uint64_t base = 0, u0 = 0;      // units of the steps before; this thread's first unit of the last step
    for (uint32_t q1 = 0; q1 < a.n; q1 += step) {
        const uint32_t q0 = q1 + tid * kPlanEach;
        if (q1) fetch(q0);
        cut();
        uint32_t mine = 0;
#pragma unroll
        for (uint32_t i = 0; i < kPlanEach; ++i) {
            if (ns[i]) atomicAdd(&bucket[at[i]], ns[i]);
            mine += ns[i];
        }
        uint32_t incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl += x;
        }
        if (q1) __syncthreads();   // wsum has been read
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        const uint32_t t = lane < nwarps ? wsum[lane] : 0u;
        const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? t : 0u);
        u0 = base + before + incl - mine;
        base += __reduce_add_sync(0xffffffffu, t);
        uint64_t u = u0;
#pragma unroll
        for (uint32_t i = 0; i < kPlanEach; ++i) {
            if (q0 + i < a.n) a.seg_off[q0 + i] = u;
            u += ns[i];
        }
    }
    if (tid == 0) a.seg_off[a.n] = base;
    // bucket counts to starts (the last barrier is behind every count)
    if (warp == 0) {
        uint32_t start = 0;
#pragma unroll
        for (uint32_t i = lane; i < kBuckets / 4; i += 32) {
            if (COUNTS && i == kPlanBuckets / 4) a.work[1] = start;
            const uint4 c = reinterpret_cast<const uint4*>(bucket)[i];
            const uint32_t mine = c.x + c.y + c.z + c.w;
            uint32_t incl = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= (uint32_t)o) incl += x;
            }
            const uint32_t f = start + incl - mine;
            reinterpret_cast<uint4*>(bucket)[i] = make_uint4(f, f + c.x, f + c.x + c.y, f + c.x + c.y + c.z);
            start += __shfl_sync(0xffffffffu, incl, 31);
        }
    }
    __syncthreads();
    for (uint32_t q1 = 0; q1 < a.n; q1 += step) {
        const uint32_t q0 = q1 + tid * kPlanEach;
        if (a.n > step) {           // else the only step's values are still there
            fetch(q0);
            cut();
            u0 = q0 < a.n ? a.seg_off[q0] : 0;
        }
        uint64_t u = u0;
#pragma unroll
        for (uint32_t i = 0; i < kPlanEach; ++i) {
            if (!ns[i]) continue;
            const uint32_t to = atomicAdd(&bucket[at[i]], ns[i]);
            for (uint32_t s = 0; s < ns[i]; ++s) a.unit[to + s] = unit_record(q0 + i, lo[i], hi[i], ns[i], s, u);
            u += ns[i];
        }
    }
}

// Shared memory of the search kernel, in 32-bit words: the plane, as large as
// the rest leaves room for, then search_kernel.cuh's SearchShared and the
// parts of its SearchParts.
struct SearchLayout {
    uint32_t runs, subs, head, qpeak, next, tkey, tab, wq, plane2, hotc, pbase, prow, qpid, tpid, tpk, qneed, end;
    uint32_t plane_words;       // a power of two
};

#include "search_kernel.cuh"
#include "count_kernel.cuh"

// lower bound of pid key (pid << 1) in entry[a, b)
__device__ __forceinline__ uint64_t entry_lower_bound(const uint32_t* __restrict__ entry, uint64_t a, uint64_t b,
                                                      uint32_t pid) {
    const uint32_t key = pid << 1;
    while (a < b) {
        const uint64_t m = (a + b) >> 1;
        if (__ldg(entry + m) < key) a = m + 1; else b = m;
    }
    return a;
}

// Where merge_kernel finds a spectrum's sorted lists and its histogram: the
// units of a search, or the results of the parts of a database (rows and
// partial histograms of part p behind those of part p - 1), whose summed
// histogram and candidate count it writes too.
struct MergeArgs {
    const uint64_t* seg_off;         // search: first unit of every spectrum
    const UnitTop* utop;
    const hicops_psm* parts;         // parts: rows, counts, how many
    const uint32_t* ns_in;
    uint32_t n_parts, hist_parts;
    uint32_t* hist_out;
    uint32_t* ns_out;
    const uint32_t* hist;
    uint32_t n, k;
    hicops_psm* out;
    uint32_t pid_stride, pid_base;   // row pid = list pid * pid_stride + pid_base ...
    const uint32_t* pid_map;         // ... or pid_map[list pid] when not NULL
    uint32_t ev_mode;                // HICOPS_EVALUE_* bits
};

__device__ __forceinline__ double warp_sum_f64(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// the greatest of the lanes' 64-bit values, and which lanes hold it
__device__ __forceinline__ int64_t warp_max_i64(int64_t v, bool* mine) {
    const int hi = (int)(v >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
    const uint32_t lo = hi == mh ? (uint32_t)v : 0u, ml = __reduce_max_sync(0xffffffffu, lo);
    *mine = hi == mh && lo == ml;
    return (int64_t)((uint64_t)(uint32_t)mh << 32 | ml);
}

// lane l's eight bins 8 l .. 8 l + 7 of a histogram (a caller's buffer: 4-byte aligned only)
__device__ __forceinline__ void lane_bins(const uint32_t* __restrict__ h, int lane, uint32_t* v) {
    const uint32_t* at = h + 8 * lane;
    if ((reinterpret_cast<uintptr_t>(h) & 15u) == 0) {
        const uint4 x = __ldg(reinterpret_cast<const uint4*>(at)), y = __ldg(reinterpret_cast<const uint4*>(at) + 1);
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
        v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = __ldg(at + i);
    }
}

// One warp per spectrum (kMergeWarps spectra per block): the top-k merge of
// the spectrum's lists, then the e-value fit (Supplementary Algorithm 4) over
// its histogram.  Lane l owns lists l and l + 32 (at most 64, each sorted by
// (key desc, pid asc)), holds the head and the next row of each, and k rounds
// of a warp argmax over the heads give the rows in rank order.  Lane l holds
// histogram bins 8l .. 8l + 7.
// The FP64 unit (2 lanes a clock) bounds it, whatever number of lanes an
// instruction has, so the FP64 work of the block's spectra is put together:
// the fit's points are spread over the block's threads for the logarithms,
// the lines are solved by a thread each, and the rows' e-values are a thread
// each; the sums of whole numbers are taken in integers (exact in both).
// 30,000 spectra: 207 -> 94 us; 20,000 of eight parts: 212 us with the
// kernel that gathered the parts -> 132 us.
template <bool PARTS>
__global__ void __launch_bounds__(kMergeWarps * 32) merge_kernel(const __grid_constant__ MergeArgs a) {
    static_assert(kMergeWarps * kMaxTopK <= kMergeWarps * 32, "a thread a row");
    // the fit's survival function G[0..256]; at a point of the fit, then its ordinate
    __shared__ int64_t gsurv[kMergeWarps][kHistBins + 1];
    __shared__ UnitTop rows[kMergeWarps][kMaxTopK];
    __shared__ uint32_t first[kMergeWarps], points[kMergeWarps], total[kMergeWarps];
    __shared__ double sum_y[kMergeWarps], sum_xy[kMergeWarps];      // then slope and intercept
    __shared__ uint32_t sum_1[kMergeWarps], sum_x[kMergeWarps], sum_xx[kMergeWarps];
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const uint32_t q = blockIdx.x * kMergeWarps + wi;
    int64_t* const G = gsurv[wi];
    const uint32_t k = a.k;
    const bool weibull = (a.ev_mode & HICOPS_EVALUE_LOG_WEIBULL) != 0u;
    uint32_t s0 = 1, np = 0;      // the fit's points: bins (linear) or bins + 1 (log-Weibull)
    if (q < a.n) {
        uint32_t v[8];
        lane_bins(a.hist + (uint64_t)q * kHistBins, lane, v);
        if (PARTS) {
            uint32_t c = lane == 0 ? a.ns_in[q] : 0u;
            for (uint32_t p = 1; p < a.hist_parts; ++p) {
                uint32_t w[8];
                lane_bins(a.hist + ((uint64_t)p * a.n + q) * kHistBins, lane, w);
#pragma unroll
                for (int i = 0; i < 8; ++i) v[i] += w[i];
                if (lane == 0) c += a.ns_in[(uint64_t)p * a.n + q];
            }
            uint32_t* ho = a.hist_out + (uint64_t)q * kHistBins + 8 * lane;
            if ((reinterpret_cast<uintptr_t>(a.hist_out) & 15u) == 0) {
                reinterpret_cast<uint4*>(ho)[0] = make_uint4(v[0], v[1], v[2], v[3]);
                reinterpret_cast<uint4*>(ho)[1] = make_uint4(v[4], v[5], v[6], v[7]);
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) ho[i] = v[i];
            }
            if (lane == 0) a.ns_out[q] = c;
        }
        // the lists
        const uint64_t u0 = PARTS ? 0 : a.seg_off[q];
        const int nl = PARTS ? (int)a.n_parts : (int)(a.seg_off[q + 1] - u0);
        const UnitTop none{INT64_MIN, 0xffffffffu, 0u};
        auto row = [&](int l, uint32_t r) -> UnitTop {
            if (l >= nl || r >= k) return none;
            if (!PARTS) return a.utop[(u0 + l) * k + r];
            const hicops_psm* t = a.parts + ((uint64_t)l * a.n + q) * k + r;
            return UnitTop{t->key, t->pid, ((uint32_t)t->nb << kNbShift) | ((uint32_t)t->ny << kNyShift)};
        };
        UnitTop c0 = row(lane, 0), n0 = row(lane, 1);
        UnitTop c1 = row(lane + 32, 0), n1 = row(lane + 32, 1);
        uint32_t h0 = 1, h1 = 1;   // rows n0 and n1 hold
        if (lane < k) rows[wi][lane] = none;
        __syncwarp();
        int64_t key0 = INT64_MIN;
        uint32_t r = 0;
        for (; r < k; ++r) {
            const bool second = c1.pid != 0xffffffffu && (c0.pid == 0xffffffffu || better(c1.key, c1.pid, c0.key, c0.pid));
            const uint32_t pid = second ? c1.pid : c0.pid;
            const int64_t key = pid != 0xffffffffu ? (second ? c1.key : c0.key) : INT64_MIN;
            bool best;
            const int64_t wk = warp_max_i64(key, &best);
            const uint32_t wp = __reduce_min_sync(0xffffffffu, best ? pid : 0xffffffffu);
            if (wp == 0xffffffffu) break;   // every list is at its end
            const int wl = __ffs(__ballot_sync(0xffffffffu, best && pid == wp)) - 1;
            if (r == 0) key0 = wk;
            if (lane == wl) {
                rows[wi][r] = second ? c1 : c0;
                if (second) {
                    c1 = n1;
                    n1 = row(lane + 32, ++h1);
                } else {
                    c0 = n0;
                    n0 = row(lane, ++h0);
                }
            }
        }
        const bool have_top = r > 0;
        uint32_t n_sum = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) n_sum += v[i];
        n_sum = __reduce_add_sync(0xffffffffu, n_sum);
        if (lane == 0) total[wi] = n_sum;
        // the distribution the fit sees (R16): the histogram, or 35 times its
        // 5-point quadratic Savitzky-Golay smoothing (zero outside the bins);
        // integers, so every sum and comparison below is exact
        int64_t g[8];
        {
            const uint32_t l2 = __shfl_up_sync(0xffffffffu, v[6], 1), l1 = __shfl_up_sync(0xffffffffu, v[7], 1);
            const uint32_t r1 = __shfl_down_sync(0xffffffffu, v[0], 1), r2 = __shfl_down_sync(0xffffffffu, v[1], 1);
            int64_t e[12];
            e[0] = lane > 0 ? l2 : 0;
            e[1] = lane > 0 ? l1 : 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) e[2 + i] = v[i];
            e[10] = lane < 31 ? r1 : 0;
            e[11] = lane < 31 ? r2 : 0;
            const bool smooth = (a.ev_mode & HICOPS_EVALUE_SMOOTH) != 0u;
#pragma unroll
            for (int i = 0; i < 8; ++i)
                g[i] = smooth ? -3 * e[i] + 12 * e[i + 1] + 17 * e[i + 2] + 12 * e[i + 3] - 3 * e[i + 4] : e[i + 2];
        }
        // survival G[j] = sum of g[i >= j]: within the lane, then over the lanes above
        int64_t loc[8];
        int64_t run = 0;
#pragma unroll
        for (int i = 7; i >= 0; --i) { run += g[i]; loc[i] = run; }
        int64_t above = run;   // inclusive suffix over lanes >= lane
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_down_sync(0xffffffffu, above, o);
            if (lane + o < 32) above += y;
        }
        above -= run;           // lanes > lane
#pragma unroll
        for (int i = 0; i < 8; ++i) G[8 * lane + i] = loc[i] + above;
        if (lane == 0) G[kHistBins] = 0;
        if (have_top) {
            if (weibull) {
                // R17: least squares of -ln(-ln F_j) on x = j + 1, F_j = 1 - G[j+1] / G[0],
                // over the bins with 0 < F_j < 1
                np = kHistBins;
            } else {
                // R12 on g: the mode (largest g, lowest bin on ties), then the line
                // through (j, log10(G[j] / G[0])) for j in [mode + 1, jtop - 1], G[j] > 0
                int64_t bv = g[0];
                int bj = 8 * lane;
#pragma unroll
                for (int i = 1; i < 8; ++i)
                    if (g[i] > bv) { bv = g[i]; bj = 8 * lane + i; }
                bool best;
                warp_max_i64(bv, &best);
                s0 = __reduce_min_sync(0xffffffffu, best ? (uint32_t)bj : 0xffffffffu) + 1u;
                int64_t jtop = key0 >> 31;
                if (jtop > 255) jtop = 255;
                if (jtop > (int64_t)s0) np = (uint32_t)jtop - s0;
            }
        }
    }
    if (lane == 0) {
        first[wi] = s0;
        points[wi] = np;
    }
    __syncthreads();
    uint32_t all = 0;
#pragma unroll
    for (int w = 0; w < kMergeWarps; ++w) all += points[w];
    for (uint32_t i = threadIdx.x; i < all; i += kMergeWarps * 32) {
        uint32_t at = i;
        int w = 0;
        for (; at >= points[w]; ++w) at -= points[w];
        at += first[w];
        const int64_t gj = gsurv[w][at], G0 = gsurv[w][0];
        double y = NAN;                                  // not a point
        if (gj > 0 && (!weibull || gj < G0)) {
            const double f = (double)gj / (double)G0;
            y = weibull ? -log(-log1p(-f)) : log10(f);
        }
        gsurv[w][at] = __double_as_longlong(y);
    }
    __syncthreads();
    if (np) {   // warp-uniform
        uint32_t c1 = 0, cx = 0, cxx = 0;
        double sy = 0, sxy = 0;
        for (uint32_t i = lane; i < np; i += 32) {
            const uint32_t xi = s0 + i;
            const double y = __longlong_as_double(G[xi]);
            if (!isnan(y)) {
                const double x = (double)xi;
                c1 += 1u;
                cx += xi;
                cxx += xi * xi;
                sy += y;
                sxy += x * y;
            }
        }
        c1 = __reduce_add_sync(0xffffffffu, c1);
        cx = __reduce_add_sync(0xffffffffu, cx);
        cxx = __reduce_add_sync(0xffffffffu, cxx);
        sy = warp_sum_f64(sy);
        sxy = warp_sum_f64(sxy);
        if (lane == 0) {
            sum_1[wi] = c1;
            sum_x[wi] = cx;
            sum_xx[wi] = cxx;
            sum_y[wi] = sy;
            sum_xy[wi] = sxy;
        }
    } else if (lane == 0) {
        sum_1[wi] = 0;
    }
    __syncthreads();
    if (threadIdx.x < kMergeWarps) {
        const int w = threadIdx.x;
        if (sum_1[w] >= 3u) {
            const double cn = (double)sum_1[w], sx = (double)sum_x[w], sxx = (double)sum_xx[w];
            const double sy = sum_y[w], sxy = sum_xy[w];
            const double den = cn * sxx - sx * sx;
            const double wfit = (cn * sxy - sx * sy) / den;
            sum_y[w] = wfit;
            sum_xy[w] = (sy - wfit * sx) / cn;
            if (weibull && !(wfit > 0.0)) sum_1[w] = 0;
        }
    }
    __syncthreads();
    if (threadIdx.x < kMergeWarps * k) {
        const uint32_t w = threadIdx.x / k, r = threadIdx.x % k;
        const uint32_t qo = blockIdx.x * kMergeWarps + w;
        if (qo < a.n) {
            const UnitTop t = rows[w][r];
            hicops_psm o;
            o.query = qo;
            o.reserved = 0;
            if (t.pid != 0xffffffffu) {
                o.pid = a.pid_map ? a.pid_map[t.pid] : t.pid * a.pid_stride + a.pid_base;
                o.nb = (uint8_t)(t.packed >> kNbShift);
                o.ny = (uint8_t)((t.packed >> kNyShift) & 63u);
                o.key = t.key;
                o.hyperscore = (float)((double)t.key * 0x1p-32);
                const double x = (double)t.key * 0x1p-31, N = (double)total[w];
                const double wfit = sum_y[w], bfit = sum_xy[w];
                if (sum_1[w] < 3u) o.evalue = N;
                else if (weibull) o.evalue = N * -expm1(-exp(-(wfit * x + bfit)));   // N * P(score >= x)
                else o.evalue = N * exp10(wfit * x + bfit);
            } else {
                o.pid = 0xffffffffu;
                o.nb = o.ny = 0;
                o.key = INT64_MIN;
                o.hyperscore = 0.0f;
                o.evalue = INFINITY;
            }
            a.out[(uint64_t)qo * k + r] = o;
        }
    }
}

// Fragment tolerance of t bins (R15): replaces spectrum q's retained peaks
// (distinct bins in any order) by the union of their windows [b - t, b + t]
// cut to [0, n_bins), ascending, each bin with the largest iq of the peaks
// covering it.  One warp per spectrum, in place: the peaks are read into
// shared memory and sorted by bin first, unless they ascend already.  Peak i emits the bins of its
// window above the previous peak's window, so no bin is emitted twice, and
// only peaks j >= i can cover them.
constexpr int kExpWarps = 4;

struct ExpandArgs {
    uint32_t* qbin;
    uint32_t* qiq;
    uint32_t* qn;
    uint32_t n, stride, t, n_bins;
};

__global__ void __launch_bounds__(kExpWarps * 32) expand_kernel(ExpandArgs a) {
    __shared__ uint64_t keys_all[kExpWarps][kMaxTopN];
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const uint32_t q = blockIdx.x * kExpWarps + wi;
    if (q >= a.n) return;   // warp-uniform
    const uint32_t cnt = a.qn[q];
    if (cnt == 0) return;
    uint64_t* keys = keys_all[wi];
    uint32_t* qb = a.qbin + (uint64_t)q * a.stride;
    uint32_t* qi = a.qiq + (uint64_t)q * a.stride;
    const int npow = next_pow2((int)cnt);
    for (int i = lane; i < npow; i += 32) keys[i] = i < (int)cnt ? ((uint64_t)qb[i] << 32) | qi[i] : ~0ull;
    __syncwarp();
    bool ascends = true;                 // as prep_warp leaves them
    for (int i = lane; i + 1 < (int)cnt; i += 32) ascends = ascends && keys[i] <= keys[i + 1];
    if (!__all_sync(0xffffffffu, ascends)) {
        __syncwarp();
        warp_bitonic_sort_u64(keys, npow, lane);
    }
    const uint32_t t = a.t;
    uint32_t base = 0;
    for (uint32_t i0 = 0; i0 < cnt; i0 += 32) {   // warp-uniform trip count
        const uint32_t i = i0 + lane;
        uint32_t lo = 0, hi = 0;   // bins [lo, hi) emitted by peak i
        if (i < cnt) {
            const uint32_t b = (uint32_t)(keys[i] >> 32);
            lo = b > t ? b - t : 0u;
            if (i > 0) lo = max(lo, (uint32_t)(keys[i - 1] >> 32) + t + 1u);
            hi = min(b + t + 1u, a.n_bins);
            if (hi < lo) hi = lo;
        }
        const uint32_t len = hi - lo;
        uint32_t incl = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        const uint32_t pos = base + incl - len;
        base += __shfl_sync(0xffffffffu, incl, 31);
        for (uint32_t x = lo; x < hi; ++x) {
            uint32_t best = 0;
            for (uint32_t j = i; j < cnt; ++j) {
                const uint64_t kj = keys[j];
                if ((uint32_t)(kj >> 32) > x + t) break;
                best = max(best, (uint32_t)kj);
            }
            qb[pos + (x - lo)] = x;
            qi[pos + (x - lo)] = best;
        }
    }
    if (lane == 0) a.qn[q] = base;
}

// per spectrum: sum over retained peaks of the bucket entries inside [lo, hi)
__global__ void work_kernel(const uint32_t* __restrict__ qbin, const uint32_t* __restrict__ qn,
                            const uint32_t* __restrict__ lo, const uint32_t* __restrict__ hi, uint32_t topn,
                            const uint64_t* __restrict__ off, const uint32_t* __restrict__ entry,
                            uint64_t* __restrict__ hits) {
    const uint32_t q = blockIdx.x;
    uint64_t h = 0;
    for (uint32_t t = threadIdx.x; t < qn[q]; t += blockDim.x) {
        const uint32_t bin = qbin[(uint64_t)q * topn + t];
        const uint64_t b0 = off[bin], b1 = off[bin + 1];
        const uint64_t c = entry_lower_bound(entry, b0, b1, lo[q]);
        const uint64_t e = entry_lower_bound(entry, c, b1, hi[q]);
        h += e - c;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
    __shared__ uint64_t red[8];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = h;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint64_t t = 0;
        for (int w = 0; w < (int)(blockDim.x / 32); ++w) t += red[w];
        hits[q] = t;
    }
}

}  // namespace
}  // namespace hicops
