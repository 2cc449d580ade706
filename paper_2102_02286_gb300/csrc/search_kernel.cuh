// filter_2 + score + heap of superstep 3 (paper: Eq. 4 terms k32'..k34,
// Supplementary Algorithm 3), included by search_kernels.cuh.
//
// One persistent CTA pulls work units (spectrum q, peptide-id segment) from a
// device counter.  The segment is walked in super-chunks of whole skip-table
// columns (kChunk peptide ids each).  Of the tens of thousands of index
// entries a unit reads, a few dozen peptides reach min_shared, so the pass
// over the entries only finds which peptides can, and those are scored
// afterwards from the forward index (each peptide's own list of ion bins):
//   pass A  every index entry of the ordinary peaks' runs sets its peptide's
//           bit in a bit-plane in shared memory; an entry whose bit was set
//           is a repeat and goes to its warp's queue, which is emptied with
//           every lane busy into an open-addressing table of (peptide,
//           repeats).  In a wide window (deep) a super-chunk spans more
//           peptides than the plane has bits, and a repeat has to find its
//           bit in a second plane set before it counts;
//   scan    only in a unit whose hot slices can qualify a peptide of one
//           ordinary hit (or none): the plane together with the bitmaps;
//   select  peptides of the table that can reach min_shared with their hot
//           bits go to the unit's queue (their ordinary hits are known, or
//           bounded from above when deep);
//   drain   at the unit's end, or when the queue runs full: the hot bits are
//           checked, then eight lanes read each remaining peptide's ion bins
//           (16-byte loads) and look them up in a table of the spectrum's
//           retained bins: nb, ny and S are exact, the key K = LF[nb] + LF[ny]
//           + LS[S] enters the histogram and the warp's top-k list.
// Should the repeats not fit their table, the super-chunk is halved, down to
// one column, which is then searched with one counter a peptide.
//
// What bounds it: the latencies and the issue slots of pass A (one shared
// atomic and about 16 instructions an entry; DRAM moves 580 KB a spectrum, a
// third of the time at full rate) and, in spectra with thousands of scored
// peptides, the drain.  Against the form that logged every entry and replayed
// the log (one bit a peptide in two planes, super-chunks of 13 columns): 30k
// spectra of 100 peaks at +-500 Da on 13.0 M peptides 15.7 -> 8.3 ms, 6k of 150
// peaks on 11.7 M peptides 5.2 -> 3.5 ms, 12k of 50-500 peaks at mixed
// tolerances 4.9 -> 3.1 ms; with windows cut by cost (plan_kernel) 7.6, 2.6 and
// 2.9 ms.

constexpr int kMaxHot = 6;                 // bitmap slices (b or y bitmap of a hot bucket) per spectrum
constexpr int kMaxWarps = 16;              // CTAs of up to 512 threads
constexpr uint32_t kSub = 8;               // lanes that walk a run together (8 groups of 4 entries: 128 bytes)
constexpr uint32_t kSlotBits = 11;
constexpr uint32_t kSlots = 1u << kSlotBits;   // repeat counters of a super-chunk
constexpr uint32_t kProbes = 64;           // slots tried before the table counts as full
constexpr uint32_t kHeads = 2048;          // chains of the retained bins' table
constexpr uint32_t kKeysAim = 700;         // peptides of the repeat table aimed at
constexpr uint32_t kQueue = 1152;          // a unit's queue of peptides to score
constexpr uint32_t kWarpQueue = 144;       // a warp's repeats waiting for the table
constexpr uint32_t kPlane2Bits = 11;       // words of the second plane (2^16 bits)
constexpr uint32_t kPlane2Words = 1u << kPlane2Bits;
constexpr float kPlane2Aim = 6500.0f;      // repeats it takes (they collide n n / 2^17 times)
constexpr uint32_t kNoEnd = 0x7fffffffu;    // length of the run that closes the list
constexpr uint32_t kOffBits = 24;          // peptide offset inside a super-chunk (repeat table key)
constexpr uint32_t kDirectNeed = 0x80u;    // queue flag: found by a scan of every peptide
constexpr uint32_t kMinPlaneWords = 4096;  // smallest plane worth another CTA on the SM (8 columns)
constexpr uint32_t kSmemPerSm = 233472;    // shared memory of an SM; each CTA also takes 1 KB of it

struct SearchArgs {
    const uint32_t* qbin;
    const uint32_t* qiq;
    const uint32_t* qn;
    uint32_t stride;            // qbin / qiq words per spectrum
    const uint4* unit;          // [units] the units in the order they are taken
    const uint64_t* n_units;    // their number
    const BinInfo* bins;        // [n_bins] bucket of every bin
    const uint32_t* entry;      // pid << 1 | isY
    const uint32_t* skip;
    uint32_t skip_stride;
    const uint32_t* hot_b;
    const uint32_t* hot_y;
    uint64_t hot_words;
    const uint64_t* fwd_off;    // [P + 1] forward lists, in groups of 4
    const uint4* fwd;           // bin << 1 | isY
    const int64_t* lf;
    const int64_t* ls;
    uint32_t s_max;             // last valid index of ls
    uint32_t min_shared;
    uint32_t k;
    uint32_t target_entries;    // entries aimed for per super-chunk
    UnitTop* utop;              // [units * k]
    uint32_t* hist;             // [n * 256]
    uint32_t* nscored;          // [n]
    unsigned long long* work;   // unit counter
    SearchLayout lay;
};

__device__ __forceinline__ bool better(int64_t ka, uint32_t pa, int64_t kb, uint32_t pb) {
    return ka > kb || (ka == kb && pa < pb);
}

// Where a CTA is in its unit (the same in every thread).
struct UnitState {
    uint32_t c, e;                    // the super-chunk's columns
    uint32_t m;                       // columns of a super-chunk
    uint32_t deep;                    // repeats pass the second plane before the table
    uint32_t taken;                   // the next unit is taken
    uint32_t slot;                    // of the current unit
};

struct SearchShared {
    const uint32_t* slice[kMaxHot];   // bitmap rows of the spectrum's hot slices
    uint32_t hist[kHistBins];
    int64_t lf[kMaxLen + 1];
    uint32_t wsum[kMaxWarps], wruns[kMaxWarps];
    int wn[kMaxWarps];                // length of each warp's top-k list
    uint32_t nkeys;                   // peptides in the repeat table
    int over;                         // it was full (or holds more than the queue takes)
    int no_room;                      // the queue may not take what the repeat table holds (-1: it is empty)
    uint32_t nq, npass;               // peptides in the queue, and of them past the hot-bit check
    int nnorm, nhotc, nslices, nhotpeaks;
    uint4 unit[2];                    // the current unit and the one taken next (alternating): spectrum, segment,
                                      // unit number
    uint64_t t_next;                  // its place in the order
    int have;                         // there is one
    uint32_t per, total;              // pieces of an octet's share, and of all
    UnitState st;                     // the current unit's, across the calls that need every register
};

// All shared memory is dynamic: the plane first (its address is then a
// constant of the atomics), SearchShared behind it and the parts of the
// layout.  Functions that are not inlined reach it through these, so that
// their accesses are shared-memory instructions too.
__device__ __forceinline__ uint32_t* search_smem() {
    extern __shared__ __align__(16) uint32_t smem32[];
    return smem32;
}
__device__ __forceinline__ SearchShared& search_shared(const SearchArgs& a) {
    return *reinterpret_cast<SearchShared*>(search_smem() + a.lay.plane_words);
}

// The parts of dynamic shared memory, and what the scoring of a unit needs.
struct SearchParts {
    uint4* runs;          // [maxp + 1] the super-chunk's non-empty runs: first group, groups, the first piece's
                          // start from the first group (its line's: 0 or below); then one without end
    uint2* subs;          // [nsub] where each octet's share starts: its run, and its first piece there
    uint32_t* head;       // [kHeads / 2] pairs of 16-bit chain heads of the retained bins' table: peak + 1, or 0
    uint2* qpeak;         // [maxp] the retained peaks: bin, quantised intensity
    uint16_t* next;       // [maxp] the next peak of the chain + 1, or 0
    int64_t* tkey;        // [nwarps * k] the warps' best candidates, sorted by (key desc, pid asc)
    uint32_t* tab;        // [kSlots] (offset << (32 - kOffBits)) | repeats
    uint32_t* wq;         // [nwarps * kWarpQueue] repeats on their way to it
    uint32_t* plane2;     // [kPlane2Words]
    uint32_t* hotc;       // [maxp] the bins of the hot peaks
    uint32_t* pbase;      // [maxp] first group of each ordinary peak's bucket
    uint32_t* prow;       // [maxp] its skip-table row
    uint32_t* qpid;       // [kQueue]
    uint32_t* tpid;       // [nwarps * k]
    uint32_t* tpk;        // [nwarps * k]
    uint8_t* qneed;       // [kQueue] hot bits needed, and kDirectNeed
    uint32_t* plane;      // [plane_words] (a power of two)
};

__device__ __forceinline__ SearchParts search_parts(const SearchLayout& l) {
    uint32_t* const base = search_smem();
    SearchParts p;
    p.runs = reinterpret_cast<uint4*>(base + l.runs);
    p.subs = reinterpret_cast<uint2*>(base + l.subs);
    p.head = base + l.head;
    p.qpeak = reinterpret_cast<uint2*>(base + l.qpeak);
    p.next = reinterpret_cast<uint16_t*>(base + l.next);
    p.tkey = reinterpret_cast<int64_t*>(base + l.tkey);
    p.tab = base + l.tab;
    p.wq = base + l.wq;
    p.plane2 = base + l.plane2;
    p.hotc = base + l.hotc;
    p.pbase = base + l.pbase;
    p.prow = base + l.prow;
    p.qpid = base + l.qpid;
    p.tpid = base + l.tpid;
    p.tpk = base + l.tpk;
    p.qneed = reinterpret_cast<uint8_t*>(base + l.qneed);
    p.plane = base;
    return p;
}

__device__ __forceinline__ uint32_t hash_u32(uint32_t x) { return x * 2654435761u; }

// The match of one ion bin, as nb | ny | S: a chained table by the bin modulo
// kHeads, where most bins find an empty head and few more than one peak.
__device__ __forceinline__ uint32_t match_ion(const SearchParts& sp, uint32_t ion) {
    const uint32_t bin = ion >> 1;   // pads are 0xffffffff: bin 2^31 - 1, in no spectrum
    uint32_t c = 0;
    uint32_t i = reinterpret_cast<const uint16_t*>(sp.head)[bin & (kHeads - 1u)];
    while (i) {
        const uint2 pk = sp.qpeak[i - 1u];
        if (pk.x == bin) {
            c = pk.y + ((ion & 1u) ? (1u << kNyShift) : (1u << kNbShift));
            break;
        }
        i = sp.next[i - 1u];
    }
    return c;
}
__device__ __forceinline__ uint32_t match_group(const SearchParts& sp, const uint4& x) {
    return match_ion(sp, x.x) + match_ion(sp, x.y) + match_ion(sp, x.z) + match_ion(sp, x.w);
}

// The key of a peptide's nb | ny | S.
template <class Args, class Shared>
__device__ __forceinline__ int64_t score_key(const Args& a, const Shared& sh, uint32_t c) {
    uint32_t S = c & kSMask;
    if (S > a.s_max) S = a.s_max;   // unreachable for a consistent index
    return sh.lf[c >> kNbShift] + sh.lf[(c >> kNyShift) & 63u] + __ldg(a.ls + S);
}

// The lanes' scored peptides (nb | ny | S in c, the key K): histogram, the
// warp's top-k list (lanes in turn).  Every lane of the warp calls it.
template <class Shared>
__device__ __forceinline__ void rank_lanes(Shared& sh, int k, int64_t* tkey, uint32_t* tpid, uint32_t* tpk, bool ok,
                                           uint32_t pid, uint32_t c, int64_t K) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    tkey += warp * k;
    tpid += warp * k;
    tpk += warp * k;
    bool pend = false;
    if (ok) {
        const int64_t hb = K >> 31;
        atomicAdd(&sh.hist[hb > 255 ? 255 : (hb < 0 ? 0 : hb)], 1u);
        const int n = sh.wn[warp];
        pend = n < k || better(K, pid, tkey[k - 1], tpid[k - 1]);
    }
    unsigned pm = __ballot_sync(0xffffffffu, pend);
    while (pm) {
        const int l = __ffs(pm) - 1;
        pm &= pm - 1;
        if (lane == l) {
            const int n = sh.wn[warp];
            if (n < k || better(K, pid, tkey[k - 1], tpid[k - 1])) {
                int pos = n < k ? n : k - 1;
                while (pos > 0 && better(K, pid, tkey[pos - 1], tpid[pos - 1])) {
                    tkey[pos] = tkey[pos - 1];
                    tpid[pos] = tpid[pos - 1];
                    tpk[pos] = tpk[pos - 1];
                    --pos;
                }
                tkey[pos] = K;
                tpid[pos] = pid;
                tpk[pos] = c;
                if (n < k) sh.wn[warp] = n + 1;
            }
        }
        __syncwarp();
    }
}

__device__ __forceinline__ uint32_t hits_of(uint32_t c) { return (c >> kNbShift) + ((c >> kNyShift) & 63u); }

__device__ __forceinline__ void score_lanes(const SearchArgs& a, SearchShared& sh, const SearchParts& sp, bool ok,
                                            uint32_t pid, uint32_t c) {
    ok = ok && hits_of(c) >= a.min_shared;
    rank_lanes(sh, (int)a.k, sp.tkey, sp.tpid, sp.tpk, ok, pid, c, ok ? score_key(a, sh, c) : INT64_MIN);
}

// A peptide is taken when its hot bits reach what its ordinary hits leave to
// min_shared (need); in a unit whose plane was scanned (once) a peptide of
// min_shared - 1 hot bits or more came from the scan (kDirectNeed), so the
// repeat table's entry for it is dropped.
__device__ __forceinline__ bool hot_check(const SearchArgs& a, const SearchShared& sh, uint32_t pid, uint32_t nd,
                                          bool once) {
    const bool scanned = (nd & kDirectNeed) != 0u;
    const uint32_t need = nd & ~kDirectNeed;
    if (!need && (scanned || !once)) return true;
    const int nslices = sh.nslices;
    uint32_t hw[kMaxHot], h = 0;   // every slice's word in flight at once
#pragma unroll
    for (int s = 0; s < kMaxHot; ++s) hw[s] = s < nslices ? __ldg(sh.slice[s] + (pid >> 5)) : 0u;
#pragma unroll
    for (int s = 0; s < kMaxHot; ++s) h += (hw[s] >> (pid & 31)) & 1u;
    return h >= need && (scanned || !once || h + 1u < a.min_shared);
}

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Scores cnt peptides pid[0..cnt) with the octets of the calling warp and of
// the nocts octets in all: octet o takes pid[o], pid[o + nocts], ...  Two
// peptides' first 64 ion bins (two 16-byte groups a lane) are in flight an
// octet; after eight peptides a lane's worth of results is scored.  oct0 is
// the lowest of the warp's octets, so that trips are warp-uniform.
__device__ __forceinline__ void score_list(const SearchArgs& a, SearchShared& sh, const SearchParts& sp,
                                           const uint32_t* pids, uint32_t cnt, uint32_t oct, uint32_t oct0,
                                           uint32_t nocts) {
    const uint32_t lane = threadIdx.x & 31, sl = lane & 7u;
    const uint4 none = make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu);
    for (uint32_t i0 = 0; i0 + oct0 < cnt; i0 += 8 * nocts) {
        // lane sl of the octet looks up item i0 + sl * nocts + oct
        const uint32_t it = i0 + sl * nocts + oct;
        uint32_t ng = 0;
        uint64_t g0 = 0;
        if (it < cnt) {
            const uint32_t pid = pids[it];
            g0 = __ldg(a.fwd_off + pid);
            ng = (uint32_t)(__ldg(a.fwd_off + pid + 1) - g0);
            // (the lists' lines on their way while the first two are matched)
            if (ng) prefetch_l2(a.fwd + g0);
            if (ng > 8u) prefetch_l2(a.fwd + g0 + 8u);
            if (ng > 16u) prefetch_l2(a.fwd + g0 + 16u);
        }
        uint32_t c = 0;
#pragma unroll 1
        for (uint32_t h = 0; h < 8 && i0 + h * nocts + oct0 < cnt; h += 2) {   // warp-uniform
            uint4 x[2], y[2];
            uint32_t nn[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int src = (int)((lane & 24u) + h) + j;
                const uint64_t gg = __shfl_sync(0xffffffffu, g0, src);
                nn[j] = __shfl_sync(0xffffffffu, ng, src);
                x[j] = sl < nn[j] ? __ldg(a.fwd + gg + sl) : none;
                y[j] = sl + 8u < nn[j] ? __ldg(a.fwd + gg + sl + 8u) : none;
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                uint32_t r = match_group(sp, x[j]);
                if (__any_sync(0xffffffffu, nn[j] > 8u)) r += match_group(sp, y[j]);
                if (__any_sync(0xffffffffu, nn[j] > 16u)) {   // more than 64 ion bins
                    const uint64_t gg = __shfl_sync(0xffffffffu, g0, (int)((lane & 24u) + h) + j);
#pragma unroll 1
                    for (uint32_t g = sl + 16u; __any_sync(0xffffffffu, g < nn[j]); g += 8u)
                        r += match_group(sp, g < nn[j] ? __ldg(a.fwd + gg + g) : none);
                }
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);   // fields cannot overflow
                if (sl == h + (uint32_t)j) c = r;
            }
        }
        score_lanes(a, sh, sp, it < cnt, it < cnt ? pids[it] : 0u, c);
    }
}

// Scores the unit's queue with the whole block and empties it (every thread
// calls it, behind a barrier after the last append; it ends with one).  The
// peptides past the hot-bit check are gathered in the warps' queues, which
// are empty between two passes.
__device__ __noinline__ void drain_queue(const SearchArgs& a) {
    SearchShared& sh = search_shared(a);
    const bool once = (uint32_t)sh.nslices + 1u >= a.min_shared;   // the plane was scanned
    const SearchParts sp = search_parts(a.lay);
    uint32_t* const pass = sp.wq;
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    const uint32_t cnt = min(sh.nq, kQueue);
    for (uint32_t i0 = tid & ~31u; i0 < cnt; i0 += blockDim.x) {   // warp-uniform trips
        const uint32_t i = i0 + lane;
        bool ok = i < cnt;
        uint32_t pid = 0;
        if (ok) {
            pid = sp.qpid[i];
            ok = hot_check(a, sh, pid, sp.qneed[i], once);
        }
        if (ok) pass[atomicAdd(&sh.npass, 1u)] = pid;
    }
    __syncthreads();
    // consecutive peptides go to different warps
    const uint32_t nwarps = blockDim.x >> 5;
    score_list(a, sh, sp, pass, sh.npass, (lane >> 3) * nwarps + (tid >> 5), tid >> 5, 4u * nwarps);
    __syncthreads();
    if (tid == 0) sh.nq = sh.npass = 0u;
    __syncthreads();
}

// Appends the lane's peptide to the unit's queue; false when it is full.
__device__ __forceinline__ bool push(const SearchArgs& a, SearchShared& sh, const SearchParts& sp, uint32_t pid,
                                     uint32_t need) {
    const uint32_t at = atomicAdd(&sh.nq, 1u);
    if (!(need & ~kDirectNeed)) prefetch_l2(a.fwd_off + pid);   // (it is sure to be scored)
    if (at >= kQueue) return false;   // (the counter stays past the end)
    sp.qpid[at] = pid;
    sp.qneed[at] = (uint8_t)need;
    return true;
}

// One more repeat of the peptide at offset off.
__device__ __forceinline__ void add_repeat(SearchShared& sh, const SearchParts& sp, uint32_t off) {
    uint32_t s = hash_u32(off) >> (32 - kSlotBits);
    for (uint32_t probe = 0; probe < kProbes; ++probe) {
        const uint32_t old = atomicCAS(&sp.tab[s], 0u, (off << (32 - kOffBits)) | 1u);
        if (old == 0u) {
            atomicAdd(&sh.nkeys, 1u);
            return;
        }
        if ((old >> (32 - kOffBits)) == off) {   // (a peptide has at most 126 ions: 8 bits hold its repeats)
            atomicAdd(&sp.tab[s], 1u);
            return;
        }
        s = (s + 1u) & (kSlots - 1u);
    }
    sh.over = 1;
}

// The plane of a super-chunk (first peptide pb, words in use, peptides [x0,
// x1)) together with the hot bitmaps: queues the peptides seen once or more
// with at least min_shared - 1 hot bits, and, when the hot peaks alone can
// reach min_shared, unseen ones with that many, and clears the plane.  Lane l
// of a warp takes 4 words at a time (16-byte reads).  When the queue is full
// every warp stops where it is, the block scores the queue, and they go on.
// Every thread calls it.
__device__ __noinline__ void scan_plane(const SearchArgs& a, uint32_t pb, uint32_t x0, uint32_t x1, uint32_t words) {
    SearchShared& sh = search_shared(a);
    const SearchParts sp = search_parts(a.lay);
    uint32_t* const plane = sp.plane;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const uint32_t min_shared = a.min_shared;
    const int nslices = sh.nslices;
    const bool hot_alone = sh.nhotpeaks >= (int)min_shared;
    const uint4 zero4 = make_uint4(0u, 0u, 0u, 0u);
    const bool all = !hot_alone && (uint32_t)nslices + 1u == min_shared;   // the intersection of the plane and every slice
    // below 5 the counts here are exact: nothing is left to check
    const uint32_t need = kDirectNeed | (min_shared <= 4u ? 0u : min_shared - 1u);
    const uint32_t step = 128u * nwarps;
    uint32_t w = warp * 128u + 4u * lane;   // the lane's next words
    uint32_t cand[4];
    bool held = false;      // candidates of the last step are left (the queue was full)
    // (entries outside the super-chunk may have set bits past its words)
    for (uint32_t i = words + threadIdx.x; i < a.lay.plane_words; i += blockDim.x)
        plane[((pb >> 5) + i) & (a.lay.plane_words - 1u)] = 0u;
    for (;;) {
        bool full = false;
        while (held || w - 4u * lane < words) {   // warp-uniform
            if (!held) {
                uint4 v = zero4;
                if (w < words) {
                    uint4* const at = reinterpret_cast<uint4*>(plane + (((pb >> 5) + w) & (a.lay.plane_words - 1u)));
                    v = *at;
                    v = make_uint4(__brev(v.x), __brev(v.y), __brev(v.z), __brev(v.w));   // the plane's bits run from the top
                    *at = zero4;
                }
                const bool look = w < words && (hot_alone || (v.x | v.y | v.z | v.w) != 0u);
                if (all) {
                    // (three slices' words in flight: min_shared is 4 in most searches)
#pragma unroll 1
                    for (int s = 0; s < nslices; s += 3) {
                        const uint4 h0 = look ? __ldg(reinterpret_cast<const uint4*>(sh.slice[s] + (pb >> 5) + w)) : zero4;
                        uint4 h1 = h0, h2 = h0;
                        if (look && s + 1 < nslices) h1 = __ldg(reinterpret_cast<const uint4*>(sh.slice[s + 1] + (pb >> 5) + w));
                        if (look && s + 2 < nslices) h2 = __ldg(reinterpret_cast<const uint4*>(sh.slice[s + 2] + (pb >> 5) + w));
                        v.x &= h0.x & h1.x & h2.x, v.y &= h0.y & h1.y & h2.y;
                        v.z &= h0.z & h1.z & h2.z, v.w &= h0.w & h1.w & h2.w;
                    }
                    cand[0] = v.x, cand[1] = v.y, cand[2] = v.z, cand[3] = v.w;
                } else {
                    // per peptide its hot bits' number: two low bits b1, b2, and b3 = 4 or more
                    uint32_t b1[4] = {0u, 0u, 0u, 0u}, b2[4] = {0u, 0u, 0u, 0u}, b3[4] = {0u, 0u, 0u, 0u};
#pragma unroll 2
                    for (int s = 0; s < nslices; ++s) {
                        const uint4 h = look ? __ldg(reinterpret_cast<const uint4*>(sh.slice[s] + (pb >> 5) + w)) : zero4;
                        const uint32_t hw[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const uint32_t k1 = b1[i] & hw[i];
                            b1[i] ^= hw[i];
                            b3[i] |= b2[i] & k1;
                            b2[i] ^= k1;
                        }
                    }
                    auto at_least = [](uint32_t c1, uint32_t c2, uint32_t c3, uint32_t t) {
                        // (a superset for t above 4: the queue's check is exact)
                        return t == 0 ? 0xffffffffu : t == 1 ? (c1 | c2 | c3) : t == 2 ? (c2 | c3)
                               : t == 3 ? ((c2 & c1) | c3) : c3;
                    };
                    const uint32_t seen[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        cand[i] = seen[i] & at_least(b1[i], b2[i], b3[i], min_shared - 1u);
                        if (hot_alone && look) cand[i] |= ~seen[i] & at_least(b1[i], b2[i], b3[i], min_shared);
                    }
                }
            }
            held = false;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t gp = pb + ((w + (uint32_t)i) << 5);
                while (cand[i] && !held) {
                    const uint32_t pid = gp + (uint32_t)__ffs(cand[i]) - 1u;
                    if (pid - x0 < x1 - x0 && !push(a, sh, sp, pid, need)) held = true;   // (peptides [x0, x1) only)
                    else cand[i] &= cand[i] - 1u;
                }
            }
            held = __any_sync(0xffffffffu, held);
            if (held) {
                full = true;
                break;
            }
            w += step;
        }
        if (!__syncthreads_or(full)) break;
        drain_queue(a);
    }
}

// A column [x0, x1) whose repeats overflow their list, with one 32-bit counter
// a peptide, in parts of the plane's size (the plane is all zero before and
// after).  The column's runs are in place.  Every thread calls it.
__device__ __noinline__ void direct_column(const SearchArgs& a, uint32_t x0, uint32_t x1) {
    SearchShared& sh = search_shared(a);
    const SearchParts sp = search_parts(a.lay);
    uint32_t* const plane = sp.plane;
    const uint32_t tid = threadIdx.x, part = a.lay.plane_words;
    const uint32_t min_shared = a.min_shared, nslices = (uint32_t)sh.nslices;
    const bool hot_alone = sh.nhotpeaks >= (int)min_shared;
    for (uint32_t pb = x0; pb < x1; pb += part) {
        const uint32_t span = min(part, x1 - pb);
        for (int t = 0; sp.runs[t].y != kNoEnd; ++t) {   // (the run without end closes the list)
            const uint4 r = sp.runs[t];
            for (uint32_t g = tid; g < r.y; g += blockDim.x) {
                const uint4 e = __ldg(reinterpret_cast<const uint4*>(a.entry) + r.x + g);
                const uint32_t e4[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint32_t o = (e4[i] >> 1) - pb;   // (a pad is past every span)
                    if (o < span) atomicAdd(&plane[o], 1u);
                }
            }
        }
        __syncthreads();
        uint32_t i = tid;
        for (;;) {
            bool full = false;
            for (; i < span; i += blockDim.x) {
                const uint32_t ord = plane[i];
                if (((ord && ord + nslices >= min_shared) || hot_alone) &&
                    !push(a, sh, sp, pb + i, kDirectNeed | (ord < min_shared ? min_shared - ord : 0u))) {
                    full = true;
                    break;
                }
                plane[i] = 0u;
            }
            if (!__syncthreads_or(full)) break;
            drain_queue(a);
        }
    }
}

// A run [ra, rb) of a bucket (positions relative to its 16-byte aligned start
// at group base) is read as whole groups of 4 entries.  The extra entries at
// either end lie in the same bucket outside the run's columns, or are the
// bucket's pad slots; both fall outside every peptide range the run is
// searched for.  Its pieces are the 128-byte lines it touches: octets that
// read whole lines take 61 cycles a step of two pieces from DRAM, octets
// that straddle them 83 to 116 (measured on the reads and atomics alone).
struct Run {
    uint32_t start, len;   // first group, groups
    __device__ __forceinline__ Run(uint32_t base, uint32_t ra, uint32_t rb)
        : start(base + (ra >> 2)), len(ra == rb ? 0u : ((rb + 3u) >> 2) - (ra >> 2)) {}
    __device__ __forceinline__ uint32_t pieces() const {
        return len ? (start + len + kSub - 1u) / kSub - start / kSub : 0u;
    }
};

// Predicated accesses of the pass over the entries, without branches.
// 16-byte group g of the index when ok; the first word is all ones otherwise.
__device__ __forceinline__ uint4 load_group(const uint32_t* entry, uint32_t g, bool ok) {
    uint4 v;
    v.x = 0xffffffffu;   // (the others stay what they are then)
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t@p ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];\n\t}"
                 : "+r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(reinterpret_cast<const uint4*>(entry) + g), "r"((uint32_t)ok));
    return v;
}
// stores v at shared address at when ok is not 0; the address behind it then
__device__ __forceinline__ uint32_t put_shared(uint32_t at, uint32_t v, uint32_t ok) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p st.shared.u32 [%0], %1;\n\t@p add.u32 %0, %0, 4;\n\t}"
                 : "+r"(at) : "r"(v), "r"(ok) : "memory");
    return at;
}

// The end of unit u of spectrum q: its top-k, where every item of the warps'
// sorted lists finds its rank among all of them, and its histogram added to the
// spectrum's.  Every thread calls it, behind a barrier after the last score.
template <int THREADS, class Args, class Shared>
__device__ __forceinline__ void unit_out(const Args& a, Shared& sh, const int64_t* tkey, const uint32_t* tpid,
                                         const uint32_t* tpk, uint32_t q, uint32_t u) {
    constexpr int nwarps = THREADS / 32;
    const int tid = threadIdx.x, lane = tid & 31;
    const int k = (int)a.k;
    for (uint32_t i = tid; i < (uint32_t)(nwarps * k); i += THREADS) {
        const uint32_t w = i / (uint32_t)k, r = i % (uint32_t)k;
        if (r >= (uint32_t)sh.wn[w]) continue;
        UnitTop row;
        row.key = tkey[i];
        row.pid = tpid[i];
        row.packed = tpk[i];
        uint32_t rank = r;
        for (uint32_t x = 0; x < (uint32_t)nwarps && rank < (uint32_t)k; ++x) {
            if (x == w) continue;
            const uint32_t n = (uint32_t)sh.wn[x];
            for (uint32_t y = 0; y < n; ++y) {
                if (!better(tkey[x * k + y], tpid[x * k + y], row.key, row.pid)) break;
                ++rank;
            }
        }
        if (rank < (uint32_t)k) a.utop[(uint64_t)u * k + rank] = row;
    }
    if (tid < k) {
        int total = 0;
#pragma unroll
        for (int w = 0; w < nwarps; ++w) total += sh.wn[w];
        if (tid >= total) {
            UnitTop row;
            row.key = INT64_MIN;
            row.pid = 0xffffffffu;
            row.packed = 0u;
            a.utop[(uint64_t)u * k + tid] = row;
        }
    }
    uint32_t mine = 0;
    for (int jb = tid; jb < (int)kHistBins; jb += THREADS) {
        const uint32_t h = sh.hist[jb];
        if (h) {
            atomicAdd(&a.hist[(uint64_t)q * kHistBins + jb], h);
            mine += h;
            sh.hist[jb] = 0;
        }
    }
    mine = __reduce_add_sync(0xffffffffu, mine);
    if (lane == 0 && mine) atomicAdd(&a.nscored[q], mine);
}

constexpr int search_min_ctas(int threads) { return threads <= 256 ? 3 : threads <= 384 ? 2 : 1; }

template <int THREADS, int PPT>
__global__ void __launch_bounds__(THREADS, search_min_ctas(THREADS)) search_kernel(const __grid_constant__ SearchArgs a) {
    SearchShared& sh = search_shared(a);
    constexpr int nwarps = THREADS / 32;
    constexpr uint32_t nsub = THREADS / kSub;
    constexpr int kG = 2;               // pieces in flight a thread
    const SearchParts sp = search_parts(a.lay);
    uint32_t* const plane = sp.plane;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // (a count_kernel behind this one may start where CTAs of this one have ended)
    asm volatile("griddepcontrol.launch_dependents;");
    for (uint32_t i = tid; i < a.lay.plane_words; i += THREADS) plane[i] = 0u;
    for (uint32_t i = tid; i < kSlots; i += THREADS) sp.tab[i] = 0u;
    for (uint32_t i = tid; i < kPlane2Words; i += THREADS) sp.plane2[i] = 0u;
    for (uint32_t i = tid; i < kHeads / 2; i += THREADS) sp.head[i] = 0u;
    for (int i = tid; i < (int)kHistBins; i += THREADS) sh.hist[i] = 0;
    for (int i = tid; i <= (int)kMaxLen; i += THREADS) sh.lf[i] = a.lf[i];
    UnitState st;
    st.slot = 0;
    // (thread 0) the unit at place t of the order becomes the CTA's next one
    auto set_unit = [&](uint64_t t) {
        sh.have = t < *a.n_units;
        if (sh.have) sh.unit[st.slot ^ 1u] = __ldg(a.unit + t);
    };
    if (tid == 0) {
        set_unit(blockIdx.x);   // the first by block index, then the counter's
        sh.nkeys = 0u;
        sh.over = 0;
    }
    // The calls below take what registers they like: the unit's state waits in
    // shared memory (every one of them has a barrier).
    auto save = [&]() {
        if (tid == 0) sh.st = st;
    };
    auto restore = [&]() { st = sh.st; };
    for (;;) {
        if (tid == 0) {
            sh.nnorm = 0;
            sh.nhotc = 0;
            sh.nslices = 0;
            sh.nhotpeaks = 0;
        }
        __syncthreads();
        if (!sh.have) break;
        st.slot ^= 1u;
        if (tid < nwarps) sh.wn[tid] = 0;      // (nothing is appended or scored before the next barriers)
        if (tid == 0) sh.nq = sh.npass = 0u;
        st.taken = 0;
        // the retained peaks: hot (bitmap) or ordinary (skip table), and all
        // of them into the hash of the spectrum's bins
        {
            const uint32_t q = sh.unit[st.slot].x, np = a.qn[q];
            const uint32_t* qb = a.qbin + (uint64_t)q * a.stride;
            const uint32_t* qi = a.qiq + (uint64_t)q * a.stride;
            for (uint32_t t = tid; t < np; t += THREADS) {
                const uint32_t bin = qb[t], iq = qi[t];
                const BinInfo bi = a.bins[bin];
                // (the peak becomes its chain's head: half a word, so by compare and swap)
                const uint32_t h = bin & (kHeads - 1u), half = 16u * (h & 1u);
                uint32_t seen = sp.head[h >> 1], was;
                do {
                    was = seen;
                    seen = atomicCAS(&sp.head[h >> 1], was, (was & ~(0xffffu << half)) | ((t + 1u) << half));
                } while (seen != was);
                sp.qpeak[t] = make_uint2(bin, iq);
                sp.next[t] = (uint16_t)(was >> half);
                if (bi.hot >= 0) {
                    sp.hotc[atomicAdd(&sh.nhotc, 1)] = bin;
                } else if (bi.row >= 0) {
                    const int s = atomicAdd(&sh.nnorm, 1);
                    sp.pbase[s] = bi.group;
                    sp.prow[s] = (uint32_t)bi.row;
                }
            }
        }
        __syncthreads();
        if (sh.nhotc) {   // uniform
            if (warp == 0) {
                // Bitmap slices for the hot peaks, the densest first (a lane
                // a hot peak, in rounds of an arg-max over their entries in
                // the segment's columns).  With min_shared - 1 slices or more
                // the plane has to be scanned for peptides of one ordinary hit
                // or none, which costs what streaming 1/8 of the segment's
                // peptides does: when the rest hold fewer entries, only
                // min_shared - 2 slices are taken and the rest are streamed
                // like ordinary peaks, as are those that get no slice at all
                // (all of them at min_shared 2: a scan would queue every hit).
                // Which hot peaks get slices does not change any result.
                const int nhc = sh.nhotc;
                const uint32_t lo = sh.unit[st.slot].y, hi = sh.unit[st.slot].z;
                const uint32_t c0 = lo >> kChunkShift, c1 = min(((hi - 1u) >> kChunkShift) + 1u, a.skip_stride - 1u);
                int ns = 0, nh = 0;   // warp-uniform
                for (int p0 = 0; p0 < nhc; p0 += 32) {   // (32 at a time: of more, the later ones are hardly ever taken)
                    BinInfo bi{0u, -1, -1, 0u};
                    uint32_t n = 0;
                    bool left = p0 + lane < nhc;
                    if (left) {
                        bi = a.bins[sp.hotc[p0 + lane]];
                        const uint32_t* sk = a.skip + (uint64_t)bi.row * a.skip_stride;
                        n = __ldg(sk + c1) - __ldg(sk + c0);
                    }
                    const int need = (int)(bi.flags & 1u) + (int)((bi.flags >> 1) & 1u);
                    float rest = (float)__reduce_add_sync(0xffffffffu, n >> 4) * 16.0f;   // entries of the peaks left
                    bool open = true;
                    while (open) {
                        const uint32_t most = __reduce_max_sync(0xffffffffu, left ? n + 1u : 0u);
                        if (!most) break;
                        const int w = __ffs(__ballot_sync(0xffffffffu, left && n + 1u == most)) - 1;
                        const int nd = __shfl_sync(0xffffffffu, need, w);
                        // the cap: min_shared - 2 while the rest are few (all of them, not only these 32)
                        const bool few = a.min_shared <= 2u || (nhc <= 32 && rest < (float)(hi - lo) * 0.125f);
                        if (ns + nd > (few ? min(kMaxHot, max((int)a.min_shared - 2, 0)) : kMaxHot)) open = false;
                        if (open) {
                            if (lane == w) {
                                int p = ns;
                                if (bi.flags & 1u) sh.slice[p++] = a.hot_b + (uint64_t)bi.hot * a.hot_words;
                                if (bi.flags & 2u) sh.slice[p] = a.hot_y + (uint64_t)bi.hot * a.hot_words;
                                left = false;
                            }
                            ns += nd;
                            ++nh;
                            rest -= (float)(most - 1u);
                        }
                    }
                    if (left) {
                        const int s = atomicAdd(&sh.nnorm, 1);
                        sp.pbase[s] = bi.group;
                        sp.prow[s] = (uint32_t)bi.row;
                    }
                }
                if (lane == 0) {
                    sh.nslices = ns;
                    sh.nhotpeaks = nh;
                }
            }
            __syncthreads();
        }
        // a thread owns the ordinary peaks tid * ppt .. + ppt - 1
        auto skip_at = [&](uint32_t (&r)[PPT], uint32_t col) {
            const int nnorm = sh.nnorm, ppt = (nnorm + THREADS - 1) / THREADS;
#pragma unroll
            for (int i = 0; i < PPT; ++i) {
                const int t = tid * ppt + i;
                r[i] = 0;
                if (i < ppt && t < nnorm)
                    r[i] = __ldg(a.skip + (uint64_t)sp.prow[t] * a.skip_stride + min(col, a.skip_stride - 1u));
            }
        };
        // Prefix of the runs' pieces (kSub groups each) and of the non-empty
        // runs over the block, in two halves around a barrier.  A super-
        // chunk's runs are [ra, rb) of the peaks' buckets.  Octet s of the
        // block takes pieces [s per, (s + 1) per) of all; per is returned.
        auto scan_1 = [&](const uint32_t (&ra)[PPT], const uint32_t (&rb)[PPT]) {
            const int nnorm = sh.nnorm, ppt = (nnorm + THREADS - 1) / THREADS;
            uint32_t sum = 0, cnt = 0;
#pragma unroll
            for (int i = 0; i < PPT; ++i) {
                const int t = tid * ppt + i;
                if (i < ppt && t < nnorm && ra[i] != rb[i]) {
                    sum += Run(sp.pbase[t], ra[i], rb[i]).pieces();
                    ++cnt;
                }
            }
            uint2 incl = make_uint2(sum, cnt);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t x = __shfl_up_sync(0xffffffffu, incl.x, o), y = __shfl_up_sync(0xffffffffu, incl.y, o);
                if (lane >= o) {
                    incl.x += x;
                    incl.y += y;
                }
            }
            if (lane == 31) {
                sh.wsum[warp] = incl.x;
                sh.wruns[warp] = incl.y;
            }
            return make_uint2(incl.x - sum, incl.y - cnt);
        };
        auto scan_2 = [&](uint2 run, const uint32_t (&ra)[PPT], const uint32_t (&rb)[PPT]) {
            const int nnorm = sh.nnorm, ppt = (nnorm + THREADS - 1) / THREADS;
            uint32_t total = 0, nruns = 0;
#pragma unroll
            for (int w = 0; w < nwarps; ++w) {
                const uint32_t p = sh.wsum[w], r = sh.wruns[w];
                if (w < warp) {
                    run.x += p;
                    run.y += r;
                }
                total += p;
                nruns += r;
            }
            const uint32_t per = (total + nsub - 1u) / nsub;
#pragma unroll
            for (int i = 0; i < PPT; ++i) {
                const int t = tid * ppt + i;
                if (i < ppt && t < nnorm && ra[i] != rb[i]) {
                    const Run r(sp.pbase[t], ra[i], rb[i]);
                    const uint32_t len = r.pieces();
                    sp.runs[run.y] = make_uint4(r.start, r.len, 0u - r.start % kSub, 0u);
                    for (uint32_t s = (run.x + per - 1u) / per; s * per < run.x + len; ++s)   // the octets that start here
                        sp.subs[s] = make_uint2(run.y, s * per - run.x);
                    run.x += len;
                    ++run.y;
                }
            }
            if (tid == 0) {
                sp.runs[nruns] = make_uint4(0u, kNoEnd, 0u, 0u);
                sh.per = per;
                sh.total = total;
            }
        };
        // Columns per super-chunk: what the plane holds (one bit a peptide),
        // about target_entries entries, and about kKeysAim repeats.  The
        // repeats of a window of W peptides and n entries are about n n / W
        // (twice what independent hits would give: measured 1.9 to 2.4 on the
        // workloads' databases).  When a peptide of one ordinary hit cannot
        // qualify and the window needs several such super-chunks, they are
        // made wider than the plane (deep): peptides that share a bit only
        // add repeats, about n n / 2 bits (at min_shared 2 each would be scored).  A repeat whose peptide needs three
        // ordinary hits or more then has to find its bit in the second plane
        // set (by an earlier repeat of its own, or of one that shares that
        // bit) before it counts, so the table only sees what is left of them,
        // and a peptide's ordinary hits are at most its count + 2.  The hits
        // that score are exact in any case.
        const uint32_t col_end = ((sh.unit[st.slot].z - 1) >> kChunkShift) + 1;
        st.c = sh.unit[st.slot].y >> kChunkShift;
        st.deep = 0;
        {
            uint32_t r0[PPT], r1[PPT];
            skip_at(r0, st.c);
            skip_at(r1, col_end);
            uint32_t s = 0;
#pragma unroll
            for (int i = 0; i < PPT; ++i) s += r1[i] - r0[i];
            s = __reduce_add_sync(0xffffffffu, s);
            if (lane == 0) sh.wsum[warp] = s;
            __syncthreads();
            float total = 0.0f;
#pragma unroll
            for (int w = 0; w < nwarps; ++w) total += (float)sh.wsum[w];
            const uint32_t ncols = max(col_end - st.c, 1u);
            const float per = total / (float)ncols;                   // entries a column
            const float rep = per * per / (float)kChunk;              // repeats a column
            auto cols = [&](float aim, float bits, uint32_t most) {   // rep m + (per m)^2 / 2 bits = aim
                const float q = bits > 0.0f ? per * per / (2.0f * bits) : 0.0f;
                float w = q > 0.0f ? (sqrtf(rep * rep + 4.0f * q * aim) - rep) / (2.0f * q) : aim / fmaxf(rep, 1e-6f);
                w = fminf(w, (float)a.target_entries / fmaxf(per, 1e-6f));
                return (uint32_t)fmaxf(1.0f, fminf(w, (float)min(most, ncols)));
            };
            st.m = cols((float)kKeysAim, 0.0f, a.lay.plane_words / (kChunk / 32));
            if ((uint32_t)sh.nslices + 2u <= a.min_shared && a.min_shared > 2u && st.m < ncols) {
                const uint32_t md = cols(kPlane2Aim, 32.0f * (float)a.lay.plane_words, (1u << kOffBits) / kChunk - 1u);
                if (md > st.m) {
                    st.m = md;
                    st.deep = 1;
                }
            }
            const uint32_t nsc = (ncols + st.m - 1u) / st.m;          // even super-chunks
            st.m = (ncols + nsc - 1u) / nsc;
            __syncthreads();   // wsum is reused by the scans
        }
        // the unit taken next, once the last super-chunk comes up (and once a
        // unit, though its end may be redone)
        auto take_unit = [&]() {
            if (st.e == col_end && !st.taken) {
                st.taken = 1;
                if (tid == 0) sh.t_next = (uint64_t)gridDim.x + atomicAdd(a.work, 1ull);
            }
        };
        // the first super-chunk from column st.c on
        auto start = [&]() {
            uint32_t r0[PPT], r1[PPT];
            st.e = min(st.c + st.m, col_end);
            take_unit();
            skip_at(r0, st.c);
            skip_at(r1, st.e);
            const uint2 excl = scan_1(r0, r1);
            __syncthreads();
            scan_2(excl, r0, r1);
            __syncthreads();
        };
        if (st.c < col_end) start();
        while (st.c < col_end) {
            const uint32_t x0 = max(sh.unit[st.slot].y, st.c << kChunkShift);
            const uint32_t x1 = (uint32_t)min((uint64_t)sh.unit[st.slot].z, (uint64_t)st.e << kChunkShift);
            const uint32_t pb = x0 & ~127u;                       // the plane's first peptide
            // plane words in use
            const uint32_t words = min(((x1 - pb + 127u) >> 5) & ~3u, a.lay.plane_words);
            // ---- pass A.  kSub lanes take a contiguous share of the runs'
            // pieces, one 16-byte group of 4 entries a lane and piece, kG
            // pieces in flight, two at a time through the plane.
            const uint32_t per = sh.per;
            const uint32_t oct = (uint32_t)tid / kSub, sl = (uint32_t)tid % kSub;
            const uint32_t mine = oct * per < sh.total ? min(per, sh.total - oct * per) : 0u;   // the octet's pieces
            const uint4* run = sp.runs;                  // the next piece's run
            uint4 cur = make_uint4(0u, kNoEnd, 0u, 0u);  // cur.z: the piece's first group, from the run's
            if (mine) {
                const uint2 at = sp.subs[oct];
                run += at.x;
                cur = *run;
                cur.z += at.y * kSub;
            }
            const bool more = st.e < col_end;
            uint32_t r1[PPT], r2[PPT];                            // the next super-chunk's runs
            if (more) {
                skip_at(r1, st.e);                                // in flight during pass A
                skip_at(r2, min(st.e + st.m, col_end));
            }
            // Peptide pid has bit 31 - pid % 32 of the plane's word pid / 32
            // modulo its words, so that a left shift by pid brings it to the
            // sign.  Entries past the super-chunk's end or before its start (a
            // run's rounding, a bucket's pads) set bits like any other: they
            // can only add repeats, and theirs are left out of the count.
            const uint32_t mask = 4u * a.lay.plane_words - 4u;   // of byte addresses
            uint32_t* const wq = sp.wq + warp * kWarpQueue;
            uint32_t qn = 0;                                     // repeats in the warp's queue
            for (uint32_t done = 0;; done += (uint32_t)kG) {     // (the same trips in every thread)
                uint4 ev[kG];
                uint32_t rep = 0;                                // bit 4 kG - 1 - i: entry i's bit was set before
                const bool last = done >= per;
                if (!last) {
#pragma unroll
                    for (int j = 0; j < kG; ++j) {
                        const uint4 nx = run[1];
                        if ((int)cur.z >= (int)cur.y) {
                            ++run;
                            cur = nx;
                        }
                        ev[j] = load_group(a.entry, cur.x + cur.z + sl, done + (uint32_t)j < mine && cur.z + sl < cur.y);
                        cur.z += kSub;
                    }
#pragma unroll
                    for (int j = 0; j < kG; ++j) {
                        // (a group inside a run starts with a real entry)
                        const uint32_t top = ev[j].x != 0xffffffffu ? 0x80000000u : 0u;
                        const uint32_t en[4] = {ev[j].x, ev[j].y, ev[j].z, ev[j].w};
                        uint32_t old[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            old[i] = atomicOr(reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(plane) + ((en[i] >> 4) & mask)),
                                              __funnelshift_r(top, 0u, en[i] >> 1));
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            rep = __funnelshift_l(__funnelshift_l(0u, old[i], en[i] >> 1), rep, 1);
                        if (!top) rep &= ~15u;
                    }
                }
                do {
                    // places in the queue: a prefix over the lanes' counts, bit
                    // by bit; more than it holds go one a lane at a time
                    uint32_t take = rep, n1 = 0, total = 0;
                    const uint32_t n = __popc(rep);
                    const unsigned lt = (1u << lane) - 1u;
#pragma unroll
                    for (int b = 0; b < 5; ++b) {
                        const unsigned m = __ballot_sync(0xffffffffu, (n >> b) & 1u);
                        n1 += (uint32_t)__popc(m & lt) << b;
                        total += (uint32_t)__popc(m) << b;
                    }
                    if (total > kWarpQueue) {
                        take = rep & (0u - rep);
                        const unsigned m = __ballot_sync(0xffffffffu, take != 0u);
                        n1 = (uint32_t)__popc(m & lt);
                        total = (uint32_t)__popc(m);
                    }
                    // the warp's queue into the table, when these do not fit and at the end
                    if (qn && (last || qn + total > kWarpQueue)) {
                        __syncwarp();
                        // kR repeats a lane, their hot words and second-plane
                        // atomics in flight together
                        constexpr int kR = (kWarpQueue + 31) / 32;
                        uint32_t pid[kR], h = 0, in = 0;   // h: four bits of hot bits a repeat; in: those that count
#pragma unroll
                        for (int r = 0; r < kR; ++r) {
                            pid[r] = lane + 32u * r < qn ? wq[lane + 32u * r] >> 1 : x1;
                            if (pid[r] - x0 < x1 - x0) in |= 1u << r;      // inside the super-chunk
                        }
                        if (st.deep) {
                            const uint32_t nslices = (uint32_t)sh.nslices;
                            if (nslices + 2u == a.min_shared)              // else three hits are needed in any case
                                for (uint32_t s = 0; s < nslices; ++s) {
                                    uint32_t hw[kR];
#pragma unroll
                                    for (int r = 0; r < kR; ++r)
                                        hw[r] = (in >> r) & 1u ? __ldg(sh.slice[s] + (pid[r] >> 5)) : 0u;
#pragma unroll
                                    for (int r = 0; r < kR; ++r) h += ((hw[r] >> (pid[r] & 31u)) & 1u) << (4 * r);
                                }
                            uint32_t old[kR];
#pragma unroll
                            for (int r = 0; r < kR; ++r) {
                                const uint32_t x = hash_u32(pid[r]);
                                old[r] = 0xffffffffu;
                                if (((in >> r) & 1u) && ((h >> (4 * r)) & 15u) + 2u < a.min_shared)
                                    old[r] = atomicOr(&sp.plane2[x >> (32 - kPlane2Bits)], 1u << ((x >> 15) & 31u));
                            }
#pragma unroll
                            for (int r = 0; r < kR; ++r)
                                if (!((old[r] >> ((hash_u32(pid[r]) >> 15) & 31u)) & 1u)) in &= ~(1u << r);
                        }
                        while (__any_sync(0xffffffffu, in != 0u)) {        // few are left: one a lane and step
                            uint32_t p = 0;
#pragma unroll
                            for (int r = kR - 1; r >= 0; --r)
                                if ((in >> r) & 1u) p = pid[r];
                            if (in) add_repeat(sh, sp, p - pb);
                            in &= in - 1u;
                        }
                        __syncwarp();
                        qn = 0;
                    }
                    if (total) {
                        uint32_t to = (uint32_t)__cvta_generic_to_shared(wq) + 4u * (qn + n1);
#pragma unroll
                        for (int i = 0; i < 4 * kG; ++i) {
                            const uint4& v = ev[i / 4];
                            to = put_shared(to, i % 4 == 0 ? v.x : i % 4 == 1 ? v.y : i % 4 == 2 ? v.z : v.w,
                                            take & (1u << (4 * kG - 1 - i)));
                        }
                        qn += total;
                    }
                    rep &= ~take;
                } while (__any_sync(0xffffffffu, rep != 0u));
                if (last) break;
            }
            if (!more && tid == 0) set_unit(sh.t_next);
            uint2 excl = make_uint2(0u, 0u);
            if (more) excl = scan_1(r1, r2);
            // (the or makes every warp's mark before the barrier count)
            if (__syncthreads_or(sh.over || sh.nkeys > kQueue)) {
                // too many repeats: nothing of this super-chunk was used yet.
                // A single column is searched with one counter a peptide;
                // else half as many columns from here on.
                if (tid == 0) {
                    sh.over = 0;
                    sh.nkeys = 0u;
                }
                for (uint32_t i = tid; i < kSlots; i += THREADS) sp.tab[i] = 0u;
                for (uint32_t i = tid; i < kPlane2Words; i += THREADS) sp.plane2[i] = 0u;
                for (uint32_t i = tid; i < a.lay.plane_words; i += THREADS) plane[i] = 0u;
                __syncthreads();
                if (st.e - st.c == 1) {
                    save();
                    direct_column(a, x0, x1);
                    restore();
                    st.c = st.e;
                } else {
                    st.m = (st.e - st.c + 1) / 2;
                }
                if (st.c < col_end) start();
                continue;
            }
            if (more) scan_2(excl, r1, r2);    // (pass A is behind the barrier: the runs are free)
            // ---- the plane: its peptides of enough hot bits, and cleared
            if ((uint32_t)sh.nslices + 1u >= a.min_shared) {
                // peptides hit once (or never) may qualify through their hot bits
                save();
                scan_plane(a, pb, x0, x1, words);
                restore();
            } else {
                uint4* p4 = reinterpret_cast<uint4*>(plane);
                for (uint32_t i = tid; i < a.lay.plane_words / 4; i += THREADS) p4[i] = make_uint4(0u, 0u, 0u, 0u);
                if (st.deep) {
                    p4 = reinterpret_cast<uint4*>(sp.plane2);
                    for (uint32_t i = tid; i < kPlane2Words / 4; i += THREADS) p4[i] = make_uint4(0u, 0u, 0u, 0u);
                }
            }
            if (tid == 0) {   // (nothing is appended between here and the barrier)
                sh.no_room = sh.nkeys == 0u ? -1 : sh.nq + sh.nkeys > kQueue;
                sh.nkeys = 0u;
            }
            __syncthreads();
            // ---- select: the warp's share of the table (there is room for
            // all of it in the queue; nothing is appended before the drain)
            if (sh.no_room >= 0) {   // uniform: the table is not empty
                if (sh.no_room) {
                    save();
                    drain_queue(a);
                    restore();
                }
                const uint32_t nslices = (uint32_t)sh.nslices, pb2 = max(sh.unit[st.slot].y, st.c << kChunkShift) & ~127u;
                for (uint32_t s0 = (uint32_t)warp * 128u; s0 < kSlots; s0 += 4 * THREADS) {
                    uint4* const t4 = reinterpret_cast<uint4*>(sp.tab + s0) + lane;   // 4 slots a lane
                    const uint4 v4 = *t4;
                    if ((v4.x | v4.y | v4.z | v4.w) == 0u) continue;
                    *t4 = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint32_t v = i == 0 ? v4.x : i == 1 ? v4.y : i == 2 ? v4.z : v4.w;
                        const uint32_t ord = (v & ((1u << (32 - kOffBits)) - 1u)) + 1u + st.deep;   // (at most)
                        if (v && ord + nslices >= a.min_shared)
                            push(a, sh, sp, pb2 + (v >> (32 - kOffBits)), ord < a.min_shared ? a.min_shared - ord : 0u);
                    }
                }
            }
            st.c = st.e;
            st.e = min(st.e + st.m, col_end);
            take_unit();
            // (a warp's next repeats may go into another's share of the table)
            if (st.c < col_end && sh.no_room >= 0) __syncthreads();
        }
        if (tid == 0 && !st.taken)   // an empty segment (a window split into more units than it has peptides)
            set_unit((uint64_t)gridDim.x + atomicAdd(a.work, 1ull));
        __syncthreads();
        if (sh.nq) {   // uniform: the appends are behind the barrier
            save();
            drain_queue(a);
            restore();
        }
        unit_out<THREADS>(a, sh, sp.tkey, sp.tpid, sp.tpk, sh.unit[st.slot].x, sh.unit[st.slot].w);
        for (uint32_t i = tid; i < kHeads / 2; i += THREADS) sp.head[i] = 0u;
    }
}
