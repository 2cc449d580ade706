// The search of units in which many peptides qualify, included by
// search_kernels.cuh behind search_kernel.cuh: with min_shared 1 (every hit is
// scored), with min_shared 2, and on grids so coarse that many of a column's
// peptides share several bins with the spectrum.  search_kernel.cuh's form
// reads the forward list of every peptide it scores, a dozen sectors of memory
// and some hundred instructions; that pays while dozens of a unit's peptides
// qualify.  Here every entry of every retained peak in a column (kChunk
// peptides) is added to its peptide's counter (nb | ny | S) in shared memory.
// A counter that reaches min_shared is queued, and what the queue holds at the
// column's end is scored as it stands, a lane a peptide.  When more qualify than
// the queue takes, the rest of the unit looks at every counter instead.  The
// planner decides by a spectrum's expected hits a peptide (Cost) and puts these
// units behind the others.
//
// A column's counters are 64 KB: three CTAs an SM of 256 threads (of 384 threads
// the same; two of 512: 2.4 against 2.1 ms).  Where there are units of both
// kinds, its CTAs start as search_kernel's leave their SMs, so that one's last
// units run beside the other's first (500 spectra at min_shared 2: 2.1 -> 1.8 ms).
// What bounds it: the latencies of a column's passes, about 3 us where few
// entries lie in it, and the issue of both passes.  13.0 M peptides, 500 spectra
// of 100 peaks at +-500 Da, scored from an entry log / from forward lists / here:
// min_shared 1 7.5 / 53 / 4.4 ms, 2 2.2 / 6.4 / 1.8 ms; 50 spectra on a grid of
// 1 Da, min_shared 4, 2.3 / 12.8 / 0.9 ms.

// Expected hits a peptide from which on a spectrum's units are counted.
// min_shared 2, from 0.02 / 0.04 / 0.05 / 0.08 on: 500 spectra of 100 peaks 1.89 /
// 1.79 / 1.74 / 2.20 ms, of 20 peaks 0.52 / 0.55 / 0.76 / 0.79, 2,000 of 10 peaks
// 0.94 / 0.79 / 0.75 / 0.73.  min_shared 3, from 0.13 / 0.17 / 0.21 / 0.27 on: 300 of
// 275 peaks on a grid of 0.02 Da 1.57 / 1.32 / 1.50 / 1.48, 200 of 100 peaks on 0.1 Da
// 1.31 / 1.49 / 1.59 / 1.79.  Above, from 0.20 / 0.25 / 0.30 on, 200 of 100 peaks: 0.1 Da
// and min_shared 6 0.87 / 0.64 / 0.64, 0.2 Da and 4 1.44 / 1.44 / 1.67, 6 1.26 / 1.26 /
// 2.25.
constexpr float kCountShare2 = 0.04f;
constexpr float kCountShare3 = 0.19f;
constexpr float kCountShare = 0.25f;
// With min_shared 3 and above it, only indexes whose average spectrum has this
// many are looked at (count_from): the call is spared a launch for the others.
constexpr float kCountGrid3 = 0.09f;
constexpr float kCountGrid = 0.18f;
constexpr uint32_t kLook = 32;             // counters a lane looks at together

struct CountLayout {
    uint32_t runs, subs, base, row, iq, queue, tkey, tpid, tpk, shared, end;   // in 32-bit words; the counters come first
};

struct CountArgs {
    const uint32_t* qbin;
    const uint32_t* qiq;
    const uint32_t* qn;
    uint32_t stride;            // qbin / qiq words per spectrum
    const uint4* unit;          // the units in the order they are taken
    const unsigned long long* first;   // the first of this kernel's
    const uint64_t* n_units;    // the number of all
    const BinInfo* bins;
    const uint32_t* entry;
    const uint32_t* skip;
    uint32_t skip_stride;
    const int64_t* lf;
    const int64_t* ls;
    uint32_t s_max;
    uint32_t min_shared;
    uint32_t k;
    UnitTop* utop;
    uint32_t* hist;
    uint32_t* nscored;
    unsigned long long* work;   // unit counter
    CountLayout lay;
};

struct CountShared {
    uint32_t hist[kHistBins];
    int64_t lf[kMaxLen + 1];
    uint32_t wsum[kMaxWarps], wruns[kMaxWarps];
    int wn[kMaxWarps];                // length of each warp's top-k list
    uint4 unit;                       // spectrum, segment, unit number
    int have, n;                      // there is one; its peaks
    uint32_t nq;                      // peptides of the column that reached min_shared
    uint32_t per, total;              // pieces of an octet's share, and of all
};

constexpr int kCountThreads = 256;
constexpr int kCountCtas = 3;          // an SM at most
constexpr uint32_t kCountEach = 4;     // peptides of the queue a thread
constexpr uint32_t kCountQueue = kCountEach * kCountThreads;

template <int PPT>
__global__ void __launch_bounds__(kCountThreads, kCountCtas) count_kernel(const __grid_constant__ CountArgs a) {
    constexpr int THREADS = kCountThreads, nwarps = THREADS / 32;
    constexpr uint32_t nsub = THREADS / kSub;
    constexpr int kG = 4;               // pieces in flight a thread
    uint32_t* const cnt = search_smem();
    CountShared& sh = *reinterpret_cast<CountShared*>(cnt + a.lay.shared);
    uint4* const runs = reinterpret_cast<uint4*>(cnt + a.lay.runs);    // a column's: first group, groups, the first
                                                                       // piece's start (as in SearchParts), intensity
    uint2* const subs = reinterpret_cast<uint2*>(cnt + a.lay.subs);
    uint32_t* const pbase = cnt + a.lay.base;
    uint32_t* const prow = cnt + a.lay.row;
    uint32_t* const piq = cnt + a.lay.iq;
    int64_t* const tkey = reinterpret_cast<int64_t*>(cnt + a.lay.tkey);
    uint16_t* const queue = reinterpret_cast<uint16_t*>(cnt + a.lay.queue);   // [kCountQueue] counters
    uint32_t* const tpid = cnt + a.lay.tpid;
    uint32_t* const tpk = cnt + a.lay.tpk;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (uint32_t i = tid; i < kChunk; i += THREADS) cnt[i] = 0u;
    for (int i = tid; i < (int)kHistBins; i += THREADS) sh.hist[i] = 0;
    for (int i = tid; i <= (int)kMaxLen; i += THREADS) sh.lf[i] = a.lf[i];
    auto set_unit = [&](uint64_t t) {
        t += *a.first;
        sh.have = t < *a.n_units;
        if (sh.have) sh.unit = __ldg(a.unit + t);
        sh.n = 0;
        sh.nq = 0;
    };
    if (tid == 0) set_unit(blockIdx.x);   // the first by block index, then the counter's
    for (;;) {
        __syncthreads();
        if (!sh.have) break;
        const uint4 u = sh.unit;
        uint64_t t_next = 0;
        if (tid == 0) t_next = (uint64_t)gridDim.x + atomicAdd(a.work, 1ull);
        if (tid < nwarps) sh.wn[tid] = 0;
        {
            const uint32_t np = a.qn[u.x];
            for (uint32_t t = tid; t < np; t += THREADS) {
                const BinInfo bi = a.bins[a.qbin[(uint64_t)u.x * a.stride + t]];
                if (bi.row >= 0) {
                    const int s = atomicAdd(&sh.n, 1);
                    pbase[s] = bi.group;
                    prow[s] = (uint32_t)bi.row;
                    piq[s] = a.qiq[(uint64_t)u.x * a.stride + t];
                }
            }
        }
        __syncthreads();
        // a thread owns the peaks tid * ppt .. + ppt - 1
        const int n = sh.n, ppt = (n + THREADS - 1) / THREADS;
        const uint32_t c0 = u.y >> kChunkShift, col_end = ((u.z - 1u) >> kChunkShift) + 1u;
        uint32_t ra[PPT], rb[PPT];          // the next column's runs
        auto skip_at = [&](uint32_t (&r)[PPT], uint32_t col) {
#pragma unroll
            for (int i = 0; i < PPT; ++i) {
                const int t = tid * ppt + i;
                r[i] = 0;
                if (i < ppt && t < n)
                    r[i] = __ldg(a.skip + (uint64_t)prow[t] * a.skip_stride + min(col, a.skip_stride - 1u));
            }
        };
        // prefix of their pieces and of the non-empty ones over the block, in two halves around a barrier
        uint2 excl;
        auto scan_1 = [&]() {
            uint32_t sum = 0, some = 0;
#pragma unroll
            for (int i = 0; i < PPT; ++i) {
                const int t = tid * ppt + i;
                if (i < ppt && t < n && ra[i] != rb[i]) {
                    sum += Run(pbase[t], ra[i], rb[i]).pieces();
                    ++some;
                }
            }
            uint2 incl = make_uint2(sum, some);
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
            excl = make_uint2(incl.x - sum, incl.y - some);
        };
        auto scan_2 = [&](uint32_t col) {   // the runs of column col, and the ends of the one behind it
            uint32_t total = 0, nruns = 0;
#pragma unroll
            for (int w = 0; w < nwarps; ++w) {
                const uint32_t p = sh.wsum[w], r = sh.wruns[w];
                if (w < warp) {
                    excl.x += p;
                    excl.y += r;
                }
                total += p;
                nruns += r;
            }
            const uint32_t per = (total + nsub - 1u) / nsub;
#pragma unroll
            for (int i = 0; i < PPT; ++i) {
                const int t = tid * ppt + i;
                if (i < ppt && t < n && ra[i] != rb[i]) {
                    const Run r(pbase[t], ra[i], rb[i]);
                    const uint32_t len = r.pieces();
                    prefetch_l2(reinterpret_cast<const uint4*>(a.entry) + r.start);
                    if (len > 1u) prefetch_l2(reinterpret_cast<const uint4*>(a.entry) + r.start + r.len - 1u);
                    runs[excl.y] = make_uint4(r.start, r.len, 0u - r.start % kSub, piq[t]);
                    for (uint32_t s = (excl.x + per - 1u) / per; s * per < excl.x + len; ++s)   // the octets that start here
                        subs[s] = make_uint2(excl.y, s * per - excl.x);
                    excl.x += len;
                    ++excl.y;
                }
                ra[i] = rb[i];
            }
            if (tid == 0) {
                runs[nruns] = make_uint4(0u, kNoEnd, 0u, 0u);
                sh.per = per;
                sh.total = total;
            }
            skip_at(rb, col + 2u);
        };
        skip_at(ra, c0);
        skip_at(rb, c0 + 1u);
        scan_1();
        __syncthreads();
        scan_2(c0);
        __syncthreads();
        bool queued = true;       // the counters that reach min_shared are queued as they do
        for (uint32_t c = c0; c < col_end; ++c) {
            const uint32_t x0 = max(u.y, c << kChunkShift);
            const uint32_t span = (uint32_t)min((uint64_t)u.z, (uint64_t)(c + 1u) << kChunkShift) - x0;
            const bool next = c + 1u < col_end;
            // ---- count: kSub lanes take a contiguous share of the runs' pieces
            {
                const uint32_t per = sh.per, oct = (uint32_t)tid / kSub, sl = (uint32_t)tid % kSub;
                const uint32_t mine = oct * per < sh.total ? min(per, sh.total - oct * per) : 0u;
                const uint4* run = runs;
                uint4 cur = make_uint4(0u, kNoEnd, 0u, 0u);
                if (mine) {
                    const uint2 at = subs[oct];
                    run += at.x;
                    cur = *run;
                    cur.z += at.y * kSub;
                }
                for (uint32_t done = 0; done < mine; done += (uint32_t)kG) {
                    uint4 ev[kG];
                    uint32_t iq[kG];
#pragma unroll
                    for (int j = 0; j < kG; ++j) {
                        if ((int)cur.z >= (int)cur.y) cur = *++run;
                        iq[j] = cur.w;
                        ev[j] = load_group(a.entry, cur.x + cur.z + sl, done + (uint32_t)j < mine && cur.z + sl < cur.y);
                        cur.z += kSub;
                    }
                    uint32_t reach = 0;      // bit 4 j + i: entry i of piece j brought its counter to min_shared
#pragma unroll
                    for (int j = 0; j < kG; ++j) {
                        if (ev[j].x == 0xffffffffu) continue;      // (a group inside a run starts with a real entry)
                        const uint32_t en[4] = {ev[j].x, ev[j].y, ev[j].z, ev[j].w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const uint32_t o = (en[i] >> 1) - x0;  // (a pad is past every span)
                            if (o >= span) continue;
                            const uint32_t add = iq[j] + (en[i] & 1u ? 1u << kNyShift : 1u << kNbShift);
                            if (!queued) atomicAdd(cnt + o, add);
                            else if (hits_of(atomicAdd(cnt + o, add)) + 1u == a.min_shared) reach |= 1u << (4 * j + i);
                        }
                    }
                    if (reach) {
                        uint32_t at = atomicAdd(&sh.nq, (uint32_t)__popc(reach));
#pragma unroll
                        for (int j = 0; j < kG; ++j) {
                            const uint32_t en[4] = {ev[j].x, ev[j].y, ev[j].z, ev[j].w};
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                if (reach & (1u << (4 * j + i))) {
                                    if (at < kCountQueue) queue[at] = (uint16_t)((en[i] >> 1) - x0);
                                    ++at;
                                }
                        }
                    }
                }
            }
            if (next) scan_1();
            __syncthreads();
            if (queued) {
                const uint32_t nq = sh.nq;
                uint32_t o[kCountEach], w[kCountEach];
#pragma unroll
                for (uint32_t j = 0; j < kCountEach; ++j) {
                    const uint32_t i = (uint32_t)tid + j * THREADS;
                    o[j] = i < nq && nq <= kCountQueue ? queue[i] : 0u;
                    w[j] = i < nq ? cnt[o[j]] : 0u;
                }
                __syncthreads();
                if (tid == 0) sh.nq = 0;
                queued = nq <= kCountQueue;          // (else the rest of the unit by looking)
                if (queued) {
                    if (next) scan_2(c + 1u);
                    for (uint32_t i = (uint32_t)tid; 4u * i < span; i += THREADS)
                        reinterpret_cast<uint4*>(cnt)[i] = make_uint4(0u, 0u, 0u, 0u);
                    int64_t K[kCountEach];
#pragma unroll
                    for (uint32_t j = 0; j < kCountEach; ++j)
                        K[j] = (uint32_t)tid + j * THREADS < nq ? score_key(a, sh, w[j]) : INT64_MIN;
#pragma unroll
                    for (uint32_t j = 0; j < kCountEach; ++j)
                        if ((uint32_t)(tid & ~31) + j * THREADS < nq)   // warp-uniform
                            rank_lanes(sh, (int)a.k, tkey, tpid, tpk, (uint32_t)tid + j * THREADS < nq, x0 + o[j], w[j], K[j]);
                    __syncthreads();
                    continue;
                }
            }
            if (next) scan_2(c + 1u);       // (the count is behind the barrier: the runs are free)
            // ---- look at every counter, and clear it
            for (uint32_t b0 = (uint32_t)warp * 32u * kLook; b0 < span; b0 += THREADS * kLook) {
                uint4* const v4 = reinterpret_cast<uint4*>(cnt + b0) + lane;
                uint32_t look = 0;                 // bit 4 j + i: word i of the lane's vector j qualifies
#pragma unroll
                for (uint32_t j = 0; j < kLook / 4; ++j) {
                    const uint4 v = v4[32 * j];
                    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (uint32_t i = 0; i < 4; ++i) look |= hits_of(w[i]) >= a.min_shared ? 1u << (4 * j + i) : 0u;
                }
                // the qualifying words dealt to the lanes in turn, two a lane
                // and step, whose reads of the score table are in flight together
                const uint32_t have = (uint32_t)__popc(look);
                uint32_t incl = have;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += x;
                }
                const uint32_t all = __shfl_sync(0xffffffffu, incl, 31);
                for (uint32_t r0 = 0; r0 < all; r0 += 64u) {
                    uint32_t w[2], o[2];
                    int64_t K[2];
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const uint32_t r = r0 + 32u * (uint32_t)j + (uint32_t)lane;
                        uint32_t from = 0;         // the lane that has the r-th: as many end at or before it
#pragma unroll
                        for (uint32_t x = 16; x; x >>= 1)
                            if (__shfl_sync(0xffffffffu, incl, (int)(from + x - 1u)) <= r) from += x;
                        uint32_t m = __shfl_sync(0xffffffffu, look, (int)from);
                        uint32_t left = r - __shfl_sync(0xffffffffu, incl - have, (int)from);
                        uint32_t i = 0;            // the place of its bit, number left of the lane's
#pragma unroll
                        for (uint32_t x = 16; x; x >>= 1) {
                            const uint32_t below = (uint32_t)__popc(m & ((1u << x) - 1u));
                            if (below <= left) {
                                left -= below;
                                m >>= x;
                                i += x;
                            }
                        }
                        o[j] = b0 + 128u * (i >> 2) + 4u * from + (i & 3u);
                        w[j] = r < all ? cnt[o[j]] : 0u;
                        K[j] = r < all ? score_key(a, sh, w[j]) : INT64_MIN;
                    }
#pragma unroll
                    for (int j = 0; j < 2; ++j)
                        if (j == 0 || r0 + 32u < all)
                            rank_lanes(sh, (int)a.k, tkey, tpid, tpk, r0 + 32u * (uint32_t)j + (uint32_t)lane < all,
                                       x0 + o[j], w[j], K[j]);
                }
#pragma unroll
                for (uint32_t j = 0; j < kLook / 4; ++j) v4[32 * j] = make_uint4(0u, 0u, 0u, 0u);
            }
            __syncthreads();
        }
        unit_out<THREADS>(a, sh, tkey, tpid, tpk, u.x, u.w);
        if (tid == 0) set_unit(t_next);
    }
    // the search that this kernel may have started beside has ended before this one does
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
