// gpz_sort.cuh -- the stable counting sort of one block's 1024 particles by
// segment id and the run-length code it yields (Sections 4.2 and 4.3), by a
// CTA of 128 threads: shared by the tile compression kernel
// (gpz_qse_tile.cuh) and the 64-bit one (gpz_wide_fast.cu).  Thread (warp w,
// lane l) owns particles 256 w + 32 r + l, r = 0..7.
#pragma once

#include "gpz_internal.cuh"

namespace gpz {

constexpr int kTileThreads = 128;              // one CTA per particle block
constexpr int kTileWarps = kTileThreads / 32;
constexpr int kTileRounds = kBlock / kTileThreads;  // particles per thread
constexpr int kTileBins = kMaxBins / kTileThreads;  // histogram bins per thread in the scan
static_assert(kTileBins == 4, "two words of 16-bit counts; four deltas or counts fit a 64-bit word");

// The per-warp histograms ([kTileWarps][512] 16-bit counts), whose space later
// takes the sorted order (one word per particle).
constexpr uint32_t kSortHistBytes = (uint32_t)kTileWarps * kMaxBins * 2u;
static_assert(kSortHistBytes >= kBlock * 4u, "the sorted order overlays the histograms");

// Ranking a warp's round of 32 keys: match takes time in proportion to the
// distinct keys (23 cycles of its SM-wide unit per round on scan data, 45 on
// uniform positions), a shared atomic in proportion to the most lanes on one
// bank; the first round's distinct keys decide for the others.  (Thresholds 14
// / 20 / 24 on a 2^26 x 6 snapshot: 0.388 / 0.393 / 0.405 ms.)
constexpr int kMatchMaxDistinct = 16;

struct alignas(16) SortShared {
    uint32_t tn[kTileWarps];               // per warp: particles | non-empty bins << 16
    uint32_t last[kTileWarps];             // ... its last non-empty bin
    uint32_t cmax[kTileWarps], dmax[kTileWarps];  // ... largest count and delta
    uint32_t unsure;                       // some warp's ranks need the check of the sorted order; zeroed
};

namespace {

// Clears the warp's row of counts.
__device__ __forceinline__ void clear_hist_row(uint16_t* hist) {
    uint4* h4 = reinterpret_cast<uint4*>(hist + (threadIdx.x >> 5) * kMaxBins) + (threadIdx.x & 31);
#pragma unroll
    for (int k = 0; k < kMaxBins / 256; ++k) h4[32 * k] = make_uint4(0u, 0u, 0u, 0u);
}

// Each particle's rank among the earlier particles of its warp with the same
// key (below 512), into bits 16 and up of key[r]; the warp's counts into its
// row of hist (zeroed before).  With shared atomics the old count that comes
// back is the rank; within one round the lanes of equal keys get distinct
// ranks in the order in which the hardware serves them, which
// sorted_order() checks (stability).
template <class Valid>
__device__ __forceinline__ void rank_keys(uint32_t (&key)[kTileRounds], uint16_t* hist, Valid valid, SortShared& S) {
    const int lane = threadIdx.x & 31;
    uint16_t* myhist = hist + (threadIdx.x >> 5) * kMaxBins;
    uint32_t peers = __match_any_sync(0xffffffffu, valid(0) ? key[0] : 0xffffffffu);
    if (valid(0)) myhist[key[0]] = (uint16_t)__popc(peers);  // every peer stores the same count
    const uint32_t rank0 = __popc(peers & lanemask_lt());
    const int distinct = __popc(__ballot_sync(0xffffffffu, valid(0) && rank0 == 0u));
    key[0] |= rank0 << 16;
    __syncwarp();
    if (distinct > kMatchMaxDistinct) {
        if (lane == 0) S.unsure = 1u;
        uint32_t* h32 = reinterpret_cast<uint32_t*>(myhist);  // two bins per word
#pragma unroll
        for (int r = 1; r < kTileRounds; ++r) {
            if (valid(r)) {
                const uint32_t sh = (key[r] & 1u) << 4;
                const uint32_t old = atomicAdd(h32 + (key[r] >> 1), 1u << sh);
                key[r] |= ((old >> sh) & 0xffffu) << 16;
            }
            __syncwarp();  // the next round's counts come after this one's
        }
    } else {
#pragma unroll
        for (int r = 1; r < kTileRounds; ++r) {
            peers = __match_any_sync(0xffffffffu, valid(r) ? key[r] : 0xffffffffu);
            uint32_t before = 0u;
            if (valid(r)) before = myhist[key[r]];
            __syncwarp();
            if (valid(r)) myhist[key[r]] = (uint16_t)(before + __popc(peers));
            __syncwarp();
            key[r] |= (before + __popc(peers & lanemask_lt())) << 16;
        }
    }
}

// The run-length code as a thread sees it: the counts of its bins
// kTileBins * t .. and what the bins before them add up to.
struct SortRuns {
    uint32_t c[kTileBins], tot;
    uint32_t excl;                   // particles | runs << 16 in the bins before
    uint32_t prev;                   // the last non-empty bin before (0 when none: a first id's delta is the id)
    uint32_t U, maxcnt, maxdelta;    // runs of the block, its largest count and delta
};

// The scan over (bin, warp), between barriers: after it hist holds every
// warp's first sorted position per bin.  Counts are 16-bit, two per word; none
// of their sums exceeds 1024.
__device__ __forceinline__ SortRuns scan_bins(uint16_t* hist, SortShared& S) {
    constexpr int NW = kTileWarps;
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    const uint32_t b0 = (uint32_t)kTileBins * t;
    SortRuns q;
    uint2 row[NW], sum = make_uint2(0u, 0u);
#pragma unroll
    for (int ww = 0; ww < NW; ++ww) {
        row[ww] = *reinterpret_cast<const uint2*>(hist + ww * kMaxBins + b0);
        sum.x += row[ww].x;
        sum.y += row[ww].y;
    }
    q.c[0] = sum.x & 0xffffu;
    q.c[1] = sum.x >> 16;
    q.c[2] = sum.y & 0xffffu;
    q.c[3] = sum.y >> 16;
    uint32_t nz = 0u, cm = 0u, mylast = 0u;
    q.tot = 0u;
#pragma unroll
    for (int k = 0; k < kTileBins; ++k) {
        q.tot += q.c[k];
        nz += q.c[k] ? 1u : 0u;
        cm = max(cm, q.c[k]);
        if (q.c[k]) mylast = b0 + k;
    }
    // one scan of both: the counts sum to at most 1024 and the non-empty bins
    // to at most 512, so they share a word
    const uint32_t mine = q.tot | (nz << 16), incl = warp_incl_sum(mine);
    cm = __reduce_max_sync(0xffffffffu, cm);
    // the last non-empty bin before this thread's, in its warp
    const uint32_t filled = __ballot_sync(0xffffffffu, q.tot != 0u), below = filled & lanemask_lt();
    q.prev = __shfl_sync(0xffffffffu, mylast, below ? 31 - __clz(below) : 0);
    if (!below) q.prev = 0u;
    const uint32_t wlast = __shfl_sync(0xffffffffu, mylast, filled ? 31 - __clz(filled) : 0);
    if (lane == 31) {
        S.tn[w] = incl;
        S.last[w] = wlast;
        S.cmax[w] = cm;
    }
    __syncthreads();
    uint32_t all = 0u;
    q.excl = incl - mine;
    q.maxcnt = 0u;
#pragma unroll
    for (int ww = 0; ww < NW; ++ww) {
        const uint32_t v = S.tn[ww];
        if (ww < w) {
            q.excl += v;
            q.prev = max(q.prev, S.last[ww]);
        }
        all += v;
        q.maxcnt = max(q.maxcnt, S.cmax[ww]);
    }
    q.U = all >> 16;
    uint32_t dm = 0u, start = q.excl & 0xffffu, pv = q.prev, first[kTileBins];
#pragma unroll
    for (int k = 0; k < kTileBins; ++k) {
        first[k] = start;
        start += q.c[k];
        if (q.c[k]) {
            dm = max(dm, b0 + k - pv);
            pv = b0 + k;
        }
    }
    // each warp's first position: the bin's plus the counts of the warps before it
    if (q.tot) {
        uint2 run = make_uint2(first[0] | (first[1] << 16), first[2] | (first[3] << 16));
#pragma unroll
        for (int ww = 0; ww < NW; ++ww) {
            *reinterpret_cast<uint2*>(hist + ww * kMaxBins + b0) = run;
            run.x += row[ww].x;
            run.y += row[ww].y;
        }
    }
    dm = __reduce_max_sync(0xffffffffu, dm);
    if (lane == 0) S.dmax[w] = dm;
    __syncthreads();
    q.maxdelta = 0u;
#pragma unroll
    for (int ww = 0; ww < NW; ++ww) q.maxdelta = max(q.maxdelta, S.dmax[ww]);
    return q;
}

// ORs the low n (<= 44) bits of v into the shared words at a bit position.
__device__ __forceinline__ void or_bits(uint32_t* words, uint32_t pos, unsigned long long v, uint32_t n) {
    const uint32_t lo = (uint32_t)v, hi = (uint32_t)(v >> 32), wi = pos >> 5, end = (pos & 31u) + n;
    if (n) atomicOr(words + wi, __funnelshift_l(0u, lo, pos));
    if (end > 32u) atomicOr(words + wi + 1, __funnelshift_l(lo, hi, pos));
    if (end > 64u) atomicOr(words + wi + 2, __funnelshift_l(hi, 0u, pos));
}

// The thread's deltas (wd bits each) and counts (wc bits), ORed into the
// cleared words of the block's two arrays, the first of which starts at word hdr.
__device__ __forceinline__ void or_runs(uint32_t* stage, const SortRuns& q, uint32_t hdr, uint32_t wd, uint32_t wc) {
    if (!q.tot) return;
    const uint32_t b0 = (uint32_t)kTileBins * threadIdx.x;
    unsigned long long dv = 0ull, cv = 0ull;
    uint32_t nd = 0u, nc = 0u, pv = q.prev;
#pragma unroll
    for (int k = 0; k < kTileBins; ++k) {
        if (q.c[k]) {
            dv |= (unsigned long long)(b0 + k - pv) << nd;
            cv |= (unsigned long long)q.c[k] << nc;
            nd += wd;
            nc += wc;
            pv = b0 + k;
        }
    }
    const uint32_t k0 = q.excl >> 16;  // index of the thread's first run
    or_bits(stage, 32u * hdr + k0 * wd, dv, nd);
    or_bits(stage, 32u * (hdr + ceil_words(q.U * wd)) + k0 * wc, cv, nc);
}

// A particle's sorted position; key becomes key | position << 16.
__device__ __forceinline__ uint32_t sorted_position(uint32_t& key, const uint16_t* hist) {
    const uint32_t k9 = key & 0xffffu;
    const uint32_t dest = hist[(threadIdx.x >> 5) * kMaxBins + k9] + (key >> 16);
    key = k9 | (dest << 16);
    return dest;
}

// Whether the sort was stable: (key, index) then increases strictly along the
// sorted positions.  Called after a barrier behind the last use of hist,
// which `order` overlays; with `want` order[j] & 1023 is afterwards the
// particle at sorted position j.
template <class Valid>
__device__ __forceinline__ bool sorted_order(const uint32_t (&key)[kTileRounds], uint32_t* order, Valid valid, int i0,
                                             int n_b, bool want, const SortShared& S) {
    const int t = threadIdx.x, lane = t & 31;
    const bool unsure = S.unsure != 0u;
    if (unsure || want) {
#pragma unroll
        for (int r = 0; r < kTileRounds; ++r)
            if (valid(r)) order[key[r] >> 16] = ((key[r] & 0xffffu) << 10) | (uint32_t)(i0 + 32 * r);
        __syncthreads();
    }
    if (!unsure) return true;
    bool bad = false;
#pragma unroll
    for (int k = 0; k < kBlock / (4 * kTileThreads); ++k) {
        const int j = 4 * (t + kTileThreads * k);
        const uint4 v = reinterpret_cast<const uint4*>(order)[t + kTileThreads * k];
        uint32_t next = __shfl_down_sync(0xffffffffu, v.x, 1);
        if (lane == 31) next = j + 4 < kBlock ? order[j + 4] : 0xffffffffu;
        bad |= j + 1 < n_b && v.x >= v.y;
        bad |= j + 2 < n_b && v.y >= v.z;
        bad |= j + 3 < n_b && v.z >= v.w;
        bad |= j + 4 < n_b && v.w >= next;
    }
    return !__syncthreads_or(bad);
}

}  // namespace

}  // namespace gpz
