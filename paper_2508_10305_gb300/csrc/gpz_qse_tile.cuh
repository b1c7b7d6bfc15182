// gpz_qse_tile.cuh -- the per-block body of the shared-memory tile
// compression kernel (Sections 4.1-4.3), used by the single-array kernel
// (gpz_qse_tile.cu, which describes the design), the interleaved-record
// kernel (gpz_aos.cu) and the batched kernel (gpz_batch_tile.cuh).  Idx
// gives the block within its array (b()) and its entry for the general list
// (id()).
#pragma once

#include <type_traits>

#include "gpz_qse_block.cuh"
#include "gpz_sort.cuh"

namespace gpz {

// The input tile, which the encoded block's staging words later overlay: an
// encoding is kept only when it is shorter than the raw block's 1 + F n_b
// words, so it fits the tile.  Its layouts: rows of 1024 values, one per
// field (16-byte aligned fields); the same with four words more, a row
// starting with the 16-byte unit that holds the block's first value, so that
// the values lie as they do in memory, 0 to 3 words into the row (fields of
// any alignment); the block's interleaved records as they are in memory.
// The second layout is a kernel of its own: with its shifts in the code, the
// aligned case took 0.405 instead of 0.391 ms on a 2^26 x 6 snapshot.
enum : int { kTileAligned, kTileUnaligned, kTileRecords };
__host__ __device__ constexpr uint32_t tile_row(int layout) { return layout == kTileUnaligned ? kBlock + 4u : kBlock; }
__host__ __device__ constexpr uint32_t tile_region_bytes(int F, int layout) {
    return (uint32_t)F * tile_row(layout) * 4u;
}

// Dynamic shared memory: the tile and the sort's histograms.  With five and
// more aligned fields, where shared memory sets the residency, the
// histograms take the place of the tile's first row once a warp has quantised
// its particles (a warp's row of counts is as long as its part of the row),
// and the staging words start behind them: records are at most 128 bits, so
// an encoded block fits the other rows.
__host__ __device__ constexpr bool tile_overlays_hist(int F, int layout) { return layout == kTileAligned && F >= 5; }
constexpr uint32_t kTileMaxEncWords = 1u + 8u + 2u + 144u + 176u + 32u * kFastRecordBits;
static_assert(4u * kBlock >= 1u + 5u + 2u + 144u + 176u + 32u * 115u && 5u * kBlock >= kTileMaxEncWords,
              "five fields (23 bits each) and more: the encoded block fits behind the first row");
static_assert(kSortHistBytes == kBlock * 4u, "the histograms take one row");
__host__ __device__ constexpr uint32_t tile_smem_bytes(int F, int layout) {
    return tile_region_bytes(F, layout) + (tile_overlays_hist(F, layout) ? 0u : kSortHistBytes);
}

// Resident CTAs per SM the kernels are compiled for: what shared memory
// allows (227 KB, 1 KB reserved per CTA, about 0.6 KB of static memory), at
// most nine (56 registers per thread), eight from five fields on (64
// registers): the counts that measured best, although from three fields on
// 140 to 600 bytes of a thread's values then live in local memory (see
// gpz_qse_tile.cu for fewer and more CTAs).
constexpr int kTileMaxCtas = 9;
__host__ __device__ constexpr int tile_ctas(int F, int layout) {
    const int by_smem = (int)((227u * 1024u) / (tile_smem_bytes(F, layout) + 1024u + 640u));
    const int most = F >= 5 ? kTileMaxCtas - 1 : kTileMaxCtas;
    return by_smem < most ? by_smem : most;
}

namespace {

// One field's constants for the block, derived once by lane f of warp 0.
struct alignas(16) TileField {
    float mn, inv;             // block minimum, reciprocal step
    uint32_t wf, cmask;        // bits in the record and their mask
    uint32_t rot, kmask;       // segId: the code rotated left by rot, under kmask (its place in the key)
    float s, ebchk;            // step, verification threshold
    uint32_t bits;             // code width
    uint32_t row;              // tile word of value 0 (unaligned layout)
    uint32_t pad[2];
};

struct alignas(16) TileShared : SortShared {
    uint4 blk;                             // flags, record width, key bits
    uint64_t bar;                          // mbarrier of the tile's bulk copies
    uint32_t fallback;                     // kFb... bits
    uint2 ext[kMaxFields];                 // the block's extremes (order keys; (0, 0): a non-finite value)
    TileField fc[kMaxFields];
};

constexpr uint32_t kFbGeneral = 1u;    // a fallback candidate that could change its field's width: general path
constexpr uint32_t kFbRaw = 2u;        // a value without a candidate in the bound: the block is stored raw
constexpr uint32_t kTfNonFinite = 1u;  // a non-finite value: stored raw
constexpr uint32_t kTfBig = 2u;        // a code reaches 2^23: general path
constexpr uint32_t kTfVerify = 4u;     // some field's first candidates need their check

// Warp 0, every lane: the fields' constants (lane f) from the block's
// extremes e, the step constants p and the tile word of its value 0: q0 = floor(fma(x - min, 1/s, 1/2)) is
// monotone in x, so when every value keeps its first candidate the largest
// code is q0 of the block maximum.
template <int F>
__device__ __forceinline__ void tile_constants(const uint2 e, const FieldParams& p, int G, uint32_t row, TileShared& S) {
    constexpr int P = F < 3 ? F : 3;
    const int lane = threadIdx.x;
    const bool fl = lane < F;
    uint32_t bits = 0u;
    bool big = false, exact = true;
    float mn = 0.0f;
    const bool nonfinite = fl && e.x == 0u;
    if (fl && e.x != 0u) {
        block_field_width(e.x, e.y, p, bits, big, exact);
        const float m0 = from_order_key(e.x);
        mn = m0 == 0.0f ? 0.0f : m0;  // a zero minimum is stored as +0
    }
    const uint32_t g = lane < P ? min((uint32_t)G, bits) : 0u;
    const uint32_t wf = bits - g;  // a position axis' segOffset bits, an extra field's whole code
    const uint32_t g1 = __shfl_sync(0xffffffffu, g, 1), g2 = __shfl_sync(0xffffffffu, g, 2);
    const uint32_t ks = lane == 0 ? g1 + g2 : (lane == 1 ? g2 : 0u);  // the segId bits of the axes after this one
    const uint32_t W = __reduce_add_sync(0xffffffffu, wf), keybits = __reduce_add_sync(0xffffffffu, g);
    const uint32_t flags = (__any_sync(0xffffffffu, nonfinite) ? kTfNonFinite : 0u) |
                           (__any_sync(0xffffffffu, big) ? kTfBig : 0u) |
                           (__any_sync(0xffffffffu, !exact) ? kTfVerify : 0u);
    if (fl) {
        TileField& c = S.fc[lane];
        c.mn = mn;
        c.inv = p.inv;
        c.wf = wf;
        c.row = row;
        c.cmask = (1u << (wf & 31u)) - 1u;
        c.rot = (ks - wf) & 31u;
        c.kmask = ((1u << g) - 1u) << ks;
        c.s = p.s;
        c.ebchk = p.ebchk;
        c.bits = bits;
    }
    if (lane == 0) S.blk = make_uint4(flags, W, keybits, 0u);
}

// The block stored raw, from its tile: a second read of the input through L2
// (write_raw) by 128 threads made a 2^24 x 6 snapshot with a NaN in every block
// 0.378 -> 0.413 ms; 0.345 this way.
template <int F, int LAY>
__device__ __forceinline__ void tile_write_raw(const QseArgs& a, const float* tile, const TileShared& S, uint32_t b,
                                               int n_b) {
    const int t = threadIdx.x;
    uint32_t* out = a.temp + (size_t)b * a.slot_words;
    if (t == 0) out[0] = 1u;
#pragma unroll
    for (int f = 0; f < F; ++f) {
        const float* row = tile + (LAY == kTileUnaligned ? (int)S.fc[f].row : f * kBlock);
        for (int i = t; i < n_b; i += kTileThreads)
            out[1 + f * n_b + i] = __float_as_uint(LAY == kTileRecords ? tile[i * F + f] : row[i]);
    }
    raw_done<F, kTileThreads>(a, b, n_b, t);
}

// Steps 3 to 5 for a block whose records are at most 32 NR bits wide (NR = 2
// or 4): the common case keeps two registers per record instead of four.
template <int F, bool FULL, int LAY, int NR, class Idx>
__device__ __forceinline__ void tile_encode(const QseArgs& a, uint8_t* dsm, TileShared& S, Idx idx, int n_b,
                                            uint32_t flags, uint32_t W) {
    constexpr int P = F < 3 ? F : 3;
    constexpr int R = kTileRounds;
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    constexpr bool OVER = tile_overlays_hist(F, LAY);
    uint32_t* stage = reinterpret_cast<uint32_t*>(dsm + (OVER ? kSortHistBytes : 0u));
    uint16_t* hist = reinterpret_cast<uint16_t*>(dsm + (OVER ? 0u : tile_region_bytes(F, LAY))); 
    uint32_t* order = reinterpret_cast<uint32_t*>(hist);                            // [1024] the sorted order, later
    const int i0 = 32 * R * w + lane;  // this thread's particles: i0 + 32 r
    auto valid = [&](int r) { return FULL || i0 + 32 * r < n_b; };

    // ---- 3. quantise from the tile, key and record in one pass.  A code is
    // the low bits of u = 2^23 + q: the rotation puts its segId at the key
    // place (the exponent bits of u fall outside kmask), the mask takes its
    // segOffset.
    uint32_t key[R], rw[R][NR];
    // MODE 0: first candidates, known to pass.  1: first candidates, checked;
    // true when one fails.  2: every candidate; S.fallback takes what they call for.
    auto quantise = [&](auto mode) {
        constexpr int MODE = decltype(mode)::value;
        const float* tile = reinterpret_cast<const float*>(dsm);
        bool pend = false;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            key[r] = 0u;
#pragma unroll
            for (int k = 0; k < NR; ++k) rw[r][k] = 0u;
        }
        constexpr int UNROLL = MODE == 2 ? 1 : F;  // the rare pass stays a loop
#pragma unroll UNROLL
        for (int f = 0; f < F; ++f) {
            const uint4 c0 = reinterpret_cast<const uint4*>(&S.fc[f])[0];
            const uint4 c1 = reinterpret_cast<const uint4*>(&S.fc[f])[1];
            const float mn = __uint_as_float(c0.x), inv = __uint_as_float(c0.y);
            const float* row = tile + (LAY == kTileUnaligned ? (int)S.fc[f].row : f * kBlock) + i0;
            const uint32_t wf = c0.z, cmask = c0.w, rot = c1.x, kmask = c1.y;
            const float s = __uint_as_float(c1.z), ebchk = __uint_as_float(c1.w);
            // the smallest and the largest code of the field's width: a fallback
            // candidate below the one or above the other could change the width
            float half = 0.0f, top = 0.0f;
            if (MODE == 2) {
                const uint32_t bits = S.fc[f].bits;
                half = __uint2float_rn((1u << bits) >> 1);
                top = __uint2float_rn((1u << bits) - 1u);
            }
            auto value = [&](int r) { return LAY == kTileRecords ? tile[(i0 + 32 * r) * F + f] : row[32 * r]; };
            auto place = [&](int r, uint32_t ub) {
                if (MODE == 2 || f < P) key[r] |= __funnelshift_l(ub, ub, rot) & kmask;
                // append below the record so far (field 0 ends most significant)
#pragma unroll
                for (int k = NR - 1; k > 0; --k) rw[r][k] = __funnelshift_l(rw[r][k - 1], rw[r][k], wf);
                rw[r][0] = (rw[r][0] << wf) | (ub & cmask);
            };
            if (MODE == 2) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float x = value(r);
                    const float tt = __fmaf_rn(__fsub_rn(x, mn), inv, 0.5f);
                    const float u = __fadd_rd(tt, 8388608.0f);  // 2^23 + floor(t), t < 2^23 here
                    uint32_t ub = __float_as_uint(u);
                    const float q = __fsub_rn(u, 8388608.0f);
                    auto ok = [&](float c) { return fabsf(__fsub_rn(x, __fmaf_rn(c, s, mn))) <= ebchk; };
                    if (valid(r) && !ok(q)) {  // the next candidates, in the format's order
                        if (q > 0.0f && ok(__fsub_rn(q, 1.0f))) {
                            if (q == half) atomicOr(&S.fallback, kFbGeneral);
                            ub -= 1u;
                        } else if (ok(__fadd_rn(q, 1.0f))) {
                            if (q == top) atomicOr(&S.fallback, kFbGeneral);
                            ub += 1u;
                        } else {
                            atomicOr(&S.fallback, kFbRaw);
                        }
                    }
                    place(r, ub);
                }
            } else {  // the same, two values at a time
                const f32x2 mn2 = pack2(mn, mn), neg2 = pack2(-mn, -mn), inv2 = pack2(inv, inv), s2 = pack2(s, s);
#pragma unroll
                for (int r = 0; r < R; r += 2) {
                    const f32x2 x = pack2(value(r), value(r + 1));
                    const f32x2 tt = fma2_rn(add2_rn(x, neg2), inv2, pack2(0.5f, 0.5f));
                    const f32x2 u = add2_rd(tt, pack2(8388608.0f, 8388608.0f));
                    if (MODE == 1) {  // x - x^ as one rounding of x^ (-1) + x
                        const f32x2 xh = fma2_rn(add2_rn(u, pack2(-8388608.0f, -8388608.0f)), s2, mn2);
                        float d0, d1;
                        unpack2(fma2_rn(xh, pack2(-1.0f, -1.0f), x), d0, d1);
                        pend |= valid(r) && !(fabsf(d0) <= ebchk);
                        pend |= valid(r + 1) && !(fabsf(d1) <= ebchk);
                    }
                    float u0, u1;
                    unpack2(u, u0, u1);
                    place(r, __float_as_uint(u0));
                    place(r + 1, __float_as_uint(u1));
                }
            }
        }
        return pend;
    };
    if (!(flags & kTfVerify)) {
        quantise(std::integral_constant<int, 0>{});
    } else if (__any_sync(0xffffffffu, quantise(std::integral_constant<int, 1>{}))) {
        quantise(std::integral_constant<int, 2>{});  // rare: once more
        if (lane == 0 && a.fallback_count) atomicAdd(a.fallback_count, 1u);
    }

    if (OVER) {  // the warp's part of the first row becomes its counts
        __syncwarp();
        clear_hist_row(hist);
        __syncwarp();
    }
    // ---- 4. counting sort: warp-local ranks, round after round
    rank_keys(key, hist, valid, S);
    __syncthreads();  // C: every value quantised (the tile is dead) and ranked
    if (const uint32_t all = S.fallback) {
        if (t == 0) a.general_list[atomicAdd(a.general_count, 1u)] = idx.id() | (all & kFbRaw ? kRawBlock : 0u);
        return;
    }
    const uint32_t hdr = 1u + (uint32_t)F + (uint32_t)((F + 3) >> 2);
    const uint32_t rwords = ceil_words((uint32_t)n_b * W);
    {
        // the staging words, assembled by OR, overlay the tile: clear what
        // the block can need (deltas <= 512 x 9 bits, counts <= 512 x 11)
        const uint32_t need = min((hdr + 144u + 176u + rwords + 3u) >> 2,
                                  (tile_region_bytes(F, LAY) - (OVER ? kSortHistBytes : 0u)) / 16u);
        uint4* s4 = reinterpret_cast<uint4*>(stage);
        for (uint32_t k = t; k < need; k += kTileThreads) s4[k] = make_uint4(0u, 0u, 0u, 0u);
    }

    // ---- 4b. scan over (bin, warp): sorted positions and the run-length code
    const SortRuns runs = scan_bins(hist, S);

    // ---- encoded size; raw when not smaller (keeps the bound size a bound)
    const uint32_t U = runs.U, wd = bit_width(runs.maxdelta), wc = bit_width(runs.maxcnt);
    const uint32_t dwords = ceil_words(U * wd), cwords = ceil_words(U * wc);
    const uint32_t enc = hdr + dwords + cwords + rwords;
    const uint32_t b = idx.b();
    if (enc >= 1u + (uint32_t)F * (uint32_t)n_b) {
        write_raw<F, kTileThreads>(a, b, n_b, t);
        return;
    }

    // ---- 5. block header and the three arrays (Section 4.3), assembled in the
    // cleared staging words -- each thread ORs in the deltas and counts of its
    // bins and its records at their positions -- then one bulk copy to the
    // temporary slot
    if (t == 0) stage[0] = (U << 1) | (wd << 12) | (wc << 17);
    if (t >= 1 && t <= F) stage[t] = __float_as_uint(S.fc[t - 1].mn);
    if (t < ((F + 3) >> 2)) {
        uint32_t word = 0;
#pragma unroll
        for (int f = 0; f < F; ++f)
            if ((f >> 2) == t) word |= S.fc[f].bits << (8 * (f & 3));
        stage[1 + F + t] = word;
    }
    or_runs(stage, runs, hdr, wd, wc);
    {
        const uint32_t rbase = 32u * (hdr + dwords + cwords);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (!valid(r)) continue;
            const uint32_t dest = sorted_position(key[r], hist);
            if (W == 0u) continue;
            const uint32_t bp = rbase + dest * W, end = (bp & 31u) + W;
            uint32_t* at = stage + (bp >> 5);
            // the record is W bits, least significant word first, zero above W
            atomicOr(at, __funnelshift_l(0u, rw[r][0], bp));
#pragma unroll
            for (int k = 1; k <= NR; ++k)
                if (end > 32u * k)
                    atomicOr(at + k, __funnelshift_l(rw[r][k - 1], k < NR ? rw[r][k < NR ? k : 0] : 0u, bp));
        }
    }
    fence_proxy_async_shared();  // the staging words are read by a bulk copy (async proxy)
    __syncthreads();
    if (t == 0) bulk_s2g_start(a.temp + (size_t)b * a.slot_words, stage, ((enc + 3u) & ~3u) * 4u);
    if (!sorted_order(key, order, valid, i0, n_b, a.perm != nullptr, S) || Idx::kUnstable) {
        if (t == 0) a.general_list[atomicAdd(a.general_count, 1u)] = idx.id();  // not stable: the general kernel redoes it
    } else {
        if (t == 0) store_size(a.sizes, a.sums, a.sum_shift, b, enc);
        if (a.perm) {
            const uint64_t first = (uint64_t)b * kBlock;
            for (int j = t; j < n_b; j += kTileThreads) a.perm[first + j] = (uint32_t)first + (order[j] & 1023u);
        }
    }
    if (t == 0) bulk_s2g_wait();
}

}  // namespace

// kTileRecords: the input is interleaved records (a.interleaved), 16-byte
// aligned; value (f, i) lies at i * F + f of the tile.
template <int F, bool FULL, bool PRE, int LAY, class Idx>
__device__ __forceinline__ void qse_block_tile(const QseArgs& a, uint8_t* dsm, TileShared& S, Idx idx) {
    constexpr bool AOS = LAY == kTileRecords, UNAL = LAY == kTileUnaligned;
    constexpr uint32_t ROW = tile_row(LAY);
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    const uint32_t b = idx.b();  // the block within its array
    const uint64_t first = (uint64_t)b * kBlock;
    const int n_b = FULL ? kBlock : (int)(a.n - first);
    float* tile = reinterpret_cast<float*>(dsm);  // [F] rows of input (the block's records if AOS)

    // ---- 1. the tile: one bulk copy per field (lane f of warp 0; one copy of
    // the whole run of records if AOS), of every 16-byte unit that holds a
    // value of the block and lies inside the array; the values of the array's
    // first and last unit, where those are cut, by plain loads
    // words in field f's row before value 0
    auto shift = [&](int f) { return !UNAL ? 0u : (uint32_t)(reinterpret_cast<uintptr_t>(a.fields[f]) >> 2) & 3u; };
    // first unit and past the last, counted from the row's start (values of
    // the row: words s .. s + n_b - 1; of the array: words from s - first)
    auto units = [&](uint32_t s, uint32_t& lo, uint32_t& hi) {
        lo = UNAL && first == 0 && s ? 1u : 0u;
        hi = (uint32_t)n_b >> 2;
        if (!UNAL) return;
        const uint64_t left = a.n - first;  // the array's values from here on
        hi = min((s + (uint32_t)n_b + 3u) >> 2, (uint32_t)min((s + left) >> 2, (uint64_t)(ROW / 4u)));
        hi = max(hi, lo);
    };
    const uint32_t nrec = (uint32_t)(F * n_b) & ~3u;  // AOS: words of the records' whole units
    if (w == 0) {
        if (lane == 0) {
            mbar_init(&S.bar, AOS ? 1 : F);
            S.fallback = 0u;
            S.unsure = 0u;
        }
        __syncwarp();
        if (AOS) {
            if (lane == 0) {
                mbar_arrive_expect_tx(&S.bar, nrec * 4u);
                if (nrec) bulk_g2s(tile, a.fields[0] + first * F, nrec * 4u, &S.bar);
            }
        } else if (lane < F) {
            const uint32_t s = shift(lane);
            uint32_t lo, hi;
            units(s, lo, hi);
            mbar_arrive_expect_tx(&S.bar, (hi - lo) * 16u);
            if (hi > lo)
                bulk_g2s(tile + lane * ROW + 4u * lo, a.fields[lane] + first - s + 4u * lo, (hi - lo) * 16u, &S.bar);
        }
    }
    if (AOS) {
        if (!FULL && t < 4) {
            const uint32_t k = nrec + t;
            if (k < (uint32_t)(F * n_b)) tile[k] = __ldcs(a.fields[0] + first * F + k);
        }
    } else if ((UNAL || !FULL) && t < 8 * F) {  // up to three words at either end of the row
        const int f = t >> 3;
        const uint32_t s = shift(f), end = s + (uint32_t)n_b;
        uint32_t lo, hi;
        units(s, lo, hi);
        const uint32_t k = (t & 4) ? 4u * hi + (t & 3) : s + (t & 3);
        if (k >= s && k < end && ((t & 4) || k < 4u * lo)) tile[f * ROW + k] = __ldcs(a.fields[f] + first + (k - s));
    }
    if (!tile_overlays_hist(F, LAY)) clear_hist_row(reinterpret_cast<uint16_t*>(dsm + tile_region_bytes(F, LAY)));
    // the range pass's results; the tile above was complete before this call's
    // work began, or the launch is an ordinary one (launch_qse_tile's `early`)
    if (PRE) wait_for_previous_kernel();
    // ---- 2. the field constants from the block's extremes: those of the
    // range pass (loaded with the step constants while the tile is in
    // flight), or found in the tile, a warp per field
    if constexpr (!PRE) {
        __syncthreads();  // the mbarrier and the plainly loaded values
        if (!mbar_wait_bounded(&S.bar, 0, a.status)) return;
        for (int f = w; f < F; f += kTileWarps) {
            float lo = INFINITY, hi = -INFINITY;
            float p0 = 0.0f, p1 = 0.0f, p2 = 0.0f, p3 = 0.0f;  // become NaN if a value is NaN or infinite (x * 0)
            const uint32_t sh = shift(f);
            if (FULL && !AOS && sh == 0u) {
                const float4* v4 = reinterpret_cast<const float4*>(tile + f * ROW) + lane;
#pragma unroll
                for (int k = 0; k < kBlock / 128; ++k) {
                    const float4 v = v4[32 * k];
                    lo = fminf(lo, fminf(fminf(v.x, v.y), fminf(v.z, v.w)));
                    hi = fmaxf(hi, fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)));
                    p0 = __fmaf_rn(v.x, 0.0f, p0);
                    p1 = __fmaf_rn(v.y, 0.0f, p1);
                    p2 = __fmaf_rn(v.z, 0.0f, p2);
                    p3 = __fmaf_rn(v.w, 0.0f, p3);
                }
            } else {
#pragma unroll 8
                for (int i = lane; i < n_b; i += 32) {
                    const float v = AOS ? tile[i * F + f] : tile[f * ROW + sh + i];
                    lo = fminf(lo, v);
                    hi = fmaxf(hi, v);
                    p0 = __fmaf_rn(v, 0.0f, p0);
                }
            }
            const float probe = __fadd_rn(__fadd_rn(p0, p1), __fadd_rn(p2, p3));
            const uint32_t lk = __reduce_min_sync(0xffffffffu, lo == INFINITY ? 0xffffffffu : order_key(lo));
            const uint32_t hk = __reduce_max_sync(0xffffffffu, hi == -INFINITY ? 0u : order_key(hi));
            const bool nonfinite = __any_sync(0xffffffffu, probe != probe);
            if (lane == 0) S.ext[f] = nonfinite ? make_uint2(0u, 0u) : make_uint2(lk, hk);
        }
        __syncthreads();  // the extremes
    }
    if (w == 0) {
        uint2 e = make_uint2(0u, 0u);
        FieldParams p = {};
        if (lane < F) {
            e = PRE ? load_after_wait(a.bext + (size_t)b * F + lane) : S.ext[lane];
            p = a.d_params ? a.d_params[lane] : a.params[lane];
        }
        tile_constants<F>(e, p, a.G, lane < F ? (uint32_t)lane * ROW + shift(lane) : 0u, S);
    }
    __syncthreads();  // the constants (with a range pass also the mbarrier and the plainly loaded values)
    if (PRE && !mbar_wait_bounded(&S.bar, 0, a.status)) return;  // no copy may outlive the CTA
    const uint4 blk = S.blk;
    const uint32_t flags = blk.x, W = blk.y;
    if (flags & kTfNonFinite) {
        tile_write_raw<F, LAY>(a, tile, S, b, n_b);
        return;
    }
    if ((flags & kTfBig) || W > kFastRecordBits) {
        if (t == 0) a.general_list[atomicAdd(a.general_count, 1u)] = idx.id();
        return;
    }
    if (F <= 2 || W <= 64u)  // two fields of codes below 2^23 never need more
        tile_encode<F, FULL, LAY, 2>(a, dsm, S, idx, n_b, flags, W);
    else
        tile_encode<F, FULL, LAY, 4>(a, dsm, S, idx, n_b, flags, W);
}

}  // namespace gpz
