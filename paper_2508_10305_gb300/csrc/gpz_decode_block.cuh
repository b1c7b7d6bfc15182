// gpz_decode_block.cuh -- the per-block body of GPZ decompression (Section
// 3.2: the reverse of compression, without sorting), shared by the
// single-stream kernel (gpz_decode.cu) and the batched kernel
// (gpz_batch_decode.cu).  See gpz_decode.cu for the design.
#pragma once

#include "gpz_internal.cuh"

namespace gpz {


constexpr int kDecWarps = kDecThreads / 32;
constexpr int kDecGroups = kBlock / (4 * kDecThreads);  // groups of four positions per thread: 4t.. of each 4 kDecThreads
constexpr int kDecRuns = kMaxBins / kDecThreads;        // runs per thread
static_assert(kDecRuns == 4, "a thread's four counts fit a 64-bit window");
// deltas (<= 512 x 9 bits) + counts (<= 512 x 11 bits) + records (<= 1024 x
// 128 bits, wider ones are read from the stream)
__host__ __device__ constexpr uint32_t dec_stage_words(int F) {
    return 144u + 176u + 32u * (31u * (uint32_t)F < 128u ? 31u * (uint32_t)F : 128u);
}
// Resident CTAs per SM: 40 registers per thread for up to three fields (whose
// staged words leave room for twelve CTAs), 48 for more.  8 / 10 / 12 CTAs:
// 10^8 x 3 scan points 0.383 / 0.368 / 0.357 ms, a 2^26 x 6 snapshot 0.340 /
// 0.317 / 0.352 ms.
__host__ __device__ constexpr int dec_ctas(int F) { return F <= 3 ? 12 : 10; }
// words read past the staged ones: a value or record is extracted from a
// window of words that may reach past its array; those bits are never used
constexpr uint32_t kDecStagePad = 8u;


__device__ __forceinline__ uint32_t mask_bits(uint32_t w) { return w >= 32u ? 0xffffffffu : ((1u << w) - 1u); }

// Values k .. k + 3 of a fixed-length array of width w (<= 11) held in shared
// memory (the words after the last value's may lie past the array: their
// bits are masked off).
__device__ __forceinline__ void extract4_s(const uint32_t* A, uint32_t k, uint32_t w, uint32_t (&v)[4]) {
    const uint32_t p = k * w;
    const uint32_t* a = A + (p >> 5);
    const uint32_t x0 = a[0], x1 = a[1], x2 = a[2], m = (1u << w) - 1u;
    uint32_t lo = __funnelshift_r(x0, x1, p), hi = __funnelshift_r(x1, x2, p);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        v[i] = lo & m;
        lo = __funnelshift_r(lo, hi, w);
        hi >>= w;
    }
}

// (float)q for q < 2^23 with two full-rate operations.
__device__ __forceinline__ float small_u2f(uint32_t q) {
    return __fsub_rn(__uint_as_float(q + 0x4B000000u), 8388608.0f);
}

// The doubles of four floats, on the integer pipe: fp64 conversions kept
// their pipe 78% busy (2^23 x 6 values: 0.116 -> 0.093 ms, with positions
// strided so that a warp's 8-byte stores are consecutive).  Normal magnitudes only move their fields; a group
// with any other value takes the second form.
__device__ __forceinline__ double widen_any(float v) {
    const uint32_t u = __float_as_uint(v), sign = u & 0x80000000u;
    uint32_t m = u & 0x7fffffffu;
    if (m >= 0x7f800000u)  // infinite, NaN
        return __hiloint2double((int)(sign | ((m >> 3) + 0x70000000u)), (int)(u << 29));
    if (m == 0u) return __hiloint2double((int)sign, 0);
    uint32_t bias = 0x38000000u;
    if (m < 0x00800000u) {  // subnormal: to a leading one at bit 23
        const int sh = __clz(m) - 8;
        m <<= sh;
        bias -= (uint32_t)sh << 20;
    }
    return __hiloint2double((int)(sign | ((m >> 3) + bias)), (int)(m << 29));
}
__device__ __forceinline__ void widen4(const float* v, double* d) {
    bool other = false;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const uint32_t u = __float_as_uint(v[e]), m = u & 0x7fffffffu;
        other |= m - 0x00800000u >= 0x7f000000u;
        d[e] = __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(u << 29));
    }
    if (other) {
#pragma unroll
        for (int e = 0; e < 4; ++e) d[e] = widen_any(v[e]);
    }
}

// Store four consecutive values at out[first .. first + 3], 16-byte aligned.
__device__ __forceinline__ void store4(float* out, uint64_t first, const float* v, int left) {
    float* dst = out + first;
    if (left >= 4) {
        __stcs(reinterpret_cast<float4*>(dst), make_float4(v[0], v[1], v[2], v[3]));
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (e < left) dst[e] = v[e];
    }
}

// Interleaved output: a block's values in record order in shared memory,
// value (j, f) at word j * F + f: consecutive lanes' records are F words
// apart, a bank conflict of gcd(F, 32) ways.
template <int F>
__device__ __forceinline__ int rec_slot(int j, int f) { return j * F + f; }
template <int F>
constexpr uint32_t rec_words() { return (uint32_t)(kBlock * F); }

// x = fma((float)q, step, min) of four codes.
__device__ __forceinline__ void rebuild4(const uint32_t* q, uint32_t bits, float s, float mn, float* v) {
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = __fmaf_rn(bits <= 23u ? small_u2f(q[e]) : __uint2float_rn(q[e]), s, mn);
}

// Where a block's values go: fp32 fields, 16-byte aligned or of any alignment,
// fp64 fields, or interleaved fp32 records.
enum : int { kOut32, kOutAny, kOut64, kOutRecords };

// The positions a thread rebuilds, in groups of four: four consecutive ones,
// stored with 16-byte stores, into aligned fields; otherwise one of each run
// of kDecThreads, so that a warp's 4-byte (8-byte) stores, or its words in the
// record stage, are consecutive.  (Into odd rows of a
// 10^7 x 6 snapshot: 53 us; with 4-byte stores of four consecutive positions
// per lane 55, with 16-byte units completed by shuffles from the next lane
// 68; aligned rows 50.)
__host__ __device__ constexpr bool out_strided(int out) { return out != kOut32; }
template <int OUT>
__device__ __forceinline__ int out_pos(int g, int e) {
    const int t = threadIdx.x;
    return out_strided(OUT) ? t + kDecThreads * (4 * g + e) : 4 * (t + kDecThreads * g) + e;
}

// The values of group g's positions of field f, in the block starting at
// particle `base`, those below n_b.
template <int F, int OUT>
__device__ __forceinline__ void store_group(const DecArgs& a, int f, int g, const float* v, uint64_t base, int n_b,
                                            float* recs) {
    if (!out_strided(OUT)) {
        const int j = out_pos<OUT>(g, 0);
        store4(a.out[f], base + j, v, n_b - j);
        return;
    }
    double d[4];
    if (OUT == kOut64) widen4(v, d);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int j = out_pos<OUT>(g, e);
        if (j >= n_b) continue;
        if (OUT == kOutRecords)
            recs[rec_slot<F>(j, f)] = v[e];
        else if (OUT == kOut64)
            __stcs(reinterpret_cast<double*>(a.out[f]) + base + j, d[e]);
        else
            __stcs(a.out[f] + base + j, v[e]);
    }
}

// Records wider than 128 bits (rare): every code is read field by field from
// the stream itself; the block header is re-read here so that the common path
// passes nothing through memory.
template <int F, int OUT>
__device__ __forceinline__ void decode_wide(const DecArgs& a, const uint32_t* blk, uint32_t rwords_off,
                                            uint32_t rwords, uint32_t W, uint32_t G, int grp, int n_b, uint64_t base,
                                            const uint32_t (&key)[4], float* recs) {
    constexpr int P = F < 3 ? F : 3;
    const uint32_t* R = blk + rwords_off;
    // walk the fields from the top of the record down: field 0 is most significant
    uint32_t kacc[F], racc[F], wfv[F], gv[F];
    {
        uint32_t r = 0, k = 0;
        for (int f = F - 1; f >= 0; --f) {
            const uint32_t bf = (__ldg(blk + 1 + F + (f >> 2)) >> (8 * (f & 3))) & 0xffu;
            const uint32_t g = f < P ? min(G, bf) : 0u;
            gv[f] = g;
            wfv[f] = f < P ? bf - g : bf;
            racc[f] = r;
            kacc[f] = k;
            r += wfv[f];
            k += g;
        }
    }
    for (int f = 0; f < F; ++f) {
        const uint32_t bf = (__ldg(blk + 1 + F + (f >> 2)) >> (8 * (f & 3))) & 0xffu;
        const float mnf = __uint_as_float(__ldg(blk + 1 + f));
        const float sf = __uint_as_float(__ldg(a.stream + kHeaderWords + 2 * f + 1));
        const uint32_t cm = mask_bits(wfv[f]), gm = mask_bits(gv[f]);
        uint32_t qv[4];
        for (int e = 0; e < 4; ++e) {
            uint32_t code = 0u;
            const int j = out_pos<OUT>(grp, e);
            if (cm && j < n_b) {
                const uint32_t p = (uint32_t)j * W + racc[f];
                const uint32_t wi = p >> 5, sh = p & 31u;
                const uint32_t lo = __ldg(R + wi);
                const uint32_t hi = (sh + wfv[f] > 32u) && (wi + 1 < rwords) ? __ldg(R + wi + 1) : 0u;
                code = __funnelshift_r(lo, hi, sh) & cm;
            }
            qv[e] = f < P ? (code | (((key[e] >> kacc[f]) & gm) << wfv[f])) : code;
        }
        float v[4];
        rebuild4(qv, bf, sf, mnf, v);
        store_group<F, OUT>(a, f, grp, v, base, n_b, recs);
    }
}

struct DecCore {  // everything a block's decoding keeps in shared memory but its staged words
    uint16_t uniq[kMaxBins];
    uint32_t mask[32];
    uint32_t warp_uc[kDecWarps];  // per warp: id sum | count sum << 14
    uint32_t bad;
    // the block's constants, checked by warp 0 and read by every warp
    uint32_t ok, raw, U, wd, wc, W, keybits, G;
    uint4 lay[kMaxFields];      // per field: bits in the record and their mask, segId bits of a position
                                // axis, segId mask shifted above the segOffset bits
    float4 ms[kMaxFields];      // per field: block minimum, step, the code width's bits (as an integer), 0
};

template <int F>
struct DecShared : DecCore {
    static constexpr uint32_t kWords = dec_stage_words(F);
    uint64_t bar;  // the staging bulk copy
    // the block's words after its header, from word `shift` (the source's
    // offset from a 16-byte boundary, 0..3)
    alignas(16) uint32_t stage[kWords + kDecStagePad + 4];
};

// The same for interleaved output: the stage also takes the block's values
// in record order once its words are consumed.
constexpr uint32_t cmax(uint32_t x, uint32_t y) { return x > y ? x : y; }
template <int F>
struct DecSharedRec : DecCore {
    static constexpr uint32_t kWords = cmax(dec_stage_words(F), rec_words<F>());  // a raw block whole
    uint64_t bar;
    alignas(16) uint32_t stage[kWords + kDecStagePad + 4];
};

// Groups g0 .. g0 + NG - 1 of four positions (keys key[g - g0]): their records
// from the staged words, then the codes of fields F-1 .. 0, consumed from the
// least significant end: field F-1 sits at bit 0 of the record and field 0 at
// the top.  rr holds a record in its low bits (NR words, W <= 32 NR); after each field the record is shifted right by the field's width
// and the key right by the axis' segId bits.  q = segId * 2^o + segOffset for
// a position axis, the whole code otherwise.  Words past the record array
// (inside the staging pad) hold bits above W, which are never consumed.
// kOutRecords: sync() once every record is in registers, then the values go to
// recs.
template <int F, int NG, int NR, int OUT, class Sync>
__device__ __forceinline__ void decode_groups(const DecArgs& a, const DecCore& L, const uint32_t* sR, uint32_t W,
                                              int g0, uint32_t (&key)[NG][4], uint64_t base, int n_b,
                                              float* recs, Sync sync) {
    constexpr int P = F < 3 ? F : 3;
    uint32_t rr[NG][4][NR];
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const uint32_t p = (uint32_t)out_pos<OUT>(g0 + g, e) * W;
            const uint32_t* at = sR + (p >> 5);
            uint32_t x = at[0];
#pragma unroll
            for (int k = 0; k < NR; ++k) {
                const uint32_t y = at[k + 1];
                rr[g][e][k] = __funnelshift_r(x, y, p);
                x = y;
            }
        }
    sync();
#pragma unroll
    for (int f = F - 1; f >= 0; --f) {
        const uint4 lay = L.lay[f];
        const float4 ms = L.ms[f];
        const uint32_t wf = lay.x, cm = lay.y;
        const bool small = __float_as_uint(ms.z) <= 23u;  // uniform: codes below 2^23 convert with one add
        float v[NG][4];
#pragma unroll
        for (int g = 0; g < NG; ++g)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                uint32_t q = rr[g][e][0] & cm;
                if (f < P) {
                    q |= (key[g][e] << wf) & lay.w;
                    key[g][e] >>= lay.z;
                }
                v[g][e] = __uint_as_float(q);
                if (f > 0) {
#pragma unroll
                    for (int k = 0; k < NR; ++k)
                        rr[g][e][k] = k + 1 < NR ? __funnelshift_r(rr[g][e][k], rr[g][e][k + 1 < NR ? k + 1 : k], wf)
                                                 : rr[g][e][k] >> wf;
                }
            }
        if (small) {
#pragma unroll
            for (int g = 0; g < NG; ++g)
#pragma unroll
                for (int e = 0; e < 4; ++e) v[g][e] = __fmaf_rn(small_u2f(__float_as_uint(v[g][e])), ms.y, ms.x);
        } else {
#pragma unroll
            for (int g = 0; g < NG; ++g)
#pragma unroll
                for (int e = 0; e < 4; ++e) v[g][e] = __fmaf_rn(__uint2float_rn(__float_as_uint(v[g][e])), ms.y, ms.x);
        }
#pragma unroll
        for (int g = 0; g < NG; ++g) store_group<F, OUT>(a, f, g0 + g, v[g], base, n_b, recs);
    }
}


// Where a CTA gets its block's index: the grid (one CTA per block), or a
// shared-memory slot (the batched kernel's block within its chunk) re-read at
// each use, so that the index holds no register through the block code.
struct DecGridBlock {
    __device__ __forceinline__ uint32_t b() const { return blockIdx.x; }
};
struct DecSlotBlock {
    const volatile uint32_t* slot;
    __device__ __forceinline__ uint32_t b() const { return *slot; }
};

// The format checks and the block's constants (warp 0 alone; every lane
// calls): from the stream header words hv (lane k holds word k), the block's
// first words bw (lane k holds word k, up to the block header's end) and the
// steps (lane f holds field f's), and the block's table entries; into S.
template <int F>
__device__ __forceinline__ void decode_checks(const DecArgs& a, DecCore& S, uint32_t hv, uint32_t bw, float step,
                                              bool inside, uint32_t b, uint32_t off, uint32_t end,
                                              uint32_t payload_words, int n_b) {
    constexpr int P = F < 3 ? F : 3;
    const int lane = threadIdx.x & 31;
    const uint32_t hdr = 1u + (uint32_t)F + (uint32_t)((F + 3) >> 2);
    const uint32_t nw = end - off;
        bool ok = true;
    switch (lane) {
        case 0: ok = hv == kMagic; break;
        case 1: ok = hv == kVersion; break;
        case 2: ok = hv == (uint32_t)F; break;
        case 3: ok = hv <= (uint32_t)kMaxSegBits; break;
        case 4: ok = hv == (uint32_t)kBlock; break;
        case 5: ok = hv <= 1u; break;
        case 6: ok = hv == (uint32_t)(a.n & 0xffffffffull); break;
        case 7: ok = hv == (uint32_t)(a.n >> 32); break;
        case 8: ok = hv == a.nblocks; break;
        case 9: break;
        default: ok = lane >= 10 + 6 || hv == 0u; break;
    }
    const uint32_t G = __shfl_sync(0xffffffffu, hv, 3);
    ok = __all_sync(0xffffffffu, ok) && inside && !(b == 0 && off != 0) &&
         !(b + 1 == a.nblocks && end != payload_words) && end != off;
    // the block header: mode word, minima, width bytes
    const uint32_t mode = __shfl_sync(0xffffffffu, bw, 0);
    const bool raw = ok && (mode & 1u);
    if (raw) ok = mode == 1u && nw == 1u + (uint32_t)F * (uint32_t)n_b;
    // lane f holds field f: its code width, minimum and step, and its
    // layout -- bits in the record, segId bits and mask
    const bool fl = lane < F;
    const uint32_t wword = __shfl_sync(0xffffffffu, bw, (1 + F + (lane >> 2)) & 31);
    const uint32_t bits = fl ? (wword >> (8 * (lane & 3))) & 0xffu : 0u;
    const float mn = __uint_as_float(__shfl_sync(0xffffffffu, bw, (1 + lane) & 31));
    const uint32_t bf = bits <= 31u ? bits : 0u;
    const uint32_t g = lane < P ? min(G, bf) : 0u;
    const uint32_t wf = fl ? bf - g : 0u;
    uint32_t U = 0, wd = 0, wc = 0, W = 0, keybits = 0;
    if (ok && !raw) {
        U = (mode >> 1) & 0x7ffu;
        wd = (mode >> 12) & 31u;
        wc = (mode >> 17) & 31u;
        ok = (mode >> 22) == 0u && nw >= hdr && !__any_sync(0xffffffffu, bits > 31u);
        // padding bytes of the last width word are zero
        const uint32_t lastw = __shfl_sync(0xffffffffu, bw, hdr - 1);
        if ((F & 3) != 0) ok = ok && (lastw >> (8 * (F & 3))) == 0u;
        keybits = __reduce_add_sync(0xffffffffu, g);
        W = __reduce_add_sync(0xffffffffu, wf);
        // ids are below 2^keybits and counts at most 1024, so their widths
        // are at most keybits and 11 bits: the deltas and counts then fit
        // the words reserved for them in the staging area
        ok = ok && U >= 1u && U <= (uint32_t)n_b && U <= (1u << keybits) && wd <= keybits && wc <= 11u &&
             nw == hdr + ceil_words(U * wd) + ceil_words(U * wc) + ceil_words((uint32_t)n_b * W);
    }
    if (lane == 0) {
        S.ok = ok;
        S.raw = raw;
        S.U = U;
        S.wd = wd;
        S.wc = wc;
        S.W = W;
        S.keybits = keybits;
        S.G = G;
    }
    if (fl) {
        S.lay[lane] = make_uint4(wf, mask_bits(wf), g, mask_bits(g) << wf);  // g + wf = bits <= 31
        S.ms[lane] = make_float4(mn, step, __uint_as_float(bf), 0.0f);
    }
}

// The block's values, staged in record order (rec_slot) from a 16-byte
// boundary, to out[0] (every thread, after the values are staged): one bulk
// copy of the whole 16-byte units when the records are 16-byte aligned.
template <int F>
__device__ __forceinline__ void store_records(const DecArgs& a, const float* recs, uint32_t b, int n_b) {
    fence_proxy_async_shared();  // the values are read by a bulk copy (async proxy)
    __syncthreads();             // every value is staged
    const int t = threadIdx.x, total = n_b * F;
    float* dst = a.out[0] + (uint64_t)b * kBlock * F;
    const bool vec = (reinterpret_cast<uintptr_t>(dst) & 15u) == 0;
    const int bulk = vec ? total & ~3 : 0;
    if (t == 0 && bulk) bulk_s2g_start(dst, recs, (uint32_t)bulk * 4u);
    for (int k = bulk + t; k < total; k += kDecThreads) dst[k] = recs[k];
    if (t == 0 && bulk) bulk_s2g_wait();
}

// Decode a block whose constants warp 0 has published in S (after a
// barrier): stage holds the block's words after its header, blk the block in
// the stream (read directly for raw blocks and records wider than 128 bits).
// kOutRecords: the values go to interleaved records at out[0]; recs (16-byte
// aligned, rec_words<F>() words) takes them once the stage's words, which it
// overlays, are consumed.
template <int F, int OUT>
__device__ __forceinline__ void decode_tail(const DecArgs& a, DecCore& S, uint32_t* stage, float* recs,
                                            const uint32_t* blk, uint32_t b, int n_b) {
    constexpr bool OUT64 = OUT == kOut64, AOS = OUT == kOutRecords;
    uint16_t* uniq = S.uniq;
    uint32_t* mask = S.mask;
    uint32_t& s_bad = S.bad;
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    const uint32_t hdr = 1u + (uint32_t)F + (uint32_t)((F + 3) >> 2);
    if (!S.ok) {
        if (t == 0) set_status(a.status, kStCorrupt);
        return;  // uniform across the CTA
    }

    // ---- 2. raw block: the values from the staged words, which start at word
    // hdr of the block, those before and after them from the stream; eight of a
    // thread in flight at once.  (2^24 x 6 raw values: 0.287 ms with 128 threads
    // that load and store a value at a time, 0.181 with eight loads in flight but
    // all from the stream, 0.134 from the stage.)
    if (S.raw) {
        constexpr int N = kBlock / kDecThreads;
        const uint32_t total = (uint32_t)(F * n_b);
        const uint32_t nst =
            total + 1u > hdr ? min(total + 1u - hdr, AOS ? DecSharedRec<F>::kWords : DecShared<F>::kWords) : 0u;
        auto value = [&](uint32_t m) {  // value m of the block, at its word m + 1
            const uint32_t k = m + 1u - hdr;
            return k < nst ? stage[k] : __ldg(blk + 1u + m);
        };
        if (AOS) {  // field-major in the stream: gather each record's fields
            float* dst = a.out[0] + (uint64_t)b * kBlock * F;
            for (uint32_t k0 = t; k0 < total; k0 += N * kDecThreads) {
                uint32_t v[N];
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    const uint32_t k = k0 + i * kDecThreads, j = k / F, f = k - j * F;
                    v[i] = k < total ? value(f * n_b + j) : 0u;
                }
#pragma unroll
                for (int i = 0; i < N; ++i)
                    if (k0 + i * kDecThreads < total) dst[k0 + i * kDecThreads] = __uint_as_float(v[i]);
            }
            return;
        }
        const uint64_t first = (uint64_t)b * kBlock + t;
        constexpr int UNROLL = OUT64 ? 1 : F;  // unrolled, the doubles' conversions cost encoded blocks 2% (registers)
#pragma unroll UNROLL
        for (int f = 0; f < F; ++f) {
            float v[N];
#pragma unroll
            for (int i = 0; i < N; ++i)
                v[i] = t + i * kDecThreads < n_b ? __uint_as_float(value(f * n_b + t + i * kDecThreads)) : 0.0f;
            double d[N];
            if (OUT64) {
                widen4(v, d);
                widen4(v + 4, d + 4);
            }
#pragma unroll
            for (int i = 0; i < N; ++i) {
                if (t + i * kDecThreads >= n_b) continue;
                if (OUT64)
                    __stcs(reinterpret_cast<double*>(a.out[f]) + first + i * kDecThreads, d[i]);
                else
                    __stcs(a.out[f] + first + i * kDecThreads, v[i]);
            }
        }
        return;
    }

    const uint32_t U = S.U, wd = S.wd, wc = S.wc, W = S.W, keybits = S.keybits;
    const uint32_t dwords = ceil_words(U * wd), cwords = ceil_words(U * wc), rwords = ceil_words((uint32_t)n_b * W);
    const uint32_t idlimit = 1u << keybits;

    // the deltas, counts and (when at most 128 bits wide) the records are in
    // the staging area, contiguous as in the stream
    const bool fast = W <= 128u;  // then dwords + cwords + rwords <= the staged words
    const uint32_t* sR = stage + dwords + cwords;
    const uint32_t k0 = (uint32_t)kDecRuns * t;
    const int nrun = (int)min((uint32_t)kDecRuns, U > k0 ? U - k0 : 0u);  // this thread's runs

    // ---- 3. unique ids and run starts
    {
        uint32_t d[kDecRuns], c[kDecRuns], su = 0u, sc = 0u;
        extract4_s(stage, min(k0, U), wd, d);
        extract4_s(stage + dwords, min(k0, U), wc, c);
        bool bad = false;
#pragma unroll
        for (int k = 0; k < kDecRuns; ++k) {
            if (k < nrun) {
                bad |= c[k] == 0u || (d[k] == 0u && k0 + k > 0u);
                su += d[k];
                sc += c[k];
            }
        }
        // one scan of both sums; a thread's ids beyond 511 or counts beyond
        // 1024 already make the block corrupt, and without them a warp's id sum
        // is below 2^14 and its count sum at most 2^15
        if (su > 511u || sc > 1024u) {
            bad = true;
            su = sc = 0u;
        }
        const uint32_t iuc = warp_incl_sum(su | (sc << 14));
        if (lane == 31) S.warp_uc[w] = iuc;
        __syncthreads();
        uint32_t u = (iuc & 0x3fffu) - su, st = (iuc >> 14) - sc, total = 0;
#pragma unroll
        for (int ww = 0; ww < kDecWarps; ++ww) {
            const uint32_t uc = S.warp_uc[ww];
            if (ww < w) {
                u += uc & 0x3fffu;
                st += uc >> 14;
            }
            total += uc >> 14;
        }
#pragma unroll
        for (int k = 0; k < kDecRuns; ++k) {
            if (k < nrun && !bad) {
                u += d[k];
                if (u >= idlimit || st >= (uint32_t)n_b) {
                    bad = true;
                } else {
                    uniq[k0 + k] = (uint16_t)u;
                    atomicOr(&mask[st >> 5], 1u << (st & 31u));
                }
                st += c[k];
            }
        }
        if (t == 0 && total != (uint32_t)n_b) bad = true;
        if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(&s_bad, 1u);
    }
    __syncthreads();
    if (s_bad) {
        if (t == 0) set_status(a.status, kStCorrupt);
        return;
    }

    // ---- 4. the run of position j is the number of run starts up to j, less
    // one: every warp scans the 32 mask words itself (no further barrier; lane
    // i holds word i and the starts before it).  Consecutive positions of a
    // group lie in one word; strided ones in one word per warp.  Position 0
    // starts a run, so every index is in 0..U-1.
    uint32_t key[kDecGroups][4];
    {
        const uint32_t mw = mask[lane];
        const uint32_t pc = __popc(mw);
        const uint32_t pre = warp_incl_sum(pc) - pc;
#pragma unroll
        for (int g = 0; g < kDecGroups; ++g) {
            if (out_strided(OUT)) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int word = out_pos<OUT>(g, e) >> 5;  // the same for the whole warp
                    const uint32_t m = __shfl_sync(0xffffffffu, mw, word) & lanemask_le();
                    key[g][e] = uniq[__shfl_sync(0xffffffffu, pre, word) + __popc(m) - 1u];
                }
            } else {
                const int j = out_pos<OUT>(g, 0);
                const uint32_t word = __shfl_sync(0xffffffffu, mw, j >> 5);
                uint32_t run = __shfl_sync(0xffffffffu, pre, j >> 5) + __popc(word & ((1u << (j & 31)) - 1u)) - 1u;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    run += (word >> ((j & 31) + e)) & 1u;
                    key[g][e] = uniq[run];
                }
            }
        }
    }
    const uint64_t base = (uint64_t)b * kBlock;
    auto sync = [] {
        if (AOS) __syncthreads();
    };
    if (!fast) {
        sync();  // the staged deltas and counts are consumed
#pragma unroll
        for (int g = 0; g < kDecGroups; ++g)
            decode_wide<F, OUT>(a, blk, hdr + dwords + cwords, rwords, W, S.G, g, n_b, base, key[g], recs);
    } else if (F <= 3 && W <= 32u && OUT != kOut64) {
        // one word per record (10^8 x 3 scan points, most of them: 0.344 -> 0.319 ms)
        decode_groups<F, kDecGroups, 1, OUT>(a, S, sR, W, 0, key, base, n_b, recs, sync);
    } else if (W <= 64u && OUT != kOut64) {
        decode_groups<F, kDecGroups, 2, OUT>(a, S, sR, W, 0, key, base, n_b, recs, sync);
    } else if (AOS) {  // every record in registers before the first value is staged
        decode_groups<F, kDecGroups, 4, OUT>(a, S, sR, W, 0, key, base, n_b, recs, sync);
    } else {  // a group at a time: fewer registers (fp64 output 94 -> 84 us on a 2^23 x 6 stream)
#pragma unroll 1
        for (int g = 0; g < kDecGroups; ++g) {
            uint32_t kg[1][4];
#pragma unroll
            for (int e = 0; e < 4; ++e) kg[0][e] = g == 0 ? key[0][e] : key[kDecGroups - 1][e];
            if (OUT == kOut64 && W <= 64u)
                decode_groups<F, 1, 2, OUT>(a, S, sR, W, g, kg, base, n_b, recs, sync);
            else
                decode_groups<F, 1, 4, OUT>(a, S, sR, W, g, kg, base, n_b, recs, sync);
        }
    }
    if (AOS) store_records<F>(a, recs, b, n_b);
}


// kOutRecords: out[0] receives interleaved records of F fields (Sh then a
// DecSharedRec<F>).  PREHW: lanes 0, 1, 2 of every warp pass in hw_pre the
// words round trip 1 would load (the payload size and the block's two table
// entries), loaded earlier by the caller.
template <int F, int OUT, bool PREHW, class Sh, class Idx>
__device__ __forceinline__ void decode_block(const DecArgs& a, Sh& S, Idx idx, uint32_t hw_pre = 0u) {
    uint32_t* stage = S.stage;
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    const uint32_t* Sw = a.stream;
    const uint32_t b = idx.b();
    const int n_b = (int)((a.n - (uint64_t)b * kBlock) < (uint64_t)kBlock ? (a.n - (uint64_t)b * kBlock) : (uint64_t)kBlock);
    const uint64_t table_start = kHeaderWords + 2ull * F;
    const uint64_t payload_start = table_start + a.nblocks + 1;
    const uint32_t hdr = 1u + (uint32_t)F + (uint32_t)((F + 3) >> 2);
    if (t < 32) S.mask[t] = 0u;
    if (t == 0) S.bad = 0u;

    // ---- 1. where the block is (every warp, one round trip): the payload
    // size and the block's two table entries, checked only as far as staging
    // the block safely needs
    const bool header_fits = payload_start <= a.total_words;
    uint32_t hw = 0;
    if (PREHW)
        hw = header_fits && lane < 3 ? hw_pre : 0u;
    else if (header_fits && lane < 3)
        hw = __ldg(lane == 0 ? Sw + 9 : Sw + table_start + b + (uint32_t)(lane - 1));
    const uint32_t payload_words = __shfl_sync(0xffffffffu, hw, 0);
    const uint32_t off = __shfl_sync(0xffffffffu, hw, 1);
    const uint32_t end = __shfl_sync(0xffffffffu, hw, 2);
    const bool inside =
        header_fits && payload_start + payload_words <= a.total_words && off <= end && end <= payload_words;
    const uint32_t* blk = Sw + payload_start + off;
    const uint32_t nw = end - off;
    // round trip 2: warp 0 fetches the stream header, the block header and the
    // steps (all in bounds once the block is inside the stream), and the
    // block's words after its header are staged in shared memory (all of them
    // when they fit; the deltas and counts always fit) by one bulk copy that
    // thread 0 issues, its last few words by plain loads where the copy's
    // 16-byte units would reach past the stream
    uint32_t hv = 0, bw = 0;
    float step = 0.0f;
    if (w == 0) {
        if (lane < kHeaderWords) hv = __ldg(Sw + lane);  // the host checked total_words >= kHeaderWords
        if (inside && (uint32_t)lane < min(hdr, nw)) bw = __ldg(blk + lane);
        if (header_fits && lane < F) step = __uint_as_float(__ldg(Sw + kHeaderWords + 2 * lane + 1));
    }
    // the copy: 16-byte units from the boundary at or below the first word,
    // as many as end inside the stream; the words after them by plain loads
    const uint32_t* src = blk + hdr;
    const uint32_t shift = (uint32_t)((reinterpret_cast<uintptr_t>(src) >> 2) & 3u);
    uint32_t nst = 0, units = 0;
    if (inside && nw > hdr) {
        nst = min(nw - hdr, Sh::kWords);
        const uint64_t avail = a.total_words - (uint64_t)(src - Sw) + shift;  // words from the boundary to the stream's end
        units = (uint32_t)(min((uint64_t)(nst + shift + 3u), avail) >> 2);
        if (units * 4u < shift) units = 0;
    }
    if (units && t == 0) {
        mbar_init(&S.bar, 1);
        mbar_arrive_expect_tx(&S.bar, units * 16u);
        bulk_g2s(S.stage, src - shift, units * 16u, &S.bar);
    }
    const uint32_t kb = units ? units * 4u - shift : 0u;  // first word not in the copy
    for (uint32_t k = kb + t; k < nst; k += kDecThreads) stage[shift + k] = __ldg(src + k);

    if (w == 0) decode_checks<F>(a, S, hv, bw, step, inside, b, off, end, payload_words, n_b);
    __syncthreads();
    if (units && !__syncthreads_and(mbar_wait_bounded(&S.bar, 0, a.status))) return;  // uniform
    decode_tail<F, OUT>(a, S, stage + shift, reinterpret_cast<float*>(stage), blk, b, n_b);
}

}  // namespace gpz
