// gpz_wide.cuh -- what the kernels of the 64-bit form share (gpz_wide.cu,
// gpz_wide_fast.cu): argument blocks, order keys, and the first-candidate
// condition.
#pragma once

#include "gpz_internal.cuh"

namespace gpz {

constexpr int kWideThreads = 256;
constexpr int kWideWarps = kWideThreads / 32;
constexpr uint32_t kWideMaxBits = 53;
constexpr unsigned long long kWideLimit = 1ull << 53;  // codes stay below 2^53
constexpr double kWideLimitD = 9007199254740992.0;     // 2^53
constexpr uint32_t kWideDcWords = 144u + 176u;         // deltas (<= 9 bits) and counts (<= 11 bits) of <= 512 runs

struct WideParams {
    double eb, s, inv, ebchk;
};

struct WideRangeArgs {
    const double* fields[kMaxFields];
    uint64_t n;
    int F;
    uint32_t* temp;           // [nblocks][slot_words]: each block's extremes go to the start of its slot
    uint32_t slot_words;
    unsigned long long* res;  // [F][2]: max of ~key (the minimum), max of key, over the non-NaN values; zeroed
};

struct WideQseArgs {
    const double* fields[kMaxFields];
    uint64_t n;
    int F, G;
    WideParams params[kMaxFields];
    uint32_t* temp;  // [nblocks][slot_words]
    uint32_t slot_words;
    uint32_t* sizes;  // [nblocks]
    uint32_t* sums;   // as QseArgs
    uint32_t sum_shift;
    uint32_t* perm;   // [n] or nullptr
    int pre;          // the range pass has put each block's extremes at the start of its slot
    uint32_t nblocks;
    uint32_t* general_list;   // [nblocks] blocks left to the general kernel
    uint32_t* general_count;  // zeroed
};

// A block's extremes of one field over its values, as the range pass leaves
// them: max of ~key, max of key (wide_key); (0, 0) when one is not finite.

struct WideDecArgs {
    const uint32_t* stream;
    uint64_t total_words;
    double* out[kMaxFields];
    uint64_t n;
    int F;
    uint32_t nblocks;
    uint32_t* status;
};

__device__ __forceinline__ unsigned long long wide_key(unsigned long long u) {
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

__device__ __forceinline__ double wide_from_key(unsigned long long k) {
    return __longlong_as_double((long long)((k >> 63) ? (k & 0x7fffffffffffffffull) : ~k));
}

// Maximum over the warp (every lane calls it): the largest high word, then
// the largest low word among the lanes that hold it (two redux operations).
__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) {
    const uint32_t hi = (uint32_t)(v >> 32), lo = (uint32_t)v;
    const uint32_t mh = __reduce_max_sync(0xffffffffu, hi);
    const uint32_t ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
    return ((unsigned long long)mh << 32) | ml;
}

__device__ __forceinline__ uint32_t bit_width64(unsigned long long v) { return 64u - (uint32_t)__clzll((long long)v); }

__device__ __forceinline__ unsigned long long mask64(uint32_t w) { return w >= 64u ? ~0ull : ((1ull << w) - 1ull); }

// floor(t) for 0 <= t < 2^53, on the integer pipe: the significand shifted
// right by the fraction bits the exponent leaves below the binary point.
__device__ __forceinline__ unsigned long long code_floor(double t) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(t);
    const int e = (int)(u >> 52) - 1023;  // t >= 0
    const unsigned long long m = (u & 0xfffffffffffffull) | 0x10000000000000ull;
    return e < 0 ? 0ull : (e >= 52 ? m : (m >> (52 - e)));
}

// When the first candidate needs no check.  With u = 2^-53, D = x - min >= 0,
// r = D / s and the three roundings of t = fma(RN(D), RN(1/s), 1/2):
// |q - r| <= 1/2 + e, e <= 3.01 u r + u/2; the reconstruction
// X = q s + min rounds to x^ with |x^ - X| <= u |X|, and the check's
// difference rounds once more.  So |RN(x - x^)| <= (s (1/2 + e) + u |X|)(1 + u).
// With s <= eb (63/32)(1 + u), r <= 2^40 (then e < 3.7e-4) and
// |X| <= max|x| + s <= eb (2^45 + 2) (then u |X| / eb < 0.0040), this is
// below 0.990 eb, under the threshold eb (1 - 2^-51) -- the 1/64 margin of
// the step absorbs the rounding.  eb >= 2^-1000 keeps every quantity normal
// (a subnormal difference is exact; a subnormal x^ errs by 2^-1075 at most).
__device__ __forceinline__ bool first_candidate_exact(double bmin, double bmax, const WideParams& p) {
    return p.eb >= 0x1p-1000 && __dsub_ru(bmax, bmin) <= p.s * 0x1p40 &&
           fmax(fabs(bmin), fabs(bmax)) <= p.eb * 0x1p45;
}

// A block stored raw: its values as they are, field after field; a thread has
// all of its values of a field in flight.
template <int F, int TH>
__device__ __forceinline__ void wide_write_raw(const WideQseArgs& a, uint32_t b, int n_b, int t) {
    constexpr int N = kBlock / TH;
    const uint64_t first = (uint64_t)b * kBlock;
    uint32_t* out = a.temp + (size_t)b * a.slot_words;
    if (t == 0) out[0] = 1u;
#pragma unroll 1
    for (int f = 0; f < F; ++f) {
        const unsigned long long* src = reinterpret_cast<const unsigned long long*>(a.fields[f] + first);
        unsigned long long v[N];
#pragma unroll
        for (int k = 0; k < N; ++k) v[k] = t + k * TH < n_b ? __ldg(src + t + k * TH) : 0ull;
#pragma unroll
        for (int k = 0; k < N; ++k) {
            if (t + k * TH >= n_b) continue;
            uint32_t* at = out + 1 + 2 * (f * n_b + t + k * TH);
            at[0] = (uint32_t)v[k];
            at[1] = (uint32_t)(v[k] >> 32);
        }
    }
    if (a.perm)
        for (int i = t; i < n_b; i += TH) a.perm[first + i] = (uint32_t)(first + i);
    if (t == 0) store_size(a.sizes, a.sums, a.sum_shift, b, 1u + 2u * (uint32_t)F * (uint32_t)n_b);
}

// Stages 1-3 of the blocks the common path takes, the others into the
// general list (gpz_wide_fast.cu).
cudaError_t launch_wide_fast(const WideQseArgs& a, cudaStream_t s);
cudaError_t prepare_wide_fast(int F);  // its attributes on the current device
// Tests: three fields, every block's sort failing its check.
cudaError_t launch_wide_fast_unstable(const WideQseArgs& a, cudaStream_t s);

}  // namespace gpz
