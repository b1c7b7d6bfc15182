// gpz_wide_fast.cu -- stages 1-3 of the 64-bit form (gpz_wide.cu describes it)
// for the blocks that nearly all data consists of: finite values whose first
// candidates need no check (first_candidate_exact; codes of at most 41 bits)
// and an encoding smaller than the raw block.  A block with a value that is not
// finite is stored raw here, the others go to a list for the general kernel.
// With an absolute bound the extremes have to be found first, and a block that
// is then left has been read for nothing; most of those show in the first 512
// values of a field and are left there and then.  2^22 x 6 doubles at 1e-12
// absolute 0.624 -> 0.541 ms (0.595 with the general kernel alone), with a NaN
// in every block 0.310 -> 0.178 (0.250).
//
// One CTA of 128 threads per block.  Nothing but the particles' keys is held:
//   1. the block's extremes (the range pass's, or found here) give every
//      field's constants and code width, warp 0 alone;
//   2. the position axes are read and quantised for the keys, which are ranked
//      and scanned (gpz_sort.cuh);
//   3. every field is read again (the block is still in L2) and quantised, and
//      its code is ORed into the staging words at the particle's sorted
//      position, which leave by one bulk copy.
// GB300's fp64 rate would set the pace (a warp's operation takes 16 cycles of
// its SM, and a code needs a subtraction and a multiply-add), so codes are
// computed in fixed point and only those within 10 * 2^-14 of a step of the
// next one, 0.1%, in fp64 (wide_code).
// 4*10^6 x 6 doubles at a relative bound of 1e-12: 0.299 ms in the general
// kernel (0.241 without its needless fp64 operations), 0.115 here: 20,200 warp
// instructions per block instead of 29,600, 60% of the issue slots busy.
#include "gpz_sort.cuh"
#include "gpz_wide.cuh"

namespace gpz {

namespace {

// Code width limit: first_candidate_exact allows a range of 2^40 steps.
constexpr uint32_t kWfBits = 41u;

__host__ __device__ constexpr uint32_t wf_stage_words(int F) {
    return (1u + 2u * (uint32_t)F + 2u + 144u + 176u + 32u * kWfBits * (uint32_t)F + 3u) & ~3u;
}
__host__ __device__ constexpr uint32_t wf_smem_bytes(int F) { return 4u * wf_stage_words(F) + kSortHistBytes; }
__host__ __device__ constexpr int wf_ctas(int F) {
    const int by_smem = (int)((227u * 1024u) / (wf_smem_bytes(F) + 1024u + 1024u));
    return by_smem < 6 ? by_smem : 6;
}

struct alignas(16) WfField {
    unsigned long long nxm, m;       // -min and 1/s in fixed point (wide_code)
    unsigned long long vmask;        // the code's bits in the record
    double mn, inv;
    uint32_t rs, wf, roff, ks;       // shift base, bits in the record and their place, the segId's place in the key
    uint32_t bits, pad[3];
};

struct WfShared : SortShared {
    uint32_t ok, nonfinite, W;
    ulonglong2 ext[kMaxFields];
    WfField fc[kMaxFields];
};

// The format's first candidate in fp64.
__device__ __noinline__ unsigned long long wide_code_fp64(unsigned long long x, double mn, double inv) {
    return code_floor(__fma_rn(__dsub_rn(__longlong_as_double((long long)x), mn), inv, 0.5));
}

// A double's bits as a multiple of 2^k, toward zero, where rs = 1085 + k: the
// 53-bit significand, 10 places up, shifted right (|value| < 2^61 * 2^k).
__device__ __forceinline__ unsigned long long wide_fixed(unsigned long long x, uint32_t rs) {
    const uint32_t hi = (uint32_t)(x >> 32), lo = (uint32_t)x;
    const uint32_t mh = __funnelshift_l(lo, (hi & 0xfffffu) | 0x100000u, 10), ml = lo << 10;
    unsigned long long v = ((unsigned long long)mh << 32) | ml;
    asm("shr.u64 %0, %0, %1;" : "+l"(v) : "r"(rs - ((hi >> 20) & 0x7ffu)));  // a shift beyond 63 gives 0 (zero, subnormal)
    const unsigned long long sign = (unsigned long long)((long long)x >> 63);
    return (v ^ sign) - sign;
}

// The first candidate q = floor(RN(fma(RN(x - min), inv, 1/2))) of a block
// that first_candidate_exact accepts, in fixed point.  k = floor(log2 s) - 15:
//   X = x / 2^k and XM = min / 2^k toward zero (|x| <= 2^45 eb: below 2^61), so
//   D = X - XM is off by less than 2 and, both being monotone, not negative;
//   m = inv * 2^(k + 78), exact (53 significant bits, in [2^62, 2^63]);
//   T = D m / 2^64 + 2^13 = 2^14 (x - min) inv + 2^13, up to: less than 3 for
//   the partial products left out, 1 for D (2 m / 2^64 <= 1), 2.2 for the
//   rounding of x - min (2^-53 of at most 2^40.1 steps) and 2 for that of the
//   multiply-add (half of 2^-12).
// So when T's low 14 bits are at least 10 away from a carry either way, T >> 14
// is the rounded value's floor; otherwise fp64 decides.
// (rs, nxm, m: c's, held in registers.)
__device__ __forceinline__ unsigned long long wide_code(unsigned long long x, uint32_t rs, unsigned long long nxm,
                                                        unsigned long long m, const WfField& c) {
    const unsigned long long D = wide_fixed(x, rs) + nxm;
    const uint32_t dl = (uint32_t)D, dh = (uint32_t)(D >> 32), ml = (uint32_t)m, mh = (uint32_t)(m >> 32);
    const unsigned long long T = (unsigned long long)dh * mh + ((unsigned long long)__umulhi(dl, mh) + 8192u) +
                                 (unsigned long long)__umulhi(dh, ml);
    if ((((uint32_t)T + 10u) & 16383u) < 20u) return wide_code_fp64(x, c.mn, c.inv);
    return T >> 14;
}

// Whether extremes of some of a field's values (max of ~key, max of key)
// are finite and already go beyond what first_candidate_exact accepts (limits
// by their exponents; any answer will do, the general kernel takes any block).
__device__ __forceinline__ bool out_of_reach(unsigned long long nmin, unsigned long long kmax, const WideParams& p) {
    const double lo = wide_from_key(~nmin), hi = wide_from_key(kmax);
    auto bits = [](double v) { return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull; };
    const unsigned long long m = max(bits(lo), bits(hi));
    return m < 0x7ff0000000000000ull &&
           (m > bits(p.eb) + (45ull << 52) || bits(__dsub_rn(hi, lo)) > bits(p.s) + (40ull << 52));
}

}  // namespace

// UNSTABLE (tests only): every block's sort fails its check.
template <int F, bool UNSTABLE = false>
__global__ void __launch_bounds__(kTileThreads, wf_ctas(F)) gpz_wide_fast_kernel(const __grid_constant__ WideQseArgs a) {
    extern __shared__ __align__(128) uint8_t dsm[];
    __shared__ WfShared S;
    constexpr int P = F < 3 ? F : 3, R = kTileRounds;
    constexpr unsigned long long kNegInf = ~0xfff0000000000000ull, kPosInf = 0xfff0000000000000ull;  // order keys
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    const uint32_t b = blockIdx.x;
    const uint64_t first = (uint64_t)b * kBlock;
    const int n_b = (int)min((uint64_t)kBlock, a.n - first);
    uint32_t* stage = reinterpret_cast<uint32_t*>(dsm);
    uint16_t* hist = reinterpret_cast<uint16_t*>(dsm + 4u * wf_stage_words(F));
    uint32_t* order = reinterpret_cast<uint32_t*>(hist);  // later
    uint32_t* out = a.temp + (size_t)b * a.slot_words;
    const int i0 = 32 * R * w + lane;  // this thread's particles: i0 + 32 r
    auto valid = [&](int r) { return i0 + 32 * r < n_b; };
    auto field = [&](int f) { return reinterpret_cast<const unsigned long long*>(a.fields[f]) + first; };

    // ---- 1. the block's extremes and the fields' constants
    if (t == 0) S.unsure = 0u;
    {
        uint4* h4 = reinterpret_cast<uint4*>(hist);
#pragma unroll
        for (int k = 0; k < (int)kSortHistBytes / 16 / kTileThreads; ++k) h4[t + kTileThreads * k] = make_uint4(0u, 0u, 0u, 0u);
    }
    if (!a.pre) {
        bool leave = false;
        for (int f = w; f < F && !leave; f += kTileWarps) {
            const unsigned long long* x = field(f);
            unsigned long long nmin = 0ull, kmax = 0ull;
            auto take = [&](unsigned long long v) {
                const unsigned long long key = wide_key(v);
                nmin = max(nmin, ~key);
                kmax = max(kmax, key);
            };
            if (n_b == kBlock) {
                unsigned long long v[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) v[k] = __ldg(x + lane + 32 * k);
#pragma unroll
                for (int k = 0; k < 16; ++k) take(v[k]);
                // half of the warp's first field tells most blocks that
                // first_candidate_exact cannot accept
                if (f == w && __any_sync(0xffffffffu, out_of_reach(nmin, kmax, a.params[f]))) {
                    leave = true;
                    break;
                }
#pragma unroll
                for (int k = 0; k < 16; ++k) v[k] = __ldg(x + lane + 512 + 32 * k);
#pragma unroll
                for (int k = 0; k < 16; ++k) take(v[k]);
            } else {
                for (int i = lane; i < n_b; i += 32) take(__ldg(x + i));
            }
            nmin = warp_max_u64(nmin);
            kmax = warp_max_u64(kmax);
            if (lane == 0)
                S.ext[f] = ~nmin > kNegInf && kmax < kPosInf ? make_ulonglong2(nmin, kmax) : make_ulonglong2(0ull, 0ull);
        }
        if (__syncthreads_or(leave)) {
            if (t == 0) a.general_list[atomicAdd(a.general_count, 1u)] = b;
            return;
        }
    }
    if (w == 0) {
        const bool fl = lane < F;
        ulonglong2 e = make_ulonglong2(0ull, 0ull);
        WideParams p = {};
        if (fl) {
            e = a.pre ? *(reinterpret_cast<const ulonglong2*>(out) + lane) : S.ext[lane];
            p = a.params[lane];
        }
        uint32_t bits = 0u;
        bool ok = true;
        double mn = 0.0;
        const unsigned long long su = (unsigned long long)__double_as_longlong(p.s);
        const unsigned long long iu = (unsigned long long)__double_as_longlong(p.inv);
        const int k = (int)((su >> 52) & 0x7ffu) - 1023 - 15;              // floor(log2 s) - 15
        const int up = (int)((iu >> 52) & 0x7ffu) - 1075 + k + 78;         // m's shift: 10 or 11 for a normal 1/s
        if (fl) {
            ok = e.y != 0ull && (up == 10 || up == 11);  // finite; no step beyond 2^1022
            const double lo = wide_from_key(~e.x), hi = wide_from_key(e.y);
            mn = lo == 0.0 ? 0.0 : lo;  // a zero minimum is stored as +0
            ok = ok && first_candidate_exact(lo, hi, p);
            // first candidates are monotone in the value: the maximum's is the largest
            if (ok) bits = bit_width64(code_floor(__fma_rn(__dsub_rn(hi, mn), p.inv, 0.5)));
            ok = ok && bits <= kWfBits;
        }
        const bool nonfinite = __any_sync(0xffffffffu, fl && e.y == 0ull);
        ok = __all_sync(0xffffffffu, ok);
        const uint32_t g = lane < P ? min((uint32_t)a.G, bits) : 0u, wf = bits - g;
        const uint32_t g1 = __shfl_sync(0xffffffffu, g, 1), g2 = __shfl_sync(0xffffffffu, g, 2);
        const uint32_t W = __reduce_add_sync(0xffffffffu, wf), upto = warp_incl_sum(wf);
        if (fl && ok) {
            WfField& c = S.fc[lane];
            c.rs = (uint32_t)(1085 + k);
            c.nxm = 0ull - wide_fixed((unsigned long long)__double_as_longlong(mn), c.rs);
            c.m = ((iu & 0xfffffffffffffull) | 0x10000000000000ull) << up;  // inv * 2^(k + 78)
            c.vmask = mask64(wf);
            c.mn = mn;
            c.inv = p.inv;
            c.wf = wf;
            c.roff = W - upto;  // field F-1 least significant
            c.ks = lane == 0 ? g1 + g2 : (lane == 1 ? g2 : 0u);
            c.bits = bits;
        }
        if (lane == 0) {
            S.ok = ok;
            S.nonfinite = nonfinite;
            S.W = W;
        }
    }
    __syncthreads();
    if (S.nonfinite) {
        wide_write_raw<F, kTileThreads>(a, b, n_b, t);
        return;
    }
    if (!S.ok) {
        if (t == 0) a.general_list[atomicAdd(a.general_count, 1u)] = b;
        return;
    }
    const uint32_t W = S.W;
    const uint32_t hdr = 1u + 2u * (uint32_t)F + (uint32_t)((F + 3) >> 2);
    const uint32_t rwords = ceil_words((uint32_t)n_b * W);
    {
        // the staging words, assembled by OR: clear what the block can need
        const uint32_t need = min((hdr + 144u + 176u + rwords + 3u) >> 2, wf_stage_words(F) / 4u);
        uint4* s4 = reinterpret_cast<uint4*>(stage);
        for (uint32_t k = t; k < need; k += kTileThreads) s4[k] = make_uint4(0u, 0u, 0u, 0u);
    }

    // ---- 2. keys of the position axes, ranks, runs
    uint32_t key[R];
#pragma unroll
    for (int r = 0; r < R; ++r) key[r] = 0u;
#pragma unroll 1
    for (int f = 0; f < P; ++f) {
        const WfField& c = S.fc[f];
        const unsigned long long nxm = c.nxm, m = c.m;
        const uint32_t rs = c.rs, wf = c.wf, ks = c.ks;
        const unsigned long long* x = field(f) + i0;
        unsigned long long v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = valid(r) ? __ldg(x + 32 * r) : 0ull;
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (valid(r)) key[r] |= (uint32_t)(wide_code(v[r], rs, nxm, m, c) >> wf) << ks;
    }
    rank_keys(key, hist, valid, S);
    __syncthreads();  // ranked
    const SortRuns runs = scan_bins(hist, S);
    const uint32_t U = runs.U, wd = bit_width(runs.maxdelta), wc = bit_width(runs.maxcnt);
    const uint32_t dwords = ceil_words(U * wd), cwords = ceil_words(U * wc);
    const uint32_t enc = hdr + dwords + cwords + rwords;
    if (enc >= 1u + 2u * (uint32_t)F * (uint32_t)n_b) {  // stored raw
        if (t == 0) a.general_list[atomicAdd(a.general_count, 1u)] = b;
        return;
    }

    // ---- 3. header, runs, and every field's codes at their sorted positions
    if (t == 0) stage[0] = (U << 1) | (wd << 12) | (wc << 17);
    if (t < 2 * F) {
        const unsigned long long u = (unsigned long long)__double_as_longlong(S.fc[t >> 1].mn);
        stage[1 + t] = (t & 1) ? (uint32_t)(u >> 32) : (uint32_t)u;
    }
    if (t < ((F + 3) >> 2)) {
        uint32_t word = 0;
#pragma unroll
        for (int f = 0; f < F; ++f)
            if ((f >> 2) == t) word |= S.fc[f].bits << (8 * (f & 3));
        stage[1 + 2 * F + t] = word;
    }
    or_runs(stage, runs, hdr, wd, wc);
    uint32_t at[R];  // each record's first bit in the staging words
#pragma unroll
    for (int r = 0; r < R; ++r) at[r] = valid(r) ? 32u * (hdr + dwords + cwords) + sorted_position(key[r], hist) * W : 0u;
#pragma unroll 1
    for (int f = 0; f < F; ++f) {
        const WfField& c = S.fc[f];
        const unsigned long long nxm = c.nxm, m = c.m, vmask = c.vmask;
        const uint32_t rs = c.rs, wf = c.wf, roff = c.roff;
        if (wf == 0u) continue;  // uniform
        const unsigned long long* x = field(f) + i0;
        unsigned long long v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = valid(r) ? __ldg(x + 32 * r) : 0ull;
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (valid(r)) or_bits(stage, at[r] + roff, wide_code(v[r], rs, nxm, m, c) & vmask, wf);
    }
    fence_proxy_async_shared();  // the staging words are read by a bulk copy (async proxy)
    __syncthreads();
    if (t == 0) bulk_s2g_start(out, stage, ((enc + 3u) & ~3u) * 4u);
    if (!sorted_order(key, order, valid, i0, n_b, a.perm != nullptr, S) || UNSTABLE) {
        if (t == 0) a.general_list[atomicAdd(a.general_count, 1u)] = b;  // not stable: the general kernel redoes it
    } else {
        if (t == 0) store_size(a.sizes, a.sums, a.sum_shift, b, enc);
        if (a.perm)
            for (int j = t; j < n_b; j += kTileThreads) a.perm[first + j] = (uint32_t)first + (order[j] & 1023u);
    }
    if (t == 0) bulk_s2g_wait();
}

namespace {

template <int F, bool UNSTABLE = false>
cudaError_t prepare_wide_fast_f() {
    auto kern = gpz_wide_fast_kernel<F, UNSTABLE>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wf_smem_bytes(F));
    return e != cudaSuccess ? e : cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
}

template <int F>
cudaError_t launch_wide_fast_f(const WideQseArgs& a, cudaStream_t s) {
    gpz_wide_fast_kernel<F><<<a.nblocks, kTileThreads, wf_smem_bytes(F), s>>>(a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_wide_fast(const WideQseArgs& a, cudaStream_t s) {
    switch (a.F) {
        case 1: return launch_wide_fast_f<1>(a, s);
        case 2: return launch_wide_fast_f<2>(a, s);
        case 3: return launch_wide_fast_f<3>(a, s);
        case 4: return launch_wide_fast_f<4>(a, s);
        case 5: return launch_wide_fast_f<5>(a, s);
        case 6: return launch_wide_fast_f<6>(a, s);
        case 7: return launch_wide_fast_f<7>(a, s);
        case 8: return launch_wide_fast_f<8>(a, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_wide_fast_unstable(const WideQseArgs& a, cudaStream_t s) {
    if (a.F != 3) return cudaErrorInvalidValue;
    const cudaError_t e = prepare_wide_fast_f<3, true>();
    if (e != cudaSuccess) return e;
    gpz_wide_fast_kernel<3, true><<<a.nblocks, kTileThreads, wf_smem_bytes(3), s>>>(a);
    return cudaGetLastError();
}

cudaError_t prepare_wide_fast(int F) {
    switch (F) {
        case 1: return prepare_wide_fast_f<1>();
        case 2: return prepare_wide_fast_f<2>();
        case 3: return prepare_wide_fast_f<3>();
        case 4: return prepare_wide_fast_f<4>();
        case 5: return prepare_wide_fast_f<5>();
        case 6: return prepare_wide_fast_f<6>();
        case 7: return prepare_wide_fast_f<7>();
        case 8: return prepare_wide_fast_f<8>();
    }
    return cudaErrorInvalidValue;
}

}  // namespace gpz
