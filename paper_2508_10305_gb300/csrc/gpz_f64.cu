// gpz_f64.cu -- fp64 input and output (Section 5.1: the paper down-casts fp64
// input to fp32 when that suffices for the error bound; otherwise the 64-bit
// form of gpz_wide.cu, Section 5.2).  Compression rounds every value to fp32 on the GPU and
// compresses the fp32 values with each field's bound reduced by the largest
// rounding error over its finite values, eb' = eb - max |x - RN32(x)|, so
// that every decompressed value lies within eb of its fp64 input.  One
// prepass kernel writes the fp32 copy (in the workspace) and finds, per
// field, the fp64 extremes of the non-NaN values and the largest rounding
// error; the host reads those (the call synchronises once), forms eb' (a
// relative bound is taken over the fp64 range) and calls gpz_compress with
// absolute bounds on the copy -- or, when some eb' is not positive, calls the
// 64-bit form with the bounds eb.  Decompression of a version-1 stream runs
// the block decoder storing fp64 (each value widened exactly from its fp32
// reconstruction); a version-2 stream goes to gpz_decompress_wide.
#include <cmath>
#include <cstring>

#include "gpz.h"
#include "gpz_host.hpp"
#include "gpz_internal.cuh"

using namespace gpz;
using namespace gpz::host;

namespace gpz {

constexpr int kF64Threads = 256;

// Order key of a double's bits: unsigned order equals numeric order (NaN excluded).
__device__ __forceinline__ unsigned long long order_key64(unsigned long long u) {
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

// Order key of a finite float (-0 < +0), as the range pass stores extremes.
__device__ __forceinline__ uint32_t f64_order_key32(float x) {
    const uint32_t u = __float_as_uint(x);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// ---------------------------------------------------------------- prepass
//
// A warp per (field, block of 1024 values): the fp32 copy, the block's fp32
// extremes for the fused kernel (as the range pass stores them), and the
// field's res[3f] = ~order key of the fp64 minimum, res[3f+1] = key of the maximum
// (over the non-NaN values), res[3f+2] = bits of the largest |x - RN32(x)|
// over the finite values (non-negative, so its bits order as the value); res
// must start as zeros.
//
// Bound by HBM and instruction issue.  A value's rounding takes about 25
// integer and fp32 instructions; the exact 64-bit extremes and errors, three
// times as many, are only updated for groups of four values per lane that a
// filter lets through: rounding is monotone, so a new fp64 minimum has an fp32
// value at most the smallest so far, and an fp32 approximation of the error
// (relative error below 2^-23) tells which error can be the largest.  CTAs
// take runs of consecutive blocks, so that the filters of a field warm up
// once.  2^23 x 6 doubles: 0.152 -> 0.115 ms
// (0.6 GB, 5.2 TB/s; 3 / 4 / 5 / 6 CTAs per SM 0.121 / 0.115 / 0.120 / 0.220),
// and the fused kernel behind it 0.105 -> 0.063 ms with the extremes given.

struct F64Shared {
    unsigned long long res[kMaxFields][3];
};

// RN32 of a double's bits; bits of |v - r|, exact in double.
static __device__ __noinline__ float f64_round_any(unsigned long long u) {
    return __double2float_rn(__longlong_as_double((long long)u));
}
static __device__ __noinline__ unsigned long long f64_small_error(unsigned long long u, float r) {
    return (unsigned long long)__double_as_longlong(fabs(__longlong_as_double((long long)u) - (double)r));
}

// Folds the order key of one value (its bits u) into the exact extremes.
__device__ __forceinline__ void f64_extremes(unsigned long long u, unsigned long long& kmin, unsigned long long& kmax) {
    if ((u << 1) > 0xffe0000000000000ull) return;  // NaN
    const unsigned long long k = order_key64(u);
    kmin = min(kmin, k);
    kmax = max(kmax, k);
}

// The exact rounding error of one finite value (bits u, rounded to r), as the
// bits of a double.
__device__ __forceinline__ unsigned long long f64_error(unsigned long long u, float r) {
    const int e = (int)((u >> 52) & 0x7ffu), e32 = e - 1023 + 127;
    const uint32_t rb = __float_as_uint(r);
    if (e == 0x7ff) return 0ull;                                                // infinite or NaN
    if (((rb >> 23) & 0xffu) == 0xffu) return 0x7ff0000000000000ull;            // rounded past the fp32 range
    if (e32 < 1) return f64_small_error(u, r);                                  // zero or fp32-subnormal magnitude
    // |v - r| = |rem - (up ? 2^29 : 0)| * 2^(e-1075), exact in double, as its
    // bit pattern; the rounding went up when r's last bits say so
    const uint32_t rem = (uint32_t)u & 0x1fffffffu;
    const bool up = (rb & 0x7fffffu) != ((uint32_t)(u >> 29) & 0x7fffffu);
    const uint32_t res = up ? 0x20000000u - rem : rem;  // < 2^29
    if (!res) return 0ull;
    const int p = 31 - __clz(res);  // position of the leading bit
    return ((unsigned long long)(e - 52 + p) << 52) | (((unsigned long long)res << (52 - p)) & 0xfffffffffffffull);
}

__device__ __forceinline__ unsigned long long warp_reduce64(unsigned long long v, bool want_max) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
        v = want_max ? max(v, w) : min(v, w);
    }
    return v;
}

__global__ void __launch_bounds__(kF64Threads, 4) gpz_f64_prepass_kernel(const __grid_constant__ F64Args a) {
    __shared__ F64Shared S;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < kMaxFields) {
        S.res[tid][0] = ~0ull;
        S.res[tid][1] = S.res[tid][2] = 0ull;
    }
    __syncthreads();
    const uint64_t nb = (a.n + kBlock - 1) / kBlock, items = nb * (uint64_t)a.F;
    const uint64_t per = (items + gridDim.x - 1) / gridDim.x;  // this CTA's run of consecutive items
    const uint64_t end = min(items, (uint64_t)(blockIdx.x + 1) * per);
    int field = -1;
    unsigned long long kmin = ~0ull, kmax = 0ull, dmax = 0ull;  // exact, per lane, over `field`
    float rmin = INFINITY, rmax = -INFINITY, thr = 0.0f;        // the filters, the same in every lane
    auto flush = [&] {
        if (field < 0) return;
        kmin = warp_reduce64(kmin, false);
        kmax = warp_reduce64(kmax, true);
        dmax = warp_reduce64(dmax, true);
        if (lane == 0) {
            atomicMin(&S.res[field][0], kmin);
            atomicMax(&S.res[field][1], kmax);
            atomicMax(&S.res[field][2], dmax);
        }
    };
    for (uint64_t it = (uint64_t)blockIdx.x * per + warp; it < end; it += kF64Threads / 32) {
        const int f = (int)(it / nb);
        const uint64_t b = it - (uint64_t)f * nb;
        if (f != field) {
            flush();
            field = f;
            kmin = ~0ull;
            kmax = dmax = 0ull;
            rmin = INFINITY;
            rmax = -INFINITY;
            thr = 0.0f;
        }
        const unsigned long long* x = reinterpret_cast<const unsigned long long*>(a.in[f]) + b * kBlock;
        float* y = a.out32[f] + b * kBlock;  // 16-byte aligned
        const int n_b = (int)min((uint64_t)kBlock, a.n - b * kBlock);
        const bool vec = n_b == kBlock && (reinterpret_cast<uintptr_t>(x) & 15u) == 0;
        // lane's values of group k: two pairs when the block is whole and
        // aligned; else four values a warp apart, those past the block
        // standing for its first value
        auto load = [&](int k, unsigned long long (&v)[4]) {
            if (vec) {
                const ulonglong2* p = reinterpret_cast<const ulonglong2*>(x) + 64 * k + lane;
                const ulonglong2 p0 = __ldcs(p), p1 = __ldcs(p + 32);
                v[0] = p0.x;
                v[1] = p0.y;
                v[2] = p1.x;
                v[3] = p1.y;
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int i = 128 * k + 32 * j + lane;
                    v[j] = __ldcs(x + (i < n_b ? i : 0));
                }
            }
        };
        float blo = INFINITY, bhi = -INFINITY;
        bool nonfinite = false;
        unsigned long long next[4];
        load(0, next);
#pragma unroll 1
        for (int k = 0; k < kBlock / 128; ++k) {
            if (128 * k >= n_b) break;
            unsigned long long v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = next[j];
            if (128 * (k + 1) < n_b) load(k + 1, next);
            float r[4], g[4];
            bool slow = false;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                // fp32-normal magnitude (below the last binade): round to nearest
                // even on the bits; the error is res units of 2^(e32-179)
                const uint32_t hi = (uint32_t)(v[j] >> 32), low = (uint32_t)v[j];
                const uint32_t m = __funnelshift_l(low, hi, 3) + 0x40000000u;  // e32 << 23 | fraction
                const uint32_t rem = low & 0x1fffffffu;
                const uint32_t rb = m + ((rem + 0x0fffffffu + (m & 1u)) >> 29);
                const bool in = ((hi >> 20) & 0x7ffu) - 897u < 253u;  // 1 <= e32 <= 253
                const int res = abs((int)(rem - ((rb - m) << 29)));
                g[j] = __fmul_rn(__int2float_rn(res), __uint_as_float(m & 0x7f800000u));
                r[j] = __uint_as_float((rb & 0x7fffffffu) | (hi & 0x80000000u));
                slow |= !in;
            }
            if (slow) {  // zeros, subnormals, the last binade and beyond, NaN: every value once more
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    r[j] = f64_round_any(v[j]);
                    g[j] = 0.0f;
                    nonfinite |= !(fabsf(r[j]) <= 3.402823466e38f);
                }
            }
            const float lo4 = fminf(fminf(r[0], r[1]), fminf(r[2], r[3]));
            const float hi4 = fmaxf(fmaxf(r[0], r[1]), fmaxf(r[2], r[3]));
            const float g4 = fmaxf(fmaxf(g[0], g[1]), fmaxf(g[2], g[3]));
            if (vec) {
                float2* q = reinterpret_cast<float2*>(y) + 64 * k + lane;
                q[0] = make_float2(r[0], r[1]);
                q[32] = make_float2(r[2], r[3]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int i = 128 * k + 32 * j + lane;
                    if (i < n_b) y[i] = r[j];
                }
            }
            blo = fminf(blo, lo4);
            bhi = fmaxf(bhi, hi4);
            const bool px = slow || lo4 <= rmin || hi4 >= rmax;
            if (__any_sync(0xffffffffu, px)) {
                if (px) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) f64_extremes(v[j], kmin, kmax);
                }
                rmin = fminf(rmin, warp_min_f32(lo4));
                rmax = fmaxf(rmax, warp_max_f32(hi4));
            }
            const bool pd = slow || (g4 > 0.0f && g4 >= thr);
            if (__any_sync(0xffffffffu, pd)) {
                if (pd) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) dmax = max(dmax, f64_error(v[j], r[j]));
                }
                // errors below the largest approximation by more than both
                // approximations' error cannot be the largest
                thr = fmaxf(thr, __fmul_rn(warp_max_f32(g4), 1.0f - 0x1p-21f));
            }
        }
        blo = warp_min_f32(blo);
        bhi = warp_max_f32(bhi);
        nonfinite = __any_sync(0xffffffffu, nonfinite);
        if (lane == 0)
            a.bext[b * (uint64_t)a.F + f] =
                nonfinite ? make_uint2(0u, 0u) : make_uint2(f64_order_key32(blo), f64_order_key32(bhi));
    }
    flush();
    __syncthreads();
    if (tid < a.F && S.res[tid][0] != ~0ull) {
        atomicMax(a.res + 3 * tid, ~S.res[tid][0]);
        atomicMax(a.res + 3 * tid + 1, S.res[tid][1]);
        atomicMax(a.res + 3 * tid + 2, S.res[tid][2]);
    }
}

}  // namespace gpz

namespace {

constexpr uint64_t kF64Align = 256;
constexpr uint64_t kResBytes = 256;  // 3 x 8 fields x 8 bytes

uint64_t f32_ld(uint64_t n) { return align_up(n, 4); }
uint64_t f32_bytes(uint64_t n, int F) { return align_up(4ull * f32_ld(n) * (uint64_t)F, kF64Align); }
unsigned f64_grid(uint64_t n, int F) {
    const uint64_t want = (nblocks_of(n) * (uint64_t)F + kF64Threads / 32 - 1) / (kF64Threads / 32);  // a warp per block and field
    const uint64_t cap = 152ull * 4ull;  // one wave: 4 CTAs per SM of a GB300
    return (unsigned)(want < 1 ? 1 : (want < cap ? want : cap));
}

double from_key64(unsigned long long k) {
    const unsigned long long u = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    double d;
    std::memcpy(&d, &u, 8);
    return d;
}

}  // namespace

extern "C" {

uint64_t gpz_compress_f64_workspace_size(uint64_t n, int n_fields) {
    const uint64_t c = gpz_compress_workspace_size(n, n_fields);
    if (c == 0) return 0;
    const uint64_t narrow = align_up(c, kF64Align) + kResBytes + f32_bytes(n, n_fields);
    const uint64_t wide = wide_workspace_size(n, n_fields);  // the 64-bit form, when fp32 cannot hold the bound
    return narrow > wide ? narrow : wide;
}

uint64_t gpz_decompress_f64_workspace_size(uint64_t n, int n_fields) {
    (void)n;
    if (n_fields < 1 || n_fields > kMaxFields) return 0;
    return align_up(gpz_decompress_workspace_size(), kF64Align);  // the status word
}

gpz_status gpz_compress_f64(const double* const* d_fields, uint64_t n, const gpz_params* p, void* d_out,
                            uint64_t out_capacity, uint64_t* d_out_size, uint64_t* h_out_size, uint32_t* d_perm,
                            void* d_ws, uint64_t ws_size, double* h_eb_used, void* stream) {
    // everything that either form checks: wide_compress takes its arguments as
    // checked, and the data decides which form runs
    if (!p || p->n_fields < 1 || p->n_fields > kMaxFields || p->seg_bits < 0 || p->seg_bits > kMaxSegBits ||
        (p->mode != GPZ_EB_ABS && p->mode != GPZ_EB_REL) || !d_out || !aligned(d_out, 4) ||
        (d_perm && !aligned(d_perm, 4)))
        return GPZ_ERR_INVALID_ARG;
    const int F = p->n_fields;
    for (int f = 0; f < F; ++f)
        if (!(p->eb[f] > 0.0) || !std::isfinite(p->eb[f])) return GPZ_ERR_INVALID_ARG;
    if (n > 0) {
        if (!d_fields) return GPZ_ERR_INVALID_ARG;
        for (int f = 0; f < F; ++f)
            if (!d_fields[f] || (reinterpret_cast<uintptr_t>(d_fields[f]) & 7u)) return GPZ_ERR_INVALID_ARG;
    }
    const uint64_t need = gpz_compress_f64_workspace_size(n, F);
    if (need == 0) return GPZ_ERR_INVALID_ARG;
    if (!d_ws || ws_size < need) return d_ws ? GPZ_ERR_CAPACITY : GPZ_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(d_ws) % kF64Align) return GPZ_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    uint8_t* ws = static_cast<uint8_t*>(d_ws);
    const uint64_t cws = align_up(gpz_compress_workspace_size(n, F), kF64Align);
    unsigned long long* res = reinterpret_cast<unsigned long long*>(ws + cws);
    float* y = reinterpret_cast<float*>(ws + cws + kResBytes);
    const uint64_t ld = f32_ld(n);

    // the prepass: the fp32 copy, the fp64 extremes and the largest rounding error
    if (cudaMemsetAsync(res, 0, 24ull * F, s) != cudaSuccess) return GPZ_ERR_CUDA;
    F64Args fa{};
    fa.F = F;
    fa.n = n;
    fa.res = res;
    fa.bext = reinterpret_cast<uint2*>(ws + compress_range_targets(n, F).bext);  // where compress_impl reads them
    for (int f = 0; f < F; ++f) {
        fa.in[f] = n ? d_fields[f] : nullptr;
        fa.out32[f] = y + (uint64_t)f * ld;
    }
    if (n > 0) {
        Recorder rec(s);
        rec.begin(1);
        gpz_f64_prepass_kernel<<<f64_grid(n, F), kF64Threads, 0, s>>>(fa);
        if (cudaGetLastError() != cudaSuccess) return GPZ_ERR_CUDA;
        rec.mark("f64");
    }
    unsigned long long got[3 * kMaxFields];
    if (cudaMemcpyAsync(got, res, 24ull * F, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return GPZ_ERR_CUDA;

    // the reduced absolute bounds (each step one IEEE double operation)
    double ebp[kMaxFields], ebf[kMaxFields];
    bool narrow = true;
    for (int f = 0; f < F; ++f) {
        double e = p->eb[f];
        const bool any = got[3 * f] != 0ull;  // some value is not NaN
        if (p->mode == GPZ_EB_REL && any) {
            const volatile double range = from_key64(got[3 * f + 1]) - from_key64(~got[3 * f]);
            if (range > 0.0 && std::isfinite(range)) {
                const volatile double t = p->eb[f] * range;
                if (t > 0.0 && std::isfinite(t)) e = t;
            }
        }
        double delta;
        std::memcpy(&delta, &got[3 * f + 2], 8);
        const volatile double reduced = e - delta;
        ebf[f] = e;
        ebp[f] = reduced;
        if (!(reduced > 0.0) || !std::isfinite(reduced)) narrow = false;
    }
    if (!narrow) {
        // fp32 cannot hold some field's bound: 64-bit intermediates with the bounds eb_f
        if (h_eb_used)
            for (int f = 0; f < F; ++f) h_eb_used[f] = ebf[f];
        return wide_compress(d_fields, n, F, p->seg_bits, p->mode, ebf, d_out, out_capacity, d_out_size, h_out_size,
                             d_perm, d_ws, ws_size, s);
    }
    if (h_eb_used)
        for (int f = 0; f < F; ++f) h_eb_used[f] = ebp[f];
    gpz_params q{};
    q.mode = GPZ_EB_ABS;
    q.n_fields = F;
    q.seg_bits = p->seg_bits;
    q.flags = p->flags;
    for (int f = 0; f < F; ++f) q.eb[f] = ebp[f];
    const float* fields[kMaxFields];
    for (int f = 0; f < F; ++f) fields[f] = y + (uint64_t)f * ld;
    // the compression workspace sits at the start, so gpz_sync_status(d_ws) reads its status
    // (fields_ready: the host has waited for the rounding pass)
    return compress_impl(fields, n, &q, d_out, out_capacity, d_out_size, h_out_size, d_perm, ws, cws, stream, true);
}

gpz_status gpz_decompress_f64(const void* d_in, uint64_t in_size, double* const* d_fields, int n_fields, uint64_t n,
                              void* d_ws, uint64_t ws_size, void* stream) {
    if (n_fields < 1 || n_fields > kMaxFields) return GPZ_ERR_INVALID_ARG;
    const int F = n_fields;
    if (n > 0) {
        if (!d_fields) return GPZ_ERR_INVALID_ARG;
        for (int f = 0; f < F; ++f)
            if (!d_fields[f] || (reinterpret_cast<uintptr_t>(d_fields[f]) & 7u)) return GPZ_ERR_INVALID_ARG;
    }
    const uint64_t need = gpz_decompress_f64_workspace_size(n, F);
    if (!d_ws || ws_size < need) return d_ws ? GPZ_ERR_CAPACITY : GPZ_ERR_INVALID_ARG;
    if (reinterpret_cast<uintptr_t>(d_ws) % kF64Align) return GPZ_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    if (d_in && in_size >= 8 && aligned(d_in, 4)) {
        // the stream's version word: version 2 is the 64-bit form
        uint32_t head[2] = {0u, 0u};
        if (cudaMemcpyAsync(head, d_in, 8, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            return GPZ_ERR_CUDA;
        if (head[1] == 2u) return gpz_decompress_wide(d_in, in_size, d_fields, F, n, d_ws, ws_size, stream);
    }
    // version 1: the block decoder stores fp64 directly (each value the fp32
    // reconstruction, widened exactly); the workspace holds the status word
    if (!d_in || !aligned(d_in, 4)) return GPZ_ERR_INVALID_ARG;
    if (in_size % 4 != 0 || in_size < 4ull * kHeaderWords) return GPZ_ERR_CORRUPT;
    const uint64_t nb = (n + kBlock - 1) / kBlock;
    if (nb + (uint64_t)F * n >= (1ull << 32)) return GPZ_ERR_UNSUPPORTED;
    uint32_t* status = static_cast<uint32_t*>(d_ws);
    if (cudaMemsetAsync(status, 0, 4, s) != cudaSuccess) return GPZ_ERR_CUDA;
    if (nb == 0) return GPZ_OK;
    DecArgs da{};
    da.stream = static_cast<const uint32_t*>(d_in);
    da.total_words = in_size / 4;
    for (int f = 0; f < F; ++f) da.out[f] = reinterpret_cast<float*>(d_fields[f]);  // double arrays
    da.n = n;
    da.F = F;
    da.nblocks = (uint32_t)nb;
    da.status = status;
    Recorder rec(s);
    rec.begin(1);
    if (launch_decompress64(da, s) != cudaSuccess) return GPZ_ERR_CUDA;
    rec.mark("decompress");
    return GPZ_OK;
}

}  // extern "C"
