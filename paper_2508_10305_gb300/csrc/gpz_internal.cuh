// gpz_internal.cuh -- device-side constants, kernel argument blocks and warp
// helpers of libgpz (sm_103a).  The stream format implemented here is the one
// of include/gpz.h: a 16-word header, (eb, step) per field, a table of block
// word offsets, then one encoded or raw block per 1024 particles.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace gpz {

constexpr int kBlock = 1024;             // particles per block (Section 4.2: 32 threads x 32 points)
constexpr uint32_t kMagic = 0x315A5047u; // 'G','P','Z','1'
constexpr uint32_t kVersion = 1;
constexpr int kHeaderWords = 16;
constexpr int kMaxFields = 8;
constexpr int kMaxSegBits = 3;
constexpr int kMaxBins = 512;            // 2^(3 * kMaxSegBits) linearised segment ids
constexpr int kRow = 33;                 // padded shared-memory row of 32 values
constexpr int kPadWords = 32 * kRow;     // 1056: 1024 values in padded rows
constexpr int kQseThreads = 256;         // one CTA per particle block, 4 particles per thread
constexpr int kDecThreads = 128;         // one CTA per particle block, 8 positions per thread
constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kScanTile = kScanThreads * kScanItems;
constexpr int kRangeThreads = 256;
constexpr int kCompactWarps = 8;

// Status codes written to the workspace status word (values of gpz_status).
constexpr uint32_t kStCapacity = 2;
constexpr uint32_t kStCorrupt = 3;
constexpr uint32_t kStTimeout = 6;

// Limit of every device-side wait on another CTA, in SM cycles (about a
// second at 2 GHz): a wait that runs out records kStTimeout and the waiting
// CTA carries on without the value it waited for.
constexpr long long kWaitCycles = 1ll << 31;

struct FieldParams {
    float eb;    // RN32(eb), stored in the header
    float s;     // quantisation step RN32(eb * 63/32)
    float inv;   // RN32(1 / s): the precomputed reciprocal (Section 5.1)
    float ebchk; // RD32(eb * (1 - 2^-22)): the verification threshold
};

// Argument blocks (passed by value).
struct RangeArgs {
    const float* fields[kMaxFields];
    uint64_t n;
    int F;
    double rel[kMaxFields];
    float2* partials;           // [gridDim.x][F] (min, max)
    uint32_t* done_counter;
    FieldParams* d_params;      // out
    uint2* bext;                // out, [nblocks][F]: each block's extremes (order keys), (0, 0) if non-finite
};

struct QseArgs {
    const float* fields[kMaxFields];
    uint64_t n;
    uint32_t nblocks;
    int F;
    int G;
    int interleaved;            // fields[0] holds F-field records: field f of particle i at fields[0][i * F + f]
    FieldParams params[kMaxFields];
    const FieldParams* d_params; // device constants (relative bound) or nullptr
    const uint2* bext;          // each block's extremes from the range pass, or nullptr
    const unsigned long long* binfo; // each block's widths and flags (gpz_block_info_kernel), or nullptr
    uint32_t* temp;             // [nblocks][slot_words]
    uint32_t slot_words;
    uint32_t* sizes;            // [nblocks] words per block
    uint32_t* sums;             // total words per 2^sum_shift blocks (zeroed), or nullptr (store_size)
    uint32_t sum_shift;
    uint32_t* perm;             // [n] or nullptr
    uint32_t* status;
    uint32_t* general_list;     // [nblocks] blocks left to the general kernel, each at most once
    uint32_t* general_count;    // zeroed
    uint32_t* fallback_count;   // nullable: warps of the tile kernel that took fallback candidates (a measure, not read here)
    // Fused compaction only (gpz_qse_direct_kernel): the stream's payload,
    // the words it can hold, the per-block look-back states (zeroed) and a
    // count of the blocks that could not be placed directly.
    uint32_t* direct;
    uint64_t direct_capacity;
    unsigned long long* bstate;
    uint32_t* deferred_count;
};

// In a general-list entry (a block index below 2^30: no device holds the
// 2^40 particles of more): a block with a value that no candidate brings
// within its bound, to be stored raw.  A block is entered at most once, so the
// list of one word per block cannot overrun: by the kernel that leaves it
// before its sort, or by the check of the sorted order.
constexpr uint32_t kRawBlock = 0x40000000u;

constexpr uint32_t kPlaced = 0x80000000u;  // in a block's word count: already in the stream

// Compaction forms of the per-block code: the temporary slot only (Section
// 4.4's three steps), or fused (placed by the block itself after its
// look-back over its predecessors' published sizes).
constexpr int kCmTemp = 0, kCmDirect = 1;

struct F64Args {                // fp64 input (gpz_f64.cu)
    const double* in[kMaxFields];
    float* out32[kMaxFields];   // 16-byte aligned
    uint64_t n;
    int F;
    unsigned long long* res;    // [F][3]: ~min key, max key, largest rounding error (bits)
    uint2* bext;                // out, [nblocks][F]: each block's fp32 extremes, as RangeArgs
};

struct ScanArgs {
    const uint32_t* sizes;      // [nblocks]
    uint32_t nblocks;
    uint64_t n;                 // particles (a block's size never exceeds its raw size)
    int F;
    uint32_t* table;            // [nblocks + 1] in the stream
    unsigned long long* tile_state; // [ntiles], zeroed
    uint32_t* tile_counter;     // zeroed
    uint32_t* status;
    long long wait_cycles;      // limit of a look-back wait in SM cycles; 0: kWaitCycles
};

// How the blocks' words come to their places in the stream (Section 4.4, steps
// 2 and 3, in one kernel): every block's size was also added to the total of
// its run of 2^sum_shift blocks, so a CTA finds its offset from the totals
// before its run and the sizes before it in the run.
struct PlaceArgs {
    const uint32_t* sums;
    uint32_t sum_shift;
    uint32_t* table;            // out, [nblocks + 1]
    uint32_t raw_fields;        // words per particle of a raw block
    uint32_t log_blocks;        // blocks per CTA, log2 (set by the launch)
};

struct CompactArgs {
    const uint32_t* temp;
    uint32_t slot_words;
    const uint32_t* sizes;
    const uint32_t* table;      // [nblocks + 1]
    uint32_t* stream;           // stream base
    uint32_t payload_start;     // words
    uint32_t nblocks;
    uint64_t n;
    int F;
    int G;
    int mode;
    FieldParams params[kMaxFields];
    const FieldParams* d_params;
    unsigned long long* d_out_size; // nullable
    unsigned long long* ws_out_size; // nullable: the same size, beside the status word
    uint32_t* unplaced;         // nullable: counts the blocks this kernel moves (in-kernel compaction forms)
    uint32_t version;           // header word 1
    uint32_t ext_words;         // nonzero: the header extension is ext[0..ext_words) instead of (eb, s) per field
    uint32_t ext[4 * kMaxFields];
};

struct DecArgs {
    const uint32_t* stream;
    uint64_t total_words;
    float* out[kMaxFields];
    uint64_t n;
    int F;
    uint32_t nblocks;
    uint32_t* status;
    int interleaved;            // out[0] receives F-field records: field f of particle i at out[0][i * F + f]
};

// The constants of one field under a relative bound rel, from the field's
// range [lo, hi] (lo > hi when the field holds no value): eb = rel * (hi - lo)
// when that is a finite positive number, else eb = rel; then the step
// eb * 63/32, its reciprocal and the verification threshold, all from the
// double eb (one rounding each).
__device__ __forceinline__ FieldParams range_params(float lo, float hi, double rel) {
    double eb = rel;
    if (lo <= hi) {
        const double range = (double)hi - (double)lo;
        if (range > 0.0 && range < HUGE_VAL) {
            const double e = rel * range;
            if (e > 0.0 && e < HUGE_VAL) eb = e;
        }
    }
    FieldParams p;
    p.eb = __double2float_rn(eb);
    p.s = __double2float_rn(eb * 1.96875);
    p.inv = __double2float_rn(1.0 / (double)p.s);
    p.ebchk = __double2float_rd(eb * (1.0 - 0x1p-22));
    return p;
}

// ---------------------------------------------------------------- helpers

// fp64 operations run at 1/64 of the fp32 rate here (a warp's takes 16 cycles
// of its SM, also with every lane predicated off), so they stay out of paths
// that only move or compare bits: rare conversions sit behind a call, and
// values whose bits are worked on are loaded as integers -- masks on the bits
// of a loaded double become fp64 negations and absolute values.

// ceil(2^32 / d) for d = 1..255 (entry 0 unused), built at compile time: with
// m = ceil(2^32 / d), floor(n / d) = floor(n * m / 2^32) exactly for n < 2^18
// (the multiply's relative error stays below 2^-14 < 1/d).
struct DivMagic {
    unsigned long long m[256];
    constexpr DivMagic() : m() {
        for (int d = 1; d < 256; ++d) m[d] = ((1ull << 32) + (unsigned long long)d - 1ull) / (unsigned long long)d;
    }
};
__constant__ DivMagic kDivMagic = DivMagic();

// floor(n / d) for n < 2^18, 1 <= d <= 255.
__device__ __forceinline__ uint32_t div_small(uint32_t n, uint32_t d) {
    const unsigned long long m = kDivMagic.m[d];
    return __umulhi(n, (uint32_t)m) + ((m >> 32) ? n : 0u);
}

// A block's final size, and its share of its run's total.
__device__ __forceinline__ void store_size(uint32_t* sizes, uint32_t* sums, uint32_t shift, uint32_t b, uint32_t words) {
    sizes[b] = words;
    if (sums) atomicAdd(sums + (b >> shift), words);
}

__device__ __forceinline__ void set_status(uint32_t* st, uint32_t code) {
    atomicCAS(st, 0u, code);
}

__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

__device__ __forceinline__ uint32_t lanemask_le() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_le;" : "=r"(m));
    return m;
}

__device__ __forceinline__ int pad_idx(int j) { return (j >> 5) * kRow + (j & 31); }

__device__ __forceinline__ uint32_t bit_width(uint32_t v) { return 32u - (uint32_t)__clz(v); }

__device__ __forceinline__ uint32_t ceil_words(uint32_t bits) { return (bits + 31u) >> 5; }

__device__ __forceinline__ uint32_t warp_max_u32(uint32_t v) {
    return __reduce_max_sync(0xffffffffu, v);
}

__device__ __forceinline__ uint32_t warp_sum_u32(uint32_t v) {
    return __reduce_add_sync(0xffffffffu, v);
}

__device__ __forceinline__ float warp_min_f32(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__device__ __forceinline__ float warp_max_f32(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Inclusive prefix sum over the warp.
__device__ __forceinline__ uint32_t warp_incl_sum(uint32_t v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Inclusive prefix maximum over the warp (signed).
__device__ __forceinline__ int warp_incl_max(int v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v = max(v, t);
    }
    return v;
}

// Two fp32 values in one register pair: the packed operations round each half
// as the scalar ones do, and take one issue slot for both.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 add2_rn(f32x2 a, f32x2 b) {
    f32x2 v;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
    return v;
}
__device__ __forceinline__ f32x2 add2_rd(f32x2 a, f32x2 b) {
    f32x2 v;
    asm("add.rm.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
    return v;
}
__device__ __forceinline__ f32x2 fma2_rn(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 v;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(v) : "l"(a), "l"(b), "l"(c));
    return v;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// ---------------------------------------------------------------- mbarrier + bulk copy global -> shared

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Arrive (the one expected arrival) and announce `bytes` of bulk copies.
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0;
}

// Wait for phase `parity` of the mbarrier, for at most kWaitCycles SM
// cycles; on expiry record kStTimeout, wait once more as long (so that bulk
// copies still in flight into this CTA's shared memory are not left behind
// by an exiting CTA), and return false.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, uint32_t* status) {
    long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (clock64() - t0 > kWaitCycles) {
            set_status(status, kStTimeout);
            t0 = clock64();
            while (!mbar_try_wait(bar, parity))
                if (clock64() - t0 > kWaitCycles) break;
            return false;
        }
    }
    return true;
}

// One-dimensional bulk copy global -> shared, completing on the mbarrier.
// Both addresses 16-byte aligned, bytes a multiple of 16.  The data is read
// once: it leaves L2 first, which keeps the slots that the copy kernel reads
// next (2^26 x 6 snapshot: copy 155.9 -> 154.7 us) and the lines a decoder has
// yet to write back (10^8 x 3 scan 351 -> 344 us).
__device__ __forceinline__ void bulk_g2s(void* smem_dst, const void* gmem_src, uint32_t bytes, uint64_t* bar) {
    unsigned long long pol;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
            smem_u32(smem_dst)),
        "l"(gmem_src), "r"(bytes), "r"(smem_u32(bar)), "l"(pol)
        : "memory");
}

// ---------------------------------------------------------------- bulk copy shared -> global (async proxy)

// Orders this thread's earlier shared-memory writes before later reads of
// them by the async proxy (a bulk copy issued after a barrier).
__device__ __forceinline__ void fence_proxy_async_shared() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// One thread: copy `bytes` (a multiple of 16) from shared memory to global
// memory, both 16-byte aligned, with one bulk copy, and wait until the copy
// has read its source (so that the CTA may exit or reuse the words).
__device__ __forceinline__ void bulk_s2g_start(void* gdst, const void* ssrc, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gdst), "r"(smem_u32(ssrc)),
                 "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void bulk_s2g_wait() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_s2g(void* gdst, const void* ssrc, uint32_t bytes) {
    bulk_s2g_start(gdst, ssrc, bytes);
    bulk_s2g_wait();
}

// ---------------------------------------------------------------- acquire / release (look-back scan)

// A look-back reads other CTAs' published states with relaxed loads: the
// value it needs is in the state word itself, and a gpu-scope acquire load
// would also invalidate the SM's L1 for every CTA resident there.  A reader
// that goes on to read data the state vouches for issues one fence first.
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release_u64(unsigned long long* p, unsigned long long v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// ---------------------------------------------------------------- dependent launches

// Launch a kernel that may be set up while the kernel before it on the stream
// still ends (programmatic dependent launch).  The kernel calls
// wait_for_previous_kernel() before it writes anything and before it reads
// anything that the kernel before it, or one that this one may in turn have
// overtaken, writes; what the wait guards is read with load_after_wait (or
// plain loads), never through the read-only path, whose data must not change
// while a kernel runs.  Launched ordinarily, the same kernel's wait returns at
// once.
template <class... P, class... A>
cudaError_t launch_dependent(void (*kern)(P...), unsigned grid, unsigned threads, size_t smem, cudaStream_t s, A&&... args) {
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &attr;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kern, static_cast<P>(args)...);
}

__device__ __forceinline__ void wait_for_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ uint32_t load_after_wait(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint2 load_after_wait(const uint2* p) {
    uint2 v;
    asm volatile("ld.global.cg.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
    return v;
}

// ---------------------------------------------------------------- launch wrappers (defined in the .cu files)

cudaError_t launch_range(const RangeArgs& a, int grid, cudaStream_t s);
cudaError_t launch_qse_direct(const QseArgs& a, cudaStream_t s);  // register kernel placing blocks directly, then the general list
cudaError_t launch_qse_general(const QseArgs& a, cudaStream_t s);
// Shared-memory tile kernel, then the general list.  early: nothing that this call
// enqueued may still be writing the fields (a transpose into the workspace
// would), so the tile may be loaded while the work before it on the stream ends.
cudaError_t launch_qse_tile(const QseArgs& a, bool early, cudaStream_t s);
cudaError_t launch_qse_tile_unaligned(const QseArgs& a, bool early, cudaStream_t s);  // the same on 4-byte aligned fields
cudaError_t launch_qse_tile_aos(const QseArgs& a, bool early, cudaStream_t s); // the same on interleaved records (16-byte aligned)
cudaError_t launch_decompress_aos(const DecArgs& a, cudaStream_t s); // decompression into interleaved records
cudaError_t launch_block_info(const uint2* bext, const FieldParams* d_params, uint32_t nblocks, int F,
                              unsigned long long* binfo, cudaStream_t s);
cudaError_t launch_scan(const ScanArgs& a, cudaStream_t s, unsigned grid = 0);  // grid 0: one CTA per tile
cudaError_t launch_compact(const CompactArgs& a, cudaStream_t s);
cudaError_t launch_place(const CompactArgs& a, const PlaceArgs& p, cudaStream_t s);  // scan and copy in one
cudaError_t launch_decompress(const DecArgs& a, cudaStream_t s);

}  // namespace gpz
