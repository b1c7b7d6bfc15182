// gpz_qse.cu -- the global range pass of the relative error bound, and the
// general compression kernel for the rare blocks that the fused kernels leave
// (codes >= 2^23, records wider than 128 bits, a fallback candidate that
// changes a field's width; Sections 4.1-4.3 in gpz_qse_block.cuh).
#include "gpz_qse_block.cuh"

namespace gpz {

// ------------------------------------------------------------------ range pass (relative bound)
//
// Bound by HBM: 1.61 GB of a 2^26 x 6 snapshot in 0.256 ms (6.3 TB/s; 0.263
// before the fold at its end took all fields at once, finish_range).  Fields
// of any alignment are read with 16-byte loads: a 10^7 x 6 snapshot with odd
// rows 62 -> 56 us, 49 with that fold.  As many CTAs as make rounds of equal
// size instead of eight per SM: no change (49 us, 0.257 ms).

// One warp per (block, field) item, field-major, so that consecutive warps
// stream consecutive blocks of a field.  Each item yields the block's
// extremes for the fused kernel (order keys; (0, 0) when the block holds a
// NaN or an infinity in that field) and feeds the CTA's running extremes of
// the field over its non-NaN values.
__global__ void __launch_bounds__(kRangeThreads, 8) gpz_range_kernel(RangeArgs a) {
    __shared__ uint32_t s_lo[kMaxFields], s_hi[kMaxFields];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < kMaxFields) {
        s_lo[tid] = 0xffffffffu;
        s_hi[tid] = 0u;
    }
    __syncthreads();
    const uint64_t nb = (a.n + kBlock - 1) / kBlock;
    const uint64_t items = nb * (uint64_t)a.F;
    const uint64_t nwarps = (uint64_t)gridDim.x * (kRangeThreads / 32);
    for (uint64_t it = (uint64_t)blockIdx.x * (kRangeThreads / 32) + warp; it < items; it += nwarps) {
        const int f = (int)(it / nb);
        const uint64_t b = it - (uint64_t)f * nb;
        const float* x = a.fields[f] + b * kBlock;
        const int n_b = (int)min((uint64_t)kBlock, a.n - b * kBlock);
        float lo, hi;
        const bool nonfinite = block_extremes(x, n_b, lo, hi);
        if (lane == 0) {
            a.bext[b * (uint64_t)a.F + f] = nonfinite ? make_uint2(0u, 0u) : make_uint2(order_key(lo), order_key(hi));
            if (lo <= hi) {  // some value is not NaN
                atomicMin(&s_lo[f], order_key(lo));
                atomicMax(&s_hi[f], order_key(hi));
            }
        }
    }
    __syncthreads();
    finish_range<kRangeThreads>(a, s_lo, s_hi);
}

cudaError_t launch_range(const RangeArgs& a, int grid, cudaStream_t s) {
    gpz_range_kernel<<<grid, kRangeThreads, 0, s>>>(a);
    return cudaGetLastError();
}

// Blocks the fast kernel leaves to the general path (rare): processed by a
// persistent grid walking the list.
template <int F>
__global__ void __launch_bounds__(kThreads, 2) gpz_qse_general_kernel(QseArgs a) {
    extern __shared__ __align__(16) uint8_t dsm[];
    __shared__ QseShared S;
    wait_for_previous_kernel();
    const uint32_t count = *(volatile const uint32_t*)a.general_count;
    for (uint32_t i = blockIdx.x; i < count; i += gridDim.x) {
        const uint32_t entry = a.general_list[i], b = entry & ~kRawBlock;
        if (entry & kRawBlock)
            write_raw<F>(a, b, (int)min((uint64_t)kBlock, a.n - (uint64_t)b * kBlock), threadIdx.x);
        else if ((uint64_t)(b + 1) * kBlock <= a.n)
            qse_block_general<F, true>(a, dsm, S, b);
        else
            qse_block_general<F, false>(a, dsm, S, b);
        __syncthreads();
    }
}

// the blocks left to the general path (usually none); the grid walks the list
template <int F>
cudaError_t launch_qse_general_f(const QseArgs& a, cudaStream_t s) {
    const size_t gsmem = qse_smem_bytes(F);
    if (gsmem + sizeof(QseShared) > 48u * 1024u) {  // beyond a CTA's default limit
        const cudaError_t e =
            cudaFuncSetAttribute(gpz_qse_general_kernel<F>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gsmem);
        if (e != cudaSuccess) return e;
    }
    const unsigned ggrid = a.nblocks < 2u * 152u ? a.nblocks : 2u * 152u;
    return launch_dependent(gpz_qse_general_kernel<F>, ggrid, kThreads, gsmem, s, a);
}

cudaError_t launch_qse_general(const QseArgs& a, cudaStream_t s) {
    if (a.nblocks == 0) return cudaSuccess;
    switch (a.F) {
        case 1: return launch_qse_general_f<1>(a, s);
        case 2: return launch_qse_general_f<2>(a, s);
        case 3: return launch_qse_general_f<3>(a, s);
        case 4: return launch_qse_general_f<4>(a, s);
        case 5: return launch_qse_general_f<5>(a, s);
        case 6: return launch_qse_general_f<6>(a, s);
        case 7: return launch_qse_general_f<7>(a, s);
        case 8: return launch_qse_general_f<8>(a, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace gpz
