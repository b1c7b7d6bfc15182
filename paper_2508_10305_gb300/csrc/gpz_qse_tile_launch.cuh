// gpz_qse_tile_launch.cuh -- the single-array tile compression kernel and its
// launch, instantiated per layout of the tile (gpz_qse_tile.cu describes the
// design).
#pragma once

#include "gpz_qse_tile.cuh"

namespace gpz {

// The last block first: a ragged one runs code of its own (in the caches of
// no SM yet) and would otherwise end the kernel alone; 1.7*10^7 x 3 records
// with 43 in the last block: 102 -> 93 us.
struct LastFirst {
    static constexpr bool kUnstable = false;
    __device__ __forceinline__ uint32_t b() const { return blockIdx.x ? blockIdx.x - 1u : gridDim.x - 1u; }  // block within its array
    __device__ __forceinline__ uint32_t id() const { return b(); }  // entry for the general list
};

struct LastBlock {
    static constexpr bool kUnstable = false;
    __device__ __forceinline__ uint32_t b() const { return gridDim.x - 1u; }
    __device__ __forceinline__ uint32_t id() const { return b(); }
};

template <int F, bool PRE, int LAY, class First = LastFirst, class Last = LastBlock>
__global__ void __launch_bounds__(kTileThreads, tile_ctas(F, LAY)) gpz_qse_tile_kernel(const __grid_constant__ QseArgs a) {
    extern __shared__ __align__(128) uint8_t dsm[];
    __shared__ TileShared S;
    // the grid's last block may be ragged
    if (blockIdx.x != 0u || (uint64_t)gridDim.x * kBlock == a.n)
        qse_block_tile<F, true, PRE, LAY>(a, dsm, S, First{});
    else
        qse_block_tile<F, false, PRE, LAY>(a, dsm, S, Last{});
}

template <int F, bool PRE, int LAY, class First = LastFirst, class Last = LastBlock>
cudaError_t launch_qse_tile_fp(const QseArgs& a, bool early, cudaStream_t s) {
    const size_t smem = tile_smem_bytes(F, LAY);
    auto kern = gpz_qse_tile_kernel<F, PRE, LAY, First, Last>;
    static_assert(tile_smem_bytes(F, LAY) + sizeof(TileShared) <= 48u * 1024u, "within the default limit of a CTA");
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    if (PRE && early) {
        e = launch_dependent(kern, a.nblocks, kTileThreads, smem, s, a);
    } else {
        kern<<<a.nblocks, kTileThreads, smem, s>>>(a);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return e;
    return launch_qse_general(a, s);
}

// One layout's launches (a translation unit each, so that they compile in
// parallel: gpz_qse_tile.cu, gpz_qse_tile_unaligned.cu, gpz_aos.cu).
template <int LAY>
cudaError_t launch_qse_tile_layout(const QseArgs& a, bool early, cudaStream_t s) {
    const bool pre = a.bext != nullptr;
    switch (a.F) {
#define GPZ_CASE(FF) \
    case FF: return pre ? launch_qse_tile_fp<FF, true, LAY>(a, early, s) : launch_qse_tile_fp<FF, false, LAY>(a, early, s);
        GPZ_CASE(1)
        GPZ_CASE(2)
        GPZ_CASE(3)
        GPZ_CASE(4)
        GPZ_CASE(5)
        GPZ_CASE(6)
        GPZ_CASE(7)
        GPZ_CASE(8)
#undef GPZ_CASE
    }
    return cudaErrorInvalidValue;
}

}  // namespace gpz
