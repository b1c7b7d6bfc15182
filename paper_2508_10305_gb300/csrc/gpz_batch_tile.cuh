// gpz_batch_tile.cuh -- the batched compression kernel with the shared-memory
// tile body, instantiated per layout of the tile (gpz_batch_tile.cu,
// gpz_batch_tile_unaligned.cu: a translation unit each, so that they compile
// in parallel).
#pragma once

#include "gpz_batch_args.cuh"
#include "gpz_qse_tile.cuh"

namespace gpz {

// One CTA per block of the group: the tile kernel's code, with the chunk's
// arguments in shared memory, in the layout that every chunk of the group
// allows.
template <int F, bool PRE, int LAY, class Idx = SlotBlock>
__global__ void __launch_bounds__(kTileThreads, tile_ctas(F, LAY)) gpz_batch_tile_kernel(BatchCompressArgs g) {
    extern __shared__ __align__(128) uint8_t dsm[];
    __shared__ TileShared S;
    __shared__ QseArgs A;
    __shared__ uint32_t slot[2];  // block within its chunk, global block id
    const uint32_t gb = g.block_first + blockIdx.x;
    load_chunk_args(g, __ldg(g.block_map + gb), gb, A, slot);
    __syncthreads();
    const Idx idx{slot};
    if ((uint64_t)(idx.b() + 1) * kBlock <= A.n)
        qse_block_tile<F, true, PRE, LAY>(A, dsm, S, idx);
    else
        qse_block_tile<F, false, PRE, LAY>(A, dsm, S, idx);
}

template <int F, bool PRE, int LAY>
cudaError_t launch_batch_tile_fp(const BatchCompressArgs* a, int grid, cudaStream_t s) {
    auto kern = gpz_batch_tile_kernel<F, PRE, LAY>;
    if (!a) {  // the kernel's attributes
        const cudaError_t e =
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tile_smem_bytes(F, LAY));
        if (e != cudaSuccess) return e;
        return cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    }
    kern<<<grid, kTileThreads, tile_smem_bytes(F, LAY), s>>>(*a);
    return cudaGetLastError();
}

// Launch for field count F, or (a == nullptr) set the attributes of F's kernels.
template <int LAY>
cudaError_t batch_tile_layout(const BatchCompressArgs* a, int F, int grid, cudaStream_t s) {
    switch (F) {
#define GPZ_CASE(FF)                                                                      \
    case FF: {                                                                            \
        if (a) return a->pre ? launch_batch_tile_fp<FF, true, LAY>(a, grid, s)            \
                             : launch_batch_tile_fp<FF, false, LAY>(a, grid, s);          \
        const cudaError_t e = launch_batch_tile_fp<FF, true, LAY>(nullptr, 0, s);         \
        return e != cudaSuccess ? e : launch_batch_tile_fp<FF, false, LAY>(nullptr, 0, s); \
    }
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
