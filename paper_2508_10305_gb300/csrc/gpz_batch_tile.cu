// gpz_batch_tile.cu -- the batched tile compression kernel on groups of chunks with
// 16-byte aligned fields (gpz_batch_tile.cuh).
#include "gpz_batch_tile.cuh"

namespace gpz {

cudaError_t batch_tile_aligned(const BatchCompressArgs* a, int F, int grid, cudaStream_t s) {
    return batch_tile_layout<kTileAligned>(a, F, grid, s);
}

}  // namespace gpz
