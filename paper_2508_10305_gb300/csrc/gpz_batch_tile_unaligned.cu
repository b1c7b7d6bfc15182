// gpz_batch_tile_unaligned.cu -- the batched tile compression kernel on groups of chunks with
// fields of any (4-byte) alignment (gpz_batch_tile.cuh).
#include "gpz_batch_tile.cuh"

namespace gpz {

cudaError_t batch_tile_unaligned(const BatchCompressArgs* a, int F, int grid, cudaStream_t s) {
    return batch_tile_layout<kTileUnaligned>(a, F, grid, s);
}

}  // namespace gpz
