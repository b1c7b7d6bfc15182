// gpz_qse_tile_unaligned.cu -- the tile compression kernel on fields of any
// (4-byte) alignment, as the rows of an [F, n] array are when n is not a
// multiple of four.  A 10^7 x 6 snapshot with odd rows (relative bound):
// 120 us in the register kernel that took them before, 86 us here (84 us with
// aligned rows).
#include "gpz_qse_tile_launch.cuh"

namespace gpz {

cudaError_t launch_qse_tile_unaligned(const QseArgs& a, bool early, cudaStream_t s) {
    return launch_qse_tile_layout<kTileUnaligned>(a, early, s);
}

}  // namespace gpz
