// gpz_qse_tile.cu -- the fused compression kernel (quantisation, sorting,
// encoding; Sections 4.1-4.3) of single-array calls, with the block's input in shared memory instead of registers.
//
// One CTA of 128 threads owns one block of 1024 particles, eight per thread:
//   - lane f of warp 0 loads field f's 1024 values into a shared tile with one
//     bulk copy, completing on an mbarrier (the few values of a ragged last
//     block beyond a multiple of four are loaded by plain loads);
//   - lanes 0..F-1 of warp 0 derive their field's constants (minimum, code
//     width, segment split, place in the key) once, into shared memory: with a
//     relative bound from the block extremes of the range pass, loaded with
//     the field's step constants in one round trip while the tile is in
//     flight; otherwise from the tile, a warp per field;
//   - each thread quantises its 8 particles of every field from the tile;
//   - once every value is quantised the tile is dead, and the encoded
//     block's staging words are assembled in the same bytes, then written to
//     the block's temporary slot by one bulk copy.
// What bounds it: instruction issue (71% of the issue slots busy with three
// fields, 62% with six) and shared-memory wavefronts (55% and 69% of their
// peak).
// Why 128 threads: whatever a block costs
// per warp rather than per particle (the constants' loads, the scan over
// (bin, warp), the barriers) halves against 256 threads of four particles,
// and eight independent particles per thread hide more latency than the
// second half of the warps did.  Per block 4,740 warp instructions instead of
// 7,200 (six fields), 1,330 shared-memory wavefronts instead of 1,980.
// Measured on a 2^26 x 6 snapshot (relative bound): 0.577 -> 0.472 ms; on
// 10^8 x 3 scan points (absolute bound): 0.750 -> 0.533 ms.
// Ranks: match runs once per distinct key of a warp's 32 and its unit was 62%
// busy on the snapshot.  Where the keys are mostly distinct the ranks are
// the old counts that shared atomics return; the order in which the hardware
// serves the lanes of one instruction is not defined, so the sorted order is
// checked and a block it fails goes to the general kernel (none has).  The
// snapshot 0.472 -> 0.391 ms, 2^25 x 3 uniform positions 0.340 -> 0.170 ms.
// Two values at a time (packed fp32 operations): the scan 0.498 -> 0.487 ms, a
// snapshot at a tight bound (checked candidates) 0.135 -> 0.131, others equal.
// (The decoder got slower with them: 0.318 -> 0.324 on the snapshot.)
// Fallback candidates (values whose rounding is near the bound) are coded in
// place, in a second pass of the warps that have one, instead of redoing the
// block in the general kernel: the scan (2% of its blocks) 0.533 -> 0.502 ms.
// Residency: for three fields nine CTAs per SM (56 registers) measured best, 7
// / 8 / 9 / 10 / 12 CTAs: 0.565 / 0.544 / 0.533 / 0.540 / 0.550 ms on the scan
// (and with the later steps 7 / 8 / 9: 0.539 / 0.518 / 0.502 ms).  For six fields
// shared memory decides: with the histograms in the tile's first row eight
// CTAs fit instead of seven, the snapshot 0.396 -> 0.377 ms.
//
// With a relative bound the block's extremes come from the range pass and
// must bound the block's values (they are exact there): codes are monotone in
// the value, so every code then fits the width derived from the maximum, and
// every key stays below 2^keybits, which the histogram's indexing relies on.
//
// Blocks the fast path cannot take (a fallback candidate that could change
// its field's width, or none that passes, a code >= 2^23, a record > 128 bits) go to the general kernel's list; blocks
// with a non-finite value or no gain are stored raw -- both exactly as in
// gpz_qse_block.cuh.
#include "gpz_qse_tile_launch.cuh"

namespace gpz {

// Fields that are all 16-byte aligned take the kernel without shifts.
cudaError_t launch_qse_tile(const QseArgs& a, bool early, cudaStream_t s) {
    if (a.nblocks == 0) return cudaSuccess;
    if (a.interleaved) return launch_qse_tile_aos(a, early, s);  // gpz_aos.cu
    for (int f = 0; f < a.F; ++f)
        if (reinterpret_cast<uintptr_t>(a.fields[f]) & 15u) return launch_qse_tile_unaligned(a, early, s);
    return launch_qse_tile_layout<kTileAligned>(a, early, s);
}

}  // namespace gpz
