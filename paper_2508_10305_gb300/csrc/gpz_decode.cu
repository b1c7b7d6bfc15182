// gpz_decode.cu -- GPZ decompression (Section 3.2, last paragraph: the
// reverse of compression without sorting; Table 1 "Decompression").
//
// One CTA of 128 threads per 1024-particle block; thread t rebuilds sorted
// positions 4t..4t+3 and 512+4t..512+4t+3.  Per CTA:
//   1. the block's table entries (one round trip), then its words after the
//      block header by one bulk copy into shared memory (an mbarrier with a
//      bounded wait), while warp 0 checks the stream header, the table
//      entries and the block header;
//   2. raw block: copy the stored values;
//   3. encoded block: every thread extracts its four deltas and four counts
//      from two 64-bit windows; a CTA-wide prefix sum gives the unique
//      segment ids and the run starts, which are marked in a 1024-bit mask;
//   4. the run of position j is the number of run starts <= j (popcount of
//      the mask prefix); its key is the run's id; the record at bit j*W
//      gives the segment offsets and extra-field codes; every value is
//      rebuilt as fma(q, step, min) and stored, four consecutive ones at once.
// What bounds it: with six fields HBM (2.06 GB of a 2^26-particle snapshot in
// 0.313 ms, 6.6 TB/s), with three the issue slots (67% busy) and the integer
// pipe (71%).  Why 128 threads: what a block costs per warp rather than per
// position (the checks' barrier, the scan, the mask, the fields' constants)
// is half of what 256 threads of four positions paid: 6,220 -> 4,160 warp
// instructions per block with six fields, 5,070 -> 3,190 with three.
// Measured: 2^26 x 6 snapshot 0.420 -> 0.317 ms (0.313 with the later steps),
// 10^8 x 3 scan points 0.514 -> 0.358 ms (0.319).
// Every read stays inside the stream, every failed check sets
// GPZ_ERR_CORRUPT in the status word, and the kernel never traps.
#include "gpz_decode_block.cuh"

namespace gpz {

// Where the arguments lie is a matter of measurement: read from the parameter
// bank for aligned fields and doubles (2^26 x 6: 0.319 -> 0.314 ms, 2^23 x 6
// doubles 0.084 -> 0.079), from a copy for fields of any alignment, whose stores index
// the field pointers more often (3*10^7 x 3: 0.128 from the bank, 0.113 from a copy).
template <int F, int OUT>
__global__ void __launch_bounds__(kDecThreads, dec_ctas(F)) gpz_decompress_kernel(const __grid_constant__ DecArgs a) {
    __shared__ DecShared<F> S;
    decode_block<F, OUT, false>(a, S, DecGridBlock{});
}
template <int F>
__global__ void __launch_bounds__(kDecThreads, dec_ctas(F)) gpz_decompress_any_kernel(DecArgs a) {
    __shared__ DecShared<F> S;
    decode_block<F, kOutAny, false>(a, S, DecGridBlock{});
}

template <int F, int OUT>
void launch_decompress_f(const DecArgs& a, cudaStream_t s) {
    if constexpr (OUT == kOutAny)
        gpz_decompress_any_kernel<F><<<a.nblocks, kDecThreads, 0, s>>>(a);
    else
        gpz_decompress_kernel<F, OUT><<<a.nblocks, kDecThreads, 0, s>>>(a);
}

template <int OUT>
cudaError_t launch_decompress_out(const DecArgs& a, cudaStream_t s) {
    if (a.nblocks == 0) return cudaSuccess;
    switch (a.F) {
        case 1: launch_decompress_f<1, OUT>(a, s); break;
        case 2: launch_decompress_f<2, OUT>(a, s); break;
        case 3: launch_decompress_f<3, OUT>(a, s); break;
        case 4: launch_decompress_f<4, OUT>(a, s); break;
        case 5: launch_decompress_f<5, OUT>(a, s); break;
        case 6: launch_decompress_f<6, OUT>(a, s); break;
        case 7: launch_decompress_f<7, OUT>(a, s); break;
        case 8: launch_decompress_f<8, OUT>(a, s); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

static bool all_aligned(const DecArgs& a) {
    for (int f = 0; f < a.F; ++f)
        if (reinterpret_cast<uintptr_t>(a.out[f]) & 15u) return false;
    return true;
}

cudaError_t launch_decompress(const DecArgs& a, cudaStream_t s) {
    if (a.nblocks == 0) return cudaSuccess;
    if (a.interleaved) return launch_decompress_aos(a, s);  // gpz_aos.cu
    return all_aligned(a) ? launch_decompress_out<kOut32>(a, s) : launch_decompress_out<kOutAny>(a, s);
}

// The same decoder storing fp64 (gpz_decompress_f64 on a version-1 stream):
// a.out[f] holds the address of field f's double array, and every value is
// the fp32 reconstruction widened exactly.
cudaError_t launch_decompress64(const DecArgs& a, cudaStream_t s) {
    return launch_decompress_out<kOut64>(a, s);
}

}  // namespace gpz
