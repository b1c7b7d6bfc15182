// gpz_testhooks.cu -- the failure-injection hooks of include/gpz_test.h: an
// allocation-failure counter read by every device allocation of the library,
// and launches of the look-back kernels with a predecessor that never
// publishes and a short wait limit, so that tests see the bounded waits run
// out (and the GPU keep answering) without any fault; and compression with
// every block's sort treated as failing its check.
#include <atomic>
#include <vector>

#include "gpz.h"
#include "gpz_batch_core.hpp"
#include "gpz_batch_tile.cuh"
#include "gpz_host.hpp"
#include "gpz_qse_block.cuh"
#include "gpz_qse_tile_launch.cuh"
#include "gpz_test.h"

namespace gpz {
namespace host {
std::atomic<int> g_fail_allocs{0};
}  // namespace host
}  // namespace gpz

using namespace gpz;
using namespace gpz::host;

namespace gpz {

namespace {

constexpr uint32_t kTestBlocks = 2u * (uint32_t)kScanTile + 1u;  // nblocks + 1 items: three tiles
constexpr uint32_t kTestTiles = 3u;
constexpr uint64_t kA = 256;

// Workspace of the scan test: control words (status, tile counter), the tile
// states, the block sizes and the offsets (64-bit, enough for either scan).
struct ScanTestLayout {
    uint64_t ctrl = 0, states = 256, sizes, offsets, total;
    ScanTestLayout() {
        sizes = states + align_up(kTestTiles * 8ull, kA);
        offsets = sizes + align_up(kTestBlocks * 4ull, kA);
        total = offsets + align_up((kTestBlocks + 1ull) * 8ull, kA);
    }
};

__global__ void gpz_test_lookback_kernel(const unsigned long long* bstate, uint32_t b, long long limit,
                                         uint32_t* result) {
    const uint32_t off = block_lookback(bstate, b, limit);
    if (threadIdx.x == 0) *result = off == kNotPlaced ? 0u : 1u;
}

// Three fields, every block's sort failing its check.
struct UnstableFirst : LastFirst {
    static constexpr bool kUnstable = true;
};
struct UnstableLast : LastBlock {
    static constexpr bool kUnstable = true;
};
struct UnstableSlot : SlotBlock {
    static constexpr bool kUnstable = true;
};

template <bool PRE, int LAY>
cudaError_t unstable_tile_layout(const QseArgs& a, bool early, cudaStream_t s) {
    return launch_qse_tile_fp<3, PRE, LAY, UnstableFirst, UnstableLast>(a, early, s);
}

cudaError_t unstable_tile(const QseArgs& a, bool early, cudaStream_t s) {
    if (a.F != 3) return cudaErrorInvalidValue;
    if (a.interleaved) return unstable_tile_layout<false, kTileRecords>(a, early, s);
    bool al = true;
    for (int f = 0; f < 3; ++f) al = al && aligned(a.fields[f], 16);
    if (a.bext) return al ? unstable_tile_layout<true, kTileAligned>(a, early, s)
                          : unstable_tile_layout<true, kTileUnaligned>(a, early, s);
    return al ? unstable_tile_layout<false, kTileAligned>(a, early, s)
              : unstable_tile_layout<false, kTileUnaligned>(a, early, s);
}

template <bool PRE>
cudaError_t unstable_batch_layout(const BatchCompressArgs& a, cudaStream_t s) {
    auto kern = gpz_batch_tile_kernel<3, PRE, kTileUnaligned, UnstableSlot>;  // takes any fields
    kern<<<a.total_blocks, kTileThreads, tile_smem_bytes(3, kTileUnaligned), s>>>(a);
    return cudaGetLastError();
}

cudaError_t unstable_batch(const BatchCompressArgs& a, int F, cudaStream_t s) {
    if (F != 3) return cudaErrorInvalidValue;
    return a.pre ? unstable_batch_layout<true>(a, s) : unstable_batch_layout<false>(a, s);
}

// A batch of one chunk: the descriptors, then the batch's workspace, in d_ws.
gpz_status batch_of_one(const gpz_compress_chunk& d, BatchCore& c) {
    const gpz_status st = core_add_compress(c, d);
    return st != GPZ_OK ? st : core_finish(c, nullptr);
}

gpz_status sync_read_u32(const uint32_t* d, uint32_t* h, cudaStream_t s) {
    if (cudaMemcpyAsync(h, d, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess) return GPZ_ERR_CUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return GPZ_ERR_CUDA;
    return GPZ_OK;
}

}  // namespace

}  // namespace gpz

extern "C" {

int gpz_test_fail_next_allocations(int count) { return g_fail_allocs.exchange(count > 0 ? count : 0); }

uint64_t gpz_test_scan_workspace_size(void) { return ScanTestLayout().total; }

gpz_status gpz_test_scan_timeout(int batched, uint32_t wait_cycles, void* d_ws, uint64_t ws_size, void* stream) {
    const ScanTestLayout L;
    if (!d_ws || ws_size < L.total || !aligned(d_ws, kA) || wait_cycles < 1 || wait_cycles > (1u << 24))
        return GPZ_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    uint8_t* ws = static_cast<uint8_t*>(d_ws);
    uint32_t* status = reinterpret_cast<uint32_t*>(ws + L.ctrl);
    uint32_t* counter = status + 1;
    // every size 0x01010101 (clamped by the kernels to a block's largest
    // size); no tile state published; the tile counter at 1, so that the two
    // CTAs launched take tiles 1 and 2 and nobody ever processes tile 0
    if (cudaMemsetAsync(ws, 0, L.sizes, s) != cudaSuccess) return GPZ_ERR_CUDA;
    if (cudaMemsetAsync(ws + L.sizes, 1, kTestBlocks * 4ull, s) != cudaSuccess) return GPZ_ERR_CUDA;
    if (cudaMemsetAsync(counter, 1, 1, s) != cudaSuccess) return GPZ_ERR_CUDA;
    cudaError_t e;
    if (batched) {
        BatchScanArgs a{};
        a.sizes = reinterpret_cast<const uint32_t*>(ws + L.sizes);
        a.total_blocks = kTestBlocks;
        a.offsets = reinterpret_cast<unsigned long long*>(ws + L.offsets);
        a.tile_state = reinterpret_cast<unsigned long long*>(ws + L.states);
        a.tile_counter = counter;
        a.status = status;
        a.wait_cycles = wait_cycles;
        e = launch_batch_scan(a, s, kTestTiles - 1);
    } else {
        ScanArgs a{};
        a.sizes = reinterpret_cast<const uint32_t*>(ws + L.sizes);
        a.nblocks = kTestBlocks;
        a.n = (uint64_t)kTestBlocks * kBlock;
        a.F = 1;
        a.table = reinterpret_cast<uint32_t*>(ws + L.offsets);
        a.tile_state = reinterpret_cast<unsigned long long*>(ws + L.states);
        a.tile_counter = counter;
        a.status = status;
        a.wait_cycles = wait_cycles;
        e = launch_scan(a, s, kTestTiles - 1);
    }
    if (e != cudaSuccess) return GPZ_ERR_CUDA;
    uint32_t st = 0;
    const gpz_status rc = sync_read_u32(status, &st, s);
    return rc != GPZ_OK ? rc : (gpz_status)st;
}

gpz_status gpz_test_block_lookback_timeout(uint32_t block, uint32_t wait_cycles, void* d_ws, uint64_t ws_size,
                                           int* h_placed, void* stream) {
    if (!d_ws || !h_placed || block < 1 || block > 4096 || ws_size < 8ull * (block + 1) || !aligned(d_ws, kA) ||
        wait_cycles < 1 || wait_cycles > (1u << 24))
        return GPZ_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    uint8_t* ws = static_cast<uint8_t*>(d_ws);
    // states of blocks 0..block-1: none published; the result word after them
    if (cudaMemsetAsync(ws, 0, 8ull * (block + 1), s) != cudaSuccess) return GPZ_ERR_CUDA;
    uint32_t* result = reinterpret_cast<uint32_t*>(ws + 8ull * block);
    gpz_test_lookback_kernel<<<1, 32, 0, s>>>(reinterpret_cast<const unsigned long long*>(ws), block,
                                              (long long)wait_cycles, result);
    if (cudaGetLastError() != cudaSuccess) return GPZ_ERR_CUDA;
    uint32_t placed = 0;
    const gpz_status rc = sync_read_u32(result, &placed, s);
    if (rc != GPZ_OK) return rc;
    *h_placed = (int)placed;
    return GPZ_OK;
}

uint64_t gpz_test_unstable_sort_workspace_size(uint64_t n) {
    const uint64_t w = wide_workspace_size(n, 3), c = gpz_compress_workspace_size(n, 3);
    return kA + (w > c ? w : c) + 64u * 1024u + 128u * nblocks_of(n);  // a batch's workspace: c and a little per block
}

gpz_status gpz_test_unstable_sort(int form, const void* const* d_fields, uint64_t n, const gpz_params* p, void* d_out,
                                  uint64_t out_capacity, uint64_t* h_out_size, uint32_t* d_perm, void* d_ws,
                                  uint64_t ws_size, uint32_t* h_listed, void* stream) {
    if (!p || p->n_fields != 3 || p->flags != 0u || p->seg_bits < 0 || p->seg_bits > kMaxSegBits || !d_fields || n == 0 ||
        !d_out || !aligned(d_out, 16) || !h_out_size || !h_listed || !d_ws || !aligned(d_ws, kA) ||
        (d_perm && !aligned(d_perm, 4)) || form < 0 || form > 3 || (form != 0 && form != 3 && p->mode != GPZ_EB_ABS))
        return GPZ_ERR_INVALID_ARG;
    for (int f = 0; f < (form == 1 ? 1 : 3); ++f)
        if (!d_fields[f] || !aligned(d_fields[f], form == 1 ? 16 : form == 2 ? 8 : 4) || !(p->eb[f] > 0.0) ||
            !std::isfinite(p->eb[f]))
            return GPZ_ERR_INVALID_ARG;
    if (ws_size < gpz_test_unstable_sort_workspace_size(n)) return GPZ_ERR_CAPACITY;
    cudaStream_t s = (cudaStream_t)stream;
    uint32_t* words = static_cast<uint32_t*>(d_ws);  // the control words, where the list's count is
    const float* fields[3];
    for (int f = 0; f < 3; ++f)
        fields[f] = form == 1 ? static_cast<const float*>(d_fields[0]) + f : static_cast<const float*>(d_fields[f]);
    gpz_status st;
    if (form == 2) {
        const double* wide[3];
        for (int f = 0; f < 3; ++f) wide[f] = static_cast<const double*>(d_fields[f]);
        st = wide_compress(wide, n, 3, p->seg_bits, p->mode, p->eb, d_out, out_capacity, nullptr, h_out_size, d_perm,
                           d_ws, ws_size, s, false, launch_wide_fast_unstable);
        words += 2;
    } else if (form != 3) {
        st = compress_impl(fields, n, p, d_out, out_capacity, nullptr, h_out_size, d_perm, d_ws, ws_size, stream, false,
                           form == 1 ? fields[0] : nullptr, true, unstable_tile);
        words += 6;
    } else {
        gpz_compress_chunk d{};
        for (int f = 0; f < 3; ++f) d.fields[f] = fields[f];
        d.n = n;
        d.params = *p;
        d.out = d_out;
        d.out_capacity = out_capacity;
        d.perm = d_perm;
        BatchCore c;
        if ((st = batch_of_one(d, c)) != GPZ_OK) return st;
        const uint64_t desc = align_up(core_device_bytes(c), kA);
        if (ws_size < kA + desc + c.L.total) return GPZ_ERR_CAPACITY;
        std::vector<uint8_t> img(core_device_bytes(c));
        core_pack(c, img.data());
        uint8_t* ws = static_cast<uint8_t*>(d_ws);
        uint64_t* d_size = reinterpret_cast<uint64_t*>(ws + desc);
        uint8_t* bws = ws + desc + kA;
        if (cudaMemcpyAsync(ws, img.data(), img.size(), cudaMemcpyHostToDevice, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            return GPZ_ERR_CUDA;
        st = core_enqueue(c, core_device_view(c, ws), bws, d_size, s, false, unstable_batch);
        if (st == GPZ_OK && (cudaMemcpyAsync(h_out_size, d_size, 8, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                             cudaStreamSynchronize(s) != cudaSuccess))
            st = GPZ_ERR_CUDA;
        words = reinterpret_cast<uint32_t*>(bws);
    }
    return st != GPZ_OK ? st : sync_read_u32(words, h_listed, s);
}

}  // extern "C"
