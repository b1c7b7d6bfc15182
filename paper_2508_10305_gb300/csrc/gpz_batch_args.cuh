// gpz_batch_args.cuh -- how a CTA of the batched compression kernels gets the
// arguments of its block's chunk.
#pragma once

#include "gpz_batch.cuh"
#include "gpz_qse_block.cuh"

namespace gpz {

namespace {

// Per-chunk argument block of the per-block code, built in shared memory by
// the CTA's threads in parallel (d_params stays null: the constants are
// copied in, read from L2).  Thread 64 also stores the block's index within
// its chunk in *slot.
__device__ __forceinline__ void load_chunk_args(const BatchCompressArgs& g, uint32_t c, uint32_t gb, QseArgs& A,
                                                uint32_t* slot) {
    const int t = threadIdx.x;
    const BatchChunk* ch = g.chunks + c;
    if (t < kMaxFields) A.fields[t] = ch->in[t];
    if (t >= 32 && t < 32 + 4 * kMaxFields) {
        const int f = (t - 32) >> 2, k = (t - 32) & 3;
        const uint32_t* src = ch->mode ? reinterpret_cast<const uint32_t*>(g.rparams + (size_t)c * kMaxFields + f)
                                       : reinterpret_cast<const uint32_t*>(ch->params + f);
        reinterpret_cast<uint32_t*>(A.params + f)[k] = __ldcg(src + k);
    }
    if (t == 64) {
        const uint32_t base = ch->block_base;
        slot[0] = gb - base;
        slot[1] = gb;
        A.n = ch->n;
        A.nblocks = ch->nblocks;
        A.F = ch->F;
        A.G = ch->G;
        A.interleaved = 0;
        A.d_params = nullptr;
        A.bext = g.pre ? g.bext + (size_t)ch->block_base * kMaxFields : nullptr;
        A.binfo = nullptr;  // the fused kernel derives the widths from the extremes
        A.temp = g.temp + ch->temp_base;
        A.slot_words = batch_slot_words(ch->F);
        A.sizes = g.sizes + base;
        A.sums = nullptr;  // the batch has its own scan
        A.sum_shift = 0;
        A.perm = ch->perm;
        A.status = g.chunk_status + c;
        A.general_list = g.general_list;
        A.general_count = g.general_count;
        A.fallback_count = nullptr;
        A.direct = nullptr;  // the batched form keeps the three-step compaction
        A.direct_capacity = 0;
        A.bstate = nullptr;
        A.deferred_count = nullptr;
    }
}

}  // namespace

}  // namespace gpz
