// The pipelines that the tie-break kernel leaves open, shared out over the CTAs of one launch.
#pragma once

#include "cm_plan_eval.cuh"

namespace cm {

constexpr int kRestThreads = 128, kRestFlags = 1 << 13;
static_assert(kRestThreads == kTile && kRestThreads == kChunk, "BatchDev::max_tiles_per_seg counts these tiles");

// What a CTA looks at: a tile of kRestThreads candidates of a pipeline.
struct RestTile {
    SegView g;
    uint64_t base, count, w_bits;              // first candidate, candidates of the pipeline, winning cost
    volatile unsigned long long *slot;         // lowest composition found so far
    __device__ __forceinline__ void commit(uint64_t kappa) const { atomicMin((unsigned long long *)slot, (unsigned long long)kappa); }
};

// Deals out tiles, the first of every pipeline, then the second ..; a tile above a composition already found
// is skipped, and a CTA that has seen the end of every pipeline is done.  The grid is a prime, so that every
// CTA comes by every pipeline.  mine(S): depths this launch takes; work(tile): a tile, all threads.
// Returns with the CTA's threads together.
template <typename Mine, typename Work>
__device__ __forceinline__ void rest_tiles(const BatchDev &bd, uint32_t n, Mine mine, Work work) {
    __shared__ uint32_t ended[kRestFlags / 32];   // pipelines whose end this CTA has seen
    __shared__ unsigned long long found;
    for (int k = threadIdx.x; k < kRestFlags / 32; k += kRestThreads) ended[k] = 0;
    uint32_t n_ended = 0;
    for (uint64_t item = blockIdx.x; n_ended < n && item < (uint64_t)n * bd.max_tiles_per_seg; item += gridDim.x) {
        const uint32_t i = (uint32_t)(item % n);
        __syncthreads();                                            // (flags, and what the last tile left in shared memory)
        if (i < kRestFlags && ((ended[i >> 5] >> (i & 31)) & 1u)) continue;   // uniform
        const uint32_t e = bd.open[i], b = e / kMaxP, p = e % kMaxP;
        RestTile t;
        t.g = seg_view(bd, bd.winner[b].scen, bd.winner[b].seg[p]);
        t.w_bits = bd.winner[b].cost_bits;
        t.slot = reinterpret_cast<unsigned long long *>(&bd.kappa_sel[(size_t)b * kMaxP + p]);
        t.base = item / n * kRestThreads;
        t.count = walk_count(t.g);
        if (threadIdx.x == 0) found = *t.slot;
        __syncthreads();
        if (!mine(t.g.S) || t.base >= t.count || found <= walk_kappa(bd.feas, t.g.feas_first, t.base)) {   // uniform
            if (threadIdx.x == 0 && i < kRestFlags) ended[i >> 5] |= 1u << (i & 31);
            if (i < kRestFlags) ++n_ended;
            continue;
        }
        work(t);
    }
}
__device__ __forceinline__ uint32_t rest_open(const BatchDev &bd) { return (uint32_t)(*bd.n_open + 1ull); }
// Candidates evaluated, summed over a warp.
__device__ __forceinline__ void rest_count(const BatchDev &bd, unsigned long long evaluated) {
    for (int o = 16; o > 0; o >>= 1) evaluated += __shfl_xor_sync(0xffffffffu, evaluated, o);
    if ((threadIdx.x & 31) == 0 && evaluated) atomicAdd(&bd.counters[1], evaluated);
}

}  // namespace cm
