// Stable partition of a stream of elements into bins, tile by tile: the building block of the column sort
// of the mirror.
//
// A CTA holds a tile of THREADS * ITEMS elements in registers (a warp owns consecutive ones, 32 per step),
// ranks every element among the equal bins of its warp (one vote per bin bit, counters of 16 bits per
// warp and bin in shared memory), turns the counters of all warps into slots of the tile in bin order,
// drops the elements into their slots and writes the tile out in runs of one bin.  Offsets of the bins in
// the output stay in the registers of the thread that owns the bin and are carried from tile to tile, so
// a CTA that walks a long range of elements needs one offset per bin for all of it.
#pragma once
#include "common.cuh"

namespace spsyrk {

// Ranks of a warp's elements among the earlier elements of the warp with the same bin.  bin(i) is the bin of step i
// (counts where bit i of `valid` is set); `count` are the warp's counters, zero on entry, the warp's totals
// on return.  The votes run bit by bit over all steps, so that the votes of different steps overlap (with all bits of
// one step after the other a warp waits for each of its votes: 6.6 ms against 4.9 for a pass over 5.4e8 records).
template <int ITEMS, typename Bin>
__device__ __forceinline__ void bucket_rank(Bin bin, uint32_t valid, int bits, uint16_t* count, uint32_t (&rk)[ITEMS]) {
    const int lane = lane_id();
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) rk[i] = __ballot_sync(FULL_MASK, (valid >> i) & 1u);  // lanes with the same bin so far
#pragma unroll 1
    for (int bit = 0; bit < bits; ++bit) {
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const bool set = (bin(i) >> bit) & 1u;
            const unsigned bal = __ballot_sync(FULL_MASK, set);
            rk[i] &= set ? bal : ~bal;
        }
    }
    // the lowest lane of every group of equal bins moves the warp's counter
    const uint32_t below = (1u << lane) - 1u;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const bool on = (valid >> i) & 1u;
        const int leader = on ? __ffs(rk[i]) - 1 : lane;
        uint32_t prev = 0;
        if (on && lane == leader) {
            uint16_t* c = count + bin(i);
            prev = *c;
            *c = (uint16_t)(prev + __popc(rk[i]));
        }
        rk[i] = __shfl_sync(FULL_MASK, prev, leader) + __popc(rk[i] & below);
        __syncwarp();
    }
}

// Warp counters -> first slot of every (warp, bin) in the tile's bin-major order.  Thread t owns bins 4 t .. 4 t + 3
// (nbins <= 4 * THREADS, a multiple of 4); gbase are their offsets in the output, moved on by the tile's counts;
// s_goff[bin] becomes the offset of the bin minus its first slot, so that slot q of that bin goes to s_goff[bin] + q.
// Returns the number of elements.  Contains barriers (the last statement is one).  Counts fit 16 bits: a tile has
// fewer than 65536 elements.
template <int THREADS>
__device__ __forceinline__ int bucket_offsets(uint16_t* count, int nbins, uint32_t* scratch, int64_t (&gbase)[4], int64_t* s_goff) {
    constexpr int WARPS = THREADS / 32;
    const int t = threadIdx.x, lane = lane_id(), warp = t >> 5;
    const bool own = 4 * t < nbins;
    uint2 tot = make_uint2(0u, 0u);
    if (own) {
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
            const uint2 c = *reinterpret_cast<const uint2*>(count + w * nbins + 4 * t);
            tot.x += c.x;
            tot.y += c.y;
        }
    }
    const uint32_t c0 = tot.x & 0xffffu, c1 = tot.x >> 16, c2 = tot.y & 0xffffu, c3 = tot.y >> 16;
    const uint32_t mine = c0 + c1 + c2 + c3;
    const uint32_t incl = warp_inclusive_scan<uint32_t>(mine);
    if (lane == 31) scratch[warp] = incl;
    __syncthreads();
    uint32_t before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) {
        const uint32_t s = scratch[w];
        if (w < warp) before += s;
        total += s;
    }
    const uint32_t b0 = before + incl - mine, b1 = b0 + c0, b2 = b1 + c1, b3 = b2 + c2;
    if (own) {
        uint2 run = make_uint2(b0 | (b1 << 16), b2 | (b3 << 16));
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
            uint2* p = reinterpret_cast<uint2*>(count + w * nbins + 4 * t);
            const uint2 c = *p;
            *p = run;
            run.x += c.x;
            run.y += c.y;
        }
        s_goff[4 * t + 0] = gbase[0] - b0; gbase[0] += c0;
        s_goff[4 * t + 1] = gbase[1] - b1; gbase[1] += c1;
        s_goff[4 * t + 2] = gbase[2] - b2; gbase[2] += c2;
        s_goff[4 * t + 3] = gbase[3] - b3; gbase[3] += c3;
    }
    __syncthreads();
    return (int)total;
}

template <int THREADS>
__device__ __forceinline__ void bucket_clear_counts(uint16_t* count, int nbins) {
    uint4* p = reinterpret_cast<uint4*>(count);
    for (int e = threadIdx.x; e < (THREADS / 32) * nbins / 8; e += THREADS) p[e] = make_uint4(0u, 0u, 0u, 0u);
}

}  // namespace spsyrk
