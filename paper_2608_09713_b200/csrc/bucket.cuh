// Stable partition of a stream of elements into bins, tile by tile: the building block of the column sort
// of the mirror.
//
// A CTA holds a tile of THREADS * ITEMS elements in registers (a warp owns consecutive ones, 32 per step),
// ranks every element among the equal bins of its warp (counters of 16 bits per warp and bin in shared memory), turns the
// counters of all warps into slots of the tile in bin order, drops the elements into their slots, looks whether equal bins
// kept their order and writes the tile out in runs of one bin.  Offsets of the bins in
// the output stay in the registers of the thread that owns the bin and are carried from tile to tile, so
// a CTA that walks a long range of elements needs one offset per bin for all of it.
#pragma once
#include "common.cuh"

namespace spsyrk {

// What the lanes of a warp may do in any order.  The bounds-checked build takes the odd lanes first, so that what relies on
// another order is found out.  What follows comes after it.
template <typename F>
__device__ __forceinline__ void in_any_order(F f) {
#ifdef SPSYRK_CHECKED
    if (lane_id() & 1) f();
    __syncwarp();
    if (!(lane_id() & 1)) f();
#else
    f();
#endif
    __syncwarp();
}

// Ranks of a warp's elements among the elements of the warp with the same bin: what an atomic add to the warp's counter of
// the bin returns (two counters per word).  bin(i) is the bin of step i (counts where bit i of `valid` is set); `count` are
// the warp's counters, zero on entry, the warp's totals on return.  Elements of one bin get different ranks, but which of them
// comes first is up to the hardware: bucket_in_order looks at the sorted tile.  (One vote per bit of the bin and a step of the
// lowest lane for its equals before, nine votes of three instructions per 32 elements on 18-bit columns: mirror of 6.4e8
// single-precision entries 15.2 ms, now 13.9.  The radix and record passes keep their votes: with atomic adds and a look at their
// tiles they took as long, and longer where many lanes meet in one counter - banded matrix, 7.04 ms against 6.86.)
template <int ITEMS, typename Bin>
__device__ __forceinline__ void bucket_rank(Bin bin, uint32_t valid, uint16_t* count, uint32_t (&rk)[ITEMS]) {
    uint32_t* words = reinterpret_cast<uint32_t*>(count);
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const uint32_t d = bin(i), shift = (d & 1u) * 16u;
        rk[i] = 0;
        in_any_order([&] {
            if ((valid >> i) & 1u) rk[i] = (atomicAdd(words + (d >> 1), 1u << shift) >> shift) & 0xffffu;
        });
    }
}

// Puts the tile in order where bucket_rank did not: slots [0, total) hold the elements in bin order; wrong(q) tells whether slots
// q and q + 1 are of one bin and the wrong way round (an element must stand behind those that came before it), exchange(q)
// exchanges them.  `bad`: the calling thread has seen such a pair.  Every thread calls it; true if the tile was changed.
// Only elements of one step of a warp can be the wrong way round, 32 neighbours at most, which as many turns put right; what is
// out of order for another reason (an input that failed its checks) stays so.  (The lanes of a step are served in their
// order on the hardware this was measured on, so that one look is all it takes.)
template <int THREADS, typename Wrong, typename Exchange>
__device__ __forceinline__ bool bucket_in_order(bool bad, int total, Wrong wrong, Exchange exchange) {
    bool changed = false;
#pragma unroll 1
    for (int turn = 0; turn < 32; ++turn) {  // odd-even transposition
        if (!__syncthreads_or(bad)) return changed;
        changed = true;
        bad = false;
#pragma unroll 1
        for (int parity = 0; parity < 2; ++parity) {
            for (int q = 2 * threadIdx.x + parity; q + 1 < total; q += 2 * THREADS) {
                if (wrong(q)) {
                    exchange(q);
                    bad = true;
                }
            }
            __syncthreads();
        }
    }
    return changed;
}

template <typename T>
__device__ __forceinline__ void exchange_slots(T* a, int q) {
    const T t = a[q];
    a[q] = a[q + 1];
    a[q + 1] = t;
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
