// Step a6 for heavy rows whose output range [0, U) has at most 2^18 columns: the symbolic pass leaves the number of
// entries of every row, and a row goes to the kernel that suits it (route_rows_kernel):
//   rank   : a bitmap of the columns that occur, prefix population counts turn it into column -> slot, partial products
//            are added into slots.  Two walks over the lists, shared memory by the row's entries.  Sparse rows.
//   direct : accumulators indexed by column, one walk, no ranks, but every column of the range is swept: short ranges that
//            the row fills, and dense rows of binary matrices that dense8 does not take (chunk by chunk).
// A row with more entries than slots fit an SM is cut into parts of whole blocks of columns: the symbolic pass has left
// the number of entries before every block.
//   dense8 : rows of a binary matrix in which every column or many a column occurs: four 8-bit counters per word, the
//            heaviest columns counted through bit masks.
// All are launched with a CTA per row or part of one, the longest lists first, so that the GPU hands the rows out as CTAs end.
// (Persistent CTAs that drew their rows from a counter in the plan lost rows when two passes of one plan overlapped; the
// same rows dealt out beforehand took 1.14 times as long on the large power-law workload.)  In direct and dense8 a CTA
// that has finished takes over one that has not started (cluster launch control) and keeps its accumulators.
//
// Before, every heavy row went through a bitmap, 32-bit ranks and one size of slots (512 threads up to 32768 products, 1024
// above), rows with more entries than slots into global slices with L2 atomics, dense rows of binary matrices
// through a 200 KB tile with one CTA per SM.  Large power-law workload (96 000 heavy rows, 1.46e9 products, single precision):
// 15.3 ms before, 12.1 now; binary Zipf workload of 50000 rows (1.25e9 counts and similarities): 10.8 ms before, dense8
// 4.4 ms = 3.4 TB/s of output.
#pragma once
#include "transpose.cuh"

namespace spsyrk {

enum : int { ROUTE_RANK0 = 0, ROUTE_RANK1, ROUTE_RANK2, ROUTE_RANK_MID, ROUTE_RANK_BIG, ROUTE_RANK_PARTS, ROUTE_DIRECT, ROUTE_DENSE8, ROUTE_WIDE, NROUTE };

// A row of the rank kernel is cut into parts of at most slots_big entries; every part but the last has more than
// slots_big - BASE_BLOCK (a block more would not have fitted), so 2^18 columns make at most 20 parts of 21504 doubles.
constexpr int MAX_ROW_PARTS = 24;

// a row or part of one: blocks [first, end) of BASE_BLOCK columns
__host__ __device__ __forceinline__ int pack_blocks(uint32_t first, uint32_t end) { return (int)(first | end << 8); }

// What the choice needs to know; bytes are shared memory of the kernels as launched
struct RouteRule {
    uint32_t slots_small, slots_mid, slots_big;  // slots of the rank kernels
    uint32_t bits0, bits1;                       // columns of the two narrower bitmaps of the small rank kernel
    uint32_t wide;                               // ranges above this go to the chunked kernel
    uint32_t chunk;                              // columns per chunk of the direct kernel
    uint32_t dense8;                             // columns the packed counters of one row may have
    int binary;
    int masks;                                   // the rows' masks of the heavy columns stand for whole rows of the lower triangle
};

// One thread per heavy row: class 7, then class 6, each with the last rows first (they carry the longest lists).  The lists
// keep that order, so that the rows of a range are two pieces of each: a tile's place in a list comes from the tiles before it by
// look-back, as in the radix passes.  `words` ([tiles][NROUTE]) and `ticket` are zero at the start.
// lengths[NROUTE ..] are the lengths of class 7's part (its `long_rows` rows come first).
constexpr int ROUTE_THREADS = 256;
inline int64_t route_tiles(int64_t rows) { return (rows + ROUTE_THREADS - 1) / ROUTE_THREADS; }
static __global__ void __launch_bounds__(ROUTE_THREADS) route_rows_kernel(PlanDev P, RouteRule R, const int32_t* __restrict__ rows, int64_t count,
                                                                          const int32_t* __restrict__ cnt, const uint32_t* __restrict__ block_base, uint32_t blocks_per_row,
                                                                          int32_t* __restrict__ lists, int64_t cap, int2* __restrict__ rank_parts,
                                                                          int64_t long_rows, uint32_t* __restrict__ lengths, unsigned long long* words,
                                                                          unsigned long long* ticket) {
    constexpr int NW = ROUTE_THREADS / 32;
    __shared__ uint32_t s_before[NW][NROUTE];  // rows (parts) of the tile's warps before
    __shared__ int64_t s_base[NROUTE];
    __shared__ uint32_t s_tile;
    link(rows, cnt, block_base);
    if (threadIdx.x == 0) s_tile = (uint32_t)atomicAdd(ticket, 1ull);
    __syncthreads();
    const int64_t tile = s_tile, n = tile * ROUTE_THREADS + threadIdx.x;
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    int route = -1;
    int32_t rloc = 0;
    uint32_t end[MAX_ROW_PARTS];
    uint32_t parts = 0;
    if (n < count) {
        rloc = rows[count - 1 - n];
        const int64_t i = (int64_t)P.r0 + rloc;
        const uint32_t U = P.mode == SPSYRK_TRIL ? (uint32_t)i + 1u : (uint32_t)P.m;
        const uint32_t entries = (uint32_t)cnt[rloc];
        const int64_t w = P.work[rloc], deg = P.rowptr[i + 1] - P.rowptr[i];
        const uint32_t blocks = (U + BASE_BLOCK - 1) / BASE_BLOCK;
        const bool dense = entries == U;
        if (U > R.wide) {
            route = ROUTE_WIDE;
        } else if (R.binary && deg <= 255 && U <= R.dense8 && (dense || (R.masks && w >= (int64_t)U))) {
            // Rows that are not dense: rank walks all their products twice, direct has 32-bit counters; dense8 walks each once, fewer with
            // heavy columns, but looks at every column.  Numeric pass of 30 000 rows of random columns, without and with dense8: w = U 2565
            // us to 2020, 1.3 U 2999 to 1551, 2 U 3737 to 1839; of 6000 rows 147 to 126, 156 to 120, 175 to 137 (below U the two
            // are level: rank has the fewer columns to look at).  The last 3000 rows of 70 000, 150 000 and 220 000 (fewer CTAs fit an SM), 1.5 U:
            // 1819 us to 665, 4610 to 2298, 6131 to 3367.  30 000 sets of 60 of 65 536 columns of Zipf frequencies, of
            // which some lack the most frequent one: all similarities 12.0 ms to 3.1, counting included.
            route = ROUTE_DENSE8;
        } else if ((R.binary && dense) || (U <= R.chunk && w >= (int64_t)(U / 4))) {
            // One chunk: direct walks the lists once and sweeps every column, rank walks them twice and sweeps a bitmap.  Measured
            // on equal rows of doubles, direct against rank: 11000 columns and w = U/8 333 us to 242, U/4 374 to 373, U/2 472 to
            // 554; 8192 columns 218 to 154, 248 to 234, 302 to 345; 2048 columns 54 to 46, 55 to 50, 57 to 57: the line
            // lies between U/4 and U/2.  (Longer ranges in chunks of 8192 columns: 14 ms per 1e9 products for the
            // searches, barriers and sweeps of every chunk, against 6.7 in parts of the rank kernel.)
            route = ROUTE_DIRECT;
        } else if (entries <= R.slots_small) {
            route = U <= R.bits0 ? ROUTE_RANK0 : U <= R.bits1 ? ROUTE_RANK1 : ROUTE_RANK2;
        } else if (entries <= R.slots_big) {
            route = entries <= R.slots_mid ? ROUTE_RANK_MID : ROUTE_RANK_BIG;
        } else {
            // as many blocks as the slots hold (a block has fewer entries than that)
            route = ROUTE_RANK_PARTS;
            const uint32_t* base = block_base + (uint64_t)i * blocks_per_row;
            uint32_t from = 0;
            for (uint32_t b = 1; b <= blocks; ++b) {
                const uint32_t upto = b < blocks ? base[b] : entries;
                if (upto - from > R.slots_big && parts < MAX_ROW_PARTS - 1) {
                    end[parts++] = b - 1;
                    from = base[b - 1];
                }
            }
            end[parts++] = blocks;
        }
    }
    uint32_t mine = 0;  // rows (parts) of this route in the lanes before
#pragma unroll
    for (int k = 0; k < NROUTE; ++k) {
        uint32_t all;
        if (k == ROUTE_RANK_PARTS) {
            const uint32_t incl = warp_inclusive_scan<uint32_t>(parts);
            all = __shfl_sync(FULL_MASK, incl, 31);
            if (route == k) mine = incl - parts;
        } else {
            const unsigned votes = __ballot_sync(FULL_MASK, route == k);
            all = __popc(votes);
            if (route == k) mine = __popc(votes & ((1u << lane) - 1u));
        }
        if (lane == 0) s_before[warp][k] = all;
    }
    __syncthreads();
    if (threadIdx.x < NROUTE) {
        uint32_t total = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const uint32_t c = s_before[w][threadIdx.x];
            s_before[w][threadIdx.x] = total;
            total += c;
        }
        radix_publish<unsigned long long, NROUTE>(words, tile, threadIdx.x, total);
        const int64_t base = radix_look_back<unsigned long long, NROUTE>(words, tile, threadIdx.x, total, P.err);
        s_base[threadIdx.x] = base;
        if (tile == gridDim.x - 1) lengths[threadIdx.x] = (uint32_t)(base + total);
    }
    __syncthreads();
    // the place in every list at which class 6 begins, from the tile that holds its first row (or the last tile: there is none)
    if (tile == min(long_rows / ROUTE_THREADS, (int64_t)gridDim.x - 1)) {
        const int first = (int)(long_rows - tile * ROUTE_THREADS), lane_of_first = first & 31;
#pragma unroll
        for (int k = 0; k < NROUTE; ++k) {
            const uint32_t before = k == ROUTE_RANK_PARTS ? warp_reduce_sum<uint32_t>(lane < lane_of_first ? parts : 0u)
                                                          : __popc(__ballot_sync(FULL_MASK, route == k) & ((1u << lane_of_first) - 1u));
            if (first < ROUTE_THREADS && warp == first >> 5 && lane == 0) lengths[NROUTE + k] = (uint32_t)s_base[k] + s_before[warp][k] + before;
        }
        if (first >= ROUTE_THREADS && threadIdx.x < NROUTE) lengths[NROUTE + threadIdx.x] = lengths[threadIdx.x];
    }
    if (route < 0) return;
    const int64_t at = s_base[route] + s_before[warp][route] + mine;
    if (route == ROUTE_RANK_PARTS) {
        for (uint32_t k = 0; k < parts; ++k) rank_parts[at + k] = make_int2(rloc, pack_blocks(k ? end[k - 1] : 0u, end[k]));
    } else {
        lists[(int64_t)route * cap + at] = rloc;
    }
}

// What of a route's list a launch takes: two pieces (the rows of a range among those of class 7 and among those of class 6)
struct RoutePieces {
    uint32_t first[2], count[2];
    __host__ __device__ __forceinline__ uint32_t total() const { return count[0] + count[1]; }
    __host__ __device__ __forceinline__ uint32_t at(uint32_t n) const { return n < count[0] ? first[0] + n : first[1] + (n - count[0]); }
};

// For every route, both pieces of the rows [lo_row, hi_row): out[(route * 2 + piece) * 2] = first, [.. + 1] = one past the
// last.  A list is descending inside a class; one thread per bound.
static __device__ void route_positions(int t, const int32_t* lists, int64_t cap, const int2* rank_parts, const uint32_t* lengths, int64_t lo_row, int64_t hi_row,
                                       int64_t* out) {
    const int k = t >> 2, piece = (t >> 1) & 1;
    const int64_t bound = (t & 1) ? lo_row : hi_row;
    uint32_t lo = piece ? lengths[NROUTE + k] : 0u, hi = piece ? lengths[k] : lengths[NROUTE + k];
    while (lo < hi) {
        const uint32_t mid = lo + (hi - lo) / 2;
        const int64_t row = k == ROUTE_RANK_PARTS ? rank_parts[mid].x : lists[(int64_t)k * cap + mid];
        if (row >= bound) lo = mid + 1; else hi = mid;
    }
    out[t] = lo;
}

// The lists of a row, up to THREADS of them at a time, flattened through a prefix sum of their lengths
template <typename Acc, int THREADS>
struct ListBatch {
    uint32_t off[THREADS + 1];
    uint32_t start[THREADS];
    Acc a[THREADS];
    uint32_t warp_sum[THREADS / 32];
};

// Every thread brings one list (len may be 0).  Contains barriers, the last statement is one.
template <typename Acc, int THREADS>
__device__ __forceinline__ void batch_fill(ListBatch<Acc, THREADS>& B, uint32_t start, uint32_t len, Acc a) {
    const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    const uint32_t incl = warp_inclusive_scan<uint32_t>(len);
    if (lane == 31) B.warp_sum[warp] = incl;
    __syncthreads();
    const uint32_t ws = lane < THREADS / 32 ? B.warp_sum[lane] : 0u;
    const uint32_t before = warp_reduce_sum<uint32_t>(lane < warp ? ws : 0u);
    B.off[tid] = before + incl - len;
    B.start[tid] = start;
    B.a[tid] = a;
    if (tid == THREADS - 1) B.off[THREADS] = before + incl;
    __syncthreads();
}

// Every warp takes a contiguous run of the flattened items and its lanes interleave inside it: loads are coalesced and UNR
// of them in flight; a lane steps from list to list as its items advance.  fn(position in the column lists, a).
template <typename Acc, int THREADS, int UNR, typename Load, typename Apply>
__device__ __forceinline__ void batch_walk(const ListBatch<Acc, THREADS>& B, Load load, Apply apply) {
    constexpr uint32_t NW = THREADS / 32;
    const uint32_t T = B.off[THREADS];
    const uint32_t per_warp = ((T + NW - 1) / NW + 31u) & ~31u;
    const uint32_t wfirst = min((uint32_t)(threadIdx.x >> 5) * per_warp, T), last = min(wfirst + per_warp, T);
    const uint32_t first = wfirst + lane_id();
    if (first >= last) return;
    uint32_t lo = 0, hi = THREADS;  // last list whose offset is <= first
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (B.off[mid] <= first) lo = mid; else hi = mid;
    }
    uint32_t cur = lo, next = B.off[cur + 1], shift = B.start[cur] - B.off[cur];
    Acc a = B.a[cur];
    using L = decltype(load(0u));
    for (uint32_t item0 = first; item0 < last; item0 += UNR * 32) {
        L v[UNR];
        Acc av[UNR];
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
            const uint32_t item = item0 + u * 32;
            if (item < last) {
                if (item >= next) {
                    do { ++cur; } while (item >= B.off[cur + 1]);
                    next = B.off[cur + 1];
                    shift = B.start[cur] - B.off[cur];
                    a = B.a[cur];
                }
                v[u] = load(shift + item);
                av[u] = a;
            }
        }
#pragma unroll
        for (int u = 0; u < UNR; ++u)
            if (item0 + u * 32 < last) apply(v[u], av[u]);
    }
}

struct HeavyArgs {
    const int32_t* list;
    RoutePieces rows;
    const int64_t* out_begin;  // where each row's part of the output starts / ends
    const int64_t* out_end;
    int32_t* c_colidx;
    bool aligned;              // the output arrays start on 16-byte boundaries
    const int2* parts;         // parts of rows (row, pack_blocks), computed before the list
    RoutePieces part_rows;
    const uint32_t* block_base;  // [absolute row * blocks_per_row + block]: entries of the row before the block of columns
    uint32_t blocks_per_row;
};

// A row, or a part of one, by its number in the launch
__device__ __forceinline__ int2 heavy_unit(const HeavyArgs& H, uint32_t n) {
    const uint32_t np = H.part_rows.total();
    return n < np ? H.parts[H.part_rows.at(n)] : make_int2(H.list[H.rows.at(n - np)], pack_blocks(0u, 255u));  // 255: to the end
}

// The order in which dense8 takes `count` rows of a list: the first of each of 64 segments, the second of each, ...  Rows next
// to each other are equally long, and CTAs that all count while all others count, and write while all write, leave the
// memory idle half the time: 50000 dense rows 5.58 ms in the list's order, 4.36 so; 20000 rows 0.92 against 0.84; 5000 rows
// 0.110 against 0.109; 3000 rows 57.6 against 59.1 us (the longest rows first matter more).
__device__ __forceinline__ uint32_t spread_rows(uint32_t n, uint32_t count) {
    constexpr uint32_t SEGMENTS = 64, MIN_LENGTH = 64;
    const uint32_t length = count / SEGMENTS;
    return length >= MIN_LENGTH && n < length * SEGMENTS ? n % SEGMENTS * length + n / SEGMENTS : n;
}

// The rows of a CTA, one after the other: its own, then those of CTAs that have not started.  Thread 0 asks for the next CTA
// while the row is computed (clusterlaunchcontrol.try_cancel; the answer arrives in shared memory and completes a phase
// of the barrier).  After a refusal nothing is asked for any more, and a CTA does not end with a request under way.
// (With a CTA per row: dense8 on 50000 rows 4.52 ms instead of 4.38, direct on 8192 equal rows 273 us instead of 257.  The
// rank kernels, whose rows take longest, gain nothing: 12.6 against 12.5 ms on the large power-law workload.)
struct RowQueueShared {
    uint4 answer;
    unsigned long long barrier;
    int2 unit;
};
struct RowQueue {
    static constexpr uint32_t NONE = 0xffffffffu;
    RowQueueShared* s;
    uint32_t answer_at, barrier_at;  // shared-memory addresses
    uint32_t n, phase = 0;
    bool asked = false;
    bool has_first;  // this CTA has handled the launch's first row: it ends the chain

    __device__ __forceinline__ explicit RowQueue(RowQueueShared* shared) : s(shared), n(blockIdx.x), has_first(blockIdx.x == 0) {
        answer_at = (uint32_t)__cvta_generic_to_shared(&s->answer);
        barrier_at = (uint32_t)__cvta_generic_to_shared(&s->barrier);
        if (threadIdx.x == 0) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(barrier_at) : "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
    }
    __device__ __forceinline__ void ask() {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the answer before has been read
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], 16;" ::"r"(barrier_at) : "memory");
        asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];" ::"r"(answer_at), "r"(barrier_at)
                     : "memory");
        asked = true;
    }
    __device__ __forceinline__ uint32_t take(uint32_t* err) {
        if (!asked) return NONE;
        asked = false;
        uint32_t done = 0;
        for (int polls = 0; !done; ++polls) {
            if (polls == SPIN_LIMIT) {
                atomicOr(err, ERRW_INTERNAL);
                return NONE;
            }
            asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                         : "=r"(done)
                         : "r"(barrier_at), "r"(phase)
                         : "memory");
        }
        phase ^= 1u;
        uint32_t cta;
        asm volatile("{\n\t.reg .pred p;\n\t.reg .b128 h;\n\tld.shared.b128 h, [%1];\n\tmov.u32 %0, 0xffffffff;\n\t"
                     "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, h;\n\t"
                     "@p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %0, h;\n\t}"
                     : "=r"(cta)
                     : "r"(answer_at)
                     : "memory");
        if (cta == 0) has_first = true;
        return cta;
    }
    // the next row (or part of one), or -1; contains barriers, after which the row before is finished by all threads
    template <bool SPREAD>
    __device__ __forceinline__ int2 next(const HeavyArgs& H, uint32_t* err) {
        if (threadIdx.x == 0) {
            int2 r = make_int2(-1, 0);
            if (asked) n = take(err);
            if (n != NONE) {
                r = heavy_unit(H, SPREAD ? spread_rows(n, H.rows.total()) : n);  // (no parts where rows are spread)
                ask();
            }
            s->unit = r;
        }
        __syncthreads();
        const int2 r = s->unit;
        __syncthreads();
        return r;
    }
};

// The same formula in the same arithmetic as spsyrk_jaccard: the values need not be ones, so the denominator can be
// anything a sum of 64 bits holds.
template <typename V>
__device__ __forceinline__ void store_jaccard(const PlanDev& P, int64_t at, int32_t j, int32_t c, int32_t deg) {
    P.jaccard[at] = __fdiv_rn((float)c, (float)((int64_t)deg + P.adeg[j] - c));
}

// ---------------------------------------------------------------------------------------------
// rank
// ---------------------------------------------------------------------------------------------
template <typename V, int THREADS>
struct RankSmem {
    using Acc = typename AccOf<V>::type;
    static size_t bytes(uint32_t columns, uint32_t slots) {
        return (size_t)columns / 8 + (size_t)columns / 32 + (size_t)slots * sizeof(Acc) + sizeof(ListBatch<Acc, THREADS>) + 16;
    }
};

// Bound by latency and by the shared-memory pipe (an add of doubles takes 17 cycles of an SM per 32 random slots, of 32-bit
// integers 2.7): what counts is how many rows an SM has under way, so the bitmap has 16-bit ranks per 64 columns (a rank per
// 32-bit word: twice the shared memory) and the slots come in three sizes.
template <typename V, int THREADS, int CTAS>
__global__ void __launch_bounds__(THREADS, CTAS) rows_rank_kernel(PlanDev P, HeavyArgs H, uint32_t columns, uint32_t slots, V* __restrict__ c_vals) {
    using Acc = typename AccOf<V>::type;
    constexpr int NW = THREADS / 32;
    extern __shared__ __align__(16) unsigned char rk_smem[];
    __shared__ uint32_t s_warp[NW];
    unsigned long long* bits = reinterpret_cast<unsigned long long*>(rk_smem);                 // [columns / 64]
    Acc* acc = reinterpret_cast<Acc*>(bits + columns / 64);                                   // [slots]
    ListBatch<Acc, THREADS>& B = *reinterpret_cast<ListBatch<Acc, THREADS>*>(acc + slots);
    uint16_t* rank = reinterpret_cast<uint16_t*>(reinterpret_cast<unsigned char*>(acc + slots) + (sizeof(ListBatch<Acc, THREADS>) + 15) / 16 * 16);  // [columns / 64]
    const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    const bool ones = P.binary != 0;
    const ColRec<V>* __restrict__ recs = static_cast<const ColRec<V>*>(P.at_rec);
    uint32_t* bits32 = reinterpret_cast<uint32_t*>(bits);
    chain_begin();
    const int2 unit = heavy_unit(H, blockIdx.x);
    const int32_t rloc = unit.x;
    const int64_t i = (int64_t)P.r0 + rloc;
    const uint32_t whole = P.mode == SPSYRK_TRIL ? (uint32_t)i + 1u : (uint32_t)P.m;
    const uint32_t b_first = unit.y & 0xff, b_end = (uint32_t)unit.y >> 8;
    const uint32_t c0 = b_first * BASE_BLOCK, c1 = min(b_end * BASE_BLOCK, whole), U = c1 - c0;  // columns [c0, c1)
    const int64_t p0 = P.rowptr[i];
    const uint32_t deg = (uint32_t)(P.rowptr[i + 1] - p0);
    int64_t ob = H.out_begin[rloc], oe = H.out_end[rloc];
    if (c1 < whole) oe = ob + H.block_base[(uint64_t)i * H.blocks_per_row + b_end];
    if (c0 > 0) ob += H.block_base[(uint64_t)i * H.blocks_per_row + b_first];
    uint32_t entries = (uint32_t)(oe - ob);
    const uint32_t words = (U + 63u) / 64u;
    if (!SPSYRK_IN_RANGE(ob >= H.out_begin[rloc] && oe <= H.out_end[rloc] && entries <= slots && U <= columns, P.err)) entries = 0;
    for (uint32_t w = tid; w < words; w += THREADS) bits[w] = 0;  // (seen by all behind the first batch's barriers)
    auto fill = [&](uint32_t b0) {
        const bool on = b0 + tid < deg;
        uint2 d = on ? P.desc[p0 + b0 + tid] : make_uint2(0u, 0u);
        const Acc a = on ? (Acc) static_cast<const V*>(P.vals)[p0 + b0 + tid] : Acc(0);
        if (d.y > 0 && U < whole) {
            const int32_t* lst = P.at_row + d.x;
            const uint32_t hi = c1 < whole ? lower_bound_i32(lst, d.y, (int32_t)c1) : d.y;
            const uint32_t lo = c0 > 0 ? lower_bound_i32(lst, hi, (int32_t)c0) : 0u;
            d = make_uint2(d.x + lo, hi - lo);
        }
        batch_fill<Acc, THREADS>(B, d.x, d.y, a);
    };
    // the columns that occur
    for (uint32_t b0 = 0; b0 < deg; b0 += THREADS) {
        if (b0) __syncthreads();
        fill(b0);
        batch_walk<Acc, THREADS, 8>(B, [&](uint32_t q) { return P.at_row[q]; }, [&](int32_t j, Acc) {
            const uint32_t rel = (uint32_t)j - c0;
            if (SPSYRK_IN_RANGE(rel < columns, P.err)) atomicOr(&bits32[rel >> 5], 1u << (rel & 31u));
        });
    }
    for (uint32_t t = tid; t < entries; t += THREADS) acc[t] = Acc(0);
    __syncthreads();
    // ranks: a warp owns consecutive words, 32 per step
    const uint32_t per_warp = ((words + NW - 1) / NW + 31u) & ~31u;
    const uint32_t w0 = min(warp * per_warp, words), w1 = min(w0 + per_warp, words);
    uint32_t sum = 0;
    for (uint32_t w = w0 + lane; w < w1; w += 32) sum += __popcll(bits[w]);
    sum = warp_reduce_sum<uint32_t>(sum);
    if (lane == 0) s_warp[warp] = sum;
    __syncthreads();
    uint32_t run = warp_reduce_sum<uint32_t>(lane < warp ? s_warp[lane < NW ? lane : 0] : 0u);
    for (uint32_t w = w0; w < w1; w += 32) {
        const uint32_t c = w + lane < w1 ? __popcll(bits[w + lane]) : 0u;
        const uint32_t incl = warp_inclusive_scan<uint32_t>(c);
        if (w + lane < w1) rank[w + lane] = (uint16_t)(run + incl - c);
        run += __shfl_sync(FULL_MASK, incl, 31);
    }
    __syncthreads();
    // the products
    auto add = [&](uint32_t j, Acc p) {
        j -= c0;
        if (!SPSYRK_IN_RANGE(j < columns, P.err)) return;
        const uint32_t slot = rank[j >> 6] + __popcll(bits[j >> 6] & ((1ull << (j & 63u)) - 1ull));
        if (SPSYRK_IN_RANGE(slot < entries && slot < slots, P.err)) atomicAdd(&acc[slot], p);
    };
    for (uint32_t b0 = 0; b0 < deg; b0 += THREADS) {
        if (deg > THREADS) {  // (one batch: the lists are still there)
            if (b0) __syncthreads();
            fill(b0);
        }
        if (ones) batch_walk<Acc, THREADS, 8>(B, [&](uint32_t q) { return P.at_row[q]; }, [&](int32_t j, Acc) { add((uint32_t)j, Acc(1)); });
        else batch_walk<Acc, THREADS, 4>(B, [&](uint32_t q) { return recs[q]; }, [&](const ColRec<V>& r, Acc a) { add((uint32_t)r.j, acc_mul(a, (Acc)r.v)); });
    }
    __syncthreads();
    // out: sums by slot, column ids from the bitmap
    for (uint32_t t = tid; t < entries; t += THREADS) c_vals[ob + t] = (V)acc[t];
    for (uint32_t w = tid; w < words; w += THREADS) {
        unsigned long long b = bits[w];
        if (b == 0) continue;
        uint32_t r = rank[w];
        while (b) {
            const int32_t j = (int32_t)(c0 + w * 64u) + __ffsll((long long)b) - 1;
            b &= b - 1;
            if (SPSYRK_IN_RANGE(r < entries, P.err)) {
                H.c_colidx[ob + r] = j;
                if constexpr (std::is_same<V, int32_t>::value)
                    if (P.jaccard) store_jaccard<V>(P, ob + r, j, acc[r], (int32_t)deg);
            }
            ++r;
        }
    }
    chain_end();
}

// ---------------------------------------------------------------------------------------------
// direct
// ---------------------------------------------------------------------------------------------
template <typename V, int THREADS>
struct DirectSmem {
    using Acc = typename AccOf<V>::type;
    static size_t bytes(uint32_t chunk) {
        return (size_t)chunk * (sizeof(Acc) + 1) + (size_t)chunk / 32 * 4 + sizeof(ListBatch<Acc, THREADS>) + 16;
    }
};

constexpr int DIRECT_THREADS = 512;

// Bound by the adds in shared memory.  Two CTAs of 512 threads per SM: one searches and sweeps while the other adds.
// A column that occurs is marked by a plain byte store (a bitmap needs an atomic or a look first; accumulators that
// start as a special NaN need a compare-and-swap loop of their own, which took five times the built-in add).
template <typename V, int THREADS>
__global__ void __launch_bounds__(THREADS, 2) rows_direct_kernel(PlanDev P, HeavyArgs H, uint32_t chunk, V* __restrict__ c_vals) {
    using Acc = typename AccOf<V>::type;
    constexpr int NW = THREADS / 32;
    extern __shared__ __align__(16) unsigned char dr_smem[];
    __shared__ RowQueueShared s_queue;
    __shared__ uint32_t s_warp[NW];
    Acc* acc = reinterpret_cast<Acc*>(dr_smem);                                          // [chunk]
    uint8_t* occurs = reinterpret_cast<uint8_t*>(acc + chunk);                           // [chunk]
    uint32_t* votes = reinterpret_cast<uint32_t*>(occurs + chunk);                       // [chunk / 32]
    ListBatch<Acc, THREADS>& B = *reinterpret_cast<ListBatch<Acc, THREADS>*>(votes + chunk / 32);
    const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    const bool ones = P.binary != 0;
    const ColRec<V>* __restrict__ recs = static_cast<const ColRec<V>*>(P.at_rec);
    for (uint32_t t = tid; t < chunk; t += THREADS) { acc[t] = Acc(0); occurs[t] = 0; }  // (later the sweep leaves them so)
    chain_begin();
    RowQueue queue(&s_queue);
    for (;;) {
        const int32_t rloc = queue.next<false>(H, P.err).x;
        if (rloc < 0) break;
        const int64_t i = (int64_t)P.r0 + rloc;
        const uint32_t U = P.mode == SPSYRK_TRIL ? (uint32_t)i + 1u : (uint32_t)P.m;
        const int64_t p0 = P.rowptr[i];
        const uint32_t deg = (uint32_t)(P.rowptr[i + 1] - p0);
        const int64_t ob = H.out_begin[rloc], oe = H.out_end[rloc];
        const bool dense = oe - ob == (int64_t)U;  // every column occurs
        const int planes = ones && dense ? heavy_planes(P) : 0;
        const bool use_masks = planes > 0;
        const HeavyMask mine = load_heavy_mask(P, i, planes);
        uint32_t done = 0;  // entries of the chunks before
        for (uint32_t c0 = 0; c0 < U; c0 += chunk) {
            const uint32_t c1 = min(c0 + chunk, U), cn = c1 - c0;
            if (use_masks) {
                for (uint32_t t = tid; t < cn; t += THREADS) {
                    uint32_t n = 0;
#pragma unroll
                    for (int p = 0; p < HEAVY_PLANES; ++p)
                        if (p < planes) n += __popc(P.heavy_mask[p * P.mask_stride + c0 + t] & mine.w[p]);
                    acc[t] = (Acc)(int32_t)n;
                }
            }
            auto add = [&](uint32_t j, Acc p) {
                const uint32_t rel = j - c0;
                if (!SPSYRK_IN_RANGE(rel < cn, P.err)) return;
                if (!dense) occurs[rel] = 1;
                atomicAdd(&acc[rel], p);
            };
            for (uint32_t b0 = 0; b0 < deg; b0 += THREADS) {
                const bool on = b0 + tid < deg;
                uint2 d = on ? P.desc[p0 + b0 + tid] : make_uint2(0u, 0u);
                if (use_masks && on && P.heavy_id[P.colidx[p0 + b0 + tid]] != 0xff) d.y = 0;  // counted through the masks
                uint32_t lo = 0, hi = d.y;  // the list's entries in [c0, c1)
                if (d.y > 0 && U > chunk) {
                    if (c1 < U) hi = lower_bound_i32(P.at_row + d.x, d.y, (int32_t)c1);
                    if (c0 > 0) lo = lower_bound_i32(P.at_row + d.x, hi, (int32_t)c0);
                }
                const Acc a = on ? (Acc) static_cast<const V*>(P.vals)[p0 + b0 + tid] : Acc(0);
                if (b0) __syncthreads();
                batch_fill<Acc, THREADS>(B, d.x + lo, hi - lo, a);
                if (ones) batch_walk<Acc, THREADS, 8>(B, [&](uint32_t q) { return P.at_row[q]; }, [&](int32_t j, Acc) { add((uint32_t)j, Acc(1)); });
                else batch_walk<Acc, THREADS, 4>(B, [&](uint32_t q) { return recs[q]; }, [&](const ColRec<V>& r, Acc av) { add((uint32_t)r.j, acc_mul(av, (Acc)r.v)); });
            }
            __syncthreads();
            // entries of every group of 32 columns, their prefix sums; a warp owns consecutive groups
            const uint32_t words = (cn + 31u) / 32u;
            const uint32_t per_warp = (words + NW - 1) / NW;
            const uint32_t w0 = min(warp * per_warp, words), w1 = min(w0 + per_warp, words);
            uint32_t tot = cn, run = 0;
            if (!dense) {
                uint32_t sum = 0;
                for (uint32_t w = w0; w < w1; ++w) {
                    const uint32_t t = w * 32u + lane;
                    const unsigned b = __ballot_sync(FULL_MASK, t < cn && occurs[t] != 0);
                    if (lane == 0) votes[w] = b;
                    sum += __popc(b);
                }
                if (lane == 0) s_warp[warp] = sum;
                __syncthreads();
                const uint32_t ws = lane < NW ? s_warp[lane] : 0u;
                run = warp_reduce_sum<uint32_t>(lane < warp ? ws : 0u);
                tot = warp_reduce_sum<uint32_t>(ws);
            }
            for (uint32_t w = w0; w < w1; ++w) {
                const uint32_t b = dense ? 0xffffffffu : votes[w];
                const uint32_t t = w * 32u + lane;
                if (((b >> lane) & 1u) && t < cn) {
                    const int64_t at = ob + done + (dense ? t : run + __popc(b & ((1u << lane) - 1u)));
                    const Acc v = acc[t];
                    acc[t] = Acc(0);
                    occurs[t] = 0;
                    if (SPSYRK_IN_RANGE(at < oe, P.err)) {
                        c_vals[at] = (V)v;
                        H.c_colidx[at] = (int32_t)(c0 + t);
                        if constexpr (std::is_same<V, int32_t>::value)
                            if (P.jaccard) store_jaccard<V>(P, at, (int32_t)(c0 + t), v, (int32_t)deg);
                    }
                }
                run += __popc(b);
            }
            done += tot;
            __syncthreads();
        }
    }
    chain_end(queue.has_first);
}

// ---------------------------------------------------------------------------------------------
// dense8
// ---------------------------------------------------------------------------------------------
template <int THREADS>
struct Dense8Smem {
    static size_t bytes(uint32_t columns) { return ((size_t)columns + 15) / 16 * 16 + 16 + sizeof(ListBatch<int32_t, THREADS>); }
};

// A row of a binary matrix with at most 255 nonzeros: every count is at most the row's own length, so a word holds
// four counters and a row is one tile.  The counters start at the overlap of the rows' heavy-column masks (read as
// planes of 32 columns, four rows j at a time), the remaining lists, short ones, are walked, and a dense row leaves four
// entries per thread: groups of four are aligned in the output, where the row starts at any offset.  Of another row the
// counters that are not zero leave, 32 columns per step of a warp.
template <typename V, int THREADS, int CTAS>
__global__ void __launch_bounds__(THREADS, CTAS) rows_dense8_kernel(PlanDev P, HeavyArgs H, uint32_t columns, V* __restrict__ c_vals) {
    extern __shared__ __align__(16) unsigned char d8_smem[];
    __shared__ RowQueueShared s_queue;
    __shared__ uint32_t s_warp[THREADS / 32];
    uint32_t* acc = reinterpret_cast<uint32_t*>(d8_smem);  // four columns per word
    ListBatch<int32_t, THREADS>& B = *reinterpret_cast<ListBatch<int32_t, THREADS>*>(d8_smem + ((size_t)columns + 15) / 16 * 16 + 16);
    const int tid = threadIdx.x;
    const int planes = heavy_planes(P);
    chain_begin();
    RowQueue queue(&s_queue);
    for (;;) {
        const int32_t rloc = queue.next<true>(H, P.err).x;
        if (rloc < 0) break;
        const int64_t i = (int64_t)P.r0 + rloc;
        const uint32_t U = P.mode == SPSYRK_TRIL ? (uint32_t)i + 1u : (uint32_t)P.m;
        const int64_t p0 = P.rowptr[i];
        const uint32_t deg = (uint32_t)(P.rowptr[i + 1] - p0);  // at most 255: one batch
        const int64_t ob = H.out_begin[rloc];
        const uint32_t words = (U + 3u) / 4u;
        uint2 d = (uint32_t)tid < deg ? P.desc[p0 + tid] : make_uint2(0u, 0u);
        if (planes > 0) {
            if (d.y > 0 && P.heavy_id[P.colidx[p0 + tid]] != 0xff) d.y = 0;  // counted through the masks
            const HeavyMask mine = load_heavy_mask(P, i, planes);
            for (uint32_t w = tid; w < words; w += THREADS) {
                uint32_t n0 = 0, n1 = 0, n2 = 0, n3 = 0;
#pragma unroll
                for (int p = 0; p < HEAVY_PLANES; ++p) {  // (planes are padded to whole groups of four rows)
                    if (p >= planes) break;
                    const uint4 k = *reinterpret_cast<const uint4*>(P.heavy_mask + p * P.mask_stride + 4 * (int64_t)w);
                    n0 += __popc(k.x & mine.w[p]); n1 += __popc(k.y & mine.w[p]);
                    n2 += __popc(k.z & mine.w[p]); n3 += __popc(k.w & mine.w[p]);
                }
                acc[w] = n0 | (n1 << 8) | (n2 << 16) | (n3 << 24);
            }
        } else {
            for (uint32_t w = tid; w < words; w += THREADS) acc[w] = 0;
        }
        batch_fill<int32_t, THREADS>(B, d.x, d.y, 0);
        batch_walk<int32_t, THREADS, 8>(B, [&](uint32_t q) { return P.at_row[q]; }, [&](int32_t j, int32_t) {
            if (SPSYRK_IN_RANGE((uint32_t)j < U, P.err)) atomicAdd(&acc[(uint32_t)j >> 2], 1u << (((uint32_t)j & 3u) * 8u));
        });
        __syncthreads();
        auto one = [&](uint32_t j) {
            const int32_t c = (int32_t)((acc[j >> 2] >> ((j & 3u) * 8u)) & 0xffu);
            c_vals[ob + j] = (V)c;
            H.c_colidx[ob + j] = (int32_t)j;
            if constexpr (std::is_same<V, int32_t>::value)
                if (P.jaccard) store_jaccard<V>(P, ob + j, (int32_t)j, c, (int32_t)deg);
        };
        if (H.out_end[rloc] - ob != (int64_t)U) {
            constexpr uint32_t NW = THREADS / 32;
            const int lane = lane_id(), warp = tid >> 5;
            const uint32_t steps = (U + 31u) / 32u, per_warp = (steps + NW - 1) / NW;  // of 32 columns; a warp owns consecutive ones
            const uint32_t j0 = min((uint32_t)warp * per_warp * 32u, U), j1 = min(j0 + per_warp * 32u, U);
            uint32_t sum = 0;
            for (uint32_t j = j0 + 4u * lane; j < j1; j += 128u) {
                const uint32_t left = j1 - j, q = acc[j >> 2] & (left < 4u ? (1u << (8u * left)) - 1u : 0xffffffffu);
                sum += __popc(__vcmpne4(q, 0u)) / 8;
            }
            sum = warp_reduce_sum<uint32_t>(sum);
            if (lane == 0) s_warp[warp] = sum;
            __syncthreads();
            uint32_t at = warp_reduce_sum<uint32_t>(lane < warp ? s_warp[lane < (int)NW ? lane : 0] : 0u);
            for (uint32_t j = j0 + lane; j - lane < j1; j += 32u) {
                const int32_t c = j < j1 ? (int32_t)((acc[j >> 2] >> ((j & 3u) * 8u)) & 0xffu) : 0;
                const unsigned votes = __ballot_sync(FULL_MASK, c != 0);
                const int64_t o = ob + at + __popc(votes & ((1u << lane) - 1u));
                if (c != 0 && SPSYRK_IN_RANGE(o < H.out_end[rloc], P.err)) {
                    c_vals[o] = (V)c;
                    H.c_colidx[o] = (int32_t)j;
                    if constexpr (std::is_same<V, int32_t>::value)
                        if (P.jaccard) store_jaccard<V>(P, o, (int32_t)j, c, (int32_t)deg);
                }
                at += __popc(votes);
            }
            continue;
        }
        if (!H.aligned) {
            for (uint32_t j = tid; j < U; j += THREADS) one(j);
            continue;
        }
        // columns [head, tail) leave in whole groups: (ob + j) % 4 == 0
        const uint32_t head = min((uint32_t)((4 - (ob & 3)) & 3), U), groups = (U - head) / 4u, tail = head + 4u * groups;
        if ((uint32_t)tid < head) one((uint32_t)tid);
        if ((uint32_t)tid < U - tail) one(tail + tid);
        for (uint32_t g = tid; g < groups; g += THREADS) {
            const uint32_t j = head + 4u * g;
            // counters j .. j + 3 straddle two words unless head is 0 (the word after the last group's is inside the buffer)
            const uint32_t q = __funnelshift_r(acc[j >> 2], acc[(j >> 2) + 1], (j & 3u) * 8u);
            const int32_t c[4] = {(int32_t)(q & 0xffu), (int32_t)((q >> 8) & 0xffu), (int32_t)((q >> 16) & 0xffu), (int32_t)(q >> 24)};
            *reinterpret_cast<int4*>(H.c_colidx + ob + j) = make_int4((int)j, (int)j + 1, (int)j + 2, (int)j + 3);
            if constexpr (sizeof(V) == 8) {
                double2* o = reinterpret_cast<double2*>(c_vals + ob + j);
                o[0] = make_double2(c[0], c[1]);
                o[1] = make_double2(c[2], c[3]);
            } else if constexpr (std::is_same<V, float>::value) {
                *reinterpret_cast<float4*>(c_vals + ob + j) = make_float4((float)c[0], (float)c[1], (float)c[2], (float)c[3]);
            } else {
                *reinterpret_cast<int4*>(c_vals + ob + j) = make_int4(c[0], c[1], c[2], c[3]);
                if (P.jaccard) {
                    float s[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) s[k] = __fdiv_rn((float)c[k], (float)(uint32_t)((int32_t)deg + P.adeg[j + k] - c[k]));  // (ones: the sum is a union's size)
                    *reinterpret_cast<float4*>(P.jaccard + ob + j) = make_float4(s[0], s[1], s[2], s[3]);
                }
            }
        }
    }
    chain_end(queue.has_first);
}

}  // namespace spsyrk
