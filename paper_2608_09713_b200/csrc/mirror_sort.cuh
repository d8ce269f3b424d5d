// The column sort of the mirror for 4-byte values of matrices of at most 2^24 rows, and for 8-byte values of at most
// 2^18: C_L's entries by (column, row) in two passes over memory (up to 2^18 rows) or three.
//
// A column id is cut into parts, from the low end: L bits, M bits (three passes) and H bits.
//   split : the entries, read from C_L in row order, go to one of 2^L buckets by their low part;
//   mid   : (three passes) every bucket's entries go to one of 2^M buckets each by the next part;
//   place : a CTA walks a bucket in order, ranks every entry inside its column (the high part) and writes
//           it to its place in F.  Rows arrive ascending, so rank order is row order.
// Buckets by low bits are of nearly equal size for most matrices (columns of C_L get shorter to the right,
// hubs sit together before a relabelling), so one CTA per bucket is a fair share of work, and a bucket's
// CTA needs no per-tile histogram: before `place`, the entries of every column are counted from the high
// parts that the pass before wrote beside the records (two bytes each), and with the row lengths of C_L that gives
// F's row pointers by one scan, before F is written.  A bucket that holds more than its share (a column that most rows
// store, columns a power of two apart, fewer buckets than the GPU has room for) is cut into pieces: each piece counts its columns, and
// a piece starts behind what the pieces before it hold.  Which buckets are cut is known on the GPU only, so the launches have
// room for as many pieces as there can be.  (One CTA per bucket whatever its size: 4e6 rows that all store column 0,
// 12.97 ms against 1.29; 2^18 rows over every 512th column 6.01 ms against 0.26; 2.9e8 entries of a dense triangle of
// doubles, 256 buckets on 296 places, 8.07 ms against 7.44.)  Diagonal entries travel along: the diagonal entry of
// column j is the first of its column and its place, one before the reflected entries, is where the row's own
// diagonal belongs anyway.
//
// 8-byte values travel as one 16-byte record (column, row, value), 4-byte values as (row, value) beside the
// two-byte rest of the column.
//
// A pass is bound by the load/store pipe and by what a CTA waits for at its barriers, 75 to 100 cycles per 32 entries and
// SM.  128 registers (two CTAs of 256 threads) hold a tile without spills; three to five CTAs with fewer registers
// took 1.2 to 2 times as long.  6.4e8 single-precision entries with 18-bit columns (the large power-law workload):
// the whole mirror 13.9 ms (15.2 with ranks by votes); three passes of 8-bit digits took 15.0, the (key, row) expansion that `split` does without 2.0 and
// their histograms and scans 2.8, beside the lower parts.
#pragma once
#include "bucket.cuh"

namespace spsyrk {

constexpr int MS_THREADS = 256;
constexpr int MS_WARPS = MS_THREADS / 32;
constexpr int MS_COLUMN_BITS = 24;  // widest column id; what is left of it after L >= 8 bits fits 16
constexpr int MS_MAX_BINS = 4 * MS_THREADS;  // widest part: 4 bins per thread

template <typename VB> struct MirrorSortTraits;
template <> struct MirrorSortTraits<uint64_t> {
    static constexpr int ITEMS = 12, MIN_CTAS = 2;
    using Rec = uint4;  // column, row, value
};
template <> struct MirrorSortTraits<uint32_t> {
    static constexpr int ITEMS = 16, MIN_CTAS = 2;
    using Rec = uint2;  // row, value
};
template <typename VB>
constexpr int mirror_tile() { return MS_THREADS * MirrorSortTraits<VB>::ITEMS; }

struct MirrorSortArgs {
    const int64_t* l_rowptr;
    const int32_t* l_colidx;
    const void* l_vals;
    int64_t m, n;              // rows, entries
    int lbits, mbits, hbits;   // mbits == 0: two passes
    // split: chunks of consecutive entries (a multiple of 32), one CTA each
    int64_t chunk, nchunks;
    const int32_t* step_row;   // row of every 32nd entry
    const int64_t* split_off;  // [part * nchunks + chunk], one more at the end
    // mid: every bucket of the split in pieces of about mid_cap entries, one CTA each, numbered in the order of the entries
    int64_t mid_cap;
    int mid_units;             // launched (there are at most so many)
    int32_t* mid_first;        // [(1 << L) + 1] the first piece of every bucket
    uint8_t* mid_bucket;       // [mid_units] the bucket of every piece
    const int64_t* mid_off;    // [part * mid_units + piece], one more at the end
    // records and rests of the split (two pieces: [0, a_split) and the tail) and what `place` reads
    void *rec_a, *rec_a_tail;
    int64_t a_split;
    uint16_t* high_a;
    void* rec_b;
    uint16_t* high_b;
    // place: one CTA per bucket, and one per piece of the buckets of more than `cap` entries
    int64_t nbuckets, cap;
    uint32_t max_pieces;       // launched (there are at most so many)
    uint32_t* pieces;          // pieces of all cut buckets, zero before the last split
    int32_t* first_piece;      // [nbuckets] -1: not cut
    int2* piece;               // [max_pieces] (bucket, number inside it)
    uint32_t* piece_cnt;       // [max_pieces << H] entries per column
    uint32_t* cnt;             // entries per column; zero before
    const int64_t* fstart;     // where column j's entries go in F
    int32_t* f_colidx;
    void* f_vals;
    uint32_t* err;
};

// A column id outside [0, m) (not a valid C_L) is taken for m - 1: every pass uses the same id, nothing is indexed out of range.
__device__ __forceinline__ uint32_t ms_key(int32_t j, int64_t m) { return min((uint32_t)j, (uint32_t)(m - 1)); }

// Parts of the columns of entries [e0, e1) counted into `hist[d * stride]`; part(e) is the part or 0xffffffff to skip.
template <int UNR, typename Part>
__device__ __forceinline__ void ms_count(int64_t e0, int64_t e1, int bits, uint32_t* __restrict__ hist, int64_t stride, Part part) {
    constexpr int COPIES = 4;  // warps share a copy: fewer collisions of their atomics
    __shared__ uint32_t h[COPIES][MS_MAX_BINS];
    const int nb = 1 << bits;
    for (int d = threadIdx.x; d < nb; d += MS_THREADS) {
#pragma unroll
        for (int c = 0; c < COPIES; ++c) h[c][d] = 0;
    }
    __syncthreads();
    uint32_t* mine = h[(threadIdx.x >> 5) & (COPIES - 1)];
    for (int64_t e = e0 + threadIdx.x; e < e1; e += UNR * MS_THREADS) {
        uint32_t k[UNR];
#pragma unroll
        for (int u = 0; u < UNR; ++u) k[u] = e + u * MS_THREADS < e1 ? part(e + u * MS_THREADS) : 0xffffffffu;
#pragma unroll
        for (int u = 0; u < UNR; ++u)
            if (k[u] < (uint32_t)nb) atomicAdd(&mine[k[u]], 1u);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < nb; d += MS_THREADS) {
        uint32_t t = 0;
#pragma unroll
        for (int c = 0; c < COPIES; ++c) t += h[c][d];
        hist[d * stride] = t;
    }
}

// G lanes per row: the row of every 32nd entry; whether the row stores its diagonal entry (rows are ascending: it is
// the last one); the counters that later passes add to
template <int G>
static __global__ void __launch_bounds__(256) mirror_rows_kernel(const int64_t* __restrict__ l_rowptr, const int32_t* __restrict__ l_colidx, int64_t m,
                                                                 int64_t n, int32_t* __restrict__ step_row, uint8_t* __restrict__ diagf,
                                                                 uint32_t* __restrict__ cnt, uint32_t* __restrict__ pieces, int64_t* __restrict__ scan_state,
                                                                 int64_t scan_words) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < scan_words; i += (int64_t)gridDim.x * blockDim.x) scan_state[i] = 0;
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    const int gl = threadIdx.x & (G - 1);
    if (r >= m) return;
    const int64_t p0 = max(l_rowptr[r], (int64_t)0), p1 = min(l_rowptr[r + 1], n);
    for (int64_t s = (p0 + 31) / 32 + gl; s * 32 < p1; s += G) step_row[s] = (int32_t)r;
    if (gl == 0) {
        diagf[r] = (p1 > p0 && (int64_t)l_colidx[p1 - 1] == r) ? 1 : 0;
        cnt[r] = 0;
        if (r == 0) *pieces = 0;
    }
}

// entries per (low part, chunk)
static __global__ void __launch_bounds__(MS_THREADS) mirror_split_count_kernel(MirrorSortArgs A, uint32_t* __restrict__ hist) {
    link();
    const int64_t e0 = (int64_t)blockIdx.x * A.chunk, e1 = min(e0 + A.chunk, A.n);
    const uint32_t mask = (1u << A.lbits) - 1u;
    ms_count<8>(e0, e1, A.lbits, hist + blockIdx.x, A.nchunks, [&](int64_t e) { return ms_key(A.l_colidx[e], A.m) & mask; });
}

// The pieces of the mid pass (one CTA: a thread per bucket, L = 8)
static __device__ void ms_mid_pieces(const MirrorSortArgs& A, uint32_t* scratch) {
    __shared__ uint32_t s_first[257];
    const int t = threadIdx.x;
    const int64_t len = A.split_off[(int64_t)(t + 1) * A.nchunks] - A.split_off[(int64_t)t * A.nchunks];
    uint32_t total;
    const uint32_t ex = block_exclusive_scan<uint32_t, MS_THREADS>((uint32_t)max((len + A.mid_cap - 1) / A.mid_cap, (int64_t)1), scratch, &total);
    s_first[t] = ex;
    A.mid_first[t] = (int32_t)ex;
    if (t == 0) {
        s_first[256] = total;
        A.mid_first[256] = (int32_t)total;
    }
    __syncthreads();
    for (uint32_t u = t; u < total && u < (uint32_t)A.mid_units; u += MS_THREADS) {
        int lo = 0, hi = 256;  // last bucket whose first piece is <= u
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (s_first[mid] <= u) lo = mid; else hi = mid;
        }
        A.mid_bucket[u] = (uint8_t)lo;
    }
    __syncthreads();
}
// entries of a piece of the mid pass (none behind the last piece)
__device__ __forceinline__ void ms_mid_piece(const MirrorSortArgs& A, int unit, int64_t* e0, int64_t* e1) {
    *e0 = *e1 = 0;
    if (unit >= A.mid_first[256]) return;
    const int bucket = A.mid_bucket[unit], first = A.mid_first[bucket], count = A.mid_first[bucket + 1] - first;
    const int64_t b0 = A.split_off[bucket * A.nchunks], len = A.split_off[(bucket + 1) * A.nchunks] - b0;
    *e0 = b0 + len * (unit - first) / count;
    *e1 = b0 + len * (unit - first + 1) / count;
}

static __global__ void __launch_bounds__(MS_THREADS) mirror_mid_count_kernel(MirrorSortArgs A, uint32_t* __restrict__ hist) {
    link(A.mid_first, A.mid_bucket, A.split_off, A.high_a);
    int64_t e0, e1;
    ms_mid_piece(A, blockIdx.x, &e0, &e1);
    const uint32_t mask = (1u << A.mbits) - 1u;
    ms_count<8>(e0, e1, A.mbits, hist + blockIdx.x, A.mid_units, [&](int64_t e) { return (uint32_t)A.high_a[e] & mask; });
}

// first entry of bucket b of `place` (of the end: b = nbuckets)
__device__ __forceinline__ int64_t ms_bucket_start(const MirrorSortArgs& A, int64_t b) {
    if (b >= A.nbuckets) return A.n;
    if (A.mbits == 0) return A.split_off[b * A.nchunks];
    return A.mid_off[(b >> A.lbits) * A.mid_units + A.mid_first[b & ((1 << A.lbits) - 1)]];
}

// The pieces of the buckets that are cut, by all CTAs of the pass before `place`
static __device__ void ms_place_pieces(const MirrorSortArgs& A) {
    for (int64_t b = (int64_t)threadIdx.x * gridDim.x + blockIdx.x; b < A.nbuckets; b += (int64_t)MS_THREADS * gridDim.x) {
        const int64_t len = ms_bucket_start(A, b + 1) - ms_bucket_start(A, b);
        int32_t first = -1;
        if (len > A.cap) {
            const uint32_t count = (uint32_t)((len + A.cap - 1) / A.cap);
            first = (int32_t)atomicAdd(A.pieces, count);
            for (uint32_t k = 0; k < count; ++k)
                if (SPSYRK_IN_RANGE(first + k < A.max_pieces, A.err)) A.piece[first + k] = make_int2((int)b, (int)k);
        }
        A.first_piece[b] = first;
    }
}

// What a CTA of the column counts and of `place` handles: a piece (the first max_pieces CTAs), or a bucket that is not cut
struct MirrorUnit {
    int64_t bucket, e0, e1;
    int32_t first, number;  // of a piece: the bucket's first piece, its number in the bucket; first = -1: a whole bucket
};
__device__ __forceinline__ bool ms_unit(const MirrorSortArgs& A, int64_t u, MirrorUnit* x) {
    if (u < A.max_pieces) {
        if (u >= *A.pieces) return false;
        const int2 p = A.piece[u];
        const int64_t b0 = ms_bucket_start(A, p.x), len = ms_bucket_start(A, (int64_t)p.x + 1) - b0, count = (len + A.cap - 1) / A.cap;
        *x = MirrorUnit{p.x, b0 + len * p.y / count, b0 + len * (p.y + 1) / count, (int32_t)u - p.y, p.y};
        return true;
    }
    const int64_t b = u - A.max_pieces;
    *x = MirrorUnit{b, ms_bucket_start(A, b), ms_bucket_start(A, b + 1), -1, 0};
    return A.first_piece[b] < 0;
}

// entries per column
static __global__ void __launch_bounds__(MS_THREADS) mirror_column_count_kernel(MirrorSortArgs A, const uint16_t* __restrict__ high) {
    __shared__ uint32_t h[MS_MAX_BINS];
    MirrorUnit unit;
    link(high);
    if (!ms_unit(A, blockIdx.x, &unit)) return;
    const int nb = 1 << A.hbits;
    for (int d = threadIdx.x; d < nb; d += MS_THREADS) h[d] = 0;
    __syncthreads();
    const int64_t b0 = unit.e0, b1 = unit.e1;
    // eight parts per load where the array is 16-byte aligned
    const int64_t a0 = min((b0 + 7) & ~int64_t(7), b1), a1 = max(a0, b1 & ~int64_t(7));
    auto one = [&](uint32_t x) { atomicAdd(&h[x & (nb - 1)], 1u); };
    for (int64_t e = b0 + threadIdx.x; e < a0; e += MS_THREADS) one(high[e]);
    for (int64_t e = a0 + 8 * (int64_t)threadIdx.x; e < a1; e += 8 * MS_THREADS) {
        const uint4 v = *reinterpret_cast<const uint4*>(high + e);
        one(v.x); one(v.x >> 16); one(v.y); one(v.y >> 16);
        one(v.z); one(v.z >> 16); one(v.w); one(v.w >> 16);
    }
    for (int64_t e = a1 + threadIdx.x; e < b1; e += MS_THREADS) one(high[e]);
    __syncthreads();
    const int low = A.lbits + A.mbits;
    for (int d = threadIdx.x; d < nb; d += MS_THREADS) {
        const int64_t j = unit.bucket + ((int64_t)d << low);
        if (unit.first >= 0) {
            A.piece_cnt[((int64_t)(unit.first + unit.number) << A.hbits) + d] = h[d];
            if (j < A.m && h[d]) atomicAdd(&A.cnt[j], h[d]);
        } else if (j < A.m) {
            A.cnt[j] = h[d];
        }
    }
}

// Consecutive entries of a tile that one warp owns: whole steps of 32, the same number for every warp
__device__ __forceinline__ int ms_warp_span(int64_t tile_n) { return (int)((tile_n + MS_THREADS - 1) / MS_THREADS) * 32; }

// row of the first entry of step s (of a step behind the last: the last row)
__device__ __forceinline__ int64_t ms_step_row(const MirrorSortArgs& A, int64_t s) {
    return s * 32 < A.n ? (int64_t)min((uint32_t)A.step_row[s], (uint32_t)(A.m - 1)) : A.m - 1;
}

// Shared memory of the three passes: the tile (records, with the part or rest of the column beside them), offsets, counters
template <typename VB>
struct MirrorSplitSmem {
    static constexpr int TILE = mirror_tile<VB>();
    static constexpr bool KEYS = sizeof(VB) == 4;  // the record does not hold the column: it lies beside it
    static size_t bytes(int nb) {
        return (size_t)TILE * sizeof(typename MirrorSortTraits<VB>::Rec) + (KEYS ? (size_t)TILE * 4 : 0) + (size_t)nb * 8 + (size_t)MS_WARPS * nb * 2;
    }
};

template <typename VB>
__device__ __forceinline__ typename MirrorSortTraits<VB>::Rec* ms_rec_at(void* head, void* tail, int64_t split, int64_t e) {
    using Rec = typename MirrorSortTraits<VB>::Rec;
    return e < split ? static_cast<Rec*>(head) + e : static_cast<Rec*>(tail) + (e - split);
}

template <typename VB>
__global__ void __launch_bounds__(MS_THREADS, MirrorSortTraits<VB>::MIN_CTAS) mirror_split_kernel(MirrorSortArgs A) {
    using T = MirrorSortTraits<VB>;
    using SM = MirrorSplitSmem<VB>;
    constexpr int ITEMS = T::ITEMS, TILE = SM::TILE, CHUNK = 32 * ITEMS;
    extern __shared__ __align__(16) unsigned char ms_smem[];
    __shared__ uint32_t scratch[33];
    __shared__ uint32_t s_bits[MS_WARPS][ITEMS];  // a bit where a row starts
    const int nb = 1 << A.lbits;
    typename T::Rec* s_rec = reinterpret_cast<typename T::Rec*>(ms_smem);       // [TILE] the tile in bucket order
    uint32_t* s_key = reinterpret_cast<uint32_t*>(s_rec + TILE);                // [TILE] (4-byte values)
    int64_t* s_goff = reinterpret_cast<int64_t*>(s_key + (SM::KEYS ? TILE : 0));  // [nb]
    uint16_t* count = reinterpret_cast<uint16_t*>(s_goff + nb);                 // [WARPS][nb]

    const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    // before the tile is in bucket order its space holds the rows that start in every warp's entries
    uint32_t* rows_of_warp = reinterpret_cast<uint32_t*>(ms_smem) + warp * (CHUNK + 1);
    static_assert((size_t)MS_WARPS * (CHUNK + 1) * 4 <= (size_t)TILE * sizeof(typename T::Rec), "rows fit the tile's space");
    uint32_t* bits = s_bits[warp];
    link(A.split_off, A.step_row);
    if (A.mbits == 0) ms_place_pieces(A);
    else if (blockIdx.x == 0) ms_mid_pieces(A, scratch);
    const int64_t e0 = (int64_t)blockIdx.x * A.chunk, e1 = min(e0 + A.chunk, A.n);
    const VB* __restrict__ vals = static_cast<const VB*>(A.l_vals);
    int64_t gbase[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
        gbase[k] = 4 * tid + k < nb ? A.split_off[(int64_t)(4 * tid + k) * A.nchunks + blockIdx.x] : 0;
    bucket_clear_counts<MS_THREADS>(count, nb);
    for (int64_t base = e0; base < e1; base += TILE) {
        const int64_t end = min(base + TILE, e1);
        const int span = ms_warp_span(end - base);
        const int64_t w0 = base + warp * span;  // the warp's entries: [w0, w0 + wn)
        const int wn = (int)max(min(end - w0, (int64_t)span), (int64_t)0);
        uint32_t key[ITEMS], row[ITEMS];
        VB val[ITEMS];
        {
            const int32_t* pc = A.l_colidx + w0 + lane;
            const VB* pv = vals + w0 + lane;
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) key[i] = i * 32 + lane < wn ? (uint32_t)pc[i * 32] : 0u;
#pragma unroll
            for (int i = 0; i < ITEMS; ++i) val[i] = i * 32 + lane < wn ? pv[i * 32] : VB(0);
        }
        __syncthreads();  // the last tile has left shared memory, the counters are clear
        if (wn > 0) {
            // rows of the warp's entries: a bit per row start, the ids of the rows in their order
            const int64_t r0 = ms_step_row(A, w0 >> 5), r1 = ms_step_row(A, ((w0 + wn - 1) >> 5) + 1);  // the first row, one not before the last
            const bool walk = r1 - r0 <= 2 * CHUNK;
            if (lane < ITEMS) bits[lane] = walk ? 0u : 0xffffffffu;
            if (lane == 0) rows_of_warp[0] = (uint32_t)r0;
            __syncwarp();
            if (!walk) {
                // Most rows are empty: every entry's row is searched for between the rows of two steps and entered as if it
                // began there.  (Walking along 1e7 rows, 32 at a time, took 2.4 ms for 4000 entries.)
#pragma unroll 1
                for (int i = lane; i < wn; i += 32) {
                    const int64_t e = w0 + i;
                    int64_t lo = ms_step_row(A, e >> 5), hi = ms_step_row(A, (e >> 5) + 1);
                    while (lo < hi) {  // the last row that starts at or before the entry
                        const int64_t mid = (lo + hi + 1) >> 1;
                        if (A.l_rowptr[mid] <= e) lo = mid; else hi = mid - 1;
                    }
                    rows_of_warp[i + 1] = (uint32_t)lo;
                }
            }
            int found = 1;
            for (int64_t r = r0 + 1 + lane; walk; r += 32) {
                const int64_t s = r < A.m ? A.l_rowptr[r] : INT64_MAX, x = r < A.m ? A.l_rowptr[r + 1] : INT64_MAX;
                const bool on = s > w0 && s < w0 + wn && x > s;
                const unsigned votes = __ballot_sync(FULL_MASK, on);
                if (on) {
                    const uint32_t p = (uint32_t)(s - w0);
                    const int at = found + __popc(votes & ((1u << lane) - 1u));
                    if (SPSYRK_IN_RANGE(p < (uint32_t)CHUNK && at <= CHUNK, A.err)) {
                        atomicOr(&bits[p >> 5], 1u << (p & 31));
                        rows_of_warp[at] = (uint32_t)r;
                    }
                }
                found += __popc(votes);
                if (!__all_sync(FULL_MASK, s < w0 + wn)) break;
            }
            __syncwarp();
        }
        uint32_t valid = 0;
        int before = 0;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            if (i * 32 + lane < wn) {
                const uint32_t b = bits[i];
                row[i] = rows_of_warp[before + __popc(b & (0xffffffffu >> (31 - lane)))];
                before += __popc(b);
                key[i] = ms_key((int32_t)key[i], A.m);
                valid |= 1u << i;
            }
        }
        const auto bin = [&](int i) { return key[i] & (uint32_t)(nb - 1); };
        uint32_t rk[ITEMS];
        uint16_t* mycount = count + warp * nb;
        bucket_rank<ITEMS>(bin, valid, mycount, rk);
        __syncthreads();
        const int total = bucket_offsets<MS_THREADS>(count, nb, scratch, gbase, s_goff);
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            if ((valid >> i) & 1u) {
                const uint32_t q = mycount[bin(i)] + rk[i];
                if (!SPSYRK_IN_RANGE(q < (uint32_t)TILE, A.err)) continue;
                if constexpr (SM::KEYS) {
                    s_rec[q] = make_uint2(row[i], (uint32_t)val[i]);
                    s_key[q] = key[i];
                } else {
                    s_rec[q] = make_uint4(key[i], row[i], (uint32_t)val[i], (uint32_t)(val[i] >> 32));
                }
            }
        }
        __syncthreads();
        bucket_clear_counts<MS_THREADS>(count, nb);
        const auto key_at = [&](int q) { if constexpr (SM::KEYS) return s_key[q]; else return s_rec[q].x; };
        const auto row_at = [&](int q) { if constexpr (SM::KEYS) return s_rec[q].x; else return s_rec[q].y; };
        // (rows ascend; entries of one row are of different columns, so their order does not matter)
        const auto wrong = [&](int q) { return ((key_at(q) ^ key_at(q + 1)) & (uint32_t)(nb - 1)) == 0 && row_at(q) > row_at(q + 1); };
        bool bad = false;
#pragma unroll 4
        for (int q = tid; q < total - 1; q += MS_THREADS) bad |= wrong(q);
        bucket_in_order<MS_THREADS>(bad, total, wrong, [&](int q) {
            exchange_slots(s_rec, q);
            if constexpr (SM::KEYS) exchange_slots(s_key, q);
        });
#pragma unroll 4
        for (int q = tid; q < total; q += MS_THREADS) {
            const typename T::Rec r = s_rec[q];
            uint32_t k;
            if constexpr (SM::KEYS) k = s_key[q]; else k = r.x;
            const int64_t dest = s_goff[k & (nb - 1)] + q;
            if (!SPSYRK_IN_RANGE(dest >= 0 && dest < A.n, A.err)) continue;
            *ms_rec_at<VB>(A.rec_a, A.rec_a_tail, A.a_split, dest) = r;
            A.high_a[dest] = (uint16_t)(k >> A.lbits);
        }
    }
}

// (4-byte values: 8-byte ones have at most 2^18 rows here, two passes)
struct MirrorMidSmem {
    static size_t bytes(int nb) { return (size_t)mirror_tile<uint32_t>() * (sizeof(uint2) + 2) + (size_t)nb * 8 + (size_t)MS_WARPS * nb * 2; }
};

static __global__ void __launch_bounds__(MS_THREADS, MirrorSortTraits<uint32_t>::MIN_CTAS) mirror_mid_kernel(MirrorSortArgs A) {
    using T = MirrorSortTraits<uint32_t>;
    constexpr int ITEMS = T::ITEMS, TILE = mirror_tile<uint32_t>();
    extern __shared__ __align__(16) unsigned char ms_smem[];
    __shared__ uint32_t scratch[33];
    const int nb = 1 << A.mbits;
    typename T::Rec* s_rec = reinterpret_cast<typename T::Rec*>(ms_smem);       // [TILE]
    int64_t* s_goff = reinterpret_cast<int64_t*>(s_rec + TILE);                 // [nb]
    uint16_t* count = reinterpret_cast<uint16_t*>(s_goff + nb);                 // [WARPS][nb]
    uint16_t* s_rest = count + MS_WARPS * nb;                                   // [TILE]
    const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    link(A.mid_off, A.rec_a, A.rec_a_tail, A.high_a);
    ms_place_pieces(A);
    int64_t e0, e1;
    ms_mid_piece(A, blockIdx.x, &e0, &e1);
    int64_t gbase[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) gbase[k] = 4 * tid + k < nb ? A.mid_off[(int64_t)(4 * tid + k) * A.mid_units + blockIdx.x] : 0;
    bucket_clear_counts<MS_THREADS>(count, nb);
    for (int64_t base = e0; base < e1; base += TILE) {
        const int64_t end = min(base + TILE, e1);
        const int span = ms_warp_span(end - base);
        const int64_t w0 = base + warp * span;
        const int wn = (int)max(min(end - w0, (int64_t)span), (int64_t)0);
        uint32_t rest[ITEMS], valid = 0;
        typename T::Rec rec[ITEMS];
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            rest[i] = 0;
            rec[i] = typename T::Rec{};
            if (i * 32 + lane < wn) {
                const int64_t e = w0 + i * 32 + lane;
                rec[i] = *ms_rec_at<uint32_t>(A.rec_a, A.rec_a_tail, A.a_split, e);
                rest[i] = A.high_a[e];
                valid |= 1u << i;
            }
        }
        const auto bin = [&](int i) { return rest[i] & (uint32_t)(nb - 1); };
        __syncthreads();  // the last tile has left shared memory, the counters are clear
        uint32_t rk[ITEMS];
        uint16_t* mycount = count + warp * nb;
        bucket_rank<ITEMS>(bin, valid, mycount, rk);
        __syncthreads();
        const int total = bucket_offsets<MS_THREADS>(count, nb, scratch, gbase, s_goff);
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            if ((valid >> i) & 1u) {
                const uint32_t q = mycount[bin(i)] + rk[i];
                if (!SPSYRK_IN_RANGE(q < (uint32_t)TILE, A.err)) continue;
                s_rec[q] = rec[i];
                s_rest[q] = (uint16_t)rest[i];
            }
        }
        __syncthreads();
        bucket_clear_counts<MS_THREADS>(count, nb);
        const auto wrong = [&](int q) { return ((s_rest[q] ^ s_rest[q + 1]) & (uint32_t)(nb - 1)) == 0 && s_rec[q].x > s_rec[q + 1].x; };
        bool bad = false;
#pragma unroll 4
        for (int q = tid; q < total - 1; q += MS_THREADS) bad |= wrong(q);
        bucket_in_order<MS_THREADS>(bad, total, wrong, [&](int q) {
            exchange_slots(s_rec, q);
            exchange_slots(s_rest, q);
        });
#pragma unroll 4
        for (int q = tid; q < total; q += MS_THREADS) {
            const typename T::Rec r = s_rec[q];
            const uint32_t k = s_rest[q];
            const int64_t dest = s_goff[k & (nb - 1)] + q;
            if (!SPSYRK_IN_RANGE(dest >= 0 && dest < A.n, A.err)) continue;
            static_cast<typename T::Rec*>(A.rec_b)[dest] = r;
            A.high_b[dest] = (uint16_t)(k >> A.mbits);
        }
    }
}

template <typename VB>
struct MirrorPlaceSmem {
    static size_t bytes(int nb) { return (size_t)mirror_tile<VB>() * (sizeof(VB) + 4 + 2) + (size_t)nb * 8 + (size_t)MS_WARPS * nb * 2; }
};

template <typename VB>
__global__ void __launch_bounds__(MS_THREADS, MirrorSortTraits<VB>::MIN_CTAS) mirror_place_kernel(MirrorSortArgs A) {
    using T = MirrorSortTraits<VB>;
    constexpr int ITEMS = T::ITEMS, TILE = mirror_tile<VB>();
    extern __shared__ __align__(16) unsigned char ms_smem[];
    __shared__ uint32_t scratch[33];
    const int nb = 1 << A.hbits, low = A.lbits + A.mbits;
    VB* s_val = reinterpret_cast<VB*>(ms_smem);                          // [TILE] the tile in column order
    int64_t* s_goff = reinterpret_cast<int64_t*>(s_val + TILE);          // [nb]
    uint32_t* s_row = reinterpret_cast<uint32_t*>(s_goff + nb);          // [TILE]
    uint16_t* count = reinterpret_cast<uint16_t*>(s_row + TILE);         // [WARPS][nb]
    uint16_t* s_bin = count + MS_WARPS * nb;                             // [TILE]
    const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    MirrorUnit unit;
    link(A.rec_b, A.high_b, A.fstart);
    if (!ms_unit(A, blockIdx.x, &unit)) return;
    const int64_t b0 = unit.e0, b1 = unit.e1, col0 = unit.bucket;  // column of bin 0
    int64_t gbase[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int64_t j = col0 + ((int64_t)(4 * tid + k) << low);
        gbase[k] = 4 * tid + k < nb && j < A.m ? A.fstart[j] : 0;
    }
    if (4 * tid < nb) {  // behind what the pieces before hold
#pragma unroll 4
        for (int q = 0; q < unit.number; ++q) {
            const uint4 c = *reinterpret_cast<const uint4*>(A.piece_cnt + ((int64_t)(unit.first + q) << A.hbits) + 4 * tid);
            gbase[0] += c.x; gbase[1] += c.y; gbase[2] += c.z; gbase[3] += c.w;
        }
    }
    const typename T::Rec* __restrict__ recs = static_cast<const typename T::Rec*>(A.rec_b);
    VB* __restrict__ f_vals = static_cast<VB*>(A.f_vals);
    bucket_clear_counts<MS_THREADS>(count, nb);
    for (int64_t base = b0; base < b1; base += TILE) {
        const int64_t end = min(base + TILE, b1);
        const int span = ms_warp_span(end - base);
        const int64_t w0 = base + warp * span;
        const int wn = (int)max(min(end - w0, (int64_t)span), (int64_t)0);
        uint32_t d[ITEMS], valid = 0;  // 4-byte values: the parts of the columns
        typename T::Rec rec[ITEMS];
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            if constexpr (sizeof(VB) == 4) d[i] = 0;
            rec[i] = typename T::Rec{};
            if (i * 32 + lane < wn) {
                const int64_t e = w0 + i * 32 + lane;
                rec[i] = recs[e];
                if constexpr (sizeof(VB) == 4) d[i] = A.high_b[e];
                valid |= 1u << i;
            }
        }
        const auto bin = [&](int i) { return sizeof(VB) == 4 ? d[i] : rec[i].x >> low; };
        __syncthreads();  // the last tile has left shared memory, the counters are clear
        uint32_t rk[ITEMS];
        uint16_t* mycount = count + warp * nb;
        bucket_rank<ITEMS>(bin, valid, mycount, rk);
        __syncthreads();
        const int total = bucket_offsets<MS_THREADS>(count, nb, scratch, gbase, s_goff);
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            if ((valid >> i) & 1u) {
                const uint32_t q = mycount[bin(i)] + rk[i];
                if (!SPSYRK_IN_RANGE(q < (uint32_t)TILE, A.err)) continue;
                if constexpr (sizeof(VB) == 8) {
                    s_row[q] = rec[i].y;
                    s_val[q] = (VB)rec[i].z | ((VB)rec[i].w << 32);
                } else {
                    s_row[q] = rec[i].x;
                    s_val[q] = rec[i].y;
                }
                s_bin[q] = (uint16_t)bin(i);
            }
        }
        __syncthreads();
        bucket_clear_counts<MS_THREADS>(count, nb);
        const auto wrong = [&](int q) { return s_bin[q] == s_bin[q + 1] && s_row[q] > s_row[q + 1]; };
        bool bad = false;
#pragma unroll 4
        for (int q = tid; q < total - 1; q += MS_THREADS) bad |= wrong(q);
        bucket_in_order<MS_THREADS>(bad, total, wrong, [&](int q) {
            exchange_slots(s_row, q);
            exchange_slots(s_val, q);
        });
#pragma unroll 4
        for (int q = tid; q < total; q += MS_THREADS) {
            const uint32_t bin = s_bin[q], r = s_row[q];
            const VB v = s_val[q];
            const int64_t pos = s_goff[bin] + q;
            // an entry above the diagonal (rows that are not ascending can hide one from the size step) is left out
            if ((int64_t)r >= col0 + ((int64_t)bin << low)) {
                A.f_colidx[pos] = (int32_t)r;
                f_vals[pos] = v;
            }
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Matrices of more than 2^24 rows, or of few entries for their rows: radix passes of (column, row, value) arrays (radix.cuh)
// ---------------------------------------------------------------------------------------------
// G lanes per row: the (column, row) pair of every entry; the diagonal entry, and one above the diagonal (rows that are not
// ascending can hide one from the size step), sorts past the end as column m and takes no part in the reflection
template <int G>
static __global__ void __launch_bounds__(256) mirror_expand_kernel(const int64_t* __restrict__ l_rowptr, const int32_t* __restrict__ l_colidx, int64_t m, int64_t n,
                                                                   uint32_t* __restrict__ key, uint32_t* __restrict__ row) {
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    const int gl = threadIdx.x & (G - 1);
    if (r >= m) return;
    const int64_t p0 = max(l_rowptr[r], (int64_t)0), p1 = min(l_rowptr[r + 1], n);
    constexpr int UNR = 4;
    for (int64_t p = p0 + gl; p < p1; p += UNR * G) {
        uint32_t j[UNR];
#pragma unroll
        for (int u = 0; u < UNR; ++u) j[u] = p + u * G < p1 ? (uint32_t)l_colidx[p + u * G] : 0u;
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
            if (p + u * G < p1) {
                key[p + u * G] = j[u] < (uint32_t)r ? j[u] : (uint32_t)m;
                row[p + u * G] = (uint32_t)r;
            }
        }
    }
}

// Last pass: before the entry at sorted position s of column j lie the strictly lower entries of the columns before and of this
// one, so its place in F is s + l_rowptr[j + 1].  The ends of a run of one column in the tile settle where the column's entries
// begin and end.  (Counting the columns while they are expanded, in row order, costs a random access to memory per
// entry: 34.1 ms instead of 26.9 for 4.0e8 entries of 2^27 rows.)
struct EmitMirror {
    static constexpr bool NEIGHBOURS = true;
    const int64_t* l_rowptr;
    uint32_t m;
    int32_t* f_colidx;
    uint32_t* f_vals;
    unsigned long long *seg_start, *seg_end;
    __device__ __forceinline__ void operator()(int64_t s, uint32_t j, uint32_t row, uint32_t val, uint32_t prev, uint32_t next) const {
        if (j >= m) return;
        const int64_t pos = s + l_rowptr[j + 1];
        f_colidx[pos] = (int32_t)row;
        f_vals[pos] = val;
        if (prev != j) atomicMin(&seg_start[j], (unsigned long long)s);
        if (next != j) atomicMax(&seg_end[j], (unsigned long long)s + 1ull);
    }
};

}  // namespace spsyrk
