// Step a7: F = C_L + C_L^T - D, the full symmetric CSR from the stored lower triangle.
//
// Row j of F = row j of C_L (columns <= j) followed by the reflected entries (r, c_rj) of the
// later rows r > j that store column j, ascending in r.  That second part is a transpose of the
// strictly lower triangle, done as a stable sort of the entries by column id:
//   sizes   : rows are ascending, so a row stores its diagonal iff its last entry is the diagonal and
//             holds an entry above the diagonal iff its last entry is one:
//             nnz(F) = 2 nnz(C_L) - #diagonals.
//   sort    : 4-byte values of up to 2^24 rows and small matrices go to buckets of columns and from there to their
//             places (mirror_sort.cuh); 8-byte values of more than 2^18 rows go through radix passes of 16-byte
//             records, the last of which writes F (mirror_rec.cuh); 4-byte values of more rows, or of few entries for
//             their rows, through radix passes of separate arrays (radix.cuh);
//   rows    : row lengths of F, scan -> f_rowptr (in the bucket sort before the last pass), lower parts copied.
#include <algorithm>
#include <mutex>

#include "mirror_rec.cuh"
#include "mirror_sort.cuh"

using namespace spsyrk;

namespace {

constexpr size_t ALIGN = 256;

constexpr int MIRROR_RADIX_BITS = 8;  // digits of the record passes

// 8-byte values: where buckets take two passes and records three, and below that, where both take two and buckets half the
// launches, the bucket sort is used (records against buckets, product and mirror: 70 000 rows and 9.0e6 entries 847 us to 724,
// 200 000 rows 1898 to 1763, 262 000 rows 3839 to 3727, a banded matrix of 250 000 rows 1060 to 946, a power-law one of 2^18 rows
// 37.2 ms to 35.3).  With a third bucket pass the records move in runs as short and the rests of the columns besides: 2^22 rows 35.06
// ms by records, 35.37 by three bucket passes, a banded matrix of 2e6 rows 6.85 to 7.21.
constexpr int64_t MIRROR_BUCKET_ROWS_8 = 262144;
bool mirror_by_records(int64_t m, size_t sv) { return sv == 8 && m > MIRROR_BUCKET_ROWS_8; }
struct MirrorWs {
    int64_t* partials;
    int64_t *split_state, *mid_state;  // bucket sort: status words of the scans, in one piece with `partials`, state_words long
    int64_t state_words;
    uint32_t* err;       // [0] error word, [1] number of diagonal entries, [2] finished CTAs
    uint32_t* hist;      // counts of the passes and their prefix sums
    int64_t *offsets, *mid_off;
    int32_t *mid_first, *first_piece;  // where the pieces of a bucket begin
    uint8_t* mid_bucket;
    uint32_t *pieces, *piece_cnt;
    int2* piece;
    // bucket sort
    uint8_t* diagf;      // m: 1 where the row stores its diagonal entry
    uint32_t* cnt;       // m: entries of C_L per column
    int64_t* fstart;     // m: where the entries of column j go in F
    int32_t* step_row;   // row of every 32nd entry
    void* rec;           // the records the place pass reads (nnz_l)
    void* rec_tail;      // three passes: what of the first buffer does not fit F's value array
    uint16_t* high;      // 4-byte values: the rests of the columns beside the records
    // radix passes: two sets of (column, row, value); the one the last pass does not read keeps columns and values in F
    uint32_t *key_a, *row_a, *key_b, *row_b;
    void *val_a, *val_b;
    RadixState rx;       // all zero at the start
    size_t rx_bytes;
    // record passes
    uint32_t* diagf32;   // m
    uint32_t* rowtot;    // m
    int64_t* dcount;     // m + 1: diagonal entries of the rows before (exclusive prefix sums of diagf32)
    int64_t* fbase;      // m: l_rowptr[j + 1] - dcount[j + 1]
    // the record buffer the last pass reads (nnz_l records) and the tail of the buffer that lives in F's value array
    MirrorRec *rec_keep, *rec_keep_tail;
    int32_t* tile_rows;  // 2 per tile
    unsigned long long* seg_start;  // m: first sorted position of column j's strictly lower entries
    unsigned long long* seg_end;    // m: one past the last
    uint8_t* dig_small;  // digit bytes of inputs too small to keep them in F's column array
};

// How the sort is cut (see mirror_sort.cuh)
struct MirrorSplit {
    int lbits, mbits, hbits;
    int64_t chunk, nchunks;     // split
    int64_t mid_cap, mid_units;  // mid: entries per piece, pieces at most
    int64_t cap, max_pieces;    // place: entries from which on a bucket is cut, pieces at most
    int64_t split_hist() const { return nchunks << lbits; }
    int64_t mid_hist() const { return mid_units << mbits; }
    int64_t nbuckets() const { return int64_t(1) << (lbits + mbits); }
};

// Column ids of at most so many bits take two passes: parts of nine bits leave runs of eight entries in a tile.  (Two parts of
// ten bits against three of six to eight on 1.35e8 entries: 5.6 ms against 4.6.)
constexpr int MIRROR_TWO_PASS_BITS = 18;

MirrorSplit mirror_split_for(int64_t m, int64_t nnz_l, size_t sv) {
    MirrorSplit s;
    int bits = 1;
    while (bits < MS_COLUMN_BITS && ((m - 1) >> bits) > 0) ++bits;
    if (bits <= MIRROR_TWO_PASS_BITS) {
        s.lbits = std::max(8, (bits + 1) / 2);  // at least 256 buckets: a bucket is one CTA of the last pass
        s.mbits = 0;
        s.hbits = std::max(2, bits - s.lbits);
    } else {
        s.lbits = 8;  // what is left fits 16 bits
        s.mbits = (bits - s.lbits + 1) / 2;
        s.hbits = bits - s.lbits - s.mbits;
    }
    const int64_t tile = sv == 8 ? mirror_tile<uint64_t>() : mirror_tile<uint32_t>();
    // Chunks of the split and pieces of the mid pass, one CTA each.  Below two tiles per SM the entries are shared out
    // evenly; above, a chunk is whole tiles, few enough that neighbouring CTAs write neighbouring runs (148 * 24 chunks
    // 6.6 ms for the split of 5.4e8 records, 148 * 150 to 300 6.0) and enough that the counts, one per bin and chunk, stay small.
    constexpr int64_t FEW = 148 * 2, MANY = 148 * 150;
    if (nnz_l <= FEW * tile) s.chunk = std::max<int64_t>((nnz_l + FEW - 1) / FEW, 256);
    else s.chunk = std::max<int64_t>(nnz_l / (MANY * tile), 1) * tile;
    s.chunk = (s.chunk + 31) / 32 * 32;
    s.nchunks = std::max<int64_t>((nnz_l + s.chunk - 1) / s.chunk, 1);
    // Pieces of the mid pass: four tiles or more, at most about 16384.  Every bucket has at least one.
    s.mid_cap = std::max<int64_t>(4 * tile, nnz_l / 16384);
    s.mid_units = s.mbits ? (int64_t(1) << s.lbits) + nnz_l / s.mid_cap : 0;
    // A bucket of `place` is cut above a quarter of what a CTA would get if all were equal; of few entries, above 8 to 16 tiles (gone
    // in 30 to 50 us), but not where it is less than twice the average.  A cut bucket has less than twice len / cap pieces.
    s.cap = std::max<int64_t>(nnz_l / (148 * 2 * 4), std::min<int64_t>(16 * tile, std::max<int64_t>(8 * tile, 2 * (nnz_l >> (s.lbits + s.mbits)))));
    s.max_pieces = 2 * (nnz_l / s.cap);
    return s;
}

// 4-byte values: what the first pass of the bucket sort leaves of a column must fit two bytes.  (Taking the columns of wider
// matrices in rounds of 2^24 reads all entries once per round: 2^26 rows and 2.7e8 entries 25.5 ms, 2^27 rows and
// 4.0e8 entries 59.1 ms, against 16.6 and 26.9 ms by four radix passes.)  Three passes of the bucket sort need entries for their
// buckets, 2^14 to 2^16 of them; with few per bucket the radix passes are faster, for whose every launch the entries count.
// Buckets against radix passes: 2^22 rows, 92 entries per bucket 1134 us to 494; 640 per bucket 1706 to 1293; 2176 per bucket
// 3624 to 4094.  2^20 rows, 1088 per bucket 1143 to 1111.  2^24 rows, 1280 per bucket 5221 to 5564.
constexpr int64_t MIRROR_BUCKET_FILL = 1024;
bool mirror_by_radix(int64_t m, int64_t nnz_l, size_t sv) {
    if (sv == 8) return false;
    const MirrorSplit s = mirror_split_for(m, nnz_l, sv);
    return m > (int64_t(1) << MS_COLUMN_BITS) || (s.mbits > 0 && nnz_l < MIRROR_BUCKET_FILL * s.nbuckets());
}

int64_t mirror_tail_records(int64_t m, int64_t nnz_l) { return (std::min(m, nnz_l) + 1) / 2; }

// Scratch inside the output.  Until the last pass writes it, F's memory is free.  Three passes need two record buffers
// of R nnz_l bytes each (R = 16 or 8, twice the size of a value).  The one the last pass reads must lie outside F; the
// other one lives in F's value array, which holds R / 2 * (2 nnz_l - D) bytes with D <= min(m, nnz_l) diagonal entries: the
// first nnz_l - ceil(min(m, nnz_l) / 2) records always fit, the few remaining ones go to a tail in the workspace.
// The digit bytes of the record passes (two buffers of nnz_l bytes) and the two-byte rests of the columns live in F's column
// array (4 (2 nnz_l - D) >= 4 nnz_l bytes) where the last pass does not read them.
constexpr int64_t MIRROR_DIG_SMALL = 32;  // inputs of fewer entries than this keep their digit bytes in the workspace
size_t carve(MirrorWs* w, void* ws, int64_t m, int64_t nnz_l, size_t sv) {
    char* base = static_cast<char*>(ws);
    size_t off = 0;
    auto take = [&](size_t bytes) -> void* {
        off = (off + ALIGN - 1) / ALIGN * ALIGN;
        void* p = base ? base + off : nullptr;
        off += bytes;
        return p;
    };
    const int64_t items = std::max<int64_t>(m, 1);
    const int64_t ne = std::max<int64_t>(nnz_l, 1);
    MirrorWs t{};
    t.err = (uint32_t*)take(12);
    if (mirror_by_records(m, sv)) {
        const int64_t hist_n = (int64_t)(1 << MIRROR_RADIX_BITS) * std::max<int64_t>(mirror_groups(nnz_l), 1);
        t.diagf32 = (uint32_t*)take(items * 4);
        t.rowtot = (uint32_t*)take(items * 4);
        t.dcount = (int64_t*)take((items + 1) * 8);
        t.fbase = (int64_t*)take(items * 8);
        t.seg_start = (unsigned long long*)take(items * 8);
        t.seg_end = (unsigned long long*)take(items * 8);
        t.partials = (int64_t*)take(scan_partials_count(std::max<int64_t>(items + 1, hist_n)) * 8);
        t.rec_keep = (MirrorRec*)take(ne * sizeof(MirrorRec));
        t.rec_keep_tail = (MirrorRec*)take((mirror_tail_records(m, nnz_l) + 1) * sizeof(MirrorRec));
        t.dig_small = (uint8_t*)take(2 * MIRROR_DIG_SMALL);
        t.tile_rows = (int32_t*)take(2 * std::max<int64_t>(mirror_tiles(nnz_l), 1) * 4);
        t.hist = (uint32_t*)take(hist_n * 4);
        t.offsets = (int64_t*)take((hist_n + 1) * 8);
    } else if (mirror_by_radix(m, nnz_l, sv)) {
        // F's column and value arrays hold 4 (2 nnz_l - D) >= 4 nnz_l bytes each: the columns and values of one set.  Passes write
        // A, B, A, ...: the last one reads B when their number is odd.
        const int npass = radix_passes((uint64_t)m);  // columns, and m for the diagonal entries
        const bool b_kept = npass % 2 == 1;
        t.rowtot = (uint32_t*)take(items * 4);
        t.seg_start = (unsigned long long*)take(items * 8);
        t.seg_end = (unsigned long long*)take(items * 8);
        t.partials = (int64_t*)take(scan_partials_count(items) * 8);
        t.row_a = (uint32_t*)take(ne * 4);
        t.row_b = (uint32_t*)take(ne * 4);
        uint32_t* const key = (uint32_t*)take(ne * 4);
        void* const val = take(ne * 4);
        if (b_kept) { t.key_b = key; t.val_b = val; } else { t.key_a = key; t.val_a = val; }
        const size_t words = radix_state_words(radix_tiles(nnz_l), radix_wide(nnz_l), npass);
        t.rx_bytes = (RX_MAX_PASSES * RX_BINS + RX_MAX_PASSES + words) * 8;
        t.rx.bins = (unsigned long long*)take(t.rx_bytes);
        t.rx.tickets = (uint32_t*)(t.rx.bins + RX_MAX_PASSES * RX_BINS);
        t.rx.words = t.rx.bins + RX_MAX_PASSES * RX_BINS + RX_MAX_PASSES;
    } else {
        const MirrorSplit sp = mirror_split_for(m, nnz_l, sv);
        const int64_t hist_n = std::max(sp.split_hist(), sp.mid_hist());
        t.diagf = (uint8_t*)take(items);
        t.cnt = (uint32_t*)take(items * 4);
        t.fstart = (int64_t*)take(items * 8);
        const int64_t row_words = scan_partials_count(items), split_words = scan_partials_count(sp.split_hist()), mid_words = sp.mbits ? scan_partials_count(sp.mid_hist()) : 0;
        t.state_words = row_words + split_words + mid_words;
        t.partials = (int64_t*)take(t.state_words * 8);
        t.split_state = t.partials + row_words;
        t.mid_state = t.split_state + split_words;
        t.hist = (uint32_t*)take(hist_n * 4);
        t.offsets = (int64_t*)take((sp.split_hist() + 1) * 8);
        t.mid_off = (int64_t*)take((sp.mid_hist() + 1) * 8);
        t.mid_first = (int32_t*)take(257 * 4);
        t.mid_bucket = (uint8_t*)take(sp.mid_units);
        t.first_piece = (int32_t*)take(sp.nbuckets() * 4);
        t.pieces = (uint32_t*)take(4);
        t.piece = (int2*)take(sp.max_pieces * 8);
        t.piece_cnt = (uint32_t*)take((sp.max_pieces << sp.hbits) * 4);
        t.step_row = (int32_t*)take((ne + 31) / 32 * 4);
        t.rec = take(ne * 2 * sv);
        t.rec_tail = take(sp.mbits ? (mirror_tail_records(m, nnz_l) + 1) * sizeof(uint2) : 0);
        t.high = (uint16_t*)take(sv == 8 ? 0 : ne * 2);
    }
    if (w) *w = t;
    return (off + ALIGN - 1) / ALIGN * ALIGN;
}

template <int G>
__global__ void __launch_bounds__(256) mirror_count_kernel(const int64_t* __restrict__ l_rowptr, const int32_t* __restrict__ l_colidx,
                                                           int64_t m, uint32_t* __restrict__ ucnt, uint32_t* err) {
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    const int gl = threadIdx.x & (G - 1);
    if (r >= m) return;
    const int64_t p0 = l_rowptr[r], p1 = l_rowptr[r + 1];
    if (p1 < p0 && gl == 0) atomicOr(err, ERRW_BAD_ROWPTR);  // the row total below would wrap
    constexpr int UNR = 4;
    for (int64_t p = p0 + gl; p < p1; p += UNR * G) {
        int64_t j[UNR];
#pragma unroll
        for (int u = 0; u < UNR; ++u) j[u] = p + u * G < p1 ? (int64_t)l_colidx[p + u * G] : r;  // r: neither counted nor an error
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
            if (j[u] > r || j[u] < 0) atomicOr(err, ERRW_UPPER);
            else if (j[u] < r) atomicAdd(&ucnt[j[u]], 1u);
        }
    }
}

__global__ void mirror_rowtot_kernel(const int64_t* __restrict__ l_rowptr, const uint32_t* __restrict__ ucnt, int64_t m,
                                     uint32_t* __restrict__ rowtot) {
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r < m) rowtot[r] = (uint32_t)(l_rowptr[r + 1] - l_rowptr[r]) + ucnt[r];
}

// one thread per row: the last entry tells whether the row stores its diagonal and whether it reaches above it
// (rows are ascending); err[1] counts the diagonals; the last CTA to finish (err[2] counts them) sends both to the host
__global__ void __launch_bounds__(256) mirror_last_entry_kernel(const int64_t* __restrict__ l_rowptr, const int32_t* __restrict__ l_colidx, int64_t m,
                                                                uint32_t* err, int64_t* host) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool diag = false;
    if (r < m) {
        const int64_t p0 = l_rowptr[r], p1 = l_rowptr[r + 1];
        if (p1 < p0) {
            atomicOr(err, ERRW_BAD_ROWPTR);
        } else if (p1 > p0) {
            const int64_t last = l_colidx[p1 - 1], first = l_colidx[p0];
            if (last > r || first < 0) atomicOr(err, ERRW_UPPER);
            else diag = last == r;
        }
    }
    const int diags = __syncthreads_count(diag);
    if (threadIdx.x == 0) {
        if (diags) atomicAdd(err + 1, (uint32_t)diags);
        __threadfence();
        if (atomicAdd(err + 2, 1u) == gridDim.x - 1) {
            __threadfence();
            host[0] = (int64_t)atomicAdd(err + 1, 0u);
            host[1] = (int64_t)atomicOr(err, 0u);
        }
    }
}

// G lanes per row: the lower part of row r of F is row r of C_L
template <typename V, int G>
__global__ void __launch_bounds__(256) mirror_copy_lower_kernel(const int64_t* __restrict__ l_rowptr, const int32_t* __restrict__ l_colidx,
                                                                const V* __restrict__ l_vals, int64_t m,
                                                                const int64_t* __restrict__ f_rowptr, int32_t* __restrict__ f_colidx,
                                                                V* __restrict__ f_vals) {
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    const int gl = threadIdx.x & (G - 1);
    link(f_rowptr);
    if (r >= m) return;
    const int64_t p0 = l_rowptr[r], p1 = l_rowptr[r + 1];
    const int64_t fb = f_rowptr[r] - p0;
    constexpr int UNR = 4;
    for (int64_t p = p0 + gl; p < p1; p += UNR * G) {
        int32_t j[UNR];
        V v[UNR];
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
            const int64_t pp = p + u * G;
            if (pp < p1) {
                j[u] = l_colidx[pp];
                v[u] = l_vals[pp];
            }
        }
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
            const int64_t pp = p + u * G;
            if (pp < p1) {
                f_colidx[fb + pp] = j[u];
                f_vals[fb + pp] = v[u];
            }
        }
    }
}

// The same where rows are long on average, and a few much longer than that: a warp per CHUNK consecutive entries, whose rows
// it finds from the rows of every 32nd entry.  (A warp per row keeps one warp at the longest row of a power-law matrix while the
// others are done: 6.4e8 single-precision entries, 2 400 per row, product and mirror 28.83 ms, so 28.28.)
constexpr int COPY_CHUNK = 512;
constexpr int64_t COPY_LONG_ROWS = 256;  // entries per row from which on
template <typename V>
__global__ void __launch_bounds__(256) mirror_copy_chunks_kernel(const int64_t* __restrict__ l_rowptr, const int32_t* __restrict__ l_colidx,
                                                                 const V* __restrict__ l_vals, int64_t m, int64_t nnz, const int32_t* __restrict__ step_row,
                                                                 const int64_t* __restrict__ f_rowptr, int32_t* __restrict__ f_colidx, V* __restrict__ f_vals) {
    const int lane = lane_id();
    link(step_row, f_rowptr);
    const int64_t e0 = ((int64_t)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5)) * COPY_CHUNK;
    const int64_t e1 = min(e0 + COPY_CHUNK, nnz);
    auto row_of_step = [&](int64_t e) { return (int64_t)min((uint32_t)step_row[e >> 5], (uint32_t)(m - 1)); };  // e a multiple of 32
    int64_t r = e0 < e1 ? row_of_step(e0) : 0;
    for (int64_t p = e0; p < e1;) {  // entries [p, end) are of row r; uniform in the warp
        const int64_t end = min(l_rowptr[r + 1], e1);
        const int64_t shift = f_rowptr[r] - l_rowptr[r];
        constexpr int UNR = 8;
        for (int64_t q = p + lane; q < end; q += 32 * UNR) {
            int32_t j[UNR];
            V v[UNR];
#pragma unroll
            for (int u = 0; u < UNR; ++u) {
                if (q + 32 * u < end) {
                    j[u] = l_colidx[q + 32 * u];
                    v[u] = l_vals[q + 32 * u];
                }
            }
#pragma unroll
            for (int u = 0; u < UNR; ++u) {
                if (q + 32 * u < end) {
                    f_colidx[shift + q + 32 * u] = j[u];
                    f_vals[shift + q + 32 * u] = v[u];
                }
            }
        }
        if (end >= e1) break;
        // the row that holds entry `end`: one of the next 32, or searched for up to the row of the next step
        const int64_t next = r + 1 + lane;
        const unsigned after = __ballot_sync(FULL_MASK, next >= m || l_rowptr[next] > end);
        if (after) {
            r += __ffs(after) - 1;
        } else {
            int64_t lo = r + 32, hi = ((end >> 5) + 1) * 32 < nnz ? row_of_step(((end >> 5) + 1) * 32) : m - 1;
            while (lo < hi) {  // the last row that starts at or before the entry
                const int64_t mid = (lo + hi + 1) >> 1;
                if (l_rowptr[mid] <= end) lo = mid; else hi = mid - 1;
            }
            r = lo;
        }
        p = max(end, p + 1);  // (row pointers that do not ascend: still to the end)
    }
}

int group_width(int64_t nnz, int64_t m) {
    const double avg = m > 0 ? (double)nnz / (double)m : 0.0;
    return avg <= 4 ? 4 : avg <= 8 ? 8 : avg <= 16 ? 16 : 32;
}

template <typename V>
cudaError_t mirror_copy_lower(int64_t m, int64_t nnz_l, const int64_t* l_rowptr, const int32_t* l_colidx, const void* l_vals, const int64_t* f_rowptr, int32_t* f_colidx,
                              void* f_vals, cudaStream_t st) {
#define COPY(G)                                                                                                                                       \
    return launch_linked(mirror_copy_lower_kernel<V, G>, (unsigned)((m * G + 255) / 256), 256, 0, st, l_rowptr, l_colidx, static_cast<const V*>(l_vals), m, f_rowptr, \
                         f_colidx, static_cast<V*>(f_vals))
    switch (group_width(nnz_l, m)) {
        case 4: COPY(4);
        case 8: COPY(8);
        case 16: COPY(16);
        default: COPY(32);
    }
#undef COPY
}

// row lengths of F: the row's own entries and those of its column, the diagonal once
struct MirrorRowLength {
    using Value = int64_t;
    const int64_t* l_rowptr;
    const uint32_t* cnt;
    const uint8_t* diagf;
    __device__ __forceinline__ int64_t operator()(int64_t r) const { return l_rowptr[r + 1] - l_rowptr[r] + (int64_t)cnt[r] - (int64_t)diagf[r]; }
};
struct MirrorRowStart {
    const int64_t* l_rowptr;
    const uint8_t* diagf;
    int64_t* f_rowptr;
    int64_t* fstart;
    int64_t m;
    __device__ __forceinline__ void operator()(int64_t r, int64_t ex) const {
        f_rowptr[r] = ex;
        fstart[r] = ex + (l_rowptr[r + 1] - l_rowptr[r]) - (int64_t)diagf[r];
    }
    __device__ __forceinline__ void total(int64_t t) const { f_rowptr[m] = t; }
    __device__ __forceinline__ void gave_up() const {}
};

// Measurement aid: CUDA events around the sorting passes (each with its counts and scan).
bool g_mirror_timing = false;
constexpr int MIRROR_MAX_PASSES = 4;
cudaEvent_t g_mirror_ev[MIRROR_MAX_PASSES + 1];
int g_mirror_passes = 0;

void mirror_mark(int i, cudaStream_t st) {
    if (g_mirror_timing) cudaEventRecord(g_mirror_ev[i], st);
}

template <typename VB>
spsyrk_status_t mirror_fill(const MirrorWs& w, int64_t m, int64_t nnz_l, const int64_t* l_rowptr, const int32_t* l_colidx,
                            const void* l_vals, int64_t* f_rowptr, int32_t* f_colidx, void* f_vals, cudaStream_t st) {
    // F's arrays hold records and rests during the sort.  8-byte values: both must take 16-byte accesses.  4-byte values: the rests
    // are moved one by one and the records of 8 bytes begin at the first multiple of 8, one of them fewer.
    if (sizeof(VB) == 8 && nnz_l > 0 && ((reinterpret_cast<uintptr_t>(f_vals) | reinterpret_cast<uintptr_t>(f_colidx)) & 15u)) return SPSYRK_ERR_INVALID_ARG;
    const int64_t skipped = (reinterpret_cast<uintptr_t>(f_vals) & 7u) ? 1 : 0;
    if (m == 0 || nnz_l == 0) {
        SPSYRK_CUDA_TRY(cudaMemsetAsync(f_rowptr, 0, (size_t)(m + 1) * sizeof(int64_t), st));
        return SPSYRK_OK;
    }
    const MirrorSplit sp = mirror_split_for(m, nnz_l, sizeof(VB));
    const bool three = sp.mbits > 0;  // (4-byte values only)
    const int g = group_width(nnz_l, m);
    uint16_t* const f_high = reinterpret_cast<uint16_t*>(f_colidx);
    MirrorSortArgs a{};
    a.l_rowptr = l_rowptr; a.l_colidx = l_colidx; a.l_vals = l_vals; a.m = m; a.n = nnz_l; a.chunk = sp.chunk; a.nchunks = sp.nchunks;
    a.lbits = sp.lbits; a.mbits = sp.mbits; a.hbits = sp.hbits; a.step_row = w.step_row;
    a.mid_cap = sp.mid_cap; a.mid_units = (int)sp.mid_units; a.mid_first = w.mid_first; a.mid_bucket = w.mid_bucket;
    a.nbuckets = sp.nbuckets(); a.cap = sp.cap; a.max_pieces = (uint32_t)sp.max_pieces; a.pieces = w.pieces; a.first_piece = w.first_piece;
    a.piece = w.piece; a.piece_cnt = w.piece_cnt;
    a.split_off = w.offsets; a.mid_off = w.mid_off;
    a.rec_a = three ? static_cast<void*>(static_cast<char*>(f_vals) + 4 * skipped) : w.rec;
    a.rec_a_tail = w.rec_tail;
    a.a_split = three ? nnz_l - mirror_tail_records(m, nnz_l) - skipped : nnz_l;  // (the tail has room for one more)
    a.rec_b = w.rec;
    // the rests: the last pass reads them only for 4-byte values, and then not from F's memory
    uint16_t* const last_high = sizeof(VB) == 4 ? w.high : f_high;
    a.high_b = last_high;
    a.high_a = three ? f_high : last_high;
    a.cnt = w.cnt; a.fstart = w.fstart; a.f_colidx = f_colidx; a.f_vals = f_vals; a.err = w.err;
    const size_t split_smem = MirrorSplitSmem<VB>::bytes(1 << sp.lbits), place_smem = MirrorPlaceSmem<VB>::bytes(1 << sp.hbits);
    SPSYRK_CUDA_TRY(allow_shared_memory<mirror_split_kernel<VB>>());
    SPSYRK_CUDA_TRY(allow_shared_memory<mirror_place_kernel<VB>>());
    mirror_mark(0, st);
#define ROWS(G) mirror_rows_kernel<G><<<(unsigned)((m * G + 255) / 256), 256, 0, st>>>(l_rowptr, l_colidx, m, nnz_l, w.step_row, w.diagf, w.cnt, w.pieces, w.partials, w.state_words)
    if (g <= 16) ROWS(4); else ROWS(16);
#undef ROWS
    note_launches(1);
    SPSYRK_CUDA_TRY(launch_linked(mirror_split_count_kernel, (unsigned)sp.nchunks, MS_THREADS, 0, st, a, w.hist));
    SPSYRK_CUDA_TRY(exclusive_scan_i64<uint32_t>(w.hist, sp.split_hist(), w.offsets, w.split_state, w.err, st, true));
    SPSYRK_CUDA_TRY(launch_linked(mirror_split_kernel<VB>, (unsigned)sp.nchunks, MS_THREADS, split_smem, st, a));
    mirror_mark(1, st);
    int pass = 2;
    if (three) {
        const unsigned units = (unsigned)sp.mid_units;
        SPSYRK_CUDA_TRY(launch_linked(mirror_mid_count_kernel, units, MS_THREADS, 0, st, a, w.hist));
        SPSYRK_CUDA_TRY(exclusive_scan_i64<uint32_t>(w.hist, sp.mid_hist(), w.mid_off, w.mid_state, w.err, st, true));
        const size_t mid_smem = MirrorMidSmem::bytes(1 << sp.mbits);
        SPSYRK_CUDA_TRY(allow_shared_memory<mirror_mid_kernel>());
        SPSYRK_CUDA_TRY(launch_linked(mirror_mid_kernel, units, MS_THREADS, mid_smem, st, a));
        mirror_mark(pass++, st);
    }
    const unsigned place_units = (unsigned)(sp.nbuckets() + sp.max_pieces);
    SPSYRK_CUDA_TRY(launch_linked(mirror_column_count_kernel, place_units, MS_THREADS, 0, st, a, (const uint16_t*)last_high));
    SPSYRK_CUDA_TRY(scan_launch(MirrorRowLength{l_rowptr, w.cnt, w.diagf}, m, MirrorRowStart{l_rowptr, w.diagf, f_rowptr, w.fstart, m}, w.partials, w.err, st, true));
    SPSYRK_CUDA_TRY(launch_linked(mirror_place_kernel<VB>, place_units, MS_THREADS, place_smem, st, a));
    mirror_mark(pass, st);
    g_mirror_passes = pass;
    if (nnz_l / m >= COPY_LONG_ROWS) {
        constexpr int64_t per_cta = 8 * COPY_CHUNK;
        SPSYRK_CUDA_TRY(launch_linked(mirror_copy_chunks_kernel<VB>, (unsigned)((nnz_l + per_cta - 1) / per_cta), 256, 0, st, l_rowptr, l_colidx, static_cast<const VB*>(l_vals),
                                      m, nnz_l, (const int32_t*)w.step_row, (const int64_t*)f_rowptr, f_colidx, static_cast<VB*>(f_vals)));
    } else {
        SPSYRK_CUDA_TRY(mirror_copy_lower<VB>(m, nnz_l, l_rowptr, l_colidx, l_vals, f_rowptr, f_colidx, f_vals, st));
    }
    SPSYRK_CUDA_TRY(cudaGetLastError());
#ifdef SPSYRK_CHECKED
    {
        uint32_t e = 0;  // the bounds-checked build reports a skipped access at once (synchronises)
        SPSYRK_CUDA_TRY(cudaMemcpyAsync(&e, w.err, 4, cudaMemcpyDeviceToHost, st));
        SPSYRK_CUDA_TRY(cudaStreamSynchronize(st));
        if (e & ERRW_INTERNAL) return SPSYRK_ERR_INTERNAL;
    }
#endif
    return SPSYRK_OK;
}

// row lengths of F: the row's own entries and its column's segment of the sorted order
__global__ void mirror_rowlen_kernel(const int64_t* __restrict__ l_rowptr, const unsigned long long* __restrict__ seg_start,
                                     const unsigned long long* __restrict__ seg_end, int64_t m, uint32_t* __restrict__ rowtot) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= m) return;
    const unsigned long long s = seg_start[r], e = seg_end[r];
    rowtot[r] = (uint32_t)(l_rowptr[r + 1] - l_rowptr[r]) + (e > s ? (uint32_t)(e - s) : 0u);
}

// 4-byte values of more than 2^24 rows, or of few entries per bucket
spsyrk_status_t mirror_fill_radix(const MirrorWs& ws, int64_t m, int64_t nnz_l, const int64_t* l_rowptr, const int32_t* l_colidx, const void* l_vals,
                                  int64_t* f_rowptr, int32_t* f_colidx, void* f_vals, cudaStream_t st) {
    if (nnz_l == 0) {
        SPSYRK_CUDA_TRY(cudaMemsetAsync(f_rowptr, 0, (size_t)(m + 1) * sizeof(int64_t), st));
        return SPSYRK_OK;
    }
    MirrorWs w = ws;
    if (!w.key_a) { w.key_a = reinterpret_cast<uint32_t*>(f_colidx); w.val_a = f_vals; }
    if (!w.key_b) { w.key_b = reinterpret_cast<uint32_t*>(f_colidx); w.val_b = f_vals; }
    SPSYRK_CUDA_TRY(cudaMemsetAsync(w.seg_start, 0xff, (size_t)m * 8, st));
    SPSYRK_CUDA_TRY(cudaMemsetAsync(w.seg_end, 0, (size_t)m * 8, st));
    SPSYRK_CUDA_TRY(cudaMemsetAsync(w.rx.bins, 0, w.rx_bytes, st));
    mirror_mark(0, st);
#define EXPAND(G) mirror_expand_kernel<G><<<(unsigned)((m * G + 255) / 256), 256, 0, st>>>(l_rowptr, l_colidx, m, nnz_l, w.key_b, w.row_b)
    switch (group_width(nnz_l, m)) {
        case 4: EXPAND(4); break;
        case 8: EXPAND(8); break;
        case 16: EXPAND(16); break;
        default: EXPAND(32); break;
    }
#undef EXPAND
    note_launches(1);
    const int npass = radix_passes((uint64_t)m);
    const uint32_t *key = w.key_b, *row = w.row_b, *val = static_cast<const uint32_t*>(l_vals);
    SPSYRK_CUDA_TRY(radix_bins<false>(key, nnz_l, npass, w.rx.bins, st));
    for (int p = 0; p < npass; ++p) {
        const bool to_a = p % 2 == 0;
        if (p == npass - 1) {
            const EmitMirror emit{l_rowptr, (uint32_t)m, f_colidx, static_cast<uint32_t*>(f_vals), w.seg_start, w.seg_end};
            SPSYRK_CUDA_TRY((radix_pass<uint32_t, false>(key, row, val, nullptr, nnz_l, p, w.rx, emit, w.err, st)));
        } else {
            const EmitArrays<uint32_t> emit{to_a ? w.key_a : w.key_b, to_a ? w.row_a : w.row_b, static_cast<uint32_t*>(to_a ? w.val_a : w.val_b)};
            SPSYRK_CUDA_TRY((radix_pass<uint32_t, false>(key, row, val, nullptr, nnz_l, p, w.rx, emit, w.err, st)));
            key = emit.keys; row = emit.pa; val = emit.pb;
        }
        mirror_mark(p + 1, st);
        g_mirror_passes = p + 1;
    }
    mirror_rowlen_kernel<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(l_rowptr, w.seg_start, w.seg_end, m, w.rowtot);
    note_launches(1);
    SPSYRK_CUDA_TRY(exclusive_scan_i64<uint32_t>(w.rowtot, m, f_rowptr, w.partials, w.err, st));
    SPSYRK_CUDA_TRY(mirror_copy_lower<uint32_t>(m, nnz_l, l_rowptr, l_colidx, l_vals, f_rowptr, f_colidx, f_vals, st));
    SPSYRK_CUDA_TRY(cudaGetLastError());
    return SPSYRK_OK;
}

// 1 where row r stores its diagonal entry (rows are ascending: it is the last entry)
__global__ void mirror_diag_flag_kernel(const int64_t* __restrict__ l_rowptr, const int32_t* __restrict__ l_colidx, int64_t m,
                                        uint32_t* __restrict__ diagf) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= m) return;
    const int64_t p0 = l_rowptr[r], p1 = l_rowptr[r + 1];
    diagf[r] = (p1 > p0 && (int64_t)l_colidx[p1 - 1] == r) ? 1u : 0u;
}

__global__ void mirror_fbase_kernel(const int64_t* __restrict__ l_rowptr, const int64_t* __restrict__ dcount, int64_t m,
                                    int64_t* __restrict__ fbase) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j < m) fbase[j] = l_rowptr[j + 1] - dcount[j + 1];
}

// row lengths of F when the sorted segments include the diagonal entries
__global__ void mirror_rowlen_diag_kernel(const int64_t* __restrict__ l_rowptr, const unsigned long long* __restrict__ seg_start,
                                          const unsigned long long* __restrict__ seg_end, const uint32_t* __restrict__ diagf, int64_t m,
                                          uint32_t* __restrict__ rowtot) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= m) return;
    const unsigned long long s = seg_start[r], e = seg_end[r];
    const uint32_t seg = e > s ? (uint32_t)(e - s) : 0u;
    rowtot[r] = (uint32_t)(l_rowptr[r + 1] - l_rowptr[r]) + (seg >= diagf[r] ? seg - diagf[r] : 0u);
}

template <bool FROM_CSR, bool FINAL>
cudaError_t launch_mirror_pass(const MirrorPassArgs& a, int64_t n, int shift, const int64_t* offsets, int64_t nt, cudaStream_t st) {
    constexpr int BITS = MIRROR_RADIX_BITS;
    auto kern = mirror_pass_kernel<BITS, FROM_CSR, FINAL>;
    const size_t smem = MirrorPassSmem<BITS>::bytes();
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)nt, MR_THREADS, smem, st>>>(a, n, shift, offsets, nt);
    note_launches(1);
    return cudaGetLastError();
}

// 8-byte values: records, the first pass straight from C_L
spsyrk_status_t mirror_fill_rec(const MirrorWs& w, int64_t m, int64_t nnz_l, const int64_t* l_rowptr, const int32_t* l_colidx,
                                const void* l_vals, int64_t* f_rowptr, int32_t* f_colidx, void* f_vals, cudaStream_t st) {
    constexpr int BITS = MIRROR_RADIX_BITS;
    constexpr int NB = 1 << BITS;
    const uint64_t* lv = static_cast<const uint64_t*>(l_vals);
    uint64_t* fv = static_cast<uint64_t*>(f_vals);
    // F's arrays hold records and digit bytes during the sort: both must take 16-byte accesses
    if (nnz_l > 0 && ((reinterpret_cast<uintptr_t>(f_vals) | reinterpret_cast<uintptr_t>(f_colidx)) & 15u)) return SPSYRK_ERR_INVALID_ARG;
    if (m > 0) {
        SPSYRK_CUDA_TRY(cudaMemsetAsync(w.seg_start, 0xff, (size_t)m * 8, st));
        SPSYRK_CUDA_TRY(cudaMemsetAsync(w.seg_end, 0, (size_t)m * 8, st));
        mirror_diag_flag_kernel<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(l_rowptr, l_colidx, m, w.diagf32);
        note_launches(1);
    }
    SPSYRK_CUDA_TRY(exclusive_scan_i64<uint32_t>(w.diagf32, m, w.dcount, w.partials, w.err, st));
    if (m > 0 && nnz_l > 0) {
        mirror_fbase_kernel<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(l_rowptr, w.dcount, m, w.fbase);
        note_launches(1);
        const int npass = (bits_for((uint64_t)(m - 1 > 0 ? m - 1 : 1)) + BITS - 1) / BITS;  // keys are column ids below m
        const int64_t nt = mirror_groups(nnz_l);  // histogram columns and CTAs of a pass
        const int64_t ntr = mirror_tiles(nnz_l);
        mirror_tile_rows_kernel<<<(unsigned)((2 * ntr + 255) / 256), 256, 0, st>>>(l_rowptr, m, nnz_l, ntr, w.tile_rows);
        note_launches(1);
        MirrorPassArgs a{};
        a.l_rowptr = l_rowptr; a.l_colidx = l_colidx; a.l_vals = lv; a.m = m; a.tile_rows = w.tile_rows;
        a.fbase = w.fbase; a.f_colidx = f_colidx; a.f_vals = fv; a.seg_start = w.seg_start; a.seg_end = w.seg_end;
        a.dtotal = w.dcount + m; a.err = w.err;
        g_mirror_passes = 0;
        // buffers: pass p writes records X[p] and digits Y[p]; X[npass - 2] is the one the last pass reads
        MirrorRec* const alias = reinterpret_cast<MirrorRec*>(fv);
        const int64_t alias_split = nnz_l - mirror_tail_records(m, nnz_l);
        const int64_t dig_stride = (nnz_l + 15) / 16 * 16;
        uint8_t* const dig0 = nnz_l < MIRROR_DIG_SMALL ? w.dig_small : reinterpret_cast<uint8_t*>(f_colidx);
        uint8_t* const dig1 = nnz_l < MIRROR_DIG_SMALL ? w.dig_small + MIRROR_DIG_SMALL : dig0 + dig_stride;
        auto in_keep = [&](int p) { return ((npass - 2 - p) % 2) == 0; };  // does pass p write the workspace buffer?
        for (int p = 0; p < npass; ++p) {
            const bool first = p == 0, last = p == npass - 1;
            if (first) mirror_mark(0, st);
            const unsigned hb = (unsigned)((nt + MR_HIST_TILES - 1) / MR_HIST_TILES);
            if (first) mirror_hist_key_kernel<BITS><<<hb, MR_THREADS, 0, st>>>(reinterpret_cast<const uint32_t*>(l_colidx), nnz_l, 0, w.hist, nt);
            else radix_hist_u8_kernel<BITS><<<hb, MR_THREADS, 0, st>>>(((p - 1) % 2) == 0 ? dig0 : dig1, nnz_l, w.hist, nt);
            note_launches(1);
            SPSYRK_CUDA_TRY(exclusive_scan_i64<uint32_t>(w.hist, (int64_t)NB * nt, w.offsets, w.partials, w.err, st));
            const bool src_keep = !first && in_keep(p - 1), dst_keep = in_keep(p);
            a.src = src_keep ? w.rec_keep : alias;
            a.src_tail = w.rec_keep_tail;
            a.src_split = src_keep ? nnz_l : alias_split;
            a.dst = dst_keep ? w.rec_keep : alias;
            a.dst_tail = w.rec_keep_tail;
            a.dst_split = dst_keep ? nnz_l : alias_split;
            a.next_digit = (p % 2) == 0 ? dig0 : dig1;
            cudaError_t e;
            if (first && last) e = launch_mirror_pass<true, true>(a, nnz_l, p * BITS, w.offsets, nt, st);
            else if (first) e = launch_mirror_pass<true, false>(a, nnz_l, p * BITS, w.offsets, nt, st);
            else if (last) e = launch_mirror_pass<false, true>(a, nnz_l, p * BITS, w.offsets, nt, st);
            else e = launch_mirror_pass<false, false>(a, nnz_l, p * BITS, w.offsets, nt, st);
            SPSYRK_CUDA_TRY(e);
            mirror_mark(p + 1, st);
            g_mirror_passes = p + 1;
        }
    }
    if (m > 0) {
        mirror_rowlen_diag_kernel<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(l_rowptr, w.seg_start, w.seg_end, w.diagf32, m, w.rowtot);
        note_launches(1);
    }
    SPSYRK_CUDA_TRY(exclusive_scan_i64<uint32_t>(w.rowtot, m, f_rowptr, w.partials, w.err, st));
    if (m > 0 && nnz_l > 0) SPSYRK_CUDA_TRY(mirror_copy_lower<uint64_t>(m, nnz_l, l_rowptr, l_colidx, l_vals, f_rowptr, f_colidx, f_vals, st));
    SPSYRK_CUDA_TRY(cudaGetLastError());
#ifdef SPSYRK_CHECKED
    {
        uint32_t e = 0;  // the bounds-checked build reports a skipped access at once (synchronises)
        SPSYRK_CUDA_TRY(cudaMemcpyAsync(&e, w.err, 4, cudaMemcpyDeviceToHost, st));
        SPSYRK_CUDA_TRY(cudaStreamSynchronize(st));
        if (e & ERRW_INTERNAL) return SPSYRK_ERR_INTERNAL;
    }
#endif
    return SPSYRK_OK;
}

}  // namespace

extern "C" spsyrk_status_t spsyrk_mirror(int64_t m, int64_t nnz_l, spsyrk_dtype_t dtype, const int64_t* d_l_rowptr,
                                         const int32_t* d_l_colidx, const void* d_l_vals, int64_t* d_f_rowptr,
                                         int32_t* d_f_colidx, void* d_f_vals, int64_t* nnz_full_out, void* d_workspace,
                                         size_t* workspace_bytes, void* cuda_stream) {
    if (!workspace_bytes || m < 0 || nnz_l < 0) return SPSYRK_ERR_INVALID_ARG;
    if (dtype != SPSYRK_F64 && dtype != SPSYRK_F32 && dtype != SPSYRK_I32) return SPSYRK_ERR_INVALID_ARG;
    if (m >= (int64_t(1) << 31) - 1) return SPSYRK_ERR_OVERFLOW;
    const size_t sv = dtype == SPSYRK_F64 ? 8 : 4;
    const size_t need = carve(nullptr, nullptr, m, nnz_l, sv);
    if (!d_workspace) {
        *workspace_bytes = need;
        return SPSYRK_OK;
    }
    if (*workspace_bytes < need) return SPSYRK_ERR_WORKSPACE;
    if (reinterpret_cast<uintptr_t>(d_workspace) % ALIGN) return SPSYRK_ERR_INVALID_ARG;
    if (!d_l_rowptr || !d_f_rowptr || (nnz_l > 0 && !d_l_colidx)) return SPSYRK_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    MirrorWs w;
    carve(&w, d_workspace, m, nnz_l, sv);

    if (!d_f_colidx) {  // step 2: checks and nnz(F)
        if (!nnz_full_out) return SPSYRK_ERR_INVALID_ARG;
        *nnz_full_out = 0;
        SPSYRK_CUDA_TRY(cudaMemsetAsync(w.err, 0, 12, st));
        if (m > 0) {
            ScopedHostBlock h;
            SPSYRK_CUDA_TRY(h.acquire());
            mirror_last_entry_kernel<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(d_l_rowptr, d_l_colidx, m, w.err, h.dev);
            note_launches(1);
            SPSYRK_CUDA_TRY(cudaGetLastError());
            SPSYRK_CUDA_TRY(cudaStreamSynchronize(st));
            if (h.host[1]) return status_of((uint32_t)h.host[1]);
            *nnz_full_out = 2 * nnz_l - h.host[0];
        }
        return SPSYRK_OK;
    }
    // step 3: fill
    if (!d_f_vals || (nnz_l > 0 && !d_l_vals)) return SPSYRK_ERR_INVALID_ARG;
    switch (dtype) {
        case SPSYRK_F64:
            if (mirror_by_records(m, sv)) return mirror_fill_rec(w, m, nnz_l, d_l_rowptr, d_l_colidx, d_l_vals, d_f_rowptr, d_f_colidx, d_f_vals, st);
            return mirror_fill<uint64_t>(w, m, nnz_l, d_l_rowptr, d_l_colidx, d_l_vals, d_f_rowptr, d_f_colidx, d_f_vals, st);
        default:
            if (mirror_by_radix(m, nnz_l, sv)) return mirror_fill_radix(w, m, nnz_l, d_l_rowptr, d_l_colidx, d_l_vals, d_f_rowptr, d_f_colidx, d_f_vals, st);
            return mirror_fill<uint32_t>(w, m, nnz_l, d_l_rowptr, d_l_colidx, d_l_vals, d_f_rowptr, d_f_colidx, d_f_vals, st);
    }
}


extern "C" spsyrk_status_t spsyrk_mirror_enable_timing(int on) {
    if (on && !g_mirror_timing) {
        for (int i = 0; i <= MIRROR_MAX_PASSES; ++i) SPSYRK_CUDA_TRY(cudaEventCreate(&g_mirror_ev[i]));
        g_mirror_passes = 0;
    } else if (!on && g_mirror_timing) {
        for (int i = 0; i <= MIRROR_MAX_PASSES; ++i) cudaEventDestroy(g_mirror_ev[i]);
    }
    g_mirror_timing = on != 0;
    return SPSYRK_OK;
}

extern "C" spsyrk_status_t spsyrk_mirror_timings(int* passes, float pass_ms[4]) {
    if (!passes || !pass_ms || !g_mirror_timing) return SPSYRK_ERR_INVALID_ARG;
    *passes = g_mirror_passes;
    for (int p = 0; p < g_mirror_passes; ++p) {
        pass_ms[p] = 0.f;
        SPSYRK_CUDA_TRY(cudaEventSynchronize(g_mirror_ev[p + 1]));
        SPSYRK_CUDA_TRY(cudaEventElapsedTime(&pass_ms[p], g_mirror_ev[p], g_mirror_ev[p + 1]));
    }
    return SPSYRK_OK;
}

// ------------------------------------------------------------------------------------------
// Allocation-free computation of F's row pointers and entry count (what steps 2 and 3 of
// spsyrk_mirror deliver between them).
//
// Some callers have no device memory to lend and may not create any: a plug-in running inside a
// host application that has claimed the whole GPU for its own memory pool, or a service loop that
// cannot afford the device-wide synchronisation a cudaMalloc / cudaFree may bring.  For them the
// scratch of this one step lives in a fixed array that is part of the library image, so the call
// needs nothing but its inputs and outputs.  The price: the array occupies its bytes on every GPU
// that loads the library until the process exits, and the problem size is capped.
// ------------------------------------------------------------------------------------------
namespace {

constexpr int64_t NOALLOC_MAX_ROWS = SPSYRK_NOALLOC_MAX_ROWS;
// strictly-lower counts (4 B per row), row totals (4 B per row), scan partials, one error word
constexpr size_t NOALLOC_UCNT_OFF = 0;
constexpr size_t NOALLOC_ROWTOT_OFF = NOALLOC_UCNT_OFF + (size_t)NOALLOC_MAX_ROWS * 4;
constexpr size_t NOALLOC_PARTIALS_OFF = NOALLOC_ROWTOT_OFF + (size_t)NOALLOC_MAX_ROWS * 4;
constexpr size_t NOALLOC_PARTIALS_BYTES = ((size_t)(NOALLOC_MAX_ROWS / SCAN_MIN_TILE) + 2) * 8;
constexpr size_t NOALLOC_ERR_OFF = (NOALLOC_PARTIALS_OFF + NOALLOC_PARTIALS_BYTES + 255) / 256 * 256;
constexpr size_t NOALLOC_BYTES = NOALLOC_ERR_OFF + 256;

// In host code this name is only a handle for the runtime, not a device address: the address is
// looked up once per device with cudaGetSymbolAddress and that pointer is what the kernels receive.
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_BYTES];

constexpr int NOALLOC_MAX_DEVICES = 64;
std::mutex g_noalloc_mutex;
unsigned char* g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {};

// device address of the scratch array on the current device (set up on the first call per device)
cudaError_t noalloc_scratch(unsigned char** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        g_noalloc_ptr[dev] = static_cast<unsigned char*>(p);
    }
    *out = g_noalloc_ptr[dev];
    return cudaSuccess;
}

}  // namespace

extern "C" spsyrk_status_t spsyrk_mirror_rowptr_noalloc(int64_t m, const int64_t* d_l_rowptr, const int32_t* d_l_colidx,
                                                        int64_t* d_f_rowptr, int64_t* nnz_full_out, void* cuda_stream) {
    if (m < 0 || !d_l_rowptr || !d_f_rowptr || !nnz_full_out) return SPSYRK_ERR_INVALID_ARG;
    if (m > NOALLOC_MAX_ROWS) return SPSYRK_ERR_OVERFLOW;  // beyond the fixed scratch: use spsyrk_mirror
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    unsigned char* base = nullptr;
    SPSYRK_CUDA_TRY(noalloc_scratch(&base));
    uint32_t* ucnt = reinterpret_cast<uint32_t*>(base + NOALLOC_UCNT_OFF);
    uint32_t* rowtot = reinterpret_cast<uint32_t*>(base + NOALLOC_ROWTOT_OFF);
    int64_t* partials = reinterpret_cast<int64_t*>(base + NOALLOC_PARTIALS_OFF);
    uint32_t* err = reinterpret_cast<uint32_t*>(base + NOALLOC_ERR_OFF);
    // the array keeps whatever the previous call left: clear what is accumulated into
    SPSYRK_CUDA_TRY(cudaMemsetAsync(err, 0, 4, st));
    if (m > 0) {
        SPSYRK_CUDA_TRY(cudaMemsetAsync(ucnt, 0, (size_t)m * 4, st));
        // row lengths are not known on the host here, so the widest lane grouping is used
        mirror_count_kernel<32><<<(unsigned)((m * 32 + 255) / 256), 256, 0, st>>>(d_l_rowptr, d_l_colidx, m, ucnt, err);
        mirror_rowtot_kernel<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(d_l_rowptr, ucnt, m, rowtot);
        note_launches(2);
    }
    SPSYRK_CUDA_TRY(exclusive_scan_i64<uint32_t>(rowtot, m, d_f_rowptr, partials, err, st));
    int64_t nnz = 0;
    uint32_t e = 0;
    SPSYRK_CUDA_TRY(cudaMemcpyAsync(&nnz, d_f_rowptr + m, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    SPSYRK_CUDA_TRY(cudaMemcpyAsync(&e, err, 4, cudaMemcpyDeviceToHost, st));
    SPSYRK_CUDA_TRY(cudaStreamSynchronize(st));
    if (e) return status_of(e);
    *nnz_full_out = nnz;
    return SPSYRK_OK;
}
