// Step a1: on-device CSR transpose of A into column lists whose entries are ascending by row,
// plus the per-nonzero descriptors the row kernels consume.
//
//   colptr[n+1]        column pointers (int64)
//   at_row[q], at_rec[q]  entries of the column lists, q in [colptr[k], colptr[k+1]) ascending by row: the row ids
//                      alone (what the structure passes read) and (row id, value) records (what the value passes read)
//   desc[p] = (start, len) for nonzero p = (i, k) of A: start = colptr[k]; len = number of entries
//             of column k with row <= i (the rank of i in the list, plus one).  "Rows j <= i of
//             column k" is then at_row[start, start+len).  The full-output mode also keeps the rest of
//             the list, the rows j > i, as a second descriptor (start + len, column length - len).
//
// Method: histogram of column ids and scan for colptr; then a stable LSD radix sort of the
// nonzeros by column id with (row, value, position in A) as payload.  The nonzeros enter in row
// order, so each column's segment comes out ascending by row; the last pass writes at_row and
// at_rec and scatters the descriptor, whose length is the entry's rank inside its column.  (The
// value travels with the element because reading it in the first pass is sequential, whereas
// fetching it by position in the last pass is one random access per nonzero.)
#pragma once
#include "radix.cuh"

namespace spsyrk {

// granularity of the per-row entry counts that the symbolic pass keeps for the heavy rows (columns)
constexpr uint32_t BASE_BLOCK = 8192;

constexpr int HEAVY_PLANES = 4;
constexpr int HEAVY_MAX = 32 * HEAVY_PLANES;

struct PlanDev {
    int32_t m, n;
    int64_t nnz;
    int32_t r0, r1;
    int32_t mode;
    const int64_t* rowptr;
    const int32_t* colidx;
    const void* vals;
    int64_t* colptr;
    int32_t* at_row;
    // (the values of the column lists live in the records only)
    void* at_rec;  // the same entries as interleaved (row id, value) records: ColRec<V>[nnz]
    uint2* desc;
    int64_t* work;  // per row of the range
    uint32_t* err;
    // Binary input (every stored value is exactly one): a partial product is 1 and an entry of the
    // product is an intersection count.  Then the heaviest columns (at most HEAVY_MAX, chosen by their number
    // of entries) are also kept as one bit per row, in planes of 32 columns: bit b of heavy_mask[p * mask_stride + i] =
    // row i stores heavy column 32 p + b, so that their share of a count is the population count of two rows' common
    // bits instead of one list walk each.  (On the Zipf workloads 128 columns leave 0.7 of 16 products per entry
    // to the walks, 64 columns 1.5.)
    int32_t binary;               // 0 / 1, valid after the plan's analysis
    const uint32_t* nheavy;       // heavy columns in use (0: none), device memory, written when the matrix is binary
    const uint8_t* heavy_id;      // [n] bit number of a heavy column, 0xff otherwise
    const uint32_t* heavy_mask;   // [HEAVY_PLANES][mask_stride]
    int64_t mask_stride;          // m rounded up to four
    float* jaccard;               // optional: the numeric pass also writes c / (|a_i| + |a_j| - c) here (int32 values)
    const int32_t* adeg;          // [m] stored entries per row of A (|a_i| of the Jaccard formula)
};

// ---------------------------------------------------------------------------------------------
// Analysis of a binary matrix (every stored value is one, see row_expand_kernel): choice of the heavy columns, the
// per-row bit masks.  The host does not know yet whether the matrix is binary: the CTAs return at once if it is not.
// facts[0] = 1 if some stored value differs from one; facts[1] = heavy columns; facts[32..] histogram.
// ---------------------------------------------------------------------------------------------
// histogram of the column lengths, four bins per octave
constexpr int HEAVY_BINS = 128;
__device__ __forceinline__ int heavy_bin(uint32_t d) {
    const int e = 31 - __clz(d);
    return 4 * e + (int)((d >> (e - 2)) & 3u);
}
// (few columns are that long: a look at the flag and an atomic each, beside the digit counts of the sort)
struct HeavyHistogram {
    uint32_t* facts;
    __device__ __forceinline__ void operator()(uint32_t d) const {
        if (d >= 256u && facts[0] == 0) atomicAdd(&facts[32 + heavy_bin(d)], 1u);  // lighter columns are never candidates
    }
};

// Columns of at least the threshold get a bit number; the threshold is the smallest bin such that at most HEAVY_MAX
// columns lie in it and above.  Part `part` of `parts`, BIN_THREADS threads.
static __device__ void heavy_assign(const uint32_t* __restrict__ colcnt, int64_t n, uint32_t* facts, uint8_t* heavy_id, int64_t part, int64_t parts) {
    __shared__ uint32_t s_thr;
    if (threadIdx.x < 32) {
        const int e = 31 - (int)threadIdx.x;  // lane l looks at the octave from 2^(31 - l)
        uint32_t c[4], sum = 0;
#pragma unroll
        for (int f = 0; f < 4; ++f) { c[f] = facts[32 + 4 * e + f]; sum += c[f]; }
        uint32_t above = warp_inclusive_scan<uint32_t>(sum) - sum, cand = 0xffffffffu;
#pragma unroll
        for (int f = 3; f >= 0; --f) {
            above += c[f];
            if (e >= 8 && above <= (uint32_t)HEAVY_MAX && c[f]) cand = (uint32_t)(4 + f) << (e - 2);
        }
        cand = __reduce_min_sync(FULL_MASK, cand);
        if (threadIdx.x == 0) s_thr = cand;
    }
    __syncthreads();
    const uint32_t thr = s_thr;
    if (thr == 0xffffffffu) return;  // no heavy column: nothing reads the bit numbers
    for (int64_t k = part * BIN_THREADS + threadIdx.x; k < n; k += parts * BIN_THREADS) {
        uint8_t id = 0xff;
        if (colcnt[k] >= thr) {
            const uint32_t b = atomicAdd(&facts[1], 1u);
            if (b < (uint32_t)HEAVY_MAX) id = (uint8_t)b;
        }
        heavy_id[k] = id;
    }
}

// The rows' masks, G lanes per row; the bit numbers were written by other CTAs of the same launch.
template <int G>
static __device__ void heavy_masks(const int64_t* __restrict__ rowptr, const int32_t* __restrict__ colidx, int32_t m, const uint8_t* heavy_id,
                                   uint32_t* __restrict__ heavy_mask, int64_t mask_stride, int64_t part, int64_t parts) {
    const int gl = threadIdx.x & (G - 1);
    constexpr int GROUPS = BIN_THREADS / G;
    for (int64_t base = part * GROUPS; base < m; base += parts * GROUPS) {  // uniform per CTA
        const int64_t gid = base + threadIdx.x / G;
        uint32_t mk[HEAVY_PLANES] = {};
        if (gid < m) {
            const int64_t p0 = rowptr[gid], p1 = rowptr[gid + 1];
            for (int64_t p = p0 + gl; p < p1; p += G) {
                const uint8_t id = __ldcg(heavy_id + colidx[p]);
#pragma unroll
                for (int q = 0; q < HEAVY_PLANES; ++q)
                    if ((id >> 5) == q) mk[q] |= 1u << (id & 31);  // (0xff belongs to no plane)
            }
        }
#pragma unroll
        for (int q = 0; q < HEAVY_PLANES; ++q) {
#pragma unroll
            for (int o = G / 2; o > 0; o >>= 1) mk[q] |= __shfl_xor_sync(FULL_MASK, mk[q], o);
            if (gid < m && gl == 0) heavy_mask[q * mask_stride + gid] = mk[q];
        }
    }
}

// The analysis as one of `ctas` CTAs beside the work estimate (which it does not depend on): as launches of their own
// the two steps cost every plan 6 us, binary or not.  The CTAs that start first hand out the bit numbers and
// return; the others wait for them, and then build the masks.
struct HeavyArrays {
    const uint32_t* colcnt;
    uint32_t* facts;  // [2] CTAs that have started, [3] CTAs whose share of the bit numbers is written
    uint8_t* heavy_id;
    uint32_t* heavy_mask;
    uint32_t ctas;
};
template <int G>
static __device__ void heavy_analysis(const PlanDev& P, const HeavyArrays& H) {
    __shared__ uint32_t s_ticket;
    // the matrix is not binary, or it failed its checks and has column ids that index nothing
    if (H.facts[0] != 0 || (*P.err & ERRW_BAD_CSR) != 0) return;
    if (threadIdx.x == 0) s_ticket = atomicAdd(&H.facts[2], 1u);
    __syncthreads();
    const uint32_t ticket = s_ticket, assigning = (H.ctas + 3) / 4;
    if (ticket < assigning) {
        heavy_assign(H.colcnt, P.n, H.facts, H.heavy_id, ticket, assigning);
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) atomicAdd(&H.facts[3], 1u);
        return;
    }
    if (threadIdx.x == 0) {
        int polls = 0;
        while (ld_status(&H.facts[3]) < assigning && polls < SPIN_LIMIT) ++polls;
        if (polls == SPIN_LIMIT) atomicOr(P.err, ERRW_INTERNAL);
        __threadfence();
    }
    __syncthreads();
    if (ld_status(&H.facts[1]) == 0) return;  // no heavy column: nothing reads the masks
    heavy_masks<G>(P.rowptr, P.colidx, P.m, H.heavy_id, H.heavy_mask, P.mask_stride, ticket - assigning, H.ctas - assigning);
}
// without rows to estimate the work of
template <int G>
static __global__ void __launch_bounds__(BIN_THREADS) heavy_analysis_kernel(PlanDev P, HeavyArrays H) { heavy_analysis<G>(P, H); }

// a row's bits of the heavy columns (planes in use: 32 columns each)
struct HeavyMask {
    uint32_t w[HEAVY_PLANES];
};
__device__ __forceinline__ HeavyMask load_heavy_mask(const PlanDev& P, int64_t i, int planes) {
    HeavyMask k;
#pragma unroll
    for (int p = 0; p < HEAVY_PLANES; ++p) k.w[p] = p < planes ? P.heavy_mask[p * P.mask_stride + i] : 0u;
    return k;
}
__device__ __forceinline__ int heavy_planes(const PlanDev& P) { return (int)((min(*P.nheavy, (uint32_t)HEAVY_MAX) + 31u) / 32u); }

// One entry of a column list as a record: what the light-row numeric kernel gathers (one aligned
// asynchronous copy per entry, whatever the list's offset).
template <typename V> struct ColRec;
template <> struct alignas(16) ColRec<double> { int32_t j; int32_t pad; double v; };
template <> struct alignas(8) ColRec<float> { int32_t j; float v; };
template <> struct alignas(8) ColRec<int32_t> { int32_t j; int32_t v; };

// Rows of more than so many steps of their G lanes are left to the whole CTA at the end: the longest row of a power-law
// matrix (15 711 nonzeros at 2^18 rows) kept its 16 lanes busy for most of the
// kernel's 401 us (product and mirror of that matrix 30.63 -> 30.23 ms, of 2^13 rows 352 -> 333 us, row_work_kernel's share included).
constexpr int LONG_STEPS = 8;

// G lanes per row, one sweep over the nonzeros of A: the checks of the row pointers (a row indexes nothing unless its own
// two are sane) and of the column ids (in range, strictly ascending inside the row), the column histogram (its scan gives
// colptr), the explicit row id of every nonzero (the radix sort's first payload), the row lengths, and whether
// every stored value is one.  Nothing waits for the checks: the kernels up to the plan's one synchronisation test what
// they index by, or look at the error word first.  Bound by the atomic adds of the histogram (1.4e11 per second on 6.7e7
// random columns).
template <int G, typename V>
static __global__ void __launch_bounds__(256) row_expand_kernel(const int64_t* __restrict__ rowptr, const int32_t* __restrict__ colidx,
                                                                const V* __restrict__ vals, int32_t m, int32_t n, int64_t nnz,
                                                                uint32_t* __restrict__ colcnt, uint32_t* __restrict__ rowid,
                                                                int32_t* __restrict__ adeg, uint32_t* facts, uint32_t* err) {
    __shared__ int32_t s_long[256 / G];
    __shared__ int s_nlong;
    const int64_t gid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    const int gl = threadIdx.x & (G - 1);
    bool look = __ldca(facts) == 0;  // values are looked at until one differs from one (an old zero only costs a look)
    bool other = false, is_long = false;
    auto entry = [&](int64_t p, int64_t p0, int64_t row) {
        const int32_t k = colidx[p];
        if (look) {
            other = !(vals[p] == V(1));
            look = !other;
        }
        if ((uint32_t)k >= (uint32_t)n) atomicOr(err, ERRW_BAD_COL);
        else atomicAdd(&colcnt[k], 1u);
        if (p > p0 && colidx[p - 1] >= k) atomicOr(err, ERRW_UNSORTED);
        rowid[p] = (uint32_t)row;
    };
    if (gid < m) {
        const int64_t p0 = rowptr[gid], p1 = rowptr[gid + 1];
        if (gl == 0) adeg[gid] = (int32_t)(p1 - p0);
        if (p0 > p1 || p0 < 0 || p1 > nnz) {
            atomicOr(err, ERRW_BAD_ROWPTR);
        } else if (p1 - p0 > LONG_STEPS * G) {
            is_long = true;
        } else {
            for (int64_t p = p0 + gl; p < p1; p += G) entry(p, p0, gid);
        }
    }
    if (__syncthreads_or(is_long)) {
        if (threadIdx.x == 0) s_nlong = 0;
        __syncthreads();
        if (is_long && gl == 0) s_long[atomicAdd(&s_nlong, 1)] = (int32_t)gid;
        __syncthreads();
        for (int i = 0; i < s_nlong; ++i) {
            const int64_t row = s_long[i];
            const int64_t p0 = rowptr[row], p1 = rowptr[row + 1];
            for (int64_t p = p0 + threadIdx.x; p < p1; p += 256) entry(p, p0, row);
        }
    }
    if (gid == 0 && gl == 0 && (rowptr[0] != 0 || rowptr[m] != nnz)) atomicOr(err, ERRW_BAD_ROWPTR);
    if (__any_sync(FULL_MASK, other) && lane_id() == 0) atomicOr(facts, 1u);  // (few: only the CTAs that started before the first)
}

// last radix pass of the transpose: the element at sorted position s is entry s of the column lists
template <typename VB>
struct EmitTransposeFinal {
    PlanDev P;
    uint2* desc_hi;  // null in lower-triangle mode
    __device__ __forceinline__ void operator()(int64_t s, uint32_t k, uint32_t row, VB val, uint32_t p) const {
        // A matrix that failed its checks (reported when the plan synchronises): keys that were not counted leave places of a
        // pass's output unwritten, so the next pass may bring any key and any position.
        if (k >= (uint32_t)P.n || (int64_t)p >= P.nnz) return;
        const int64_t cs = P.colptr[k];
        P.at_row[s] = (int32_t)row;
        if constexpr (sizeof(VB) == 8) static_cast<uint4*>(P.at_rec)[s] = make_uint4(row, 0u, (uint32_t)val, (uint32_t)(val >> 32));
        else static_cast<uint2*>(P.at_rec)[s] = make_uint2(row, (uint32_t)val);
        // the entries of column k with row <= i are the first rank + 1 of its list; the full-output mode also keeps
        // the rest of the list (rows > i) as a second descriptor
        const uint32_t rank1 = (uint32_t)(s - cs) + 1u;
        P.desc[p] = make_uint2((uint32_t)cs, rank1);
        if (desc_hi) desc_hi[p] = make_uint2((uint32_t)cs + rank1, (uint32_t)(P.colptr[k + 1] - cs) - rank1);
    }
};

// Restriction of the plan to output columns [s0, s1): column k's entries with row in that range are
// a contiguous piece of its (row-sorted) list, so the descriptor of every nonzero of the rows
// [r0, r1) is narrowed to that piece by two binary searches inside its full-range prefix.
template <int G>
// desc_hi (full-output mode): the rest of every column list; the block is then cut out of the whole list.
static __global__ void __launch_bounds__(256) block_desc_kernel(PlanDev P, const uint2* __restrict__ desc_full, const uint2* __restrict__ desc_hi,
                                                                uint2* __restrict__ desc_blk, int32_t s0, int32_t s1) {
    const int64_t gid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    const int gl = threadIdx.x & (G - 1);
    if (gid >= P.r1 - P.r0) return;
    const int64_t i = P.r0 + gid;
    const int64_t p0 = P.rowptr[i], p1 = P.rowptr[i + 1];
    for (int64_t p = p0 + gl; p < p1; p += G) {
        uint2 full = desc_full[p];
        if (desc_hi) full.y += desc_hi[p].y;
        const int32_t* lst = P.at_row + full.x;
        const uint32_t lo = s0 <= 0 ? 0u : lower_bound_i32(lst, full.y, s0);
        const uint32_t hi = lower_bound_i32(lst, full.y, s1);
        desc_blk[p] = make_uint2(full.x + lo, hi > lo ? hi - lo : 0u);
    }
}

constexpr int ROW_DENSE = 8;  // beside the class in cls[]: every column of the row's range is stored
// Step a2: per-row work w[i] = sum of the descriptor lengths of row i (G lanes per row), the class of the row and
// the number of rows of every class in every CTA's tile (the first half of a stable counting sort by class).
//   class 0: no work; 1..5: w <= 32, 64, 128, 256, 512 and at most 32 nonzeros (one warp, register sort)
//   6: w <= block_max (block class, bitmap accumulator); 7: larger (one 1024-thread CTA)
//   A heavy row that stores a column of every row of its range (of at most dense_range rows) is dense: it is marked here,
//   row_scatter_kernel settles its count, and a class with nothing but dense rows needs no counting kernel (50 000 such rows,
//   a CTA each that only looked at the descriptors: 311 us)
//   diag: the light-row kernels leave the diagonal products out of their item lists (lower-triangle mode
//   over the whole column range), so a light row is classed by w minus its number of nonzeros
// A group takes UNR rows at a time, so that the loads of one row do not wait for those of the row before (one at a time:
// 438 us for 4.2e6 rows of 16 nonzeros).  The CTAs behind `nblocks` do the binary analysis.  Six CTAs per SM are asked for: left
// to itself the compiler serialises the loads of long rows beside the analysis (524288 rows of a power-law matrix, whole
// plan: 859 us without the bound, 749 with it).
template <int G>
static __global__ void __launch_bounds__(BIN_THREADS, 6) row_work_kernel(PlanDev P, uint8_t* __restrict__ cls, int64_t block_max, uint32_t dense_range, bool diag, int64_t tile,
                                                                      int32_t* __restrict__ blockhist, int64_t nblocks,
                                                                      unsigned long long* __restrict__ work_total, unsigned long long* __restrict__ sparse_heavy, HeavyArrays heavy) {
    link();
    if (blockIdx.x >= nblocks) {
        heavy_analysis<G>(P, heavy);
        return;
    }
    constexpr int GROUPS = BIN_THREADS / G;
    constexpr int UNR = 4;
    constexpr int LONG_CTA = 1024;  // long rows of more nonzeros than this are walked by the whole CTA, not by a warp
    __shared__ int32_t hist[NCLASS];
    __shared__ unsigned long long cta_sum, s_work, s_sparse;
    __shared__ uint16_t s_long[BIN_MAX_TILE];
    __shared__ int s_nlong;
    if (threadIdx.x < NCLASS) hist[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        cta_sum = s_work = s_sparse = 0;
        s_nlong = 0;
    }
    __syncthreads();
    const int gl = threadIdx.x & (G - 1), group = threadIdx.x / G;
    const int64_t rows = P.r1 - P.r0;
    const int64_t t0 = (int64_t)blockIdx.x * tile, t1 = min(t0 + tile, rows);
    const bool sane = (*P.err & ERRW_BAD_CSR) == 0;  // a matrix that failed its checks has no descriptors
    unsigned long long mine = 0;    // work of the rows this thread owned
    const bool tril = P.mode == SPSYRK_TRIL;
    auto range_of = [&](int64_t r) { return tril ? (uint32_t)(P.r0 + (int32_t)r) + 1u : (uint32_t)P.m; };
    auto is_heavy = [&](int32_t deg, uint32_t w) { return deg > 32 || (diag ? w - deg : w) > 512u; };
    // (the lengths of a row's descriptors add up to less than 2^31)
    auto settle = [&](int64_t r, int32_t deg, uint32_t w, bool full) {  // one thread per row; full: it stores a column of every row of its range
        const bool dense = full && range_of(r) <= dense_range;
        P.work[r] = w;
        int c;
        const uint32_t wl = diag ? w - deg : w;  // items of a light row
        if (w == 0) c = 0;
        else if (!is_heavy(deg, w)) c = wl <= 32 ? 1 : wl <= 64 ? 2 : wl <= 128 ? 3 : wl <= 256 ? 4 : 5;
        else c = w <= block_max ? 6 : 7;
        cls[r] = (uint8_t)(c | (dense && c >= 6 ? ROW_DENSE : 0));
        atomicAdd(&hist[c], 1);
        if (c >= 6 && !dense) atomicAdd(&s_sparse, c == 6 ? 1ull : 1ull << 32);
        mine += (unsigned long long)w;
    };
    for (int64_t base = t0; base < t1; base += GROUPS * UNR) {
        int64_t p0[UNR];
        uint32_t w[UNR], full = 0;  // a bit per row
        int32_t deg[UNR];  // -1: left for the end
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
            const int64_t r = base + u * GROUPS + group;
            p0[u] = 0; deg[u] = 0;
            if (r < t1 && sane) {
                p0[u] = P.rowptr[P.r0 + r];
                deg[u] = (int32_t)(P.rowptr[P.r0 + r + 1] - p0[u]);
            }
        }
        const int32_t longest = max(max(deg[0], deg[1]), max(deg[2], deg[3]));
        static_assert(UNR == 4, "the longest of a group's rows");
        if (longest > LONG_STEPS * G) {
#pragma unroll
            for (int u = 0; u < UNR; ++u) {
                if (deg[u] > LONG_STEPS * G) {
                    if (gl == 0) s_long[atomicAdd(&s_nlong, 1)] = (uint16_t)(base + u * GROUPS + group - t0);
                    deg[u] = -1;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < UNR; ++u) w[u] = gl < deg[u] ? P.desc[p0[u] + gl].y : 0;
#pragma unroll
        for (int u = 0; u < UNR; ++u)
            for (int32_t q = gl + G; q < deg[u]; q += G) w[u] += P.desc[p0[u] + q].y;
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
#pragma unroll
            for (int o = G / 2; o > 0; o >>= 1) w[u] += __shfl_xor_sync(FULL_MASK, w[u], o);
        }
        // heavy rows: does one of the columns cover the row's range?  (a look at the largest first: light rows have little else to do here)
        if (__any_sync(FULL_MASK, longest > 32 || max(max(w[0], w[1]), max(w[2], w[3])) > 512u)) {
#pragma unroll
            for (int u = 0; u < UNR; ++u) {
                if (!is_heavy(deg[u], w[u])) continue;
                const uint32_t range = range_of(base + u * GROUPS + group);
                bool f = false;
                for (int32_t q = gl; q < deg[u]; q += G) f |= P.desc[p0[u] + q].y == range;
                full |= (uint32_t)f << u;
            }
#pragma unroll
            for (int o = G / 2; o > 0; o >>= 1) full |= __shfl_xor_sync(FULL_MASK, full, o);
        }
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
            const int64_t r = base + u * GROUPS + group;
            if (r < t1 && gl == 0 && deg[u] >= 0) settle(r, deg[u], w[u], (full >> u) & 1u);
        }
    }
    __syncthreads();
    const int nlong = s_nlong;
    // the long rows: a warp each, or (of more than LONG_CTA nonzeros) all warps together
    auto walk = [&](int64_t r, int64_t p0, int32_t deg, int32_t first, int32_t step, bool* full) {
        const uint32_t range = range_of(r);
        uint32_t w = 0;
        bool f = false;
        for (int32_t q = first; q < deg; q += step) {
            const uint32_t len = P.desc[p0 + q].y;
            w += len;
            f |= len == range;
        }
        *full = __any_sync(FULL_MASK, f);
        return warp_reduce_sum<uint32_t>(w);
    };
    for (int whole = 0; whole < 2 && nlong > 0; ++whole) {
        for (int i = whole ? 0 : threadIdx.x >> 5; i < nlong; i += whole ? 1 : BIN_THREADS / 32) {
            const int64_t r = t0 + s_long[i], p0 = P.rowptr[P.r0 + r];
            const int32_t deg = (int32_t)(P.rowptr[P.r0 + r + 1] - p0);
            if ((deg > LONG_CTA) != (whole == 1)) continue;
            bool full;
            const uint32_t w = walk(r, p0, deg, whole ? threadIdx.x : lane_id(), whole ? BIN_THREADS : 32, &full);
            if (!whole) {
                if (lane_id() == 0) settle(r, deg, w, full);
                continue;
            }
            if (lane_id() == 0) atomicAdd(&s_work, (unsigned long long)w | (unsigned long long)full << 32);
            __syncthreads();
            if (threadIdx.x == 0) {
                settle(r, deg, (uint32_t)s_work, (s_work >> 32) != 0);
                s_work = 0;
            }
            __syncthreads();
        }
    }
    const unsigned long long ws = warp_reduce_sum<unsigned long long>(mine);
    if (lane_id() == 0 && ws) atomicAdd(&cta_sum, ws);
    __syncthreads();
    if (threadIdx.x == 0 && cta_sum) atomicAdd(work_total, cta_sum);
    if (threadIdx.x == 0 && s_sparse) atomicAdd(sparse_heavy, s_sparse);
    if (threadIdx.x < NCLASS) blockhist[(int64_t)threadIdx.x * nblocks + blockIdx.x] = hist[threadIdx.x];
}

// prefix sums of the class-major counts, and where every class starts
struct BinStarts {
    int64_t* offsets;
    uint32_t nblocks;
    int64_t* class_start;  // NCLASS + 1
    __device__ __forceinline__ void operator()(int64_t i, int64_t ex) const {
        offsets[i] = ex;
        const uint32_t c = (uint32_t)i / nblocks;
        if (c * nblocks == (uint32_t)i) class_start[c] = ex;
    }
    __device__ __forceinline__ void total(int64_t t) const { class_start[NCLASS] = t; }
    __device__ __forceinline__ void gave_up() const {}
};

// Second half of the counting sort: the rows in class order (ascending inside a class), for each of them the header
// (row inside the plan's range, position of its first nonzero in A, number of nonzeros) and the words of the item map
// it needs (its items rounded up to eight; light rows only).  The counts of empty and of dense rows are settled here.
static __global__ void __launch_bounds__(BIN_THREADS) row_scatter_kernel(PlanDev P, const uint8_t* __restrict__ cls, int64_t tile,
                                                                         const int64_t* __restrict__ offsets, int64_t nblocks, bool diag,
                                                                         int32_t* __restrict__ perm, uint4* __restrict__ hdr,
                                                                         uint32_t* __restrict__ items8, int32_t* __restrict__ cnt,
                                                                         uint32_t* __restrict__ block_base, uint32_t blocks_per_row) {
    constexpr int NW = BIN_THREADS / 32;
    __shared__ int64_t running[NCLASS];
    __shared__ int32_t wcount[NW][NCLASS];
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    link(cls, offsets);
    if (threadIdx.x < NCLASS) running[threadIdx.x] = offsets[(int64_t)threadIdx.x * nblocks + blockIdx.x];
    const int64_t rows = P.r1 - P.r0;
    const int64_t t0 = (int64_t)blockIdx.x * tile, t1 = min(t0 + tile, rows);
    for (int64_t base = t0; base < t1; base += BIN_THREADS) {
        const int64_t r = base + threadIdx.x;
        int c = -1;
        int64_t p0 = 0, deg = 0, w = 0;
        if (r < t1) {
            c = cls[r] & (ROW_DENSE - 1);
            if (cls[r] & ROW_DENSE) {  // what the counting kernel would find
                const uint32_t range = P.mode == SPSYRK_TRIL ? (uint32_t)(P.r0 + r) + 1u : (uint32_t)P.m, blocks = (range + BASE_BLOCK - 1) / BASE_BLOCK;
                cnt[r] = (int32_t)range;
                for (uint32_t b = 0; b < blocks && blocks <= blocks_per_row; ++b) block_base[(uint64_t)(P.r0 + r) * blocks_per_row + b] = b * BASE_BLOCK;
            }
            p0 = P.rowptr[P.r0 + r];
            deg = P.rowptr[P.r0 + r + 1] - p0;
            w = P.work[r];
        }
        int myrank = 0;
#pragma unroll
        for (int k = 0; k < NCLASS; ++k) {
            const unsigned b = __ballot_sync(FULL_MASK, c == k);
            if (c == k) myrank = __popc(b & ((1u << lane) - 1u));
            if (lane == 0) wcount[warp][k] = __popc(b);
        }
        __syncthreads();
        if (c >= 0) {
            int64_t pos = running[c] + myrank;
            for (int v = 0; v < warp; ++v) pos += wcount[v][c];
            perm[pos] = (int32_t)r;
            hdr[pos] = make_uint4((uint32_t)r, (uint32_t)p0, (uint32_t)deg, 0u);
            items8[pos] = c >= 1 && c <= 5 ? ((uint32_t)(diag ? w - deg : w) + 7u) & ~7u : 0u;
            if (c == 0) cnt[r] = 0;
        }
        __syncthreads();
        if (threadIdx.x < NCLASS) {
            int t = 0;
            for (int v = 0; v < NW; ++v) t += wcount[v][threadIdx.x];
            running[threadIdx.x] += t;
        }
        __syncthreads();
    }
}

// What the host needs to know about a view of the plan, in the order in which it is written for the host
enum : int { PF_CLASS_START = 0, PF_MAP_ITEMS = NCLASS + 1, PF_WORK, PF_OTHER_THAN_ONE, PF_ERR, PF_SPARSE_HEAVY, PF_WORDS };
struct PlanFacts {
    const int64_t* class_start;
    const unsigned long long* work_total;
    const unsigned long long* sparse_heavy;  // rows of class 6, and in the upper half of class 7, that are not dense
    const uint32_t* facts;
    const uint32_t* err;
    int64_t* host;
    int64_t* gave_up;
    __device__ __forceinline__ void publish(int64_t map_items) const {
        int64_t w[PF_WORDS];  // all loads before the first store: one round trip, not thirteen
#pragma unroll
        for (int c = 0; c <= NCLASS; ++c) w[PF_CLASS_START + c] = class_start[c];
        w[PF_MAP_ITEMS] = map_items;
        w[PF_WORK] = (int64_t)*work_total;
        w[PF_OTHER_THAN_ONE] = (int64_t)facts[0];
        w[PF_ERR] = (int64_t)*err;
        w[PF_SPARSE_HEAVY] = (int64_t)*sparse_heavy;
#pragma unroll
        for (int c = 0; c < PF_WORDS; ++c) host[c] = w[c];
    }
};
// prefix sums of the map words; the last kernel before the plan's synchronisation
struct ItemStarts {
    int64_t* itemoff;
    int64_t n;
    PlanFacts facts;
    __device__ __forceinline__ void operator()(int64_t i, int64_t ex) const { itemoff[i] = ex; }
    __device__ __forceinline__ void total(int64_t t) const {
        itemoff[n] = t;
        facts.publish(t);
    }
    __device__ __forceinline__ void gave_up() const { *facts.gave_up = 1; }
};

}  // namespace spsyrk
