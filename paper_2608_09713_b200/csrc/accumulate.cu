// The accumulating form of the local product (Section III-A: C_ii = sum over s of SYRK(A_is);
// Algorithm 2 line 2: C_local += SYRK(A_recv)).
//
//   spsyrk_column_panel : A_s = A(:, [k0, k1)), the operand of one term of the sum;
//   spsyrk_accumulate   : Z = X + Y on sorted CSR rows, the "+=" itself.
//
// The sum works row by row: G lanes per row when rows are short, a warp (merge_windows) when they are longer, a CTA (merge_path)
// for the longest.  In the G-lane kernels, an entry's place in the merged row is
//     its own index + the number of entries of the other row below it - the matches below it,
// where a match is a column stored in both rows (it is emitted once, from X's side, with x + y).
// The other row's count is a binary search; the matches below come from a running count over the
// row, advanced G entries at a time with a vote inside the group.
#include <algorithm>

#include "common.cuh"

using namespace spsyrk;

namespace {

constexpr size_t ALIGN = 256;

int group_width(int64_t nnz, int64_t m) {
    const double avg = m > 0 ? (double)nnz / (double)m : 0.0;
    return avg <= 4 ? 4 : avg <= 8 ? 8 : avg <= 16 ? 16 : 32;
}

struct RowWs {
    uint32_t* cnt;  // m
    int64_t* partials;
    uint32_t* err;
};

size_t carve(RowWs* w, void* ws, int64_t m) {
    char* base = static_cast<char*>(ws);
    size_t off = 0;
    auto take = [&](size_t bytes) -> void* {
        off = (off + ALIGN - 1) / ALIGN * ALIGN;
        void* p = base ? base + off : nullptr;
        off += bytes;
        return p;
    };
    const int64_t items = std::max<int64_t>(m, 1);
    RowWs t;
    t.cnt = (uint32_t*)take(items * 4);
    t.partials = (int64_t*)take(scan_partials_count(items + 1) * 8);
    t.err = (uint32_t*)take(16);
    if (w) *w = t;
    return (off + ALIGN - 1) / ALIGN * ALIGN;
}

// lanes of the G-wide group this lane belongs to
template <int G>
__device__ __forceinline__ unsigned group_mask() {
    return (uint32_t)((1ull << G) - 1ull) << (lane_id() & ~(G - 1));
}

// ------------------------------------------------------------------------------ column panel
__global__ void __launch_bounds__(256) panel_count_kernel(int64_t m, const int64_t* __restrict__ rowptr,
                                                          const int32_t* __restrict__ colidx, int32_t k0, int32_t k1,
                                                          uint32_t* __restrict__ cnt) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= m) return;
    const int64_t p0 = rowptr[r];
    const uint32_t len = (uint32_t)(rowptr[r + 1] - p0);
    const uint32_t a = lower_bound_i32(colidx + p0, len, k0);
    const uint32_t b = a + lower_bound_i32(colidx + p0 + a, len - a, k1);
    cnt[r] = b - a;
}

template <typename V, int G>
__global__ void __launch_bounds__(256) panel_fill_kernel(int64_t m, const int64_t* __restrict__ rowptr,
                                                         const int32_t* __restrict__ colidx, const V* __restrict__ vals, int32_t k0,
                                                         const int64_t* __restrict__ p_rowptr, int32_t* __restrict__ p_colidx,
                                                         V* __restrict__ p_vals) {
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    const int gl = threadIdx.x & (G - 1);
    if (r >= m) return;
    const int64_t o0 = p_rowptr[r];
    const uint32_t n = (uint32_t)(p_rowptr[r + 1] - o0);
    if (n == 0) return;
    const int64_t p0 = rowptr[r];
    const int64_t src = p0 + lower_bound_i32(colidx + p0, (uint32_t)(rowptr[r + 1] - p0), k0);
    for (uint32_t t = gl; t < n; t += G) {
        p_colidx[o0 + t] = colidx[src + t];
        p_vals[o0 + t] = vals[src + t];
    }
}

// ------------------------------------------------------------------------------- sparse sum
// Walk row `self` G entries at a time; for each entry report (index, lower bound in `other`, match,
// matches before it) to `visit`.  Returns the number of matches of the row.  Loop bounds are
// uniform inside the group, so the votes see all of its lanes.
// CHECK: a row that does not ascend sets the error bit.
template <int G, bool CHECK, typename Visit>
__device__ __forceinline__ uint32_t walk_row(const int32_t* __restrict__ self, uint32_t ls, const int32_t* __restrict__ other,
                                             uint32_t lo_len, uint32_t* err, Visit visit) {
    const unsigned gmask = group_mask<G>();
    const int gl = lane_id() & (G - 1);
    const int gshift = lane_id() & ~(G - 1);
    uint32_t matched = 0;
    for (uint32_t t0 = 0; t0 < ls; t0 += G) {
        const uint32_t t = t0 + gl;
        bool match = false;
        uint32_t lb = 0;
        int32_t col = 0;
        if (t < ls) {
            col = self[t];
            if (CHECK && t > 0 && self[t - 1] >= col) atomicOr(err, ERRW_UNSORTED);
            lb = lower_bound_i32(other, lo_len, col);
            match = lb < lo_len && other[lb] == col;
        }
        const unsigned votes = (__ballot_sync(gmask, match) >> gshift) & (uint32_t)((1ull << G) - 1ull);
        if (t < ls) visit(t, lb, match, matched + __popc(votes & ((1u << gl) - 1u)), col);
        matched += __popc(votes);
    }
    return matched;
}

// Rows of more than a few entries.  A warp walks the two rows in windows of 32 ids each.  Everything up to the smaller of the
// two windows' last ids is known completely, so those entries are merged at once: an entry's place is the output position
// reached so far + its index in its own window + the entries of the other window below it (a search over the window in shared
// memory) - the matches below it (votes).  All global accesses are coalesced and a step brings in up to 64 ids with one
// round of loads.  Bound by instruction issue (rows of 131 entries: 86 % of the slots in the size step, 77 in the fill; load/store pipe 54
// and 50 %, DRAM 16 and 32).  Sums of 6e7 entries, single precision, both steps, rows of
// 33, 131, 513 and 2000 entries of both inputs: 1023, 591, 518 and 554 us.  (The merge path by a warp, eight entries a lane: 2700, 974, 683
// and 658, because a row pays for a whole tile.)
// FILL: the merged row goes to zc, zv (at most lz entries: always enough with the row pointer of the size step; keeps a
// stale one from writing outside); otherwise the rows are checked.  Returns the number of entries of the merged row.
constexpr int MERGE_WARPS = 8;
struct WindowSmem {
    int32_t x[32], y[32];
};
template <typename V, bool FILL>
__device__ __forceinline__ uint32_t merge_windows(const int32_t* __restrict__ xc, const V* __restrict__ xv, uint32_t lx, const int32_t* __restrict__ yc,
                                                  const V* __restrict__ yv, uint32_t ly, int32_t* __restrict__ zc, V* __restrict__ zv, uint32_t lz,
                                                  WindowSmem& S, uint32_t* err) {
    constexpr int32_t INF = 0x7fffffff;  // above every column id
    const uint32_t lane = lane_id();
    const unsigned lt = (1u << lane) - 1u;
    // number of ids below key among the first n (ascending) ids of a window
    auto below = [&](const int32_t* win, uint32_t n, int32_t key) -> uint32_t {
        uint32_t pos = 0;
#pragma unroll
        for (uint32_t step = 16; step > 0; step >>= 1)
            if (pos + step <= n && win[pos + step - 1] < key) pos += step;
        if (pos < n && win[pos] < key) ++pos;  // a full window with every probed id below: the last one
        return pos;
    };
    uint32_t ix = 0, iy = 0, out = 0;
    int32_t lastx = -1, lasty = -1;
    while (ix < lx || iy < ly) {  // the same for all lanes
        const uint32_t nx = min(32u, lx - ix), ny = min(32u, ly - iy);
        const int32_t xa = lane < nx ? xc[ix + lane] : INF, ya = lane < ny ? yc[iy + lane] : INF;
        S.x[lane] = xa;
        S.y[lane] = ya;
        __syncwarp();
        const int32_t bound = min(ix + 32 < lx ? S.x[31] : INF, iy + 32 < ly ? S.y[31] : INF);
        if (!FILL) {  // rows must be strictly ascending (also across windows)
            const int32_t px = lane == 0 ? lastx : S.x[lane - 1], py = lane == 0 ? lasty : S.y[lane - 1];
            if ((lane < nx && px >= xa) || (lane < ny && py >= ya)) atomicOr(err, ERRW_UNSORTED);
        }
        const bool takex = lane < nx && xa <= bound, takey = lane < ny && ya <= bound;
        const uint32_t ry = takex ? below(S.y, ny, xa) : 0u;
        const bool mx = takex && ry < ny && S.y[ry] == xa;
        const unsigned vmx = __ballot_sync(FULL_MASK, mx);
        const uint32_t cx = __popc(__ballot_sync(FULL_MASK, takex)), cy = __popc(__ballot_sync(FULL_MASK, takey));
        if (FILL) {
            const uint32_t rx = takey ? below(S.x, nx, ya) : 0u;
            const bool my = takey && rx < nx && S.x[rx] == ya;
            const unsigned vmy = __ballot_sync(FULL_MASK, my);
            const uint32_t px = out + lane + ry - __popc(vmx & lt), py = out + lane + rx - __popc(vmy & lt);
            if (takex && px < lz) {
                zc[px] = xa;
                const V v = xv[ix + lane];
                zv[px] = mx ? (V)(v + yv[iy + ry]) : v;
            }
            if (takey && !my && py < lz) {
                zc[py] = ya;
                zv[py] = yv[iy + lane];
            }
        } else {
            if (cx > 0) lastx = S.x[cx - 1];
            if (cy > 0) lasty = S.y[cy - 1];
        }
        out += cx + cy - __popc(vmx);
        ix += cx;
        iy += cy;
        __syncwarp();  // the windows are rewritten
    }
    return out;
}

// The longest rows: a CTA merges a row MERGE_TILE entries at a time along the merge path (Odeh, Green, Mwassi, Shmueli &
// Birk, "Merge Path - Parallel Merging Made Simple", 2012).  A tile holds the next ids of both rows in shared memory; a thread
// finds by a binary search where its MERGE_ITEMS entries of the merged order begin in either row and merges them one
// after the other, x before y where both store a column; such a pair is emitted once, with x + y, by the thread that has its
// x.  The emitted entries are put in order in the shared memory of the ids and written out by consecutive threads.
// Bound by the steps of a tile, one behind the other (size step: issue slots and load/store pipe 68 % each; fill 56 and 55, waits for the
// values and at the barriers).  Rows of 10 000 entries: 630 us for 6e7; the windows of a warp take less time in all for
// shorter rows, but a row's 32 entries after 32 entries keep one warp long after the others.
constexpr int MERGE_ITEMS = 8;
constexpr int MERGE_LONG_THREADS = 256;
constexpr uint32_t MERGE_TILE = MERGE_LONG_THREADS * MERGE_ITEMS;
struct MergeSmem {
    uint32_t x[MERGE_TILE + 1], y[MERGE_TILE + 1];  // the ids of a tile of either row, one more behind them as a sentinel
    uint32_t scratch[33];
    uint32_t end;  // entries of x and, in the upper half, of y in the tile
};

// As merge_windows, by all threads of the CTA.  Rows that are not strictly ascending set the error bit in the size step; their
// merge is wrong but stays inside the rows.
template <typename V, bool FILL>
__device__ __forceinline__ uint32_t merge_path(const int32_t* __restrict__ xc, const V* __restrict__ xv, uint32_t lx, const int32_t* __restrict__ yc,
                                               const V* __restrict__ yv, uint32_t ly, int32_t* __restrict__ zc, V* __restrict__ zv, uint32_t lz,
                                               MergeSmem& S, uint32_t* err) {
    constexpr int T = MERGE_LONG_THREADS;
    constexpr uint32_t NONE = 0xffffu, INF = 0xffffffffu;  // (a negative id fails the check and is merged as 0)
    static_assert(MERGE_TILE < NONE, "positions inside a tile are 16 bits");
    const int t = threadIdx.x;
    uint32_t ix = 0, iy = 0, out = 0;
    // A warp brings in consecutive ids, 32 per step, and hands each to the next lane for the check of the order.
    auto load = [&](const int32_t* __restrict__ ids, uint32_t first, uint32_t n, uint32_t* window) {
        const uint32_t base = (uint32_t)(t & ~31) * MERGE_ITEMS, lane = t & 31;
        if (base >= n) return;
        int32_t before = -1;
        if (!FILL && lane == 0 && first + base > 0) before = ids[first + base - 1];
        bool bad = false;
        int32_t id[MERGE_ITEMS];
#pragma unroll
        for (int u = 0; u < MERGE_ITEMS; ++u) id[u] = base + u * 32 + lane < n ? ids[first + base + u * 32 + lane] : 0x7fffffff;
#pragma unroll
        for (int u = 0; u < MERGE_ITEMS; ++u) {
            const uint32_t e = base + u * 32 + lane;
            if (e < n) window[e] = (uint32_t)max(id[u], 0);
            if (!FILL) {
                int32_t left = __shfl_up_sync(FULL_MASK, id[u], 1);
                if (lane == 0) left = before;
                bad |= e < n && left >= id[u];
                before = __shfl_sync(FULL_MASK, id[u], 31);
            }
        }
        if (!FILL && bad) atomicOr(err, ERRW_UNSORTED);
    };
    while (ix < lx || iy < ly) {  // the same for all threads
        const uint32_t nx = min(MERGE_TILE, lx - ix), ny = min(MERGE_TILE, ly - iy);
        load(xc, ix, nx, S.x);
        load(yc, iy, ny, S.y);
        if (t == 0) S.x[nx] = S.y[ny] = INF;
        __syncthreads();
        const uint32_t total = min(MERGE_TILE, nx + ny);
        const uint32_t d = min((uint32_t)t * MERGE_ITEMS, total), d_end = min(d + MERGE_ITEMS, total);
        uint32_t xi = d > ny ? d - ny : 0u, hi = min(d, nx);  // entries of x among the first d of the merged order
        while (xi < hi) {
            const uint32_t mid = (xi + hi) >> 1;
            if (S.x[mid] <= S.y[d - 1 - mid]) xi = mid + 1;
            else hi = mid;
        }
        uint32_t yi = d - xi;
        uint32_t a = S.x[xi], b = S.y[yi];
        if (xi > 0 && S.x[xi - 1] == b) b = S.y[++yi];  // the pair went with its x (never the sentinel: ids are at most 2^31 - 1)
        uint32_t col[MERGE_ITEMS], src[MERGE_ITEMS];  // src: position in x's window | position in y's << 16
        uint32_t n = 0;
#pragma unroll
        for (int i = 0; i < MERGE_ITEMS; ++i) {
            const bool go = xi + yi < d_end;
            const bool tx = a <= b, ty = b <= a;
            if (FILL) {
                col[i] = tx ? a : b;
                src[i] = (tx ? xi : NONE) | (ty ? yi : NONE) << 16;
            }
            if (go) {
                ++n;
                if (tx) a = S.x[min(++xi, nx)];
                if (ty) b = S.y[min(++yi, ny)];
            }
        }
        if (t == T - 1) S.end = xi | yi << 16;
        uint32_t sum;
        const uint32_t rank = block_exclusive_scan<uint32_t, T>(n, S.scratch, &sum);  // (behind its barriers the windows are read)
        const uint32_t end = S.end;
        if (FILL) {
#pragma unroll
            for (int i = 0; i < MERGE_ITEMS; ++i) {
                if (i < n) {
                    S.x[rank + i] = col[i];
                    S.y[rank + i] = src[i];
                }
            }
            __syncthreads();
            const uint32_t n_out = out < lz ? min(sum, lz - out) : 0u;
            for (uint32_t i = t; i < n_out; i += T) {
                const uint32_t s = S.y[i], sx = s & NONE, sy = s >> 16;
                V v{}, w{};
                if (sx != NONE) v = xv[ix + sx];
                if (sy != NONE) w = yv[iy + sy];
                zc[out + i] = (int32_t)S.x[i];
                zv[out + i] = sx == NONE ? w : sy == NONE ? v : (V)(v + w);
            }
        }
        __syncthreads();  // the windows are rewritten
        out += sum;
        ix += end & 0xffffu;
        iy += end >> 16;
    }
    return out;
}

// the operands of the sum and, when it is filled, the result
template <typename V>
struct SumArgs {
    int64_t m;
    const int64_t* x_rowptr;
    const int32_t* x_colidx;
    const V* x_vals;
    const int64_t* y_rowptr;
    const int32_t* y_colidx;
    const V* y_vals;
    int64_t longest;           // rows of more entries (of both inputs together) are merged by a CTA each
    uint32_t* cnt;             // size step
    const int64_t* z_rowptr;   // fill step
    int32_t* z_colidx;
    V* z_vals;
    uint32_t* err;             // size step
};

// row r by the warp (merge_windows) or by the CTA (merge_path), `leader` in one thread of it
template <typename V, bool FILL, typename Smem>
__device__ __forceinline__ void sum_row(const SumArgs<V>& A, int64_t r, int64_t x0, uint32_t lx, int64_t y0, uint32_t ly, Smem& S, bool leader) {
    const int64_t z0 = FILL ? A.z_rowptr[r] : 0;
    const uint32_t lz = FILL ? (uint32_t)(A.z_rowptr[r + 1] - z0) : 0u;
    const int32_t *xc = A.x_colidx + x0, *yc = A.y_colidx + y0;
    const V *xv = FILL ? A.x_vals + x0 : nullptr, *yv = FILL ? A.y_vals + y0 : nullptr;
    int32_t* zc = FILL ? A.z_colidx + z0 : nullptr;
    V* zv = FILL ? A.z_vals + z0 : nullptr;
    uint32_t n;
    if constexpr (std::is_same<Smem, WindowSmem>::value) n = merge_windows<V, FILL>(xc, xv, lx, yc, yv, ly, zc, zv, lz, S, A.err);
    else n = merge_path<V, FILL>(xc, xv, lx, yc, yv, ly, zc, zv, lz, S, A.err);
    if (!FILL && leader) A.cnt[r] = n;
}

// One warp per row.  A CTA has `share` consecutive rows, which its warps draw one after the other.
template <typename V, bool FILL>
__global__ void __launch_bounds__(MERGE_WARPS * 32) add_merge_kernel(SumArgs<V> A, int share) {
    __shared__ WindowSmem smem[MERGE_WARPS];
    __shared__ int s_next;
    const int warp = threadIdx.x >> 5, lane = lane_id();
    chain_begin();
    if (threadIdx.x == 0) s_next = 0;
    __syncthreads();
    const int64_t first = (int64_t)blockIdx.x * share;
    const int n = (int)min((int64_t)share, A.m - first);
    for (;;) {
        int i = 0;
        if (lane == 0) i = atomicAdd(&s_next, 1);
        i = __shfl_sync(FULL_MASK, i, 0);
        if (i >= n) break;
        const int64_t r = first + i;
        const int64_t x0 = A.x_rowptr[r], y0 = A.y_rowptr[r];
        const int64_t lx = A.x_rowptr[r + 1] - x0, ly = A.y_rowptr[r + 1] - y0;
        if (lx < 0 || ly < 0 || lx + ly > 0x7fffffffLL) {
            if (!FILL && lane == 0) {
                atomicOr(A.err, ERRW_BAD_ROWPTR);
                A.cnt[r] = 0;
            }
        } else if (lx + ly <= A.longest) {
            sum_row<V, FILL>(A, r, x0, (uint32_t)lx, y0, (uint32_t)ly, smem[warp], lane == 0);
        }
    }
    chain_end();
}

// The longer rows, a CTA each.  The rows are dealt to the CTAs in units of 1 << unit_bits, a unit of every
// gridDim.x, so that long rows which stand together go to different CTAs; a CTA has at most one unit per thread.  A unit of few
// entries has no such row: of it only the ends are looked at.
template <typename V, bool FILL>
__global__ void __launch_bounds__(MERGE_LONG_THREADS, 6) add_long_kernel(SumArgs<V> A, int unit_bits) {
    __shared__ MergeSmem smem;
    __shared__ int64_t s_unit[MERGE_LONG_THREADS];  // first rows of the units that are looked at row by row
    __shared__ int64_t s_row[MERGE_LONG_THREADS];
    __shared__ int s_units, s_rows;
    const int t = threadIdx.x;
    chain_begin();
    auto entries = [&](int64_t a, int64_t b) { return A.x_rowptr[b] - A.x_rowptr[a] + A.y_rowptr[b] - A.y_rowptr[a]; };
    if (t == 0) s_units = 0;
    __syncthreads();
    const int64_t u0 = ((int64_t)blockIdx.x + (int64_t)t * gridDim.x) << unit_bits;
    if (u0 < A.m && entries(u0, min(u0 + (1 << unit_bits), A.m)) > A.longest) s_unit[atomicAdd(&s_units, 1)] = u0;
    __syncthreads();
    const int n = s_units << unit_bits;
    for (int base = 0; base < n; base += MERGE_LONG_THREADS) {
        if (t == 0) s_rows = 0;
        __syncthreads();
        if (base + t < n) {
            const int64_t r = s_unit[(base + t) >> unit_bits] + ((base + t) & ((1 << unit_bits) - 1));
            if (r < A.m) {
                const int64_t lx = A.x_rowptr[r + 1] - A.x_rowptr[r], ly = A.y_rowptr[r + 1] - A.y_rowptr[r];
                if (lx >= 0 && ly >= 0 && lx + ly > A.longest && lx + ly <= 0x7fffffffLL) s_row[atomicAdd(&s_rows, 1)] = r;
            }
        }
        __syncthreads();
        const int rows = s_rows;
        for (int i = 0; i < rows; ++i) {
            const int64_t r = s_row[i], x0 = A.x_rowptr[r], y0 = A.y_rowptr[r];
            sum_row<V, FILL>(A, r, x0, (uint32_t)(A.x_rowptr[r + 1] - x0), y0, (uint32_t)(A.y_rowptr[r + 1] - y0), smem, t == 0);
        }
        __syncthreads();
    }
    chain_end();
}

// G lanes per row, where rows are short on average
template <int G>
__global__ void __launch_bounds__(256) add_count_kernel(SumArgs<uint32_t> A) {
    chain_begin();
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    const int gl = threadIdx.x & (G - 1);
    if (r >= A.m) return;  // whole groups leave together
    const int64_t x0 = A.x_rowptr[r], y0 = A.y_rowptr[r];
    const int64_t lx64 = A.x_rowptr[r + 1] - x0, ly64 = A.y_rowptr[r + 1] - y0;
    if (lx64 < 0 || ly64 < 0 || lx64 + ly64 > 0x7fffffffLL) {
        if (gl == 0) { atomicOr(A.err, ERRW_BAD_ROWPTR); A.cnt[r] = 0; }
        return;
    }
    if (lx64 + ly64 > A.longest) return;
    const uint32_t lx = (uint32_t)lx64, ly = (uint32_t)ly64;
    const int32_t *xc = A.x_colidx + x0, *yc = A.y_colidx + y0;
    // the sortedness of X is checked here, that of Y inside the walk
    for (uint32_t t = 1 + gl; t < lx; t += G)
        if (xc[t - 1] >= xc[t]) atomicOr(A.err, ERRW_UNSORTED);
    const uint32_t matched = walk_row<G, true>(yc, ly, xc, lx, A.err, [](uint32_t, uint32_t, bool, uint32_t, int32_t) {});
    if (gl == 0) A.cnt[r] = lx + ly - matched;
}

template <typename V, int G>
__global__ void __launch_bounds__(256) add_fill_kernel(SumArgs<V> A) {
    chain_begin();
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    if (r >= A.m) return;
    const int64_t x0 = A.x_rowptr[r], y0 = A.y_rowptr[r], z0 = A.z_rowptr[r];
    const int64_t lx64 = A.x_rowptr[r + 1] - x0, ly64 = A.y_rowptr[r + 1] - y0;
    if (lx64 + ly64 > A.longest) return;
    const uint32_t lx = (uint32_t)lx64, ly = (uint32_t)ly64;
    const uint32_t lz = (uint32_t)(A.z_rowptr[r + 1] - z0);
    const int32_t *xc = A.x_colidx + x0, *yc = A.y_colidx + y0;
    // entries of X: all are emitted, matched ones with the sum
    walk_row<G, false>(xc, lx, yc, ly, nullptr, [&](uint32_t t, uint32_t lb, bool match, uint32_t before, int32_t col) {
        const uint32_t pos = t + lb - before;
        if (pos < lz) {  // always true for the row pointer of the size step; keeps a stale one from writing outside
            A.z_colidx[z0 + pos] = col;
            const V xv = A.x_vals[x0 + t];
            A.z_vals[z0 + pos] = match ? (V)(xv + A.y_vals[y0 + lb]) : xv;
        }
    });
    // entries of Y: only the ones X does not store
    walk_row<G, false>(yc, ly, xc, lx, nullptr, [&](uint32_t t, uint32_t lb, bool match, uint32_t before, int32_t col) {
        const uint32_t pos = t + lb - before;
        if (!match && pos < lz) {
            A.z_colidx[z0 + pos] = col;
            A.z_vals[z0 + pos] = A.y_vals[y0 + t];
        }
    });
}

// row pointers from the per-row counts; the total and the error word travel to the host (synchronises)
spsyrk_status_t scan_and_total(const RowWs& w, int64_t m, int64_t* d_rowptr_out, int64_t* total, cudaStream_t st) {
    ScopedHostBlock h;
    SPSYRK_CUDA_TRY(h.acquire());
    if (m == 0) {
        SPSYRK_CUDA_TRY(cudaMemsetAsync(d_rowptr_out, 0, sizeof(int64_t), st));
        h.host[0] = h.host[1] = 0;
    } else if (scan_launch(ScanArray<uint32_t>{w.cnt}, m, ScanIntoHost{d_rowptr_out, m, w.err, h.dev}, w.partials, w.err, st) != cudaSuccess) {
        cudaStreamSynchronize(st);  // the error may be an earlier launch's: the scan is under way then and writes into the host block
        return SPSYRK_ERR_CUDA;
    }
    SPSYRK_CUDA_TRY(wait_for(st));
    if (const uint32_t e = h.errors(h.host[1])) return status_of(e);
    *total = h.host[0];
    return SPSYRK_OK;
}

template <typename V>
void launch_panel_fill(int g, int64_t m, const int64_t* rowptr, const int32_t* colidx, const void* vals, int32_t k0,
                       const int64_t* p_rowptr, int32_t* p_colidx, void* p_vals, cudaStream_t st) {
#define FILL(G)                                                                                                            \
    panel_fill_kernel<V, G><<<(unsigned)((m * G + 255) / 256), 256, 0, st>>>(m, rowptr, colidx, static_cast<const V*>(vals), k0, \
                                                                             p_rowptr, p_colidx, static_cast<V*>(p_vals))
    switch (g) {
        case 4: FILL(4); break;
        case 8: FILL(8); break;
        case 16: FILL(16); break;
        default: FILL(32); break;
    }
#undef FILL
    note_launches(1);
}

// Entries of the longest row that a warp merges: about twice its share of all, so that no warp is left with one row when the others are
// done, not fewer than half a tile of a CTA and at most two.  Power-law panels of 2^13, 2^15 and 2^16 rows, 4.5e6, 3.6e7 and 1.0e8 entries: 160, 609
// and 1189 us; with 4096 for all of them the first takes 319, with 1024 the last 1519; rows of 2000 entries 554 us, with 1024 786.
int64_t longest_of_a_warp(int64_t entries) { return std::min<int64_t>(std::max<int64_t>(entries / (148 * 24), 1024), 4096); }

// Kernels of one step of the sum, the second beside the first: lanes of a warp share a row up to a mean of 16 entries, warps take
// the rows beyond.  The line lies where rows that differ much in length turn: power-law panels of 19 entries per row 224 us by 16 lanes, 147
// by warps.  Equal rows would turn at 30 (21 entries: 1173 us by 16 lanes, 1591 by warps; 29: 968 to 1189; 33: 1023 either way).
template <typename V, bool FILL>
spsyrk_status_t launch_sum(int g, const SumArgs<V>& A, cudaStream_t st) {
    Chain ch{st, true};
    const auto lanes = [&](void (*kern)(SumArgs<V>), int width) { return ch.launch(true, kern, (unsigned)((A.m * width + 255) / 256), 256, 0, A); };
    if (g <= 16) {
        if constexpr (FILL) SPSYRK_CUDA_TRY(g == 4 ? lanes(add_fill_kernel<V, 4>, 4) : g == 8 ? lanes(add_fill_kernel<V, 8>, 8) : lanes(add_fill_kernel<V, 16>, 16));
        else SPSYRK_CUDA_TRY(g == 4 ? lanes(add_count_kernel<4>, 4) : g == 8 ? lanes(add_count_kernel<8>, 8) : lanes(add_count_kernel<16>, 16));
    }
    const int unit_bits = A.m <= 1 << 16 ? 0 : A.m <= 1 << 20 ? 2 : 5;
    const int64_t units = (A.m + (1 << unit_bits) - 1) >> unit_bits;
    const int64_t ctas = std::max<int64_t>(std::min<int64_t>(units, 148 * 12), (units + MERGE_LONG_THREADS - 1) / MERGE_LONG_THREADS);
    SPSYRK_CUDA_TRY(ch.launch(true, add_long_kernel<V, FILL>, (unsigned)ctas, MERGE_LONG_THREADS, 0, A, unit_bits));
    if (g > 16) {
        // the other rows beside the long ones; rows per CTA: one for each warp as long as all of them are at most 16 times what the
        // GPU holds, up to 32 then
        const int64_t share = std::min<int64_t>(std::max<int64_t>(A.m / (148 * 32 * 16), 1), 32) * MERGE_WARPS;
        SPSYRK_CUDA_TRY(ch.launch(true, add_merge_kernel<V, FILL>, (unsigned)((A.m + share - 1) / share), MERGE_WARPS * 32, 0, A, (int)share));
    }
    return SPSYRK_OK;
}

bool dtype_ok(spsyrk_dtype_t t) { return t == SPSYRK_F64 || t == SPSYRK_F32 || t == SPSYRK_I32; }

}  // namespace

extern "C" spsyrk_status_t spsyrk_column_panel(int64_t m, int64_t nnz, spsyrk_dtype_t dtype, const int64_t* d_rowptr,
                                               const int32_t* d_colidx, const void* d_vals, int64_t k0, int64_t k1,
                                               int64_t* d_p_rowptr, int32_t* d_p_colidx, void* d_p_vals, int64_t* nnz_out,
                                               void* d_workspace, size_t* workspace_bytes, void* cuda_stream) {
    if (!workspace_bytes || m < 0 || nnz < 0 || !dtype_ok(dtype)) return SPSYRK_ERR_INVALID_ARG;
    if (k0 < 0 || k1 < k0) return SPSYRK_ERR_INVALID_ARG;
    const size_t need = carve(nullptr, nullptr, m);
    if (!d_workspace) {
        *workspace_bytes = need;
        return SPSYRK_OK;
    }
    if (*workspace_bytes < need) return SPSYRK_ERR_WORKSPACE;
    if (reinterpret_cast<uintptr_t>(d_workspace) % ALIGN) return SPSYRK_ERR_INVALID_ARG;
    if (!d_rowptr || !d_p_rowptr || (nnz > 0 && !d_colidx)) return SPSYRK_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    RowWs w;
    carve(&w, d_workspace, m);
    // column ids are below 2^31, so larger bounds mean "to the end"
    const int32_t c0 = (int32_t)std::min<int64_t>(k0, 0x7fffffffLL), c1 = (int32_t)std::min<int64_t>(k1, 0x7fffffffLL);
    if (!d_p_colidx) {  // step 2: sizes
        if (!nnz_out) return SPSYRK_ERR_INVALID_ARG;
        SPSYRK_CUDA_TRY(cudaMemsetAsync(w.err, 0, 4, st));
        if (m > 0) {
            panel_count_kernel<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(m, d_rowptr, d_colidx, c0, c1, w.cnt);
            note_launches(1);
        }
        return scan_and_total(w, m, d_p_rowptr, nnz_out, st);
    }
    if (!d_p_vals || (nnz > 0 && !d_vals)) return SPSYRK_ERR_INVALID_ARG;
    if (m == 0) return SPSYRK_OK;
    const int g = group_width(nnz, m);
    if (dtype == SPSYRK_F64) launch_panel_fill<uint64_t>(g, m, d_rowptr, d_colidx, d_vals, c0, d_p_rowptr, d_p_colidx, d_p_vals, st);
    else launch_panel_fill<uint32_t>(g, m, d_rowptr, d_colidx, d_vals, c0, d_p_rowptr, d_p_colidx, d_p_vals, st);
    SPSYRK_CUDA_TRY(cudaGetLastError());
    return SPSYRK_OK;
}

extern "C" spsyrk_status_t spsyrk_accumulate(int64_t m, spsyrk_dtype_t dtype, int64_t nnz_x, const int64_t* d_x_rowptr,
                                             const int32_t* d_x_colidx, const void* d_x_vals, int64_t nnz_y,
                                             const int64_t* d_y_rowptr, const int32_t* d_y_colidx, const void* d_y_vals,
                                             int64_t* d_z_rowptr, int32_t* d_z_colidx, void* d_z_vals, int64_t* nnz_out,
                                             void* d_workspace, size_t* workspace_bytes, void* cuda_stream) {
    if (!workspace_bytes || m < 0 || nnz_x < 0 || nnz_y < 0 || !dtype_ok(dtype)) return SPSYRK_ERR_INVALID_ARG;
    const size_t need = carve(nullptr, nullptr, m);
    if (!d_workspace) {
        *workspace_bytes = need;
        return SPSYRK_OK;
    }
    if (*workspace_bytes < need) return SPSYRK_ERR_WORKSPACE;
    if (reinterpret_cast<uintptr_t>(d_workspace) % ALIGN) return SPSYRK_ERR_INVALID_ARG;
    if (!d_x_rowptr || !d_y_rowptr || !d_z_rowptr || (nnz_x > 0 && !d_x_colidx) || (nnz_y > 0 && !d_y_colidx))
        return SPSYRK_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    RowWs w;
    carve(&w, d_workspace, m);
    const int g = group_width(nnz_x + nnz_y, m);
    const int64_t longest = longest_of_a_warp(nnz_x + nnz_y);
    if (!d_z_colidx) {  // step 2: sizes
        if (!nnz_out) return SPSYRK_ERR_INVALID_ARG;
        SPSYRK_CUDA_TRY(cudaMemsetAsync(w.err, 0, 4, st));
        if (m > 0) {
            const spsyrk_status_t s = launch_sum<uint32_t, false>(
                g, {m, d_x_rowptr, d_x_colidx, nullptr, d_y_rowptr, d_y_colidx, nullptr, longest, w.cnt, nullptr, nullptr, nullptr, w.err}, st);
            if (s != SPSYRK_OK) return s;
        }
        return scan_and_total(w, m, d_z_rowptr, nnz_out, st);
    }
    if (!d_z_vals || (nnz_x > 0 && !d_x_vals) || (nnz_y > 0 && !d_y_vals)) return SPSYRK_ERR_INVALID_ARG;
    if (m == 0) return SPSYRK_OK;
    const auto fill = [&](auto* z_vals) {
        using V = std::remove_pointer_t<decltype(z_vals)>;
        return launch_sum<V, true>(g, {m, d_x_rowptr, d_x_colidx, static_cast<const V*>(d_x_vals), d_y_rowptr, d_y_colidx, static_cast<const V*>(d_y_vals),
                                       longest, nullptr, d_z_rowptr, d_z_colidx, z_vals, nullptr}, st);
    };
    switch (dtype) {
        case SPSYRK_F64: return fill(static_cast<double*>(d_z_vals));
        case SPSYRK_F32: return fill(static_cast<float*>(d_z_vals));
        // unsigned addition wraps modulo 2^32, which is also what two's-complement int32 addition means
        default: return fill(static_cast<uint32_t*>(d_z_vals));
    }
}
