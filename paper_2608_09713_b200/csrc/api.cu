// C ABI: spsyrk_plan / spsyrk_plan_set_rows / spsyrk_symbolic / spsyrk_numeric and helpers.
// Host-side orchestration only; every step of the path runs in the kernels of the .cuh files.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "rows_cta.cuh"
#include "rows_heavy.cuh"
#include "rows_warp.cuh"

#include <atomic>

using namespace spsyrk;

namespace spsyrk {
static std::atomic<long long> g_launches{0};
void note_launches(int n) { g_launches.fetch_add(n, std::memory_order_relaxed); }

// Allocating pinned memory takes a millisecond or more, so blocks given back are kept for the next user, up to
// HOST_POOL_MAX of 1280 bytes each.  Blocks are portable: any device's kernels may write them.
static std::mutex g_host_mutex;
static std::vector<int64_t*> g_host_pool;
constexpr size_t HOST_POOL_MAX = 64;
cudaError_t HostBlock::acquire() {
    {
        std::lock_guard<std::mutex> lock(g_host_mutex);
        if (!g_host_pool.empty()) {
            host = g_host_pool.back();
            g_host_pool.pop_back();
        }
    }
    if (!host) {
        const cudaError_t e = cudaHostAlloc(reinterpret_cast<void**>(&host), HOST_WORDS * sizeof(int64_t), cudaHostAllocMapped | cudaHostAllocPortable);
        if (e != cudaSuccess) { host = nullptr; return e; }
    }
    host[HOST_GAVE_UP] = 0;
    return cudaHostGetDevicePointer(reinterpret_cast<void**>(&dev), host, 0);
}
void HostBlock::release() {
    if (!host) return;
    {
        std::lock_guard<std::mutex> lock(g_host_mutex);
        if (g_host_pool.size() < HOST_POOL_MAX) {
            g_host_pool.push_back(host);
            host = nullptr;
        }
    }
    if (host) cudaFreeHost(host);
    host = dev = nullptr;
}
}  // namespace spsyrk

namespace {

constexpr size_t ALIGN = 256;
constexpr int64_t BLOCK_CLASS_MAX_WORK = 32768;  // class 6 (block class) up to here, class 7 above
constexpr uint32_t ROW_CHUNK_BITS_MAX_NUMERIC = 1u << 18;
constexpr uint32_t ROW_CHUNK_BITS_MAX_SYMBOLIC = 1u << 20;
constexpr size_t LARGE_SMEM_BUDGET = 200 * 1024;
constexpr int64_t MAX_PARTS = 65536;

// Shared-memory shapes of the heavy-row kernels (see heavy_shapes)
constexpr int RANK_SMALL_THREADS = 256, RANK_MID_THREADS = 512, RANK_BIG_THREADS = 1024, DENSE8_THREADS = 512, DENSE8_SHORT_THREADS = 256;
template <int T, int C> struct RankShape { static constexpr int THREADS = T, CTAS = C; };
constexpr size_t SMEM_PER_CTA = 226 * 1024, SMEM_PER_SM = 228 * 1024, SMEM_OF_A_CTA = 1024;  // the last: taken by every CTA that is resident
// slots of the largest rank kernel, one CTA per SM: doubles 21504 beside a bitmap of 2^18 columns, 23552 beside 2^17, 24576 beside 2^16
template <typename V>
uint32_t rank_slots_big(uint32_t columns) {
    using Acc = typename AccOf<V>::type;
    return std::min(columns, (uint32_t)((SMEM_PER_CTA - RankSmem<V, RANK_BIG_THREADS>::bytes(columns, 0)) / sizeof(Acc)) / 1024 * 1024);
}

size_t dtype_size(spsyrk_dtype_t t) { return t == SPSYRK_F64 ? 8 : 4; }

struct Carver {
    char* base;
    size_t off = 0;
    explicit Carver(void* b) : base(static_cast<char*>(b)) {}
    template <typename T>
    T* take(size_t count) {
        off = (off + ALIGN - 1) / ALIGN * ALIGN;
        T* p = base ? reinterpret_cast<T*>(base + off) : nullptr;
        off += count * sizeof(T);
        return p;
    }
};

uint32_t pow2_at_least(uint64_t v, uint32_t lo, uint32_t hi) {
    uint32_t p = lo;
    while (p < hi && p < v) p <<= 1;
    return p;
}

}  // namespace

struct spsyrk_plan_s {
    PlanDev dev;
    spsyrk_dtype_t dtype;
    // Full-output mode over the whole column range is computed in two parts per row: the lower part (columns
    // <= row, this object, working exactly like the lower-triangle mode) and the upper part (columns > row, the
    // `upper` view: the rest of every column list).  The two parts of a row are sorted ranges that follow
    // each other in the output, so each is a product of half the size and the light-row kernels see rows of
    // half the work.  dev.mode is the column range the kernels of a view work on; user_mode what was asked for.
    spsyrk_mode_t user_mode;
    spsyrk_plan_s* upper;   // null in lower-triangle mode
    bool upper_active;      // the current range is computed in two parts
    uint2* desc_hi;         // descriptors of the upper parts (start after the row's own entry, rest of the column)
    int32_t* cnt_tot;       // rows: entries per row, both parts
    int64_t* hi_begin;      // rows + 1: where the upper part of every row starts in the output
    int64_t* work_sum;      // rows: work of both parts
    const int64_t* out_begin;  // set by spsyrk_numeric: where each row's part starts / ends in the output
    const int64_t* out_end;
    // spsyrk_numeric_rows: the numeric launches take only positions [sub_lo[c], sub_hi[c]) of class c's row list
    bool sub_active;
    int64_t sub_lo[NCLASS], sub_hi[NCLASS];
    // one-pass mode (spsyrk_onepass_*): per-row slot sizes (upper bounds for the light rows), their prefix sums, and
    // where the sorting numeric kernel reports the counts it finds
    int32_t* ub;
    int64_t* ub_off;
    int32_t* cnt_out;
    bool have_onepass;
    HostBlock host;  // words 0..31: facts of the two views; the rest: the position search of spsyrk_numeric_rows (upper view: unused)
    int64_t route_cap;
    // workspace views
    int32_t* perm;
    uint4* hdr;  // per-row headers in class order
    uint2* desc_full;  // descriptors for the whole column range (written by the transpose)
    uint2* desc_blk;   // descriptors narrowed to the current column range
    int32_t s0, s1;    // current column range
    int32_t* cnt;
    uint8_t* cls;
    uint32_t* colcnt;
    // radix sort buffers of the transpose (nnz entries each) and its histograms
    uint32_t *rx_key_a, *rx_row_a, *rx_pos_a, *rx_key_b, *rx_row_b, *rx_pos_b;
    void *rx_val_a, *rx_val_b;
    RadixState rx;
    int32_t* blockhist;
    int64_t* offsets;
    int64_t* partials;
    int64_t *state_bin, *state_items;  // status words of the scans of the binning, cleared with the counters
    uint32_t* items8;                  // rows: map words per row in class order
    void *zero_all, *zero_bin;         // the counters every plan starts from zero; those every binning does
    size_t zero_all_bytes, zero_bin_bytes;
    int64_t* state_col;
    int64_t* class_start_dev;  // NCLASS + 1
    unsigned long long* work_total_dev;
    // heavy rows by the kernel that computes them (rows_heavy.cuh)
    int32_t* route_list;    // NROUTE lists, route_cap apart
    uint32_t* route_count;  // 2 * NROUTE list lengths (device) ...
    uint32_t route_n[NROUTE];  // ... and as the host knows them after the symbolic pass
    int2* rank_parts;       // parts of the longest rows
    uint32_t* block_base;   // entries of a heavy row before every block of columns, [row][blocks_per_row]
    uint32_t blocks_per_row;
    RoutePieces sub_route[NROUTE];  // with sub_active: the pieces of the heavy rows' lists to compute
    // status words of the scan of the counts (the last ones of count_state_words), then for both views [ticket, words of the look-back], as
    // many as their heavy rows need
    unsigned long long* count_state;
    size_t count_state_words;
    uint32_t* facts;       // binary analysis (device): differs-from-one flag, heavy columns, threshold, histogram
    uint8_t* heavy_id;
    uint32_t* heavy_mask;
    int32_t* adeg;
    int64_t* itemoff;      // rows + 1, class order: where the map words of a light row start
    int64_t map_items;     // map words the current row range needs
    uint16_t* map;         // caller's item map (spsyrk_plan_lend_map), or null
    size_t map_bytes;
    bool map_filled;       // the last symbolic pass wrote the map
    int64_t* work_prefix;  // rows + 1: exclusive prefix sums of the per-row work (spsyrk_plan_partition)
    int64_t* part_bounds;  // MAX_PARTS + 1
    // host facts
    int64_t class_start[NCLASS + 1];
    int64_t work_total;
    uint32_t sparse_heavy[2];  // rows of classes 6 and 7 whose count is not settled by the binning
    bool have_symbolic;
    bool key64;
    bool diag;  // the light-row kernels handle the diagonal apart (lower-triangle mode, whole column range)
    int sm_count;
    int device;
    // optional per-class timing of the symbolic and numeric launches
    bool timing;
    cudaEvent_t ev_sym[NCLASS + 1];
    cudaEvent_t ev_num[NCLASS + 1];
};

namespace {

size_t carve(spsyrk_plan_s* pl, spsyrk_plan_s* up, void* ws, int64_t m, int64_t n, int64_t nnz, size_t sv, bool full) {
    Carver c(ws);
    const int64_t rows = std::max<int64_t>(m, 1);  // output rows; only the column pointers, counts and bit numbers go by columns
    const int64_t nb = bin_blocks_max(rows);
    auto colptr = c.take<int64_t>(n + 1);
    auto desc = c.take<uint2>(nnz);
    auto work = c.take<int64_t>(m);
    auto perm = c.take<int32_t>(m);
    auto hdr = c.take<uint4>(m);
    auto cnt = c.take<int32_t>(m);
    auto cls = c.take<uint8_t>(rows);
    const int npass = radix_passes((uint64_t)std::max<int64_t>(n - 1, 1));
    const size_t rx_words = radix_state_words(radix_tiles(nnz), radix_wide(nnz), npass);
    // counters in one piece, so that one memset clears them: the binning's, then the plan's, then the column counts
    const int views = full ? 2 : 1;
    const size_t bin_words = views * (2 + (size_t)scan_partials_count(NCLASS * nb) + (size_t)scan_partials_count(rows));
    auto zero = c.take<int64_t>(bin_words + 32 + (32 + HEAVY_BINS) / 2 + (size_t)scan_partials_count(std::max<int64_t>(n, 1)) + (size_t)(n + 1) / 2 +
                                RX_MAX_PASSES * RX_BINS + RX_MAX_PASSES + rx_words);
    Carver cz(zero);
    auto take_words = [&](size_t words) { int64_t* q = zero ? zero + cz.off : nullptr; cz.off += words; return q; };
    auto work_total_dev = reinterpret_cast<unsigned long long*>(take_words(2));  // and the heavy rows that are not dense
    auto state_bin = take_words(scan_partials_count(NCLASS * nb)), state_items = take_words(scan_partials_count(rows));
    unsigned long long* u_work_total_dev = full ? reinterpret_cast<unsigned long long*>(take_words(2)) : nullptr;
    int64_t* u_state_bin = full ? take_words(scan_partials_count(NCLASS * nb)) : nullptr;
    int64_t* u_state_items = full ? take_words(scan_partials_count(rows)) : nullptr;
    auto err = reinterpret_cast<uint32_t*>(take_words(32));
    auto facts = reinterpret_cast<uint32_t*>(take_words((32 + HEAVY_BINS) / 2));  // [0..1] binary analysis, [32..] its histogram
    auto state_col = take_words(scan_partials_count(std::max<int64_t>(n, 1)));
    auto colcnt = reinterpret_cast<uint32_t*>(take_words((size_t)(n + 1) / 2));
    RadixState rx;
    rx.bins = reinterpret_cast<unsigned long long*>(take_words(RX_MAX_PASSES * RX_BINS));
    rx.tickets = reinterpret_cast<uint32_t*>(take_words(RX_MAX_PASSES));
    rx.words = take_words(rx_words);
    const size_t zero_words = cz.off;
    // The two buffer sets of the radix sort (key, row, position, value per nonzero) are reused: the set that
    // the last pass does not read receives the column lists that pass writes (row ids and records), and the
    // set it does read holds, once the sort is over, the block descriptors.
    const size_t set_bytes = (size_t)nnz * (12 + sv) + 4 * ALIGN;
    auto set_a = c.take<char>(set_bytes);
    auto set_b = c.take<char>(set_bytes);
    Carver ca(set_a), cb(set_b);
    auto rx_key_a = ca.take<uint32_t>(nnz);
    auto rx_row_a = ca.take<uint32_t>(nnz);
    auto rx_pos_a = ca.take<uint32_t>(nnz);
    auto rx_val_a = ca.take<char>(nnz * sv);
    auto rx_key_b = cb.take<uint32_t>(nnz);
    auto rx_row_b = cb.take<uint32_t>(nnz);
    auto rx_pos_b = cb.take<uint32_t>(nnz);
    auto rx_val_b = cb.take<char>(nnz * sv);
    const bool last_reads_a = npass >= 2 && (npass % 2) == 0;  // pass p writes set A when p is even; one pass reads the input itself (and row ids kept in set B)
    Carver c_free(last_reads_a ? set_b : set_a), c_src(last_reads_a ? set_a : set_b);
    auto at_row = c_free.take<int32_t>(nnz + 4);  // the symbolic gathers read aligned 16-byte pieces: up to 3 entries past the end
    auto at_rec = c_free.take<char>(nnz * (sv == 8 ? 16 : 8));
    auto desc_blk = c_src.take<uint2>(nnz);
    auto blockhist = c.take<int32_t>(NCLASS * nb);
    auto offsets = c.take<int64_t>(NCLASS * nb + 1);
    auto partials = c.take<int64_t>(scan_partials_count(std::max<int64_t>(rows + 1, NCLASS * nb)));
    auto class_start_dev = c.take<int64_t>(NCLASS + 1);
    auto route_count = c.take<uint32_t>(2 * 2 * NROUTE);  // of every view: the lengths, the lengths of class 7's part
    // every route but the last takes rows of ranges of at most 2^18 columns, and there are no more of those than that
    static_assert(ROUTE_WIDE == NROUTE - 1, "the list that may hold all rows is the last");
    const int64_t route_cap = std::min<int64_t>(rows, ROW_CHUNK_BITS_MAX_NUMERIC);
    auto route_list = c.take<int32_t>(ROUTE_WIDE * route_cap + rows);
    const size_t count_state_words = (size_t)scan_partials_count(rows);
    auto count_state = c.take<unsigned long long>(count_state_words + views * (1 + (size_t)route_tiles(m) * NROUTE));
    // Rows that the rank kernel takes in parts: their range has at most 2^18 columns and more than the slots hold
    const int64_t ranged = std::min<int64_t>(m, ROW_CHUNK_BITS_MAX_NUMERIC);
    const int64_t slots = rank_slots_big<double>(pow2_at_least((uint64_t)m, 1024u, ROW_CHUNK_BITS_MAX_NUMERIC)), part = slots - BASE_BLOCK;
    const bool cut = m > slots;
    // parts of all such rows: a row of U columns has fewer than U / part + 2 of them; U is the row's number or m
    const int64_t parts_of_m = cut && m <= ROW_CHUNK_BITS_MAX_NUMERIC ? m * std::min<int64_t>(m / part + 1, MAX_ROW_PARTS) : 0;
    const int64_t parts_by_row = cut ? (ranged - slots) + ((ranged - slots) * (ranged + slots + 1) / 2) / part : 0;
    const uint32_t blocks_per_row = cut ? (uint32_t)((ranged + BASE_BLOCK - 1) / BASE_BLOCK) : 0u;
    auto rank_parts = c.take<int2>(full ? std::max(parts_of_m, parts_by_row) : parts_by_row);
    auto block_base = c.take<uint32_t>(ranged * blocks_per_row);
    auto work_prefix = c.take<int64_t>(rows + 1);
    auto itemoff = c.take<int64_t>(rows + 1);
    auto heavy_id = c.take<uint8_t>(std::max<int64_t>(n, 1));
    const int64_t mask_stride = (rows + 3) / 4 * 4;
    auto heavy_mask = c.take<uint32_t>(HEAVY_PLANES * mask_stride);
    auto items8 = c.take<uint32_t>(rows);
    auto adeg = c.take<int32_t>(std::max<int64_t>(m, 1));
    auto part_bounds = c.take<int64_t>(MAX_PARTS + 1);
    auto ub = c.take<int32_t>(std::max<int64_t>(m, 1));
    auto ub_off = c.take<int64_t>(rows + 1);
    // full-output mode: the upper view's own per-row arrays and the second descriptor array
    uint2* desc_hi = nullptr;
    int64_t *u_work = nullptr, *u_itemoff = nullptr, *u_class_start_dev = nullptr, *hi_begin = nullptr, *work_sum = nullptr;
    int32_t *u_perm = nullptr, *u_cnt = nullptr, *cnt_tot = nullptr, *u_route_list = nullptr;
    int2* u_rank_parts = nullptr;
    uint32_t* u_block_base = nullptr;
    uint4* u_hdr = nullptr;
    uint8_t* u_cls = nullptr;
    if (full) {
        desc_hi = c.take<uint2>(nnz);
        u_work = c.take<int64_t>(m);
        u_perm = c.take<int32_t>(m);
        u_hdr = c.take<uint4>(m);
        u_cnt = c.take<int32_t>(m);
        u_cls = c.take<uint8_t>(rows);
        u_itemoff = c.take<int64_t>(rows + 1);
        u_class_start_dev = c.take<int64_t>(NCLASS + 1);
        cnt_tot = c.take<int32_t>(m);
        u_route_list = c.take<int32_t>(ROUTE_WIDE * route_cap + rows);
        u_rank_parts = c.take<int2>(parts_of_m);
        u_block_base = c.take<uint32_t>(parts_of_m ? ranged * blocks_per_row : 0);
        hi_begin = c.take<int64_t>(rows + 1);
        work_sum = c.take<int64_t>(m);
    }
    if (pl) {
        pl->desc_hi = desc_hi; pl->cnt_tot = cnt_tot; pl->hi_begin = hi_begin; pl->work_sum = work_sum;
        pl->route_count = route_count; pl->route_list = route_list; pl->count_state = count_state; pl->count_state_words = count_state_words; pl->rank_parts = rank_parts;
        pl->block_base = block_base; pl->blocks_per_row = blocks_per_row;
        pl->dev.mask_stride = mask_stride;
        pl->work_prefix = work_prefix; pl->part_bounds = part_bounds; pl->itemoff = itemoff;
        pl->ub = ub; pl->ub_off = ub_off;
        pl->dev.heavy_id = heavy_id; pl->dev.heavy_mask = heavy_mask; pl->facts = facts;
        pl->heavy_id = heavy_id; pl->heavy_mask = heavy_mask; pl->adeg = adeg; pl->dev.adeg = adeg;
        pl->dev.colptr = colptr; pl->dev.at_row = at_row; pl->dev.at_rec = at_rec; pl->dev.desc = desc;
        pl->dev.work = work; pl->dev.err = err;
        pl->desc_full = desc; pl->desc_blk = desc_blk;
        pl->perm = perm; pl->hdr = hdr; pl->cnt = cnt; pl->cls = cls; pl->colcnt = colcnt;
        pl->rx_key_a = rx_key_a; pl->rx_row_a = rx_row_a; pl->rx_pos_a = rx_pos_a; pl->rx_key_b = rx_key_b; pl->rx_row_b = rx_row_b;
        pl->rx_pos_b = rx_pos_b; pl->rx_val_a = rx_val_a; pl->rx_val_b = rx_val_b; pl->rx = rx;
        pl->blockhist = blockhist; pl->offsets = offsets; pl->partials = partials;
        pl->class_start_dev = class_start_dev; pl->work_total_dev = work_total_dev;
        pl->state_bin = state_bin; pl->state_items = state_items; pl->state_col = state_col; pl->items8 = items8;
        pl->zero_all = zero; pl->zero_all_bytes = zero_words * sizeof(int64_t);
        pl->route_cap = route_cap; pl->zero_bin = zero; pl->zero_bin_bytes = bin_words * sizeof(int64_t);
        pl->dev.nheavy = facts + 1;
        if (up) {
            // the upper view shares everything that describes A and the scratch space; its rows are its own
            *up = *pl;
            up->upper = nullptr;
            up->dev.desc = desc_hi; up->dev.work = u_work;
            up->perm = u_perm; up->hdr = u_hdr; up->cnt = u_cnt; up->cls = u_cls; up->itemoff = u_itemoff;
            up->class_start_dev = u_class_start_dev; up->work_total_dev = u_work_total_dev;
            up->state_bin = u_state_bin; up->state_items = u_state_items;
            up->route_count = route_count + 2 * NROUTE; up->route_list = u_route_list;
            up->rank_parts = u_rank_parts; up->block_base = u_block_base;
        }
    }
    return (c.off + ALIGN - 1) / ALIGN * ALIGN;
}

inline bool brief_rows(int64_t rows, int64_t resident) { return rows <= 16 * resident; }  // a few rows per CTA

// CTAs of a kernel that an SM holds at once, asked for once per device (and the shared memory it needs is allowed once).  One
// object per kernel.
struct Residency {
    static constexpr int DEVICES = 64;
    std::atomic<int> per_sm[DEVICES] = {};
    template <typename Kernel>
    cudaError_t get(Kernel kern, int threads, size_t smem, int device, int* out) {
        const bool known = device >= 0 && device < DEVICES;
        int n = known ? per_sm[device].load(std::memory_order_relaxed) : 0;
        if (n == 0) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, threads, smem);
            if (e != cudaSuccess) return e;
            n = std::max(n, 1);
            if (known) per_sm[device].store(n, std::memory_order_relaxed);
        }
        *out = n;
        return cudaSuccess;
    }
};

[[maybe_unused]] spsyrk_status_t read_err(spsyrk_plan_s* pl, cudaStream_t st) {
    uint32_t e = 0;
    SPSYRK_CUDA_TRY(cudaMemcpyAsync(&e, pl->dev.err, sizeof(e), cudaMemcpyDeviceToHost, st));
    SPSYRK_CUDA_TRY(cudaStreamSynchronize(st));
    return status_of(e);
}

template <int G, typename V>
void launch_row_expand_v(spsyrk_plan_s* pl, cudaStream_t st) {
    const PlanDev& P = pl->dev;
    const int64_t threads = std::max<int64_t>(P.m, 1) * G;
    row_expand_kernel<G, V><<<(unsigned)((threads + 255) / 256), 256, 0, st>>>(P.rowptr, P.colidx, static_cast<const V*>(P.vals), P.m, P.n, P.nnz,
                                                                               pl->colcnt, pl->rx_row_b, pl->adeg, pl->facts, P.err);
    note_launches(1);
}
template <int G>
void launch_row_expand(spsyrk_plan_s* pl, cudaStream_t st) {
    if (pl->dtype == SPSYRK_F64) launch_row_expand_v<G, double>(pl, st);
    else if (pl->dtype == SPSYRK_F32) launch_row_expand_v<G, float>(pl, st);
    else launch_row_expand_v<G, int32_t>(pl, st);
}

template <int G>
void launch_block_desc(spsyrk_plan_s* pl, cudaStream_t st) {
    const PlanDev& P = pl->dev;
    const int64_t threads = (int64_t)(P.r1 - P.r0) * G;
    block_desc_kernel<G><<<(unsigned)((threads + 255) / 256), 256, 0, st>>>(P, pl->desc_full, pl->user_mode == SPSYRK_FULL ? pl->desc_hi : nullptr, pl->desc_blk, pl->s0, pl->s1);
    note_launches(1);
}

// analyse: the binary analysis is due (a new plan's first view); at least two CTAs, at most what the GPU holds beside others
template <int G>
cudaError_t launch_row_work(spsyrk_plan_s* pl, bool analyse, cudaStream_t st) {
    const PlanDev& P = pl->dev;
    const int64_t rows = P.r1 - P.r0, nb = bin_blocks(rows);
    HeavyArrays heavy{pl->colcnt, pl->facts, pl->heavy_id, pl->heavy_mask, 0u};
    if (analyse) heavy.ctas = (unsigned)std::min<int64_t>(2 + std::max<int64_t>(P.n, (int64_t)P.m * G) / BIN_THREADS, (int64_t)pl->sm_count * 8);
    if (nb > 0)
        return launch_linked(row_work_kernel<G>, (unsigned)nb + heavy.ctas, BIN_THREADS, 0, st, P, pl->cls, BLOCK_CLASS_MAX_WORK, ROW_CHUNK_BITS_MAX_SYMBOLIC, pl->diag,
                             bin_tile(rows), pl->blockhist, nb, pl->work_total_dev, pl->work_total_dev + 1, heavy);
    if (analyse) {
        heavy_analysis_kernel<G><<<heavy.ctas, BIN_THREADS, 0, st>>>(P, heavy);
        note_launches(1);
    }
    return cudaGetLastError();
}

int group_width(int64_t nnz, int64_t m) {
    const double avg = m > 0 ? (double)nnz / (double)m : 0.0;
    return avg <= 4 ? 4 : avg <= 8 ? 8 : avg <= 16 ? 16 : 32;
}

// stable radix sort of the nonzeros by column id; the last pass writes the column lists and descriptors.
// VB: unsigned integer of the value's width (values are only moved)
template <typename VB>
spsyrk_status_t sort_by_column(spsyrk_plan_s* pl, cudaStream_t st) {
    const PlanDev& P = pl->dev;
    if (P.nnz == 0) return SPSYRK_OK;
    const int npass = radix_passes((uint64_t)std::max<int64_t>(P.n - 1, 1));
    SPSYRK_CUDA_TRY(radix_bins<true>(pl->colcnt, P.n, npass, pl->rx.bins, st, HeavyHistogram{pl->facts}));  // from the column counts: n numbers, not nnz keys
    const uint32_t* src_key = reinterpret_cast<const uint32_t*>(P.colidx);
    const uint32_t* src_row = pl->rx_row_b;
    const VB* src_val = static_cast<const VB*>(P.vals);
    const uint32_t* src_pos = nullptr;  // position in A: the element's own index in the first pass
    for (int p = 0; p < npass; ++p) {
        const bool to_a = (p % 2) == 0;
        uint32_t* dst_key = to_a ? pl->rx_key_a : pl->rx_key_b;
        uint32_t* dst_row = to_a ? pl->rx_row_a : pl->rx_row_b;
        uint32_t* dst_pos = to_a ? pl->rx_pos_a : pl->rx_pos_b;
        VB* dst_val = static_cast<VB*>(to_a ? pl->rx_val_a : pl->rx_val_b);
        if (p == npass - 1) {
            EmitTransposeFinal<VB> emit{P, pl->desc_hi};
            SPSYRK_CUDA_TRY((radix_pass<VB, true>(src_key, src_row, src_val, src_pos, P.nnz, p, pl->rx, emit, P.err, st)));
        } else {
            EmitArrays3<VB> emit{dst_key, dst_row, dst_val, dst_pos};
            SPSYRK_CUDA_TRY((radix_pass<VB, true>(src_key, src_row, src_val, src_pos, P.nnz, p, pl->rx, emit, P.err, st)));
        }
        src_key = dst_key;
        src_row = dst_row;
        src_val = dst_val;
        src_pos = dst_pos;
    }
    return SPSYRK_OK;
}

__global__ void add_work_kernel(const int64_t* __restrict__ a, const int64_t* __restrict__ b, int64_t rows, int64_t* __restrict__ out) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r < rows) out[r] = a[r] + b[r];
}

__global__ void plan_facts_kernel(PlanFacts f) { f.publish(0); }

// Work estimate + binning of one view's current row range (dev.desc, dev.mode and diag are set).  The facts the host
// needs are on their way to `host` when this returns.
spsyrk_status_t bin_launch(spsyrk_plan_s* pl, int64_t* host, int64_t* gave_up, bool analyse, cudaStream_t st) {
    const int64_t rows = pl->dev.r1 - pl->dev.r0, nb = bin_blocks(rows);
    pl->have_symbolic = false;
    pl->have_onepass = false;
    pl->map_filled = false;
    const PlanDev& P = pl->dev;
    const PlanFacts facts{pl->class_start_dev, pl->work_total_dev, pl->work_total_dev + 1, pl->facts, P.err, host, gave_up};
    if (P.nnz == 0) analyse = false;
    switch (group_width(P.nnz, P.m)) {
        case 4: SPSYRK_CUDA_TRY(launch_row_work<4>(pl, analyse, st)); break;
        case 8: SPSYRK_CUDA_TRY(launch_row_work<8>(pl, analyse, st)); break;
        case 16: SPSYRK_CUDA_TRY(launch_row_work<16>(pl, analyse, st)); break;
        default: SPSYRK_CUDA_TRY(launch_row_work<32>(pl, analyse, st)); break;
    }
    if (rows == 0) {
        SPSYRK_CUDA_TRY(cudaMemsetAsync(pl->class_start_dev, 0, (NCLASS + 1) * sizeof(int64_t), st));
        plan_facts_kernel<<<1, 1, 0, st>>>(facts);
        note_launches(1);
        SPSYRK_CUDA_TRY(cudaGetLastError());
        return SPSYRK_OK;
    }
    SPSYRK_CUDA_TRY(scan_launch(ScanArray<int32_t>{pl->blockhist}, NCLASS * nb, BinStarts{pl->offsets, (uint32_t)nb, pl->class_start_dev}, pl->state_bin, P.err, st, true));
    SPSYRK_CUDA_TRY(launch_linked(row_scatter_kernel, (unsigned)nb, BIN_THREADS, 0, st, P, pl->cls, bin_tile(rows), pl->offsets, nb, pl->diag, pl->perm, pl->hdr, pl->items8,
                                  pl->cnt, pl->block_base, pl->blocks_per_row));
    SPSYRK_CUDA_TRY(scan_launch(ScanArray<uint32_t>{pl->items8}, rows, ItemStarts{pl->itemoff, rows, facts}, pl->state_items, P.err, st, true));
    return SPSYRK_OK;
}

// after the synchronisation
spsyrk_status_t bin_collect(spsyrk_plan_s* pl, const HostBlock& block, const int64_t* host) {
    std::memcpy(pl->class_start, host + PF_CLASS_START, sizeof(pl->class_start));
    pl->map_items = host[PF_MAP_ITEMS];
    pl->work_total = host[PF_WORK];
    for (int k = 0; k < 2; ++k) pl->sparse_heavy[k] = (uint32_t)((uint64_t)host[PF_SPARSE_HEAVY] >> (32 * k));
    pl->dev.binary = (pl->dev.nnz > 0 && host[PF_OTHER_THAN_ONE] == 0) ? 1 : 0;
    return status_of(block.errors(host[PF_ERR]));
}

// Descriptors, work estimate and binning of the plan's current block of output rows and columns; synchronises once.
// fresh: a new plan's first call (the counters of the binning are zero already, the binary analysis is due).
spsyrk_status_t estimate_and_bin(spsyrk_plan_s* pl, bool fresh, cudaStream_t st) {
    const int64_t rows = pl->dev.r1 - pl->dev.r0;
    const bool whole = pl->s0 <= 0 && pl->s1 >= pl->dev.m;
    pl->upper_active = false;
    if (!fresh) SPSYRK_CUDA_TRY(cudaMemsetAsync(pl->zero_bin, 0, pl->zero_bin_bytes, st));
    if (whole) {
        pl->dev.desc = pl->desc_full;
        // two parts per row in full-output mode: this view does the lower parts like the lower-triangle mode
        pl->upper_active = pl->user_mode == SPSYRK_FULL && pl->upper;
        pl->dev.mode = pl->upper_active ? SPSYRK_TRIL : (int32_t)pl->user_mode;
        pl->diag = pl->dev.mode == SPSYRK_TRIL;
    } else {
        // a column range: descriptors narrowed to [s0, s1) (cut out of the whole column lists in full-output mode)
        pl->dev.desc = pl->desc_blk;
        pl->dev.mode = (int32_t)pl->user_mode;
        pl->diag = false;
        if (rows > 0 && pl->dev.nnz > 0) {
            switch (group_width(pl->dev.nnz, pl->dev.m)) {
                case 4: launch_block_desc<4>(pl, st); break;
                case 8: launch_block_desc<8>(pl, st); break;
                case 16: launch_block_desc<16>(pl, st); break;
                default: launch_block_desc<32>(pl, st); break;
            }
        }
    }
    spsyrk_status_t s = bin_launch(pl, pl->host.dev, pl->host.dev + HOST_GAVE_UP, fresh, st);
    if (s != SPSYRK_OK) return s;
    spsyrk_plan_s* up = pl->upper_active ? pl->upper : nullptr;
    if (up) {
        up->dev.r0 = pl->dev.r0; up->dev.r1 = pl->dev.r1;
        up->dev.mode = SPSYRK_FULL;  // the upper part of row i lies in (i, m): the kernels work on the range [0, m)
        up->dev.desc = pl->desc_hi;
        up->dev.jaccard = pl->dev.jaccard;
        up->diag = false;
        s = bin_launch(up, pl->host.dev + 16, pl->host.dev + HOST_GAVE_UP, false, st);
        if (s != SPSYRK_OK) return s;
        if (rows > 0) {
            add_work_kernel<<<(unsigned)((rows + 255) / 256), 256, 0, st>>>(pl->dev.work, up->dev.work, rows, pl->work_sum);
            note_launches(1);
        }
    }
    SPSYRK_CUDA_TRY(wait_for(st));
    s = bin_collect(pl, pl->host, pl->host.host);
    if (s == SPSYRK_OK && up) s = bin_collect(up, pl->host, pl->host.host + 16);
    return s;
}
static_assert(PF_WORDS <= 16, "a view's facts take sixteen words of the host block");

int64_t map_items_total(const spsyrk_plan_s* pl) { return pl->map_items + (pl->upper_active ? pl->upper->map_items : 0); }

bool use_map(const spsyrk_plan_s* pl) { return pl->map && pl->map_bytes >= (size_t)map_items_total(pl) * sizeof(uint16_t); }

template <int N, bool DIAG>
spsyrk_status_t launch_symbolic_warp_d(spsyrk_plan_s* pl, int c, Chain& ch) {
    const int64_t count = pl->class_start[c + 1] - pl->class_start[c];
    if (count <= 0) return SPSYRK_OK;
    constexpr int G = warp_class_group(N);
    constexpr int SW = symbolic_warps(N);
    constexpr int ROWS = SW * (32 / G);  // rows a CTA works on at a time
    constexpr size_t smem = (size_t)ROWS * SymbolicWarpSmem<N>::GROUP;
    auto kern = symbolic_warp_kernel<N, G, DIAG>;
    static Residency residency;
    int per_sm = 1;
    SPSYRK_CUDA_TRY(residency.get(kern, SW * 32, smem, pl->device, &per_sm));
    const int64_t want = (count + ROWS - 1) / ROWS;
    const int64_t cap = (int64_t)pl->sm_count * per_sm;
    SPSYRK_CUDA_TRY(ch.launch(want <= cap, kern, (unsigned)std::min(want, cap), SW * 32, smem, pl->dev, pl->hdr + pl->class_start[c], count, pl->cnt));
    return SPSYRK_OK;
}

template <int N>
spsyrk_status_t launch_symbolic_warp(spsyrk_plan_s* pl, int c, Chain& ch) {
    return pl->diag ? launch_symbolic_warp_d<N, true>(pl, c, ch) : launch_symbolic_warp_d<N, false>(pl, c, ch);
}

// the part of class c's row list (rows in ascending order) a numeric launch covers
inline int64_t numeric_first(const spsyrk_plan_s* pl, int c) { return pl->sub_active ? pl->sub_lo[c] : pl->class_start[c]; }
inline int64_t numeric_count(const spsyrk_plan_s* pl, int c) {
    return pl->sub_active ? pl->sub_hi[c] - pl->sub_lo[c] : pl->class_start[c + 1] - pl->class_start[c];
}

template <typename V, int N, typename Key, bool DIAG>
spsyrk_status_t launch_numeric_warp_d(spsyrk_plan_s* pl, int c, int32_t* c_colidx, void* c_vals, Chain& ch) {
    const int64_t count = numeric_count(pl, c);
    if (count <= 0) return SPSYRK_OK;
    constexpr int G = warp_class_group(N);
    constexpr int NW = numeric_warps(N);
    constexpr int ROWS = NW * (32 / G);
    constexpr size_t smem = (size_t)ROWS * NumericWarpSmem<V, N>::GROUP;
    // persistent groups: exactly as many CTAs as are resident at once, each group walks its rows with
    // a stride of the whole grid
    auto kern = numeric_warp_kernel<V, N, G, Key, DIAG>;
    static Residency residency;
    int per_sm = 1;
    SPSYRK_CUDA_TRY(residency.get(kern, NW * 32, smem, pl->device, &per_sm));
    const int64_t want = (count + ROWS - 1) / ROWS;
    const int64_t cap = (int64_t)pl->sm_count * per_sm;
    SPSYRK_CUDA_TRY(ch.launch(want <= cap, kern, (unsigned)std::min(want, cap), NW * 32, smem, pl->dev, pl->hdr + numeric_first(pl, c), count, pl->out_begin, pl->out_end,
                                                               c_colidx, static_cast<V*>(c_vals), pl->cnt_out));
    return SPSYRK_OK;
}

template <typename V, int N, typename Key>
spsyrk_status_t launch_numeric_warp(spsyrk_plan_s* pl, int c, int32_t* c_colidx, void* c_vals, Chain& ch) {
    return pl->diag ? launch_numeric_warp_d<V, N, Key, true>(pl, c, c_colidx, c_vals, ch)
                    : launch_numeric_warp_d<V, N, Key, false>(pl, c, c_colidx, c_vals, ch);
}

template <int N, typename Key, bool DIAG>
spsyrk_status_t launch_symbolic_sort_d(spsyrk_plan_s* pl, int c, Chain& ch) {
    const int64_t count = pl->class_start[c + 1] - pl->class_start[c];
    if (count <= 0) return SPSYRK_OK;
    constexpr int G = warp_class_group(N);
    constexpr int SW = symbolic_sort_warps(N);
    constexpr int ROWS = SW * (32 / G);
    constexpr size_t smem = (size_t)ROWS * SymbolicSortSmem<N>::GROUP;
    auto kern = symbolic_sort_warp_kernel<N, G, Key, DIAG>;
    static Residency residency;
    int per_sm = 1;
    SPSYRK_CUDA_TRY(residency.get(kern, SW * 32, smem, pl->device, &per_sm));
    const int64_t want = (count + ROWS - 1) / ROWS;
    const int64_t cap = (int64_t)pl->sm_count * per_sm;
    SPSYRK_CUDA_TRY(ch.launch(want <= cap, kern, (unsigned)std::min(want, cap), SW * 32, smem, pl->dev, pl->hdr + pl->class_start[c], pl->itemoff + pl->class_start[c],
                                                               count, pl->cnt, pl->map));
    return SPSYRK_OK;
}

template <int N>
spsyrk_status_t launch_symbolic_sort(spsyrk_plan_s* pl, int c, Chain& ch) {
    if (pl->key64)
        return pl->diag ? launch_symbolic_sort_d<N, uint64_t, true>(pl, c, ch) : launch_symbolic_sort_d<N, uint64_t, false>(pl, c, ch);
    return pl->diag ? launch_symbolic_sort_d<N, uint32_t, true>(pl, c, ch) : launch_symbolic_sort_d<N, uint32_t, false>(pl, c, ch);
}

template <typename V, int N, bool DIAG>
spsyrk_status_t launch_numeric_map_d(spsyrk_plan_s* pl, int c, int32_t* c_colidx, void* c_vals, Chain& ch) {
    const int64_t count = numeric_count(pl, c);
    if (count <= 0) return SPSYRK_OK;
    constexpr int G = warp_class_group(N);
    constexpr int NW = numeric_map_warps(N);
    constexpr int ROWS = NW * (32 / G);
    constexpr size_t smem = (size_t)ROWS * NumericMapSmem<V, N>::GROUP;
    auto kern = numeric_map_warp_kernel<V, N, G, DIAG>;
    static Residency residency;
    int per_sm = 1;
    SPSYRK_CUDA_TRY(residency.get(kern, NW * 32, smem, pl->device, &per_sm));
    const int64_t want = (count + ROWS - 1) / ROWS;
    const int64_t cap = (int64_t)pl->sm_count * per_sm;
    SPSYRK_CUDA_TRY(ch.launch(want <= cap, kern, (unsigned)std::min(want, cap), NW * 32, smem, pl->dev, pl->hdr + numeric_first(pl, c), pl->itemoff + numeric_first(pl, c),
                                                               count, pl->map, pl->out_begin, pl->out_end, c_colidx, static_cast<V*>(c_vals)));
    return SPSYRK_OK;
}

template <typename V, int N>
spsyrk_status_t launch_numeric_map(spsyrk_plan_s* pl, int c, int32_t* c_colidx, void* c_vals, Chain& ch) {
    return pl->diag ? launch_numeric_map_d<V, N, true>(pl, c, c_colidx, c_vals, ch)
                    : launch_numeric_map_d<V, N, false>(pl, c, c_colidx, c_vals, ch);
}

inline void mark(spsyrk_plan_s* pl, cudaEvent_t* ev, int i, const Chain& ch) {
    if (pl->timing) cudaEventRecord(ev[i], ch.st);
}

template <typename V>
void launch_numeric_map_all(spsyrk_plan_s* pl, int32_t* c_colidx, void* c_vals, Chain& ch) {
    mark(pl, pl->ev_num, 1, ch);
    launch_numeric_map<V, 32>(pl, 1, c_colidx, c_vals, ch);
    mark(pl, pl->ev_num, 2, ch);
    launch_numeric_map<V, 64>(pl, 2, c_colidx, c_vals, ch);
    mark(pl, pl->ev_num, 3, ch);
    launch_numeric_map<V, 128>(pl, 3, c_colidx, c_vals, ch);
    mark(pl, pl->ev_num, 4, ch);
    launch_numeric_map<V, 256>(pl, 4, c_colidx, c_vals, ch);
    mark(pl, pl->ev_num, 5, ch);
    launch_numeric_map<V, 512>(pl, 5, c_colidx, c_vals, ch);
    mark(pl, pl->ev_num, 6, ch);
}

template <typename V, typename Key>
void launch_numeric_warp_all(spsyrk_plan_s* pl, int32_t* c_colidx, void* c_vals, Chain& ch) {
    mark(pl, pl->ev_num, 1, ch);
    launch_numeric_warp<V, 32, Key>(pl, 1, c_colidx, c_vals, ch);
    mark(pl, pl->ev_num, 2, ch);
    launch_numeric_warp<V, 64, Key>(pl, 2, c_colidx, c_vals, ch);
    mark(pl, pl->ev_num, 3, ch);
    launch_numeric_warp<V, 128, Key>(pl, 3, c_colidx, c_vals, ch);
    mark(pl, pl->ev_num, 4, ch);
    launch_numeric_warp<V, 256, Key>(pl, 4, c_colidx, c_vals, ch);
    mark(pl, pl->ev_num, 5, ch);
    launch_numeric_warp<V, 512, Key>(pl, 5, c_colidx, c_vals, ch);
    mark(pl, pl->ev_num, 6, ch);
}

// bounds[p] = r0 + the smallest r in [0, rows] with prefix[r] * parts >= p * prefix[rows]
// (the prefix sums' error word goes to the host)
__global__ void partition_kernel(const int64_t* __restrict__ prefix, int64_t rows, int64_t parts, int64_t r0,
                                 int64_t* __restrict__ bounds, const uint32_t* __restrict__ err, int64_t* __restrict__ host) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p == 0) host[0] = (int64_t)*err;
    if (p > parts) return;
    if (p == parts) { bounds[p] = r0 + rows; return; }
    const int64_t target = p * prefix[rows];
    int64_t lo = 0, hi = rows;  // prefix is non-decreasing; prefix[rows] * parts >= target always
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (prefix[mid] * parts >= target) hi = mid; else lo = mid + 1;
    }
    bounds[p] = r0 + lo;
}

uint32_t row_chunk_bits(const spsyrk_plan_s* pl, uint32_t cap) {
    const uint64_t umax = pl->dev.mode == SPSYRK_TRIL ? (uint64_t)pl->dev.r1 : (uint64_t)pl->dev.m;
    return pow2_at_least(umax, 1024u, cap);
}

// A row's masks of the heavy columns stand for all its products: not where the columns are a part (a block, or the upper part of
// the rows in full-output mode)
bool row_masks(const spsyrk_plan_s* pl) { return pl->dev.binary && pl->diag; }

template <int THREADS, bool MASKS>
spsyrk_status_t launch_symbolic_cta_m(spsyrk_plan_s* pl, int c, Chain& ch) {
    const int64_t count = pl->class_start[c + 1] - pl->class_start[c];
    if (count <= 0 || pl->sparse_heavy[c - 6] == 0) return SPSYRK_OK;
    const uint32_t cb = row_chunk_bits(pl, ROW_CHUNK_BITS_MAX_SYMBOLIC);
    const size_t smem = CtaRowSmem<int32_t, THREADS, false>::bytes(cb, 0);
    auto kern = rows_cta_kernel<int32_t, THREADS, false, MASKS>;
    SPSYRK_CUDA_TRY((allow_shared_memory<rows_cta_kernel<int32_t, THREADS, false, MASKS>>()));
    SPSYRK_CUDA_TRY(ch.launch(brief_rows(count, (int64_t)pl->sm_count * (2048 / THREADS)), kern, (unsigned)count, THREADS, smem, pl->dev, pl->perm + pl->class_start[c], cb, 0u, pl->cnt,
                              nullptr, nullptr, nullptr, nullptr, pl->block_base, pl->blocks_per_row));
    return SPSYRK_OK;
}
template <int THREADS>
spsyrk_status_t launch_symbolic_cta(spsyrk_plan_s* pl, int c, Chain& ch) {
    return row_masks(pl) ? launch_symbolic_cta_m<THREADS, true>(pl, c, ch) : launch_symbolic_cta_m<THREADS, false>(pl, c, ch);
}

// Shared-memory shapes of the heavy-row kernels and the rule that goes with them.  The small rank kernel is launched
// for three widths of its bitmap, so that rows in the lower part of the range leave room for more CTAs per SM.
struct HeavyShapes {
    RouteRule rule;
    uint32_t columns;  // of the widest bitmap
    uint32_t dense8_columns;
};

template <typename V>
HeavyShapes heavy_shapes(const spsyrk_plan_s* pl) {
    using Acc = typename AccOf<V>::type;
    HeavyShapes h;
    h.columns = row_chunk_bits(pl, ROW_CHUNK_BITS_MAX_NUMERIC);
    const uint32_t cb = h.columns;
    RouteRule& r = h.rule;
    r.wide = ROW_CHUNK_BITS_MAX_NUMERIC;
    r.bits0 = std::min(cb, 65536u);
    r.bits1 = std::min(cb, 131072u);
    r.slots_small = std::min(cb, (uint32_t)(16384 / sizeof(Acc)));
    r.slots_mid = std::min(cb, (uint32_t)(65536 / sizeof(Acc)));
    r.slots_big = rank_slots_big<V>(cb);
    // two CTAs per SM
    r.chunk = std::min(cb, (uint32_t)((SMEM_PER_CTA / 2 - 1024 - DirectSmem<V, DIRECT_THREADS>::bytes(0)) / (sizeof(Acc) * 32 + 32 + 4)) * 32);
    const uint64_t umax = pl->dev.mode == SPSYRK_TRIL ? (uint64_t)pl->dev.r1 : (uint64_t)pl->dev.m;
    h.dense8_columns = (uint32_t)std::min<uint64_t>(umax, (SMEM_PER_CTA - Dense8Smem<DENSE8_THREADS>::bytes(0)) / 16 * 16);
    r.dense8 = h.dense8_columns;
    r.binary = pl->dev.binary;
    r.masks = row_masks(pl);
    return h;
}

int64_t heavy_rows(const spsyrk_plan_s* pl) { return pl->class_start[NCLASS] - pl->class_start[6]; }

// which kernel computes which heavy row; the counts of the symbolic pass are known
spsyrk_status_t route_heavy(spsyrk_plan_s* pl, unsigned long long* state, cudaStream_t st) {
    const int64_t count = heavy_rows(pl);
    if (count <= 0) return SPSYRK_OK;
    const HeavyShapes h = pl->dtype == SPSYRK_I32 ? heavy_shapes<int32_t>(pl) : heavy_shapes<double>(pl);
    SPSYRK_CUDA_TRY(launch_linked(route_rows_kernel, (unsigned)route_tiles(count), ROUTE_THREADS, 0, st, pl->dev, h.rule, pl->perm + pl->class_start[6], count, pl->cnt,
                                  pl->block_base, pl->blocks_per_row, pl->route_list, pl->route_cap, pl->rank_parts, pl->class_start[NCLASS] - pl->class_start[7],
                                  pl->route_count, state + 1, state));
    return SPSYRK_OK;
}

// Clears what the counting pass's last steps need zero, in one piece: the status words of the scan of the counts, then the
// state of the routing (both views).  Before the counting kernels, so that nothing stands between them and those steps.
spsyrk_status_t clear_count_state(spsyrk_plan_s* pl, int64_t rows, cudaStream_t st) {
    spsyrk_plan_s* up = pl->upper_active ? pl->upper : nullptr;
    const bool heavy = heavy_rows(pl) || (up && heavy_rows(up));
    const size_t words = heavy ? 1 + (size_t)route_tiles(heavy_rows(pl)) * NROUTE + (up ? 1 + (size_t)route_tiles(heavy_rows(up)) * NROUTE : 0) : 0;
    const size_t first = (size_t)(pl->count_state_words - scan_partials_count(rows));  // the scan's words end where the routing's begin
    if (rows > SCAN_MIN_TILE || heavy)
        SPSYRK_CUDA_TRY(cudaMemsetAsync(pl->count_state + first, 0, (pl->count_state_words - first + words) * sizeof(unsigned long long), st));
    return SPSYRK_OK;
}

// the lists of both views; without heavy rows nothing is launched and nobody looks at the list lengths
spsyrk_status_t route_views(spsyrk_plan_s* pl, cudaStream_t st) {
    spsyrk_plan_s* up = pl->upper_active ? pl->upper : nullptr;
    if (!heavy_rows(pl) && !(up && heavy_rows(up))) return SPSYRK_OK;
    unsigned long long* const state = pl->count_state + pl->count_state_words;
    const spsyrk_status_t s = route_heavy(pl, state, st);
    return s == SPSYRK_OK && up ? route_heavy(up, state + 1 + (size_t)route_tiles(heavy_rows(pl)) * NROUTE, st) : s;
}

// A launch of one CTA per row or part of one (the CTAs that start take the others over): a brief one if there are few per CTA
template <auto Kernel, typename... Args>
cudaError_t launch_rows(const spsyrk_plan_s* pl, Chain& ch, int64_t units, int threads, size_t smem, Args... args) {
    cudaError_t e = allow_shared_memory<Kernel>();
    int per_sm = 1;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, Kernel, threads, smem);
    if (e != cudaSuccess) return e;
    return ch.launch(brief_rows(units, (int64_t)pl->sm_count * std::max(per_sm, 1)), Kernel, (unsigned)units, threads, smem, args...);
}

template <typename V>
spsyrk_status_t launch_heavy(spsyrk_plan_s* pl, int32_t* c_colidx, void* c_vals, Chain& ch) {
    using Acc = typename AccOf<V>::type;
    static_assert(sizeof(Acc) == sizeof(typename AccOf<std::conditional_t<std::is_same<V, int32_t>::value, int32_t, double>>::type), "the rule's shapes");
    if (!heavy_rows(pl)) return SPSYRK_OK;
    const HeavyShapes h = heavy_shapes<V>(pl);
    V* cv = static_cast<V*>(c_vals);
    auto pieces = [&](int k) { return pl->sub_active ? pl->sub_route[k] : RoutePieces{{0u, 0u}, {pl->route_n[k], 0u}}; };
    const bool aligned = ((reinterpret_cast<uintptr_t>(c_colidx) | reinterpret_cast<uintptr_t>(c_vals) | reinterpret_cast<uintptr_t>(pl->dev.jaccard)) & 15u) == 0;
    auto args = [&](int k) {
        return HeavyArgs{pl->route_list + k * (pl->route_cap), pieces(k), pl->out_begin, pl->out_end, c_colidx, aligned,
                         pl->rank_parts, k == ROUTE_RANK_BIG ? pieces(ROUTE_RANK_PARTS) : RoutePieces{}, pl->block_base, pl->blocks_per_row};
    };
    if (const int64_t units = pieces(ROUTE_DIRECT).total()) {
        SPSYRK_CUDA_TRY((launch_rows<rows_direct_kernel<V, DIRECT_THREADS>>(pl, ch, units, DIRECT_THREADS, DirectSmem<V, DIRECT_THREADS>::bytes(h.rule.chunk), pl->dev,
                                                                            args(ROUTE_DIRECT), h.rule.chunk, cv)));
    }
    auto rank = [&](auto shape, int k, uint32_t columns, uint32_t slots) -> cudaError_t {
        using Shape = decltype(shape);
        const int64_t units = (int64_t)pieces(k).total() + (k == ROUTE_RANK_BIG ? pieces(ROUTE_RANK_PARTS).total() : 0u);
        if (!units) return cudaSuccess;
        return launch_rows<rows_rank_kernel<V, Shape::THREADS, Shape::CTAS>>(pl, ch, units, Shape::THREADS, RankSmem<V, Shape::THREADS>::bytes(columns, slots), pl->dev,
                                                                             args(k), columns, slots, cv);
    };
    SPSYRK_CUDA_TRY(rank(RankShape<RANK_BIG_THREADS, 1>{}, ROUTE_RANK_BIG, h.columns, h.rule.slots_big));
    SPSYRK_CUDA_TRY(rank(RankShape<RANK_MID_THREADS, 2>{}, ROUTE_RANK_MID, h.columns, h.rule.slots_mid));
    SPSYRK_CUDA_TRY(rank(RankShape<RANK_SMALL_THREADS, 4>{}, ROUTE_RANK2, h.columns, h.rule.slots_small));
    SPSYRK_CUDA_TRY(rank(RankShape<RANK_SMALL_THREADS, 4>{}, ROUTE_RANK1, h.rule.bits1, h.rule.slots_small));
    SPSYRK_CUDA_TRY(rank(RankShape<RANK_SMALL_THREADS, 4>{}, ROUTE_RANK0, h.rule.bits0, h.rule.slots_small));
    if (const int64_t units = pieces(ROUTE_DENSE8).total()) {
        // Short rows have little to do for many threads: six CTAs of 256 where so many fit an SM, up to about 32 000 columns, three of 512 beyond
        // (similarities of 3001 sets 203 us to 191, 8000 373 to 335, 24 000 1487 to 1359; of 40 000, five CTAs, 3405 to 3590)
        const size_t narrow = Dense8Smem<DENSE8_SHORT_THREADS>::bytes(h.dense8_columns);
        if (6 * (narrow + SMEM_OF_A_CTA + 256) <= SMEM_PER_SM)
            SPSYRK_CUDA_TRY((launch_rows<rows_dense8_kernel<V, DENSE8_SHORT_THREADS, 6>>(pl, ch, units, DENSE8_SHORT_THREADS, narrow, pl->dev, args(ROUTE_DENSE8), h.dense8_columns, cv)));
        else
            SPSYRK_CUDA_TRY((launch_rows<rows_dense8_kernel<V, DENSE8_THREADS, 3>>(pl, ch, units, DENSE8_THREADS, Dense8Smem<DENSE8_THREADS>::bytes(h.dense8_columns), pl->dev,
                                                                                   args(ROUTE_DENSE8), h.dense8_columns, cv)));
    }
    const RoutePieces wide = pieces(ROUTE_WIDE);
    for (int k = 0; k < 2; ++k) {
        if (!wide.count[k]) continue;
        constexpr int THREADS = 1024;
        const size_t fixed = CtaRowSmem<V, THREADS, true>::bytes(h.columns, 0);
        const uint32_t slots = std::min((uint32_t)((LARGE_SMEM_BUDGET - fixed) / sizeof(Acc)), h.columns);
        const size_t smem = CtaRowSmem<V, THREADS, true>::bytes(h.columns, slots);
        auto kern = rows_cta_kernel<V, THREADS, true>;
        SPSYRK_CUDA_TRY((allow_shared_memory<rows_cta_kernel<V, THREADS, true>>()));
        SPSYRK_CUDA_TRY(ch.launch(brief_rows(wide.count[k], pl->sm_count), kern, wide.count[k], THREADS, smem, pl->dev,
                                  pl->route_list + ROUTE_WIDE * pl->route_cap + wide.first[k], h.columns, slots, nullptr, pl->out_begin, pl->out_end, c_colidx, cv,
                                  nullptr, 0u));
    }
    SPSYRK_CUDA_TRY(cudaGetLastError());
    return SPSYRK_OK;
}

template <typename V>
spsyrk_status_t numeric_typed(spsyrk_plan_s* pl, int32_t* c_colidx, void* c_vals, Chain& ch) {
    if (pl->map_filled) launch_numeric_map_all<V>(pl, c_colidx, c_vals, ch);
    else if (pl->key64) launch_numeric_warp_all<V, uint64_t>(pl, c_colidx, c_vals, ch);
    else launch_numeric_warp_all<V, uint32_t>(pl, c_colidx, c_vals, ch);
    mark(pl, pl->ev_num, 7, ch);  // the heavy rows of both classes are timed as one
    const spsyrk_status_t s = launch_heavy<V>(pl, c_colidx, c_vals, ch);
    if (s != SPSYRK_OK) return s;
    mark(pl, pl->ev_num, 8, ch);
    SPSYRK_CUDA_TRY(cudaGetLastError());
#ifdef SPSYRK_CHECKED
    return read_err(pl, ch.st);  // the bounds-checked build reports a skipped access at once (synchronises)
#else
    return SPSYRK_OK;
#endif
}

__global__ void add_counts_kernel(const int32_t* __restrict__ a, const int32_t* __restrict__ b, int64_t rows, int32_t* __restrict__ out) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r < rows) out[r] = a[r] + b[r];
}

__global__ void upper_begin_kernel(const int64_t* __restrict__ c_rowptr, const int32_t* __restrict__ cnt_lo, int64_t rows,
                                   int64_t* __restrict__ hi_begin) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r < rows) hi_begin[r] = c_rowptr[r] + cnt_lo[r];
}

// prefix sums, and for the host the total, the error word and the lengths of the heavy rows' lists (both views)
struct CountsOut {
    int64_t* out;
    int64_t n;
    const uint32_t *err, *routes;
    int64_t* host;
    __device__ __forceinline__ void operator()(int64_t i, int64_t ex) const { out[i] = ex; }
    __device__ __forceinline__ void total(int64_t t) const {
        uint32_t w[1 + 2 * NROUTE];
        w[0] = *err;
#pragma unroll
        for (int k = 0; k < 2 * NROUTE; ++k) w[1 + k] = routes[k < NROUTE ? k : k + NROUTE];
        out[n] = t;
        host[0] = t;
#pragma unroll
        for (int k = 0; k < 1 + 2 * NROUTE; ++k) host[1 + k] = (int64_t)w[k];
    }
    __device__ __forceinline__ void gave_up() const { host[HOST_GAVE_UP] = 1; }
};
static_assert(2 + 2 * NROUTE <= 32, "the totals take the first half of the host block");

// prefix sums of per-row counts into out[rows + 1]; what the host needs is on its way
// (cleared: clear_count_state has been called for this scan)
cudaError_t scan_counts(spsyrk_plan_s* pl, const int32_t* counts, int64_t rows, int64_t* out, bool cleared, cudaStream_t st) {
    if (rows == 0) return cudaMemsetAsync(out, 0, sizeof(int64_t), st);
    int64_t* const state = cleared ? reinterpret_cast<int64_t*>(pl->count_state + pl->count_state_words - scan_partials_count(rows)) : pl->partials;
    return scan_launch(ScanArray<int32_t>{counts}, rows, CountsOut{out, rows, pl->dev.err, pl->route_count, pl->host.dev}, state, pl->dev.err, st, cleared);
}
// waits for it
spsyrk_status_t collect_total(spsyrk_plan_s* pl, int64_t rows, bool routes, int64_t* total, cudaStream_t st) {
    SPSYRK_CUDA_TRY(wait_for(st));
    spsyrk_plan_s* up = pl->upper_active ? pl->upper : nullptr;
    if (rows == 0) {
        *total = 0;
        if (routes) std::memset(pl->route_n, 0, sizeof(pl->route_n));
        if (routes && up) std::memset(up->route_n, 0, sizeof(up->route_n));
        return SPSYRK_OK;
    }
    const int64_t* h = pl->host.host;
    const spsyrk_status_t s = status_of(pl->host.errors(h[1]));
    if (s == SPSYRK_OK) *total = h[0];
    for (int k = 0; routes && k < NROUTE; ++k) {
        pl->route_n[k] = heavy_rows(pl) ? (uint32_t)h[2 + k] : 0u;
        if (up) up->route_n[k] = heavy_rows(up) ? (uint32_t)h[2 + NROUTE + k] : 0u;
    }
    return s;
}

// the per-class count kernels of one view (entries per row into its cnt array)
spsyrk_status_t symbolic_view(spsyrk_plan_s* pl, bool with_map, Chain& ch) {
    pl->map_filled = false;
    mark(pl, pl->ev_sym, 1, ch);
    if (with_map) launch_symbolic_sort<32>(pl, 1, ch); else launch_symbolic_warp<32>(pl, 1, ch);
    mark(pl, pl->ev_sym, 2, ch);
    if (with_map) launch_symbolic_sort<64>(pl, 2, ch); else launch_symbolic_warp<64>(pl, 2, ch);
    mark(pl, pl->ev_sym, 3, ch);
    if (with_map) launch_symbolic_sort<128>(pl, 3, ch); else launch_symbolic_warp<128>(pl, 3, ch);
    mark(pl, pl->ev_sym, 4, ch);
    if (with_map) launch_symbolic_sort<256>(pl, 4, ch); else launch_symbolic_warp<256>(pl, 4, ch);
    mark(pl, pl->ev_sym, 5, ch);
    if (with_map) launch_symbolic_sort<512>(pl, 5, ch); else launch_symbolic_warp<512>(pl, 5, ch);
    mark(pl, pl->ev_sym, 6, ch);
    spsyrk_status_t s = launch_symbolic_cta<256>(pl, 6, ch);
    if (s != SPSYRK_OK) return s;
    mark(pl, pl->ev_sym, 7, ch);
    s = launch_symbolic_cta<1024>(pl, 7, ch);
    if (s != SPSYRK_OK) return s;
    mark(pl, pl->ev_sym, 8, ch);
    return SPSYRK_OK;
}

}  // namespace

namespace {
// slot size of every row in the one-pass layout: light rows by the number of their partial products (an upper
// bound of their entries; with the diagonal handled apart: products without the diagonal ones, plus the diagonal
// entry), heavy rows by the count their own symbolic kernels just found
__global__ void onepass_slots_kernel(PlanDev P, const uint8_t* __restrict__ cls, const int32_t* __restrict__ cnt, bool diag, int64_t rows,
                                     int32_t* __restrict__ ub) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= rows) return;
    const int c = cls[r] & (ROW_DENSE - 1);
    const int64_t i = P.r0 + r;
    const int64_t deg = P.rowptr[i + 1] - P.rowptr[i];
    int64_t u = 0;
    if (c >= 6) u = cnt[r];
    else if (c >= 1) u = diag ? P.work[r] - deg + (deg > 0 ? 1 : 0) : P.work[r];
    ub[r] = (int32_t)u;  // a light row has at most 512 + 32 products
}

// G lanes per row: row r moves from its slot to its place
template <typename V, int G>
__global__ void __launch_bounds__(256) onepass_compact_kernel(const int64_t* __restrict__ src_off, const int64_t* __restrict__ dst_off, int64_t rows,
                                                              const int32_t* __restrict__ s_col, const V* __restrict__ s_val,
                                                              int32_t* __restrict__ d_col, V* __restrict__ d_val) {
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
    const int gl = threadIdx.x & (G - 1);
    if (r >= rows) return;
    const int64_t s0 = src_off[r], d0 = dst_off[r], len = dst_off[r + 1] - d0;
    constexpr int UNR = 4;
    for (int64_t p = gl; p < len; p += UNR * G) {
        int32_t j[UNR];
        V v[UNR];
#pragma unroll
        for (int u = 0; u < UNR; ++u)
            if (p + u * G < len) { j[u] = s_col[s0 + p + u * G]; v[u] = s_val[s0 + p + u * G]; }
#pragma unroll
        for (int u = 0; u < UNR; ++u)
            if (p + u * G < len) { d_col[d0 + p + u * G] = j[u]; d_val[d0 + p + u * G] = v[u]; }
    }
}

template <typename V>
void launch_onepass_compact(const spsyrk_plan_s* pl, const int64_t* dst_off, int64_t rows, int64_t nnz, const int32_t* s_col, const void* s_val,
                            int32_t* d_col, void* d_val, cudaStream_t st) {
    const double avg = rows > 0 ? (double)nnz / (double)rows : 0.0;
#define COMPACT(G) \
    onepass_compact_kernel<V, G><<<(unsigned)((rows * G + 255) / 256), 256, 0, st>>>(pl->ub_off, dst_off, rows, s_col, static_cast<const V*>(s_val), \
                                                                                  d_col, static_cast<V*>(d_val))
    if (avg <= 4) COMPACT(4); else if (avg <= 8) COMPACT(8); else if (avg <= 16) COMPACT(16); else COMPACT(32);
#undef COMPACT
    note_launches(1);
}
}  // namespace


extern "C" {

spsyrk_status_t spsyrk_plan(spsyrk_plan_t* plan, int64_t m, int64_t n, int64_t nnz, const int64_t* d_rowptr,
                            const int32_t* d_colidx, const void* d_vals, spsyrk_dtype_t dtype, spsyrk_mode_t mode,
                            int64_t row_begin, int64_t row_end, void* d_workspace, size_t* workspace_bytes,
                            void* cuda_stream) {
    if (!workspace_bytes || m < 0 || n < 0 || nnz < 0) return SPSYRK_ERR_INVALID_ARG;
    if (dtype != SPSYRK_F64 && dtype != SPSYRK_F32 && dtype != SPSYRK_I32) return SPSYRK_ERR_INVALID_ARG;
    if (mode != SPSYRK_TRIL && mode != SPSYRK_FULL) return SPSYRK_ERR_INVALID_ARG;
    if (row_begin < 0 || row_end < row_begin || row_end > m) return SPSYRK_ERR_INVALID_ARG;
    if (m >= (int64_t(1) << 31) - 1 || n >= (int64_t(1) << 31) - 1 || nnz >= (int64_t(1) << 31) - 1) return SPSYRK_ERR_OVERFLOW;
    const size_t sv = dtype_size(dtype);
    const bool full = mode == SPSYRK_FULL;
    const size_t need = carve(nullptr, nullptr, nullptr, m, n, nnz, sv, full);
    if (!d_workspace) {
        *workspace_bytes = need;
        return SPSYRK_OK;
    }
    if (!plan || !d_rowptr || (nnz > 0 && (!d_colidx || !d_vals))) return SPSYRK_ERR_INVALID_ARG;
    if (*workspace_bytes < need) return SPSYRK_ERR_WORKSPACE;
    if (reinterpret_cast<uintptr_t>(d_workspace) % ALIGN) return SPSYRK_ERR_INVALID_ARG;

    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    spsyrk_plan_s* pl = new (std::nothrow) spsyrk_plan_s();
    if (!pl) return SPSYRK_ERR_INTERNAL;
    std::memset(pl, 0, sizeof(*pl));
    PlanDev& P = pl->dev;
    P.m = (int32_t)m; P.n = (int32_t)n; P.nnz = nnz; P.r0 = (int32_t)row_begin; P.r1 = (int32_t)row_end; P.mode = (int32_t)mode;
    P.rowptr = d_rowptr; P.colidx = d_colidx; P.vals = d_vals;
    pl->dtype = dtype;
    pl->user_mode = mode;
    pl->key64 = m > (int64_t(1) << 22);
    pl->s0 = 0;
    pl->s1 = (int32_t)m;
    {
        int dev_id = 0;
        pl->sm_count = 148;
        if (cudaGetDevice(&dev_id) == cudaSuccess) cudaDeviceGetAttribute(&pl->sm_count, cudaDevAttrMultiProcessorCount, dev_id);
        pl->device = dev_id;
    }
    spsyrk_plan_s* up = nullptr;
    if (full) {
        up = new (std::nothrow) spsyrk_plan_s();
        if (!up) { delete pl; return SPSYRK_ERR_INTERNAL; }
    }
    pl->upper = up;
    carve(pl, up, d_workspace, m, n, nnz, sv, full);
    pl->upper = up;  // (the copy into the upper view happened with a null link)

    auto fail = [&](spsyrk_status_t s) {
        if (s == SPSYRK_ERR_CUDA) cudaStreamSynchronize(st);  // a kernel under way may still write into the host block
        pl->host.release();
        delete up;
        delete pl;
        return s;
    };
#define PLAN_TRY(expr) do { if ((expr) != cudaSuccess) return fail(SPSYRK_ERR_CUDA); } while (0)
    PLAN_TRY(pl->host.acquire());
    PLAN_TRY(cudaMemsetAsync(pl->zero_all, 0, pl->zero_all_bytes, st));
    // 1. one sweep over A (checks, column histogram, row ids, row lengths, values all one?); 2. transpose: the histogram's
    // scan gives colptr; stable radix sort by column; 3. work estimate, row binning and binary analysis.  One synchronisation at
    // the end: nothing of the plan is under way when the call returns.
    const int g = group_width(nnz, m);
    switch (g) {
        case 4: launch_row_expand<4>(pl, st); break;
        case 8: launch_row_expand<8>(pl, st); break;
        case 16: launch_row_expand<16>(pl, st); break;
        default: launch_row_expand<32>(pl, st); break;
    }
    PLAN_TRY(exclusive_scan_i64<uint32_t>(pl->colcnt, n, P.colptr, pl->state_col, P.err, st, true));
    spsyrk_status_t s = sv == 8 ? sort_by_column<uint64_t>(pl, st) : sort_by_column<uint32_t>(pl, st);
    if (s != SPSYRK_OK) return fail(s);
    s = estimate_and_bin(pl, true, st);
    if (s != SPSYRK_OK) return fail(s);
#undef PLAN_TRY
    *plan = pl;
    return SPSYRK_OK;
}

spsyrk_status_t spsyrk_plan_set_block(spsyrk_plan_t plan, int64_t row_begin, int64_t row_end, int64_t col_begin,
                                      int64_t col_end, void* cuda_stream) {
    if (!plan || row_begin < 0 || row_end < row_begin || row_end > plan->dev.m) return SPSYRK_ERR_INVALID_ARG;
    if (col_begin < 0 || col_end < col_begin || col_end > plan->dev.m) return SPSYRK_ERR_INVALID_ARG;
    plan->dev.r0 = (int32_t)row_begin;
    plan->dev.r1 = (int32_t)row_end;
    plan->s0 = (int32_t)col_begin;
    plan->s1 = (int32_t)col_end;
    plan->have_symbolic = false;
    return estimate_and_bin(plan, false, static_cast<cudaStream_t>(cuda_stream));
}

spsyrk_status_t spsyrk_plan_set_rows(spsyrk_plan_t plan, int64_t row_begin, int64_t row_end, void* cuda_stream) {
    if (!plan) return SPSYRK_ERR_INVALID_ARG;
    return spsyrk_plan_set_block(plan, row_begin, row_end, 0, plan->dev.m, cuda_stream);
}

spsyrk_status_t spsyrk_plan_partition(spsyrk_plan_t plan, int64_t parts, int64_t* bounds, void* cuda_stream) {
    if (!plan || !bounds || parts < 1 || parts > MAX_PARTS) return SPSYRK_ERR_INVALID_ARG;
    spsyrk_plan_s* pl = plan;
    const int64_t work_all = pl->work_total + (pl->upper_active ? pl->upper->work_total : 0);
    if (work_all > 0 && work_all > INT64_MAX / parts) return SPSYRK_ERR_OVERFLOW;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const int64_t rows = pl->dev.r1 - pl->dev.r0;
    SPSYRK_CUDA_TRY(exclusive_scan_i64<int64_t>(pl->upper_active ? pl->work_sum : pl->dev.work, rows, pl->work_prefix, pl->partials, pl->dev.err, st));
    partition_kernel<<<(unsigned)((parts + 1 + 255) / 256), 256, 0, st>>>(pl->work_prefix, rows, parts, pl->dev.r0, pl->part_bounds, pl->dev.err, pl->host.dev);
    note_launches(1);
    SPSYRK_CUDA_TRY(cudaGetLastError());
    SPSYRK_CUDA_TRY(cudaMemcpyAsync(bounds, pl->part_bounds, (size_t)(parts + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    SPSYRK_CUDA_TRY(cudaStreamSynchronize(st));
    return status_of((uint32_t)pl->host.host[0]);
}

spsyrk_status_t spsyrk_symbolic(spsyrk_plan_t plan, int64_t* d_c_rowptr, int64_t* nnz_out, void* cuda_stream) {
    if (!plan || !d_c_rowptr || !nnz_out) return SPSYRK_ERR_INVALID_ARG;
    spsyrk_plan_s* pl = plan;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const int64_t rows = pl->dev.r1 - pl->dev.r0;
    const bool with_map = use_map(pl);
    Chain ch{st, !pl->timing};
    spsyrk_status_t s = clear_count_state(pl, rows, st);
    if (s == SPSYRK_OK) s = symbolic_view(pl, with_map, ch);
    if (s != SPSYRK_OK) return s;
    const int32_t* counts = pl->cnt;
    spsyrk_plan_s* up = pl->upper_active ? pl->upper : nullptr;
    if (up) {
        up->map = with_map ? pl->map + pl->map_items : nullptr;  // the upper parts' words follow the lower parts'
        up->map_bytes = with_map ? (size_t)up->map_items * sizeof(uint16_t) : 0;
        s = symbolic_view(up, with_map, ch);
        if (s != SPSYRK_OK) return s;
    }
    s = route_views(pl, st);
    if (s != SPSYRK_OK) return s;
    if (up) {
        if (rows > 0) {
            add_counts_kernel<<<(unsigned)((rows + 255) / 256), 256, 0, st>>>(pl->cnt, up->cnt, rows, pl->cnt_tot);
            note_launches(1);
        }
        counts = pl->cnt_tot;
    }
    SPSYRK_CUDA_TRY(scan_counts(pl, counts, rows, d_c_rowptr, true, st));
    if (pl->upper_active && rows > 0) {
        // the upper part of row r starts after its lower part
        upper_begin_kernel<<<(unsigned)((rows + 255) / 256), 256, 0, st>>>(d_c_rowptr, pl->cnt, rows, pl->hi_begin);
        note_launches(1);
    }
    s = collect_total(pl, rows, true, nnz_out, st);
    if (s != SPSYRK_OK) return s;
    pl->have_symbolic = true;
    pl->map_filled = with_map;
    if (pl->upper_active) { pl->upper->have_symbolic = true; pl->upper->map_filled = with_map; }
    return SPSYRK_OK;
}

spsyrk_status_t spsyrk_numeric(spsyrk_plan_t plan, const int64_t* d_c_rowptr, int32_t* d_c_colidx, void* d_c_vals,
                               void* cuda_stream) {
    if (!plan || !d_c_rowptr) return SPSYRK_ERR_INVALID_ARG;
    spsyrk_plan_s* pl = plan;
    if (!pl->have_symbolic) return SPSYRK_ERR_SEQUENCE;
    const int64_t work_all = pl->work_total + (pl->upper_active ? pl->upper->work_total : 0);
    if (work_all > 0 && (!d_c_colidx || !d_c_vals)) return SPSYRK_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    Chain ch{st, !pl->timing};
    auto run = [&](spsyrk_plan_s* v) {
        switch (v->dtype) {
            case SPSYRK_F64: return numeric_typed<double>(v, d_c_colidx, d_c_vals, ch);
            case SPSYRK_F32: return numeric_typed<float>(v, d_c_colidx, d_c_vals, ch);
            default: return numeric_typed<int32_t>(v, d_c_colidx, d_c_vals, ch);
        }
    };
    pl->out_begin = d_c_rowptr;
    pl->out_end = pl->upper_active ? pl->hi_begin : d_c_rowptr + 1;
    spsyrk_status_t s = run(pl);
    if (s != SPSYRK_OK || !pl->upper_active) return s;
    spsyrk_plan_s* up = pl->upper;
    up->dev.jaccard = pl->dev.jaccard;
    up->out_begin = pl->hi_begin;
    up->out_end = d_c_rowptr + 1;
    return run(up);
}

namespace {
// out[(2 * c) + e] = first position of class c's row list (ascending local row ids) whose row is >= bound[e]; behind them the
// pieces of the heavy rows' lists (route_positions), where there are any
constexpr int POSITION_WORDS = 2 * NCLASS + 4 * NROUTE;
static_assert(32 + 2 * POSITION_WORDS <= HOST_GAVE_UP, "the positions of both views in the rest of the host block");
__global__ void class_positions_kernel(const int32_t* __restrict__ perm, const int64_t* __restrict__ class_start_dev, int64_t lo_row,
                                       int64_t hi_row, bool heavy, const int32_t* __restrict__ lists, int64_t cap, const int2* __restrict__ rank_parts,
                                       const uint32_t* __restrict__ lengths, int64_t* __restrict__ out) {
    const int t = threadIdx.x;
    if (t >= 2 * NCLASS) {
        if (heavy && t < POSITION_WORDS) route_positions(t - 2 * NCLASS, lists, cap, rank_parts, lengths, lo_row, hi_row, out + 2 * NCLASS);
        return;
    }
    const int c = t >> 1;
    const int64_t bound = (t & 1) ? hi_row : lo_row;
    int64_t lo = class_start_dev[c], hi = class_start_dev[c + 1];
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if ((int64_t)perm[mid] < bound) lo = mid + 1; else hi = mid;
    }
    out[t] = lo;
}
}  // namespace

spsyrk_status_t spsyrk_numeric_rows(spsyrk_plan_t plan, int64_t row_begin, int64_t row_end, const int64_t* d_c_rowptr,
                                    int32_t* d_c_colidx, void* d_c_vals, void* cuda_stream) {
    if (!plan || !d_c_rowptr) return SPSYRK_ERR_INVALID_ARG;
    spsyrk_plan_s* pl = plan;
    if (!pl->have_symbolic) return SPSYRK_ERR_SEQUENCE;
    if (row_begin < pl->dev.r0 || row_end > pl->dev.r1 || row_begin > row_end) return SPSYRK_ERR_INVALID_ARG;
    if (row_begin == row_end) return SPSYRK_OK;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    // where the rows of the range sit in every class's list: one small kernel per view and one read-back
    // The kernel writes straight into pinned host memory: a device-to-host copy would queue behind whatever the
    // caller is downloading at the moment (the point of this call is to overlap with such copies).
    int64_t* const dev_pos = pl->host.dev + 32;
    spsyrk_plan_s* views[2] = {pl, pl->upper_active ? pl->upper : nullptr};
    for (int v = 0; v < 2; ++v) {
        if (!views[v]) continue;
        class_positions_kernel<<<1, 64, 0, st>>>(views[v]->perm, views[v]->class_start_dev, row_begin - pl->dev.r0, row_end - pl->dev.r0, heavy_rows(views[v]) > 0,
                                                 views[v]->route_list, pl->route_cap, views[v]->rank_parts, views[v]->route_count,
                                                 dev_pos + v * POSITION_WORDS);
        note_launches(1);
    }
    static_assert(POSITION_WORDS <= 64, "one thread per position");
    SPSYRK_CUDA_TRY(cudaGetLastError());
    SPSYRK_CUDA_TRY(cudaStreamSynchronize(st));
    for (int v = 0; v < 2; ++v) {
        if (!views[v]) continue;
        const int64_t* pos = pl->host.host + 32 + v * POSITION_WORDS;
        views[v]->sub_active = true;
        for (int c = 0; c < NCLASS; ++c) { views[v]->sub_lo[c] = pos[2 * c]; views[v]->sub_hi[c] = pos[2 * c + 1]; }
        pos += 2 * NCLASS;
        for (int k = 0; k < NROUTE; ++k) {
            RoutePieces& r = views[v]->sub_route[k];
            for (int e = 0; e < 2; ++e) {
                r.first[e] = heavy_rows(views[v]) ? (uint32_t)pos[4 * k + 2 * e] : 0u;
                r.count[e] = heavy_rows(views[v]) ? (uint32_t)(pos[4 * k + 2 * e + 1] - pos[4 * k + 2 * e]) : 0u;
            }
        }
    }
    const spsyrk_status_t s = spsyrk_numeric(plan, d_c_rowptr, d_c_colidx, d_c_vals, cuda_stream);
    for (int v = 0; v < 2; ++v)
        if (views[v]) views[v]->sub_active = false;
    return s;
}

spsyrk_status_t spsyrk_onepass_slots(spsyrk_plan_t plan, int64_t* slot_entries, void* cuda_stream) {
    if (!plan || !slot_entries) return SPSYRK_ERR_INVALID_ARG;
    spsyrk_plan_s* pl = plan;
    if (pl->upper_active) return SPSYRK_ERR_NOT_IMPLEMENTED;  // the two-part full-output mode keeps the two-pass route
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const int64_t rows = pl->dev.r1 - pl->dev.r0;
    pl->have_onepass = false;
    // heavy rows: their counts come from their own kernels (bitmaps), as in the symbolic pass
    Chain ch{st, !pl->timing};
    spsyrk_status_t s = clear_count_state(pl, rows, st);
    if (s == SPSYRK_OK) s = launch_symbolic_cta<256>(pl, 6, ch);
    if (s != SPSYRK_OK) return s;
    s = launch_symbolic_cta<1024>(pl, 7, ch);
    if (s == SPSYRK_OK) s = route_views(pl, st);
    if (s != SPSYRK_OK) return s;
    if (rows > 0) {
        onepass_slots_kernel<<<(unsigned)((rows + 255) / 256), 256, 0, st>>>(pl->dev, pl->cls, pl->cnt, pl->diag, rows, pl->ub);
        note_launches(1);
    }
    SPSYRK_CUDA_TRY(scan_counts(pl, pl->ub, rows, pl->ub_off, true, st));
    s = collect_total(pl, rows, true, slot_entries, st);
    if (s != SPSYRK_OK) return s;
    pl->have_onepass = true;
    return SPSYRK_OK;
}

spsyrk_status_t spsyrk_onepass_numeric(spsyrk_plan_t plan, int32_t* d_slot_colidx, void* d_slot_vals, int64_t* d_c_rowptr, int64_t* nnz_out,
                                       void* cuda_stream) {
    if (!plan || !d_c_rowptr || !nnz_out) return SPSYRK_ERR_INVALID_ARG;
    spsyrk_plan_s* pl = plan;
    if (!pl->have_onepass) return SPSYRK_ERR_SEQUENCE;
    if (pl->dev.jaccard) return SPSYRK_ERR_INVALID_ARG;  // the fused similarity is written at final offsets only
    if (pl->work_total > 0 && (!d_slot_colidx || !d_slot_vals)) return SPSYRK_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const int64_t rows = pl->dev.r1 - pl->dev.r0;
    // every row is computed into its slot; the light rows report their counts (the heavy ones have theirs already)
    const bool map_was = pl->map_filled;
    pl->map_filled = false;  // the kernel that sorts in the numeric pass counts as it goes
    pl->cnt_out = pl->cnt;
    pl->out_begin = pl->ub_off;
    pl->out_end = pl->ub_off + 1;
    Chain ch{st, !pl->timing};
    spsyrk_status_t s;
    switch (pl->dtype) {
        case SPSYRK_F64: s = numeric_typed<double>(pl, d_slot_colidx, d_slot_vals, ch); break;
        case SPSYRK_F32: s = numeric_typed<float>(pl, d_slot_colidx, d_slot_vals, ch); break;
        default: s = numeric_typed<int32_t>(pl, d_slot_colidx, d_slot_vals, ch); break;
    }
    pl->cnt_out = nullptr;
    pl->map_filled = map_was;
    if (s != SPSYRK_OK) return s;
    SPSYRK_CUDA_TRY(scan_counts(pl, pl->cnt, rows, d_c_rowptr, false, st));
    return collect_total(pl, rows, false, nnz_out, st);
}

spsyrk_status_t spsyrk_onepass_row_begin(spsyrk_plan_t plan, int64_t* d_row_begin, void* cuda_stream) {
    if (!plan || !d_row_begin) return SPSYRK_ERR_INVALID_ARG;
    if (!plan->have_onepass) return SPSYRK_ERR_SEQUENCE;
    const int64_t rows = plan->dev.r1 - plan->dev.r0;
    SPSYRK_CUDA_TRY(cudaMemcpyAsync(d_row_begin, plan->ub_off, (size_t)(rows + 1) * sizeof(int64_t), cudaMemcpyDeviceToDevice,
                                    static_cast<cudaStream_t>(cuda_stream)));
    return SPSYRK_OK;
}

spsyrk_status_t spsyrk_onepass_compact(spsyrk_plan_t plan, const int64_t* d_c_rowptr, int64_t nnz, const int32_t* d_slot_colidx,
                                       const void* d_slot_vals, int32_t* d_c_colidx, void* d_c_vals, void* cuda_stream) {
    if (!plan || !d_c_rowptr || nnz < 0) return SPSYRK_ERR_INVALID_ARG;
    spsyrk_plan_s* pl = plan;
    if (!pl->have_onepass) return SPSYRK_ERR_SEQUENCE;
    if (nnz > 0 && (!d_slot_colidx || !d_slot_vals || !d_c_colidx || !d_c_vals)) return SPSYRK_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const int64_t rows = pl->dev.r1 - pl->dev.r0;
    if (rows > 0 && nnz > 0) {
        if (pl->dtype == SPSYRK_F64) launch_onepass_compact<uint64_t>(pl, d_c_rowptr, rows, nnz, d_slot_colidx, d_slot_vals, d_c_colidx, d_c_vals, st);
        else launch_onepass_compact<uint32_t>(pl, d_c_rowptr, rows, nnz, d_slot_colidx, d_slot_vals, d_c_colidx, d_c_vals, st);
    }
    SPSYRK_CUDA_TRY(cudaGetLastError());
    return SPSYRK_OK;
}

spsyrk_status_t spsyrk_plan_map_bytes(spsyrk_plan_t plan, size_t* bytes) {
    if (!plan || !bytes) return SPSYRK_ERR_INVALID_ARG;
    *bytes = (size_t)map_items_total(plan) * sizeof(uint16_t);
    return SPSYRK_OK;
}

spsyrk_status_t spsyrk_plan_lend_map(spsyrk_plan_t plan, void* d_map, size_t bytes) {
    if (!plan || (d_map && reinterpret_cast<uintptr_t>(d_map) % ALIGN)) return SPSYRK_ERR_INVALID_ARG;
    plan->map = static_cast<uint16_t*>(d_map);
    plan->map_bytes = d_map ? bytes : 0;
    plan->map_filled = false;
    plan->have_symbolic = false;
    if (plan->upper) { plan->upper->map_filled = false; plan->upper->have_symbolic = false; }
    return SPSYRK_OK;
}

spsyrk_status_t spsyrk_plan_set_jaccard(spsyrk_plan_t plan, float* d_jaccard) {
    if (!plan) return SPSYRK_ERR_INVALID_ARG;
    if (d_jaccard && plan->dtype != SPSYRK_I32) return SPSYRK_ERR_INVALID_ARG;
    plan->dev.jaccard = d_jaccard;
    if (plan->upper) plan->upper->dev.jaccard = d_jaccard;
    return SPSYRK_OK;
}

spsyrk_status_t spsyrk_plan_stats(spsyrk_plan_t plan, int64_t* work_total, int64_t class_rows[8]) {
    if (!plan) return SPSYRK_ERR_INVALID_ARG;
    if (work_total) *work_total = plan->work_total + (plan->upper_active ? plan->upper->work_total : 0);
    if (class_rows)
        for (int c = 0; c < NCLASS; ++c) class_rows[c] = plan->class_start[c + 1] - plan->class_start[c];
    return SPSYRK_OK;
}

spsyrk_status_t spsyrk_plan_buffers(spsyrk_plan_t plan, const int64_t** d_colptr, const int32_t** d_at_row,
                                    const void** d_at_rec, const int64_t** d_work) {
    if (!plan) return SPSYRK_ERR_INVALID_ARG;
    if (d_colptr) *d_colptr = plan->dev.colptr;
    if (d_at_row) *d_at_row = plan->dev.at_row;
    if (d_at_rec) *d_at_rec = plan->dev.at_rec;
    if (d_work) *d_work = plan->upper_active ? plan->work_sum : plan->dev.work;
    return SPSYRK_OK;
}

void spsyrk_destroy(spsyrk_plan_t plan) {
    if (!plan) return;
    if (plan->timing)
        for (int i = 0; i <= NCLASS; ++i) { cudaEventDestroy(plan->ev_sym[i]); cudaEventDestroy(plan->ev_num[i]); }
    plan->host.release();
    delete plan->upper;
    delete plan;
}

spsyrk_status_t spsyrk_plan_enable_timing(spsyrk_plan_t plan) {
    if (!plan) return SPSYRK_ERR_INVALID_ARG;
    if (plan->timing) return SPSYRK_OK;
    for (int i = 0; i <= NCLASS; ++i) {
        SPSYRK_CUDA_TRY(cudaEventCreate(&plan->ev_sym[i]));
        SPSYRK_CUDA_TRY(cudaEventCreate(&plan->ev_num[i]));
    }
    plan->timing = true;
    return SPSYRK_OK;
}

spsyrk_status_t spsyrk_plan_timings(spsyrk_plan_t plan, float symbolic_ms[8], float numeric_ms[8]) {
    if (!plan || !plan->timing || !symbolic_ms || !numeric_ms) return SPSYRK_ERR_INVALID_ARG;
    if (!plan->have_symbolic) return SPSYRK_ERR_SEQUENCE;
    symbolic_ms[0] = numeric_ms[0] = 0.f;
    for (int c = 1; c < NCLASS; ++c) {
        symbolic_ms[c] = numeric_ms[c] = 0.f;
        SPSYRK_CUDA_TRY(cudaEventSynchronize(plan->ev_sym[c + 1]));
        SPSYRK_CUDA_TRY(cudaEventElapsedTime(&symbolic_ms[c], plan->ev_sym[c], plan->ev_sym[c + 1]));
        if (cudaEventQuery(plan->ev_num[c + 1]) == cudaSuccess && cudaEventQuery(plan->ev_num[c]) == cudaSuccess)
            cudaEventElapsedTime(&numeric_ms[c], plan->ev_num[c], plan->ev_num[c + 1]);
    }
    cudaGetLastError();
    return SPSYRK_OK;
}

int64_t spsyrk_launch_count(void) { return (int64_t)g_launches.load(std::memory_order_relaxed); }

const char* spsyrk_status_string(spsyrk_status_t s) {
    switch (s) {
        case SPSYRK_OK: return "ok";
        case SPSYRK_ERR_INVALID_ARG: return "invalid argument";
        case SPSYRK_ERR_BAD_CSR: return "input is not canonical CSR";
        case SPSYRK_ERR_WORKSPACE: return "workspace too small";
        case SPSYRK_ERR_OVERFLOW: return "size exceeds the supported range";
        case SPSYRK_ERR_SEQUENCE: return "call sequence error";
        case SPSYRK_ERR_CUDA: return "CUDA runtime error";
        case SPSYRK_ERR_INTERNAL: return "internal error";
        case SPSYRK_ERR_NOT_IMPLEMENTED: return "not implemented";
    }
    return "unknown status";
}

}  // extern "C"
