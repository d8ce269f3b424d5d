// Shared device utilities: warp/block scans, register bitonic sort, device-wide scan,
// stable class binning.  Header-only; included by every translation unit of libspsyrk.
#pragma once
#include <cuda_runtime.h>
#include <atomic>
#include <stdint.h>
#include <type_traits>

#include "../../include/spsyrk.h"
#include "errors.h"

namespace spsyrk {

constexpr unsigned FULL_MASK = 0xffffffffu;

// Bounds-checked build (-DSPSYRK_CHECKED, a second library next to the regular one): every index into a
// shared-memory accumulator, hash or landing slot and every output offset that the kernels compute is
// tested first; a violation sets ERRW_INTERNAL in the device error word and the access is skipped, so the
// caller gets SPSYRK_ERR_INTERNAL instead of a memory fault.  In the regular build the test is `true`.
#ifdef SPSYRK_CHECKED
#define SPSYRK_IN_RANGE(cond, errptr) ((cond) ? true : (atomicOr((errptr), ::spsyrk::ERRW_INTERNAL), false))
#else
#define SPSYRK_IN_RANGE(cond, errptr) true
#endif

constexpr int NCLASS = 8;  // row / column classes produced by the binning pass

// kernel-launch bookkeeping behind spsyrk_launch_count (defined in api.cu)
void note_launches(int n);

// Pinned host memory that kernels write the facts the host waits for into (class sizes, entry counts, the error word):
// one synchronisation and no copy, where a copy into ordinary memory took 3 us of device time and as much again
// on the host, up to five in a row.  Blocks of HOST_WORDS words come from a pool (defined in api.cu).
constexpr int HOST_WORDS = 160;
constexpr int HOST_GAVE_UP = HOST_WORDS - 1;  // set by a wait that ran out while the facts were being published; cleared by acquire
struct HostBlock {
    int64_t* host = nullptr;
    int64_t* dev = nullptr;  // the same memory as kernels see it
    cudaError_t acquire();
    void release();
    // the error word that a kernel has sent along; a tile that gave up may have set its bit after that
    uint32_t errors(int64_t word) const { return (uint32_t)word | (host[HOST_GAVE_UP] ? (uint32_t)ERRW_INTERNAL : 0u); }
};
struct ScopedHostBlock : HostBlock {
    ~ScopedHostBlock() { release(); }
};

#define SPSYRK_CUDA_TRY(expr)                                  \
    do {                                                       \
        cudaError_t _e = (expr);                               \
        if (_e != cudaSuccess) return SPSYRK_ERR_CUDA;         \
    } while (0)

// Lets a kernel take all the shared memory of an SM that its static arrays leave, once per device.  A kernel that is
// launched with several sizes must not have its limit set to each of them in turn: another thread's limit can come between.
template <auto Kernel>
inline cudaError_t allow_shared_memory() {
    static std::atomic<uint64_t> done{0};  // a bit per device
    int device = 0, most = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    const uint64_t bit = device < 64 ? uint64_t(1) << device : 0;
    if (done.load(std::memory_order_relaxed) & bit) return cudaSuccess;
    cudaFuncAttributes a{};
    e = cudaFuncGetAttributes(&a, Kernel);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)a.sharedSizeBytes);
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_relaxed);
    return e;
}

// Kernels that do not depend on one another (the row classes of a pass, the two views of the full-output mode) are launched as a
// chain (programmatic dependent launch): a kernel of the chain may start when every CTA of the one before has started,
// so that small launches run side by side and the tail of one is filled by the next.  A kernel calls chain_begin first;
// one thread of it waits at the end for the kernel before, so that the last kernel's end is the end of all of
// them, which is what the next ordinary launch waits for.  (Launched the ordinary way both calls do nothing.)
__device__ __forceinline__ void chain_begin() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_end(bool this_cta) {  // true in one CTA
    if (this_cta && threadIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void chain_end() { chain_end(blockIdx.x == 0); }

// Launches, and returns the first error that has not been reported: an earlier launch by <<< >>> of the same call says nothing by itself.
template <typename... Params>
[[nodiscard]] inline cudaError_t launch_kernel(const cudaLaunchConfig_t& cfg, void (*kern)(Params...), Params... params) {
    note_launches(1);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, params...), earlier = cudaGetLastError();
    return e != cudaSuccess ? e : earlier;
}

// Waits for the stream, and returns the error of a launch that has not been reported.
inline cudaError_t wait_for(cudaStream_t st) {
    const cudaError_t launched = cudaGetLastError(), e = cudaStreamSynchronize(st);
    return launched != cudaSuccess ? launched : e;
}

// A chain of kernels that do not depend on one another (see chain_begin).  With `overlap` off every launch is an ordinary one,
// and so is that of a kernel that fills the GPU for long (`brief` false): its CTAs would start one by one as those of the
// kernel before end, and a persistent grid that shares its rows out beforehand ends with the last of them.  (All launches
// overlapped: large Erdos-Renyi product and mirror 36.0 ms against 35.1, large power-law 35.7 against 34.6; the
// 8192-row power-law product takes 378 us with and 446 without overlap.)
struct Chain {
    cudaStream_t st;
    bool overlap;
    bool first = true;
    template <typename... Params, typename... Args>
    [[nodiscard]] cudaError_t launch(bool brief, void (*kern)(Params...), unsigned grid, int threads, size_t smem, Args... args) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(grid);
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute attr{};
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = overlap && brief && !first ? 1 : 0;
        first = false;
        return launch_kernel(cfg, kern, static_cast<Params>(args)...);
    }
};

// Kernels that follow one another step by step: the next one is launched (launch_linked) while the one before it runs, so that
// its launch is over when it may start, and calls link() before it looks at anything: it waits until the kernel before has
// ended and its results can be seen.  A launch behind another saves 1 us that way, of which the plan and the mirror of a
// small matrix have twenty.  Not for the first kernel of a chain, whose next ones do not wait at their start.
// The pointers through which the kernel reads what the one before wrote are handed to it: loads through pointers that are const
// and restrict count as loads of constants, which a compiler may move ahead of the wait.
template <typename... P>
__device__ __forceinline__ void link(P&... p) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    (..., [&] { asm volatile("" : "+l"(p)::"memory"); }());
}
template <typename... Params, typename... Args>
[[nodiscard]] inline cudaError_t launch_linked(void (*kern)(Params...), unsigned grid, int threads, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return launch_kernel(cfg, kern, static_cast<Params>(args)...);
}

__host__ __device__ constexpr int ilog2_ce(int v) { return v <= 1 ? 0 : 1 + ilog2_ce(v >> 1); }

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

template <typename T>
__device__ __forceinline__ T warp_inclusive_scan(T v) {
    const int lane = lane_id();
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T t = __shfl_up_sync(FULL_MASK, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

template <typename T>
__device__ __forceinline__ T warp_reduce_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL_MASK, v, o);
    return v;
}

// Exclusive scan over the threads of a CTA.  `scratch` holds 33 elements of T in shared memory.
// Returns the exclusive prefix of `v`; *total receives the CTA-wide sum.  Contains barriers.
template <typename T, int THREADS>
__device__ __forceinline__ T block_exclusive_scan(T v, T* scratch, T* total) {
    static_assert(THREADS % 32 == 0 && THREADS <= 1024, "bad CTA size");
    constexpr int NW = THREADS / 32;
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    T incl = warp_inclusive_scan(v);
    if (lane == 31) scratch[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        T s = lane < NW ? scratch[lane] : T(0);
        T si = warp_inclusive_scan(s);
        scratch[lane] = si - s;
        if (lane == 31) scratch[32] = si;
    }
    __syncthreads();
    T res = scratch[warp] + incl - v;
    *total = scratch[32];
    __syncthreads();
    return res;
}

// ---------------------------------------------------------------------------------------
// Bitonic sort of G*R keys held in registers by groups of G lanes (G = 8, 16 or 32), R keys per
// lane, ascending.  Element e of a group lives in lane (e / R) of the group, register e % R, so
// that compare-exchanges at a distance below R stay inside a lane and the others are one
// shuffle per register.  After the call lane l of a group holds sorted elements [l*R, l*R+R).
//
// Every compare-exchange is a plain min/max: merge levels whose direction depends on the
// register index are resolved at compile time, and levels whose direction depends on the lane
// run on complemented keys in the descending lanes (x -> ~x reverses the order), so that the
// whole level is an ascending merge.
// ---------------------------------------------------------------------------------------
template <typename K>
__device__ __forceinline__ K kmin(K a, K b) { return a < b ? a : b; }
template <typename K>
__device__ __forceinline__ K kmax(K a, K b) { return a < b ? b : a; }
template <>
__device__ __forceinline__ uint32_t kmin<uint32_t>(uint32_t a, uint32_t b) { return min(a, b); }
template <>
__device__ __forceinline__ uint32_t kmax<uint32_t>(uint32_t a, uint32_t b) { return max(a, b); }

// x -> ~x for every key when `flip`, else unchanged.  ~x = -x - 1, written as x * c + d with
// (c, d) = (-1, -1) or (1, 0): an integer multiply-add, which issues on the FMA pipe and leaves the
// ALU pipe (busy with the min/max of the network) alone.
template <typename K, int R>
__device__ __forceinline__ void flip_keys(K (&x)[R], bool flip) {
    const K c = flip ? ~K(0) : K(1);
    const K d = flip ? ~K(0) : K(0);
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = x[r] * c + d;
}

template <typename K, int R, int G = 32>
__device__ __forceinline__ void group_bitonic_sort(K (&x)[R]) {
    static_assert((R & (R - 1)) == 0 && (G & (G - 1)) == 0 && G <= 32, "powers of two");
    const int gl = lane_id() & (G - 1);
    bool flipped = false;
#pragma unroll
    for (int k = 2; k <= G * R; k <<= 1) {
        if (k >= R && k < G * R) {
            // direction of this level is per lane: descending lanes work on complemented keys
            const bool want = (gl & (k / R)) != 0;
            flip_keys<K, R>(x, want != flipped);
            flipped = want;
        } else if (k == G * R && G * R > R) {
            flip_keys<K, R>(x, flipped);
            flipped = false;
        }
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j < R) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int pr = r ^ j;
                    if (pr > r) {
                        // for k < R the direction depends on r only (compile time); otherwise ascending
                        const bool up = (k < R) ? ((r & k) == 0) : true;
                        const K lo = kmin(x[r], x[pr]), hi = kmax(x[r], x[pr]);
                        x[r] = up ? lo : hi;
                        x[pr] = up ? hi : lo;
                    }
                }
            } else {
                const int lj = j / R;
                const bool lower = (gl & lj) == 0;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const K other = __shfl_xor_sync(FULL_MASK, x[r], lj);
                    x[r] = lower ? kmin(x[r], other) : kmax(x[r], other);
                }
            }
        }
    }
}

// first position in a[0, len) whose value is >= key (a ascending)
__device__ __forceinline__ uint32_t lower_bound_i32(const int32_t* __restrict__ a, uint32_t len, int32_t key) {
    uint32_t lo = 0, hi = len;
    while (lo < hi) {
        uint32_t mid = (lo + hi) >> 1;
        if (a[mid] < key) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// ---------------------------------------------------------------------------------------
// Device-wide exclusive scan in one launch, by decoupled look-back (Merrill & Garland, "Single-pass
// Parallel Prefix Scan with Decoupled Look-back", 2016):
//   out(i, sum_{r<i} in(r)) for i in [0, n): out stores the prefix; out.total(sum) once at the end; out.gave_up() if a wait ran out.
// A CTA takes its tile's number from a counter, so a tile only ever waits for tiles that running CTAs
// hold; it publishes its own sum, adds up what the tiles before it have published and publishes its
// inclusive prefix.  A status word is value << 2 | kind, so value and kind arrive together.
// `state` needs scan_partials_count(n) 64-bit words; a single tile uses none of them.
// (Three launches - tile sums, their scan, the tiles again - before: 2.5 us of device time and as much
// host time each, ten scans per product and mirror, and the input read twice.)
// ---------------------------------------------------------------------------------------
constexpr int SCAN_THREADS = 256;
constexpr int scan_items(size_t value_bytes) { return value_bytes == 8 ? 8 : 16; }
constexpr int SCAN_MIN_TILE = SCAN_THREADS * 8;
constexpr unsigned long long SCAN_PARTIAL = 1, SCAN_PREFIX = 2;  // kinds of a status word (0: nothing yet)
constexpr int SCAN_WINDOW = 256;
constexpr int SPIN_LIMIT = 1 << 24;  // polls before a wait gives up with ERRW_INTERNAL

inline int64_t scan_partials_count(int64_t n) { return (n + SCAN_MIN_TILE - 1) / SCAN_MIN_TILE + 1; }

__device__ __forceinline__ unsigned long long ld_status(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_status(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Called by one whole warp: publishes the tile's sum and returns the sum of all tiles before it.  A wait that runs out sets
// ERRW_INTERNAL and calls gave_up(): a call that reads the word back returns SPSYRK_ERR_INTERNAL; after an asynchronous one (the
// mirror's fill) nobody reads it.  The prefix is too small then, so nothing is indexed out of range.
template <typename GaveUp>
__device__ __forceinline__ int64_t scan_look_back(unsigned long long* state, int64_t tile, int64_t sum, uint32_t* err, GaveUp gave_up) {
    const int lane = lane_id();
    if (tile == 0) {
        if (lane == 0) st_status(state, ((unsigned long long)sum << 2) | SCAN_PREFIX);
        return 0;
    }
    if (lane == 0) st_status(state + tile, ((unsigned long long)sum << 2) | SCAN_PARTIAL);
    // SCAN_WINDOW tiles per step: when all tiles in flight start together the first of them is a thousand tiles away, and
    // every step is a round trip to L2 (34 million counters: 0.4 ms with 32 tiles per step).
    int64_t before = 0;
    for (int64_t last = tile - 1;; last -= SCAN_WINDOW) {  // lane l looks at tiles last - l, last - 32 - l, ...
        unsigned long long v[SCAN_WINDOW / 32];
#pragma unroll
        for (int k = 0; k < SCAN_WINDOW / 32; ++k) {
            const int64_t t = last - 32 * k - lane;
            v[k] = t >= 0 ? ld_status(state + t) : SCAN_PREFIX;
        }
        bool done = false;
#pragma unroll
        for (int k = 0; k < SCAN_WINDOW / 32; ++k) {
            if (done) continue;  // (the same for all lanes)
            const int64_t t = last - 32 * k - lane;
            for (int polls = 0; __any_sync(FULL_MASK, (v[k] & 3u) == 0); ++polls) {
                if (polls == SPIN_LIMIT) {
                    if (lane == 0) {
                        if (err) atomicOr(err, ERRW_INTERNAL);
                        gave_up();
                    }
                    v[k] |= SCAN_PREFIX;
                    break;
                }
                if ((v[k] & 3u) == 0) v[k] = ld_status(state + t);
            }
            const unsigned full = __ballot_sync(FULL_MASK, (v[k] & 3u) == SCAN_PREFIX);
            const int stop = full ? __ffs(full) - 1 : 31;  // the nearest tile whose inclusive prefix is known ends the walk
            before += warp_reduce_sum<int64_t>(lane <= stop ? (int64_t)(v[k] >> 2) : 0);
            done = full != 0;
        }
        if (done) break;
    }
    if (lane == 0) st_status(state + tile, ((unsigned long long)(before + sum) << 2) | SCAN_PREFIX);
    return before;
}

// In::Value is what an element is held as.  The tile's sum is published before the prefixes inside the tile are computed, and
// those are computed as they are stored: 40 registers, six CTAs per SM (with 64-bit prefixes in registers two CTAs:
// 0.46 ms for 34 million counters, 0.9 ms more for the large Erdos-Renyi product and mirror).
template <typename In, typename Out>
static __global__ void __launch_bounds__(SCAN_THREADS, 6) scan_kernel(In in, int64_t n, Out out, unsigned long long* __restrict__ state,
                                                                      int64_t ntiles, uint32_t* __restrict__ err) {
    using Value = typename In::Value;
    constexpr int ITEMS = scan_items(sizeof(Value));
    __shared__ int64_t s_warp[SCAN_THREADS / 32];
    __shared__ int64_t s_before;
    __shared__ uint32_t s_tile;
    link();
    int64_t tile = 0;
    if (ntiles > 1) {
        if (threadIdx.x == 0) s_tile = atomicAdd(reinterpret_cast<uint32_t*>(state + ntiles), 1u);
        __syncthreads();
        tile = s_tile;
    }
    // a warp owns consecutive elements, 32 per step: loads and stores are whole lines
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const int64_t base = tile * (SCAN_THREADS * ITEMS) + warp * (32 * ITEMS) + lane;
    const int left = (int)min(max(n - base, (int64_t)0), (int64_t)(32 * ITEMS));
    Value v[ITEMS];
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) v[it] = it * 32 < left ? in(base + it * 32) : Value(0);
    int64_t s = 0;
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) s += (int64_t)v[it];
    s = warp_reduce_sum<int64_t>(s);
    if (lane == 0) s_warp[warp] = s;
    __syncthreads();
    int64_t run = 0, tot = 0;
#pragma unroll
    for (int w = 0; w < SCAN_THREADS / 32; ++w) {
        if (w < warp) run += s_warp[w];
        tot += s_warp[w];
    }
    if (ntiles > 1) {
        if (warp == 0) {
            const int64_t b = scan_look_back(state, tile, tot, err, [&] { out.gave_up(); });
            if (lane == 0) s_before = b;
        }
        __syncthreads();
        run += s_before;
        tot += s_before;
    }
    if (tile == ntiles - 1 && threadIdx.x == 0) out.total(tot);
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        const int64_t incl = warp_inclusive_scan<int64_t>((int64_t)v[it]);
        if (it * 32 < left) out(base + it * 32, run + incl - (int64_t)v[it]);
        run += __shfl_sync(FULL_MASK, incl, 31);
    }
}

// reads an array; stores the prefixes and, behind the last one, the total
template <typename T>
struct ScanArray {
    using Value = T;
    const T* p;
    __device__ __forceinline__ T operator()(int64_t i) const { return p[i]; }
};
struct ScanInto {
    int64_t* out;
    int64_t n;
    __device__ __forceinline__ void operator()(int64_t i, int64_t ex) const { out[i] = ex; }
    __device__ __forceinline__ void total(int64_t t) const { out[n] = t; }
    __device__ __forceinline__ void gave_up() const {}
};

// the same, and the total and the error word go to the host (words 0 and 1)
struct ScanIntoHost {
    int64_t* out;
    int64_t n;
    const uint32_t* err;
    int64_t* host;
    __device__ __forceinline__ void operator()(int64_t i, int64_t ex) const { out[i] = ex; }
    __device__ __forceinline__ void total(int64_t t) const {
        const int64_t e = (int64_t)*err;
        out[n] = t;
        host[0] = t;
        host[1] = e;
    }
    __device__ __forceinline__ void gave_up() const { host[HOST_GAVE_UP] = 1; }
};

// n >= 1.  The status words are cleared here unless the caller has done so (`cleared`).
template <typename In, typename Out>
inline cudaError_t scan_launch(In in, int64_t n, Out out, int64_t* partials, uint32_t* err, cudaStream_t st, bool cleared = false) {
    constexpr int64_t tile = SCAN_THREADS * scan_items(sizeof(typename In::Value));
    const int64_t ntiles = (n + tile - 1) / tile;
    unsigned long long* const state = reinterpret_cast<unsigned long long*>(partials);
    if (ntiles > 1 && !cleared) {  // (not behind another kernel then: an ordinary launch)
        const cudaError_t e = cudaMemsetAsync(partials, 0, (size_t)(ntiles + 1) * sizeof(int64_t), st);
        if (e != cudaSuccess) return e;
        scan_kernel<In, Out><<<(unsigned)ntiles, SCAN_THREADS, 0, st>>>(in, n, out, state, ntiles, err);
        note_launches(1);
        return cudaGetLastError();
    }
    return launch_linked(scan_kernel<In, Out>, (unsigned)ntiles, SCAN_THREADS, 0, st, in, n, out, state, ntiles, err);
}

// out[i] = sum_{r<i} in[r] for i in [0, n]: out has n + 1 entries and out[n] is the total
template <typename InT>
inline cudaError_t exclusive_scan_i64(const InT* in, int64_t n, int64_t* out, int64_t* partials, uint32_t* err, cudaStream_t st,
                                      bool cleared = false) {
    if (n <= 0) return cudaMemsetAsync(out, 0, sizeof(int64_t), st);
    return scan_launch(ScanArray<InT>{in}, n, ScanInto{out, n}, partials, err, st, cleared);
}

// Rows per CTA of the binning kernels: about four CTAs per SM for small inputs, at most BIN_MAX_TILE rows.
constexpr int BIN_THREADS = 256;
constexpr int BIN_MAX_TILE = 2048;
constexpr int BIN_FEW_BLOCKS = 148 * 4;
inline int64_t bin_tile(int64_t n) {
    const int64_t t = (n + BIN_FEW_BLOCKS - 1) / BIN_FEW_BLOCKS;
    return t >= BIN_MAX_TILE ? BIN_MAX_TILE : t <= 32 ? 32 : (t + 31) / 32 * 32;
}
inline int64_t bin_blocks(int64_t n) { return n > 0 ? (n + bin_tile(n) - 1) / bin_tile(n) : 0; }
inline int64_t bin_blocks_max(int64_t n) { return n / BIN_MAX_TILE + BIN_FEW_BLOCKS + 1; }  // over every number of rows up to n

// value-type traits: accumulator type and exact conversions
template <typename V> struct AccOf { using type = double; };
template <> struct AccOf<int32_t> { using type = int32_t; };

__device__ __forceinline__ double acc_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ int32_t acc_mul(int32_t a, int32_t b) { return (int32_t)((uint32_t)a * (uint32_t)b); }
__device__ __forceinline__ double acc_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ int32_t acc_add(int32_t a, int32_t b) { return (int32_t)((uint32_t)a + (uint32_t)b); }

}  // namespace spsyrk
