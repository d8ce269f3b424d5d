// Stable least-significant-digit radix partition passes over (key, payload a, payload b) records
// held as separate arrays.  A sparse transpose is a stable sort by column id: entries that arrive
// in ascending row order leave every column's segment in ascending row order, with no atomics and
// no per-segment sort, and every pass reads and writes memory in long runs.
//
// A pass is one launch (single-pass partition with decoupled look-back: Adinets & Merrill, "Onesweep", 2022): the
// sizes of all digits of all passes are known beforehand, a CTA takes its tile's number from a counter,
// ranks its elements, publishes the tile's count of every digit, drops the elements into their slots of the
// digit-major tile in shared memory, adds up what the tiles before it have published, one thread per digit, and
// writes the tile out in runs.  In the ranking a warp owns a contiguous slice of the tile, keeps its
// elements in registers and ranks them 32 at a time (elements with equal digits find each other through one
// warp vote per digit bit, the lowest lane bumps the warp's counter); an exclusive prefix over the
// warps makes the ranks tile-wide and stable.  A tile only waits for tiles that running CTAs hold.
// (Per-tile histograms and their device-wide scan before: three more launches per pass and the keys read twice.)
#pragma once
#include <algorithm>
#include <type_traits>

#include "common.cuh"

namespace spsyrk {

constexpr int RX_THREADS = 512;
constexpr int RX_WARPS = RX_THREADS / 32;
constexpr int RX_ITEMS = 8;
constexpr int RX_TILE = RX_THREADS * RX_ITEMS;  // elements per CTA
constexpr int RX_CHUNK = RX_TILE / RX_WARPS;    // contiguous elements per warp

inline int64_t radix_tiles(int64_t n) { return n > 0 ? (n + RX_TILE - 1) / RX_TILE : 0; }

constexpr int RX_BITS = 8;
constexpr int RX_BINS = 1 << RX_BITS;
constexpr int RX_MAX_PASSES = 4;
inline int radix_passes(uint64_t max_key);

// State of a sort, all zero at its start: sizes of the digits of every pass, a tile counter per pass, and per pass, tile
// and digit a word value << 2 | kind (see scan_look_back; 32-bit words while counts stay below 2^30).
struct RadixState {
    unsigned long long* bins;  // [passes][RX_BINS]
    uint32_t* tickets;         // [RX_MAX_PASSES]
    void* words;               // [passes][tiles][RX_BINS]
};
inline bool radix_wide(int64_t n) { return n >= (int64_t(1) << 30); }
inline size_t radix_state_words(int64_t tiles, bool wide, int passes) { return (size_t)passes * tiles * RX_BINS / (wide ? 1 : 2); }  // 64-bit words

__device__ __forceinline__ uint32_t ld_status(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_status(uint32_t* p, uint32_t v) { asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory"); }

// One thread per digit: the tile's count is published with radix_publish as soon as it is known; radix_look_back returns how
// many elements of the digit the tiles before hold and publishes the sum.
template <typename S, int BINS = RX_BINS>
__device__ __forceinline__ void radix_publish(S* words, int64_t tile, int digit, uint32_t count) {
    st_status(words + tile * BINS + digit, (S)(((S)count << 2) | (tile == 0 ? (S)SCAN_PREFIX : (S)SCAN_PARTIAL)));
}
template <typename S, int BINS = RX_BINS>
__device__ __forceinline__ int64_t radix_look_back(S* words, int64_t tile, int digit, uint32_t count, uint32_t* err) {
    if (tile == 0) return 0;
    constexpr int W = 8;  // tiles per round trip
    S before = 0;
    bool done = false;
    for (int64_t last = tile - 1; !done; last -= W) {
        S v[W];
#pragma unroll
        for (int k = 0; k < W; ++k) v[k] = last - k >= 0 ? ld_status(words + (last - k) * BINS + digit) : (S)SCAN_PREFIX;
#pragma unroll
        for (int k = 0; k < W; ++k) {
            if (done) continue;
            for (int polls = 0; (v[k] & 3) == 0; ++polls) {
                if (polls == SPIN_LIMIT) {  // as in scan_look_back: the sum is too small, nothing is indexed out of range
                    if (err) atomicOr(err, ERRW_INTERNAL);
                    v[k] = (S)SCAN_PREFIX;
                    break;
                }
                v[k] = ld_status(words + (last - k) * BINS + digit);
            }
            before += v[k] >> 2;
            done = (v[k] & 3) == (S)SCAN_PREFIX;
        }
    }
    st_status(words + tile * BINS + digit, (S)(((S)(before + count) << 2) | (S)SCAN_PREFIX));
    return (int64_t)before;
}

// Sizes of all digits of 32-bit keys: in[k] elements of key k (COUNTED), or the keys themselves.  also(x) is called with
// every non-zero count (every key).
struct RadixBinsOnly {
    __device__ __forceinline__ void operator()(uint32_t) const {}
};
template <bool COUNTED, typename Also>
static __global__ void __launch_bounds__(RX_THREADS) radix_bins_kernel(const uint32_t* __restrict__ in, int64_t n, int passes, unsigned long long* __restrict__ bins,
                                                                       Also also) {
    __shared__ uint32_t h[RX_MAX_PASSES][RX_BINS];
    link(in);
    for (int d = threadIdx.x; d < RX_MAX_PASSES * RX_BINS; d += RX_THREADS) (&h[0][0])[d] = 0;
    __syncthreads();
    // a CTA counts fewer than 2^32 elements: the sum of all weights of a matrix is below 2^31, and keys are one each
    const int64_t stride = (int64_t)gridDim.x * RX_THREADS;
    constexpr int UNR = 4;
    for (int64_t e = (int64_t)blockIdx.x * RX_THREADS + threadIdx.x; e < n; e += UNR * stride) {
        uint32_t v[UNR];
#pragma unroll
        for (int u = 0; u < UNR; ++u) v[u] = e + u * stride < n ? in[e + u * stride] : 0u;
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
            if (e + u * stride >= n || (COUNTED && v[u] == 0)) continue;
            const uint32_t key = COUNTED ? (uint32_t)(e + u * stride) : v[u];
            also(v[u]);
            for (int p = 0; p < passes; ++p) atomicAdd(&h[p][(key >> (p * RX_BITS)) & (RX_BINS - 1)], COUNTED ? v[u] : 1u);
        }
    }
    __syncthreads();
    for (int d = threadIdx.x; d < passes * RX_BINS; d += RX_THREADS)
        if ((&h[0][0])[d]) atomicAdd(&bins[d], (unsigned long long)(&h[0][0])[d]);
}
template <bool COUNTED, typename Also = RadixBinsOnly>
inline cudaError_t radix_bins(const uint32_t* in, int64_t n, int passes, unsigned long long* bins, cudaStream_t st, Also also = {}) {
    if (n <= 0) return cudaSuccess;
    const int64_t ctas = std::min<int64_t>((n + RX_THREADS * 4 - 1) / (RX_THREADS * 4), 148 * 4);
    return launch_linked(radix_bins_kernel<COUNTED, Also>, (unsigned)ctas, RX_THREADS, 0, st, in, n, passes, bins, also);
}

template <int BITS, typename PB, bool HAS_PC = false>
struct RadixSmem {
    static constexpr int NB = 1 << BITS;
    static size_t bytes() {
        return (size_t)NB * 8 + (size_t)RX_TILE * sizeof(PB) + (size_t)RX_TILE * (4 + 4 + (HAS_PC ? 4 : 0)) + (size_t)RX_WARPS * NB * 4 +
               (size_t)NB * 4;
    }
};

// Emits that want to see the keys before and after theirs in the tile's order (NO_KEY at its ends): where a key's run begins and ends
constexpr uint32_t NO_KEY = 0xffffffffu;
template <typename Emit, typename = void> struct EmitNeighbours : std::false_type {};
template <typename Emit> struct EmitNeighbours<Emit, std::void_t<decltype(Emit::NEIGHBOURS)>> : std::true_type {};

// `err` is the device error word of the caller: set by a look-back that gives up (and by the bounds-checked build).
// Emit(dest, key, pa, pb) is called once per element with its position `dest` in the order sorted
// by the digits seen so far.  pa == nullptr (pb == nullptr) means "this payload is the element's own
// index".
//
// A thread keeps its RX_ITEMS elements in registers (coalesced loads straight from global memory,
// the payloads still in flight while the keys are ranked), learns each element's slot in the tile's
// digit-major order, drops key and payloads into that slot of shared memory, and the tile is then
// read back slot by slot and written out in runs.
// HAS_PC: a third payload pc (32 bits; nullptr = the element's own index) travels along and the functor is
// called as emit(dest, key, pa, pb, pc).
// An element whose position is not in [0, n) is dropped: it takes keys that were not counted (a matrix that failed its
// checks, which the caller learns of later).  Then places of the output also stay unwritten, and what the next pass reads
// there is whatever the memory held: an emit that indexes by a payload tests it.
template <int BITS, typename PB, typename Emit, bool HAS_PC, typename S>
__global__ void __launch_bounds__(RX_THREADS, 2) radix_scatter_kernel(const uint32_t* __restrict__ keys, const uint32_t* __restrict__ pa,
                                                                      const PB* __restrict__ pb, const uint32_t* __restrict__ pc,
                                                                      int64_t n, int shift, const unsigned long long* __restrict__ bins,
                                                                      S* __restrict__ words, uint32_t* __restrict__ ticket, Emit emit, uint32_t* err) {
    constexpr int NB = 1 << BITS;
    static_assert(BITS <= 12, "digit width");
    extern __shared__ __align__(16) unsigned char rx_smem[];
    __shared__ uint32_t scratch[33];
    __shared__ int64_t scratch64[33];
    __shared__ uint32_t s_tile;
    int64_t* goff = reinterpret_cast<int64_t*>(rx_smem);               // [NB]
    PB* s_pb = reinterpret_cast<PB*>(goff + NB);                       // [TILE] sorted order
    uint32_t* s_key = reinterpret_cast<uint32_t*>(s_pb + RX_TILE);     // [TILE] sorted order
    uint32_t* s_pa = s_key + RX_TILE;                                  // [TILE] sorted order
    uint32_t* s_pc = s_pa + RX_TILE;                                   // [TILE] sorted order (HAS_PC only)
    uint32_t* wcount = s_pc + (HAS_PC ? RX_TILE : 0);                  // [WARPS][NB]
    uint32_t* bin_start = wcount + RX_WARPS * NB;                      // [NB]

    const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    static_assert(NB == RX_BINS && NB <= RX_THREADS, "one thread per digit");
    // (What is read of the elements lies where the ticket says, which is drawn behind this; with their pointers handed to link
    // they were no loads of constants any more and registers were spilled: a pass over 1.7e7 nonzeros took 250 us instead of 240.)
    link();
    if (tid == 0) s_tile = atomicAdd(ticket, 1u);
    __syncthreads();
    const int64_t tile = s_tile, tile_base = tile * RX_TILE;
    const int tile_n = (int)min((int64_t)RX_TILE, n - tile_base);
    uint32_t k[RX_ITEMS], a[RX_ITEMS];
    PB b[RX_ITEMS];
#pragma unroll
    for (int i = 0; i < RX_ITEMS; ++i) {
        const int t = warp * RX_CHUNK + i * 32 + lane;
        k[i] = t < tile_n ? keys[tile_base + t] : 0u;
    }
#pragma unroll
    for (int i = 0; i < RX_ITEMS; ++i) {
        const int t = warp * RX_CHUNK + i * 32 + lane;
        a[i] = (pa && t < tile_n) ? pa[tile_base + t] : (uint32_t)(tile_base + t);
        b[i] = (pb && t < tile_n) ? pb[tile_base + t] : (PB)(tile_base + t);
    }
    for (int d = tid; d < RX_WARPS * NB; d += RX_THREADS) wcount[d] = 0;
    __syncthreads();

    uint32_t rk[RX_ITEMS];
    uint32_t* mycount = wcount + warp * NB;
#pragma unroll
    for (int i = 0; i < RX_ITEMS; ++i) {
        const int t = warp * RX_CHUNK + i * 32 + lane;
        const bool valid = t < tile_n;
        const uint32_t d = valid ? ((k[i] >> shift) & (NB - 1)) : 0u;
        // lanes with the same digit, found one bit at a time with warp votes (cheaper here than the
        // match instruction, whose unit saturates long before memory does)
        unsigned peers = __ballot_sync(FULL_MASK, valid);
#pragma unroll
        for (int bit = 0; bit < BITS; ++bit) {
            const bool set = (d >> bit) & 1u;
            const unsigned bal = __ballot_sync(FULL_MASK, set);
            peers &= set ? bal : ~bal;
        }
        const int leader = __ffs(peers) - 1;
        uint32_t prev = 0;
        if (valid && lane == leader) {
            prev = mycount[d];
            mycount[d] = prev + __popc(peers);
        }
        prev = __shfl_sync(FULL_MASK, prev, leader);
        rk[i] = (prev + __popc(peers & ((1u << lane) - 1u))) | (d << 16);
        __syncwarp();
    }
    __syncthreads();
    // exclusive prefix over the warps per digit; the digit totals are published at once
    uint32_t total_d = 0;
    if (tid < NB) {
#pragma unroll
        for (int w = 0; w < RX_WARPS; ++w) {
            const uint32_t c = wcount[w * NB + tid];
            wcount[w * NB + tid] = total_d;
            total_d += c;
        }
        radix_publish<S>(words, tile, tid, total_d);
    }
    uint32_t tot;
    const uint32_t first_d = block_exclusive_scan<uint32_t, RX_THREADS>(total_d, scratch, &tot);
    if (tid < NB) bin_start[tid] = first_d;
    __syncthreads();
    // a warp's first slot of digit d = start of the digit + the elements of the warps before it
    for (int e = tid; e < RX_WARPS * NB; e += RX_THREADS) wcount[e] += bin_start[e & (NB - 1)];
    __syncthreads();
    // elements into their slots
#pragma unroll
    for (int i = 0; i < RX_ITEMS; ++i) {
        const int t = warp * RX_CHUNK + i * 32 + lane;
        if (t < tile_n) {
            const uint32_t q = mycount[rk[i] >> 16] + (rk[i] & 0xffffu);
            if (!SPSYRK_IN_RANGE(q < (uint32_t)RX_TILE, err)) continue;
            s_key[q] = k[i];
            s_pa[q] = a[i];
            s_pb[q] = b[i];
            // the third payload is loaded only now: it would not fit the registers next to the others
            if constexpr (HAS_PC) s_pc[q] = pc ? pc[tile_base + t] : (uint32_t)(tile_base + t);
        }
    }
    // slot q of digit d goes to (elements of smaller digits) + (of this digit in the tiles before) + q - first slot of d
    int64_t tot64;
    const int64_t base_d = block_exclusive_scan<int64_t, RX_THREADS>(tid < NB ? (int64_t)ld_status(bins + tid) : 0, scratch64, &tot64);  // (not before link: a load that stays where it is)
    if (tid < NB) goff[tid] = base_d + radix_look_back<S>(words, tile, tid, total_d, err) - (int64_t)first_d;
    __syncthreads();
    for (int q = tid; q < tile_n; q += RX_THREADS) {
        const uint32_t key = s_key[q];
        const int64_t dest = goff[(key >> shift) & (NB - 1)] + q;
        if (dest < 0 || dest >= n) continue;
        if constexpr (HAS_PC) {
            emit(dest, key, s_pa[q], s_pb[q], s_pc[q]);
        } else if constexpr (EmitNeighbours<Emit>::value) {
            emit(dest, key, s_pa[q], s_pb[q], q > 0 ? s_key[q - 1] : NO_KEY, q + 1 < tile_n ? s_key[q + 1] : NO_KEY);
        } else {
            emit(dest, key, s_pa[q], s_pb[q]);
        }
    }
}

template <typename PB>
struct EmitArrays {
    uint32_t* keys;
    uint32_t* pa;
    PB* pb;
    __device__ __forceinline__ void operator()(int64_t dest, uint32_t k, uint32_t a, PB b) const {
        keys[dest] = k;
        pa[dest] = a;
        pb[dest] = b;
    }
};

template <typename PB>
struct EmitArrays3 {
    uint32_t* keys;
    uint32_t* pa;
    PB* pb;
    uint32_t* pc;
    __device__ __forceinline__ void operator()(int64_t dest, uint32_t k, uint32_t a, PB b, uint32_t c) const {
        keys[dest] = k;
        pa[dest] = a;
        pb[dest] = b;
        pc[dest] = c;
    }
};

// pass `pass` of a sort whose state has been set up (zeroed, bins counted)
template <typename PB, bool HAS_PC, typename Emit, typename S>
inline cudaError_t radix_pass_launch(const uint32_t* keys, const uint32_t* pa, const PB* pb, const uint32_t* pc, int64_t n, int pass, const RadixState& rs,
                                     Emit emit, uint32_t* err, cudaStream_t st) {
    const int64_t nt = radix_tiles(n);
    auto kern = radix_scatter_kernel<RX_BITS, PB, Emit, HAS_PC, S>;
    const size_t smem = RadixSmem<RX_BITS, PB, HAS_PC>::bytes();
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_linked(kern, (unsigned)nt, RX_THREADS, smem, st, keys, pa, pb, pc, n, pass * RX_BITS, rs.bins + pass * RX_BINS,
                         static_cast<S*>(rs.words) + (size_t)pass * nt * RX_BINS, rs.tickets + pass, emit, err);
}
template <typename PB, bool HAS_PC, typename Emit>
inline cudaError_t radix_pass(const uint32_t* keys, const uint32_t* pa, const PB* pb, const uint32_t* pc, int64_t n, int pass, const RadixState& rs, Emit emit,
                              uint32_t* err, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    return radix_wide(n) ? radix_pass_launch<PB, HAS_PC, Emit, unsigned long long>(keys, pa, pb, pc, n, pass, rs, emit, err, st)
                         : radix_pass_launch<PB, HAS_PC, Emit, uint32_t>(keys, pa, pb, pc, n, pass, rs, emit, err, st);
}

inline int bits_for(uint64_t max_value) {
    int b = 1;
    while (b < 64 && (max_value >> b)) ++b;
    return b;
}

inline int radix_passes(uint64_t max_key) { return (bits_for(max_key) + RX_BITS - 1) / RX_BITS; }

}  // namespace spsyrk
