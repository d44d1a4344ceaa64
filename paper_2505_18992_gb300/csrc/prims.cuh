// Device-wide primitives: a single-pass exclusive scan and a stable LSD radix
// sort, both with decoupled look-back (Merrill & Garland, "Single-pass Parallel
// Prefix Scan with Decoupled Look-back", 2016; Adinets & Merrill, "Onesweep",
// 2022).  Logical block ids come from an atomic ticket, so a block only ever
// waits on blocks that started before it.  Every wait is bounded (LookBack's
// spin_limit, by default kSpinLimit); running out records VPGS_ERR_TIMEOUT and
// the kernel carries on with a partial prefix, whose scatter positions are
// still bounds-checked.
#pragma once

#include <type_traits>

#include "common.cuh"
#include "profiler.h"

namespace vpgs {

VPGS_D unsigned long long ld_volatile_u64(const unsigned long long *p) {
    return *reinterpret_cast<const volatile unsigned long long *>(p);
}
VPGS_D void st_volatile_u64(unsigned long long *p, unsigned long long v) {
    *reinterpret_cast<volatile unsigned long long *>(p) = v;
}
VPGS_D uint32_t ld_volatile_u32(const uint32_t *p) {
    return *reinterpret_cast<const volatile uint32_t *>(p);
}
VPGS_D void st_volatile_u32(uint32_t *p, uint32_t v) {
    *reinterpret_cast<volatile uint32_t *>(p) = v;
}
VPGS_D uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// ---------------------------------------------------------------------------
// exclusive scan of n uint32 values: out prefix handed to a store functor
//   Load:  __device__ uint32_t operator()(int64_t i) const         (i < n)
//   Store: __device__ void operator()(int64_t i, uint32_t excl, uint32_t v) const
// The scan total is written to *total (when total != nullptr).
// n = min(n_cap, *n_dev) if n_dev else n_cap.
// Status word layout (64 bit): [63:62] flag 1 = aggregate, 2 = inclusive prefix.
// ---------------------------------------------------------------------------
// How a look-back kernel waits: polls before it gives up (VPGS_ERR_TIMEOUT), and
// whether it returns at entry when the status word already holds an error (the
// render's binning chain, whose later kernels index with earlier outputs).
struct LookBack {
    int spin_limit = kSpinLimit;
    bool stop_on_error = false;
};

constexpr unsigned long long kFlagAgg = 1ull << 62;
constexpr unsigned long long kFlagPre = 2ull << 62;
constexpr unsigned long long kValMask = (1ull << 62) - 1;

template <class Load, class Store, int ITEMS>
__global__ void __launch_bounds__(kScanThreads)
scan_kernel(Load load, Store store, int64_t n_cap, const uint32_t *n_dev, uint32_t *ticket,
            unsigned long long *look, uint32_t *total, uint32_t *status, LookBack lb) {
    constexpr int kTile = kScanThreads * ITEMS;
    grid_dep_enter();
    // (as a block: another block of this launch may record a timeout meanwhile, and threads
    // that read the word apart would leave warps to work with what the absent ones never wrote)
    if (lb.stop_on_error && __syncthreads_or(*status != 0u)) return;
    __shared__ uint32_t s_items[kTile + kTile / 32];
    __shared__ uint32_t s_warp[kScanThreads / kWarp];
    __shared__ uint32_t s_bid, s_excl;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int64_t n = n_cap;
    if (n_dev) n = min(n, (int64_t)*n_dev);
    // tiles in ticket order until they run out (the grid is sized to what fits
    // on the GPU at once, not to the capacity)
    for (;;) {
    if (tid == 0) s_bid = atomicAdd(ticket, 1u);
    __syncthreads();
    const int64_t bid = s_bid;
    const int64_t base = bid * kTile;
    if (base >= n) {
        if (bid == 0 && tid == 0 && total) *total = 0;
        return;
    }
    // striped, coalesced loads into a padded shared tile
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        int idx = j * kScanThreads + tid;
        int64_t gi = base + idx;
        s_items[idx + (idx >> 5)] = gi < n ? load(gi) : 0u;
    }
    __syncthreads();
    // blocked: thread t owns items t*ITEMS .. t*ITEMS+ITEMS-1
    uint32_t v[ITEMS];
    uint32_t tsum = 0;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        int idx = tid * ITEMS + i;
        v[i] = s_items[idx + (idx >> 5)];
        tsum += v[i];
    }
    // block exclusive scan of the thread sums
    uint32_t x = tsum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < kScanThreads / kWarp ? s_warp[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < kScanThreads / kWarp) s_warp[lane] = w;  // inclusive warp totals
    }
    __syncthreads();
    const uint32_t block_agg = s_warp[kScanThreads / kWarp - 1];
    uint32_t texcl = x - tsum + (warp > 0 ? s_warp[warp - 1] : 0u);
    // decoupled look-back, one warp: 32 predecessors per step
    if (warp == 0) {
        unsigned long long excl = 0;
        if (bid == 0) {
            if (lane == 0) st_volatile_u64(look, kFlagPre | block_agg);
        } else {
            if (lane == 0) st_volatile_u64(look + bid, kFlagAgg | block_agg);
            int64_t j0 = bid - 1;
            for (;;) {
                const int64_t j = j0 - lane;
                unsigned long long w = j >= 0 ? ld_volatile_u64(look + j) : kFlagPre;
                int spins = 0;
                bool timed_out = false;
                while (!__all_sync(0xffffffffu, (w >> 62) != 0)) {
                    if (++spins > lb.spin_limit) {
                        timed_out = true;
                        break;
                    }
                    __nanosleep(64);
                    if ((w >> 62) == 0) w = ld_volatile_u64(look + j);
                }
                if (timed_out) {
                    if (lane == 0) set_status(status, VPGS_ERR_TIMEOUT);
                    break;
                }
                const uint32_t pre = __ballot_sync(0xffffffffu, (w >> 62) == 2);
                const int last = pre ? __ffs(pre) - 1 : 31;  // nearest inclusive prefix
                unsigned long long v = lane <= last ? (w & kValMask) : 0ull;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                excl += v;
                if (pre) break;
                j0 -= 32;
            }
            if (lane == 0) st_volatile_u64(look + bid, kFlagPre | (excl + block_agg));
        }
        if (lane == 0) {
            s_excl = (uint32_t)excl;
            if (base + kTile >= n && total) *total = (uint32_t)excl + block_agg;
        }
    }
    __syncthreads();
    uint32_t run = s_excl + texcl;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        int64_t gi = base + (int64_t)tid * ITEMS + i;
        if (gi < n) store(gi, run, v[i]);
        run += v[i];
    }
    __syncthreads();  // the next tile reuses the shared arrays
    }
}

// Blocks of a kernel that fit on the current GPU at once.
inline int resident_grid(const void *kernel, int threads, size_t smem, int64_t cap_blocks) {
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, smem) != cudaSuccess || occ < 1) occ = 1;
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t g = (int64_t)occ * std::max(sms, 1);
    return (int)std::max<int64_t>(1, std::min(g, cap_blocks));
}

inline int64_t scan_blocks(int64_t n) { return (n + kScanTile - 1) / kScanTile; }

// A ticket-loop grid: what is resident, or at most per_sm blocks per SM (per_sm
// > 0; for passes whose item count is usually far below its capacity, where
// blocks past the last tile only launch, take a ticket and leave).
int device_sm_count();
inline int grid_cap(int resident, int per_sm) {
    return per_sm > 0 ? std::max(1, std::min(resident, per_sm * device_sm_count())) : resident;
}

template <class Load, class Store, int ITEMS>
cudaError_t launch_scan_as(const char *name, Load load, Store store, int64_t n_cap, const uint32_t *n_dev,
                           uint32_t *ticket, unsigned long long *look, uint32_t *total, uint32_t *status,
                           cudaStream_t stream, LookBack lb, int per_sm) {
    const int64_t tile = (int64_t)kScanThreads * ITEMS;
    int64_t nb = (n_cap + tile - 1) / tile;
    if (nb == 0) nb = 1;
    static std::atomic<int> grid_cache[kDeviceCache];  // per <Load, Store, ITEMS> and device
    const int grid_res = per_device(grid_cache, [] {
        return resident_grid((const void *)scan_kernel<Load, Store, ITEMS>, kScanThreads, 0, int64_t(1) << 30);
    });
    const int grid = (int)std::min<int64_t>(grid_cap(grid_res, per_sm), nb);
    VPGS_LAUNCH(name, stream,
                launch_k(scan_kernel<Load, Store, ITEMS>, (unsigned)grid, kScanThreads, 0, stream, load, store, n_cap,
                         n_dev, ticket, look, total, status, lb));
    return cudaGetLastError();
}

// Launch a scan over at most n_cap items.  *ticket and the scan_blocks(n_cap)
// look-back words must be zero on entry (the render's prepare kernel clears them).
// wide: tiles of kScanItemsWide items per thread (fewer tiles in the look-back
// chain, for scans of many millions of items) instead of kScanItems.
template <class Load, class Store>
cudaError_t launch_scan(const char *name, Load load, Store store, int64_t n_cap, const uint32_t *n_dev,
                        uint32_t *ticket, unsigned long long *look, uint32_t *total,
                        uint32_t *status, cudaStream_t stream, LookBack lb = LookBack{}, int per_sm = 0,
                        bool wide = false) {
    if (wide)
        return launch_scan_as<Load, Store, kScanItemsWide>(name, load, store, n_cap, n_dev, ticket, look, total,
                                                           status, stream, lb, per_sm);
    return launch_scan_as<Load, Store, kScanItems>(name, load, store, n_cap, n_dev, ticket, look, total, status,
                                                   stream, lb, per_sm);
}

// ---------------------------------------------------------------------------
// Stable LSD radix sort of (uint32 key, uint32 value) pairs.
// One kernel computes the global histograms of every pass; then one kernel per
// pass ranks and scatters ("one sweep") with per-digit decoupled look-back.
// ---------------------------------------------------------------------------
struct SortPass {
    int shift, bits;
};

// Lanes of the warp holding the same digit: one ballot per digit bit (a lane
// keeps the lanes that agree with it on every bit), which is cheaper than the
// hardware match for digits of up to 8 bits.  Items past the end (valid =
// false) match only themselves.
VPGS_D uint32_t match_digit(uint32_t d, bool valid, int bits, int lane) {
    uint32_t m = __ballot_sync(0xffffffffu, valid);
    if (!valid) m = 1u << lane;
#pragma unroll
    for (int b = 0; b < kRadixBits + 1; ++b) {
        if (b >= bits) break;  // (the same for every thread of the grid)
        const uint32_t bit = (d >> b) & 1u;
        const uint32_t bb = __ballot_sync(0xffffffffu, bit != 0u);
        m &= bit ? bb : ~bb;
    }
    return m;
}

// predecessor tiles read per look-back step of a one-sweep pass
#ifndef VPGS_LOOK_DEPTH
#define VPGS_LOOK_DEPTH 8
#endif

// one-sweep look-back word: [31:30] flag (1 = block aggregate, 2 = inclusive
// prefix), [29:0] count
constexpr uint32_t kSFlagAgg = 1u << 30;
constexpr uint32_t kSFlagPre = 2u << 30;
constexpr uint32_t kSValMask = (1u << 30) - 1u;

// DPT: digits per thread (1: digits of up to 8 bits, 2: up to 9)
// Ranking in one round of votes (the count and the rank of a key come from the same
// match) and two blocks of 120 registers per SM, which keep a tile's loads in flight
// together.  Tile pass, old -> new: 1.19M keys 21.8 -> 18.6 us, 10.3M 118 -> 97 us; three
// blocks (80 registers) 22.9 / 92 us, four (spills) 26.6 / 98 us.
#ifndef VPGS_SORT_MINB
#define VPGS_SORT_MINB 2
#endif
template <int ITEMS, int DPT>
static __global__ void __launch_bounds__(kSortThreads, VPGS_SORT_MINB)
radix_onesweep_kernel(const uint32_t *__restrict__ key_in, const uint32_t *__restrict__ val_in,
                      uint32_t *__restrict__ key_out, uint32_t *__restrict__ val_out,
                      int64_t n_cap, const uint32_t *n_dev, SortPass pass,
                      const uint32_t *__restrict__ pass_hist, uint32_t *ticket, uint32_t *look,
                      uint32_t *next_look, uint32_t *status, LookBack lb) {
    grid_dep_enter();
    if (lb.stop_on_error && __syncthreads_or(*status != 0u)) return;  // (as a block: see scan_kernel)
    constexpr int kWarps = kSortThreads / kWarp;
    constexpr int kSeg = kWarp * ITEMS;  // contiguous items per warp
    constexpr int kTile = kSortThreads * ITEMS;
    constexpr int kDigits = kRadix * DPT;
    static_assert(kSortThreads == kRadix, "a thread takes DPT consecutive digits");
    // (16-bit counts, a tile holds at most 4,096 keys, keep 512 digits within 48 KB)
    using Count = typename std::conditional<DPT == 1, uint32_t, uint16_t>::type;
    static_assert(DPT == 1 || kTile < 65536, "a tile's counts fit 16 bits");
    __shared__ Count s_cnt[kWarps][kDigits];
    __shared__ uint32_t s_glob[kRadix];
    __shared__ uint32_t s_dstart[kDigits], s_gbase[kDigits], s_wsum[kWarps];
    __shared__ uint32_t s_key[kTile], s_val[kTile];
    __shared__ uint32_t s_bid;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int64_t n = n_cap;
    if (n_dev) n = min(n, (int64_t)*n_dev);
    if (n == 0) return;
    const uint32_t mask = (1u << pass.bits) - 1u;

    // global exclusive digit offsets of this pass (every block recomputes them)
    uint32_t glob_excl[DPT], hist_sum = 0;
#pragma unroll
    for (int e = 0; e < DPT; ++e) {
        glob_excl[e] = hist_sum;
        hist_sum += pass_hist[tid * DPT + e];
    }
    {
        // inclusive scan of the threads' sums in two levels of warps
        uint32_t x = hist_sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        s_glob[tid] = x;  // inclusive within warp
        __syncthreads();
        uint32_t add = x - hist_sum;
        for (int w = 0; w < warp; ++w) add += s_glob[w * 32 + 31];
#pragma unroll
        for (int e = 0; e < DPT; ++e) glob_excl[e] += add;
    }

    // tiles in ticket order until they run out (the grid is sized to what fits
    // on the GPU at once; a tile only waits on lower tickets, held by running blocks)
    for (;;) {
    if (tid == 0) s_bid = atomicAdd(ticket, 1u);
    for (int i = tid; i < kWarps * kDigits; i += kSortThreads) (&s_cnt[0][0])[i] = 0;
    __syncthreads();
    const int64_t bid = s_bid;
    const int64_t base = bid * (int64_t)(kSortThreads * ITEMS);
    if (base >= n) return;

    // load this warp's contiguous segment, 32 consecutive keys per step
    uint32_t k[ITEMS], v[ITEMS], rk[(ITEMS + 1) / 2];
    const int64_t seg = base + (int64_t)warp * kSeg;
    const int mine = (int)min((int64_t)ITEMS, max((int64_t)0, (n - seg - lane + kWarp - 1) / kWarp));  // this lane's keys
#pragma unroll
    for (int s = 0; s < ITEMS; ++s) {
        const int64_t i = seg + s * kWarp + lane;
        k[s] = s < mine ? key_in[i] : 0u;
        v[s] = s < mine ? val_in[i] : 0u;
    }
    // each key's rank among the warp's earlier keys of its digit (16 bits: a segment has at
    // most 1,024 keys), and with it the warp's digit counts
#pragma unroll
    for (int s = 0; s < ITEMS; ++s) {
        const uint32_t d = (k[s] >> pass.shift) & mask;
        const uint32_t m = match_digit(d, s < mine, pass.bits, lane);
        const uint32_t before = s < mine ? s_cnt[warp][d] : 0u;
        __syncwarp();
        if (s < mine && (m & lanemask_lt()) == 0) s_cnt[warp][d] = (Count)(before + __popc(m));
        const uint32_t rank = before + __popc(m & lanemask_lt());
        if (s & 1) rk[s / 2] |= rank << 16;
        else rk[s / 2] = rank;
        __syncwarp();
    }
    __syncthreads();
    // block count per digit and its block-local exclusive start
    uint32_t c[DPT], csum = 0;
#pragma unroll
    for (int e = 0; e < DPT; ++e) {
        c[e] = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) c[e] += s_cnt[w][tid * DPT + e];
        csum += c[e];
    }
    {
        uint32_t x = csum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_wsum[warp] = x;
        __syncthreads();
        uint32_t add = x - csum;
        for (int w = 0; w < warp; ++w) add += s_wsum[w];
#pragma unroll
        for (int e = 0; e < DPT; ++e) {
            s_dstart[tid * DPT + e] = add;
            add += c[e];
        }
    }
    // publish, look back over earlier blocks
#pragma unroll
    for (int e = 0; e < DPT; ++e)
        st_volatile_u32(look + bid * kDigits + tid * DPT + e, (bid == 0 ? kSFlagPre : kSFlagAgg) | c[e]);
#pragma unroll
    for (int e = 0; e < DPT; ++e) {
        const int dg = tid * DPT + e;
        uint32_t excl = 0;
        if (bid > 0) {
            // kLookDepth independent loads per step shorten the dependent chain
            constexpr int kLookDepth = VPGS_LOOK_DEPTH;
            int64_t j0 = bid - 1;
            bool done = false;
            while (!done) {
                uint32_t w[kLookDepth];
#pragma unroll
                for (int i = 0; i < kLookDepth; ++i) {
                    const int64_t j = j0 - i;
                    w[i] = j >= 0 ? ld_volatile_u32(look + j * kDigits + dg) : kSFlagPre;
                }
#pragma unroll
                for (int i = 0; i < kLookDepth; ++i) {
                    if (done) break;
                    const int64_t j = j0 - i;
                    uint32_t x = w[i];
                    int spins = 0;
                    while ((x >> 30) == 0) {
                        if (++spins > lb.spin_limit) {
                            set_status(status, VPGS_ERR_TIMEOUT);
                            x = kSFlagPre;
                            break;
                        }
                        __nanosleep(32);
                        x = ld_volatile_u32(look + j * kDigits + dg);
                    }
                    excl += x & kSValMask;
                    if ((x >> 30) == 2) done = true;
                }
                j0 -= kLookDepth;
            }
            st_volatile_u32(look + bid * kDigits + dg, kSFlagPre | (excl + c[e]));
        }
        s_gbase[dg] = glob_excl[e] + excl;  // global slot of this block's first key with this digit
        // per-warp bases inside the block (block-local digit order)
        uint32_t run = s_dstart[dg];
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const uint32_t t = s_cnt[w][dg];
            s_cnt[w][dg] = (Count)run;
            run += t;
        }
    }
    __syncthreads();
    // into shared memory in digit order (stable: ranks follow the input order)
#pragma unroll
    for (int s = 0; s < ITEMS; ++s) {
        if (s < mine) {
            const uint32_t lp = s_cnt[warp][(k[s] >> pass.shift) & mask] + (rk[s / 2] >> (16 * (s & 1)) & 0xffffu);
            s_key[lp] = k[s];
            s_val[lp] = v[s];
        }
    }
    __syncthreads();
    // coalesced write-out: consecutive threads write consecutive slots of each digit run
    const int nb = (int)min((int64_t)kTile, n - base);
    for (int i = tid; i < nb; i += kSortThreads) {
        const uint32_t key = s_key[i];
        const uint32_t dg = (key >> pass.shift) & mask;
        const uint32_t pos = s_gbase[dg] + ((uint32_t)i - s_dstart[dg]);
        if ((int64_t)pos < n) {  // always true unless a look-back wait timed out
            key_out[pos] = key;
            val_out[pos] = s_val[i];
        }
    }
    if (next_look) {  // the next pass starts from zero
#pragma unroll
        for (int e = 0; e < DPT; ++e) next_look[bid * kDigits + tid * DPT + e] = 0u;
    }
    __syncthreads();  // the next tile reuses the shared arrays
    }
}

// Digits per thread of a sort over `bits` key bits: 2 for 9 bits (257 to 512 tiles), one
// pass of 9-bit digits instead of two passes, else 1.  A pass costs 7-13 us however few
// its keys, and one pass of 512 digits takes the look-back words of two of 256.  Forwards
// by one pass / by two (us): 20k small Gaussians 272 tiles 74 / 79, 512 tiles 85 / 90; 100k
// of a room 92 / 99 and 84 / 89; 400k 188 / 193 and 143 / 144.
inline int sort_dpt(int bits) { return bits == kRadixBits + 1 ? 2 : 1; }

// Split `bits` low key bits starting at `lo` into balanced passes of <= 8 (9: sort_dpt) bits.
inline int plan_passes(int lo, int bits, SortPass *out) {
    const int most = kRadixBits + (sort_dpt(bits) == 2 ? 1 : 0);
    int np = (bits + most - 1) / most;
    if (np == 0) return 0;
    int base = bits / np, extra = bits % np, s = lo;
    for (int p = 0; p < np; ++p) {
        int b = base + (p < extra ? 1 : 0);
        out[p] = {s, b};
        s += b;
    }
    return np;
}

inline int64_t sort_blocks(int64_t n, int items) {
    const int64_t tile = (int64_t)kSortThreads * items;
    return (n + tile - 1) / tile;
}

// Sort n (<= n_cap, or *n_dev) pairs from (k0, v0) using (k1, v1) as the other
// buffer.  Returns in *result_in_1 whether the sorted data ended in buffer 1.
// On entry (the producers of the keys and the render's prepare kernel see to it):
//   hist   [passes][256 * sort_dpt(bits)] global digit histograms of the n keys;
//   ticket [passes] zero;
//   look   [passes][sort_blocks(n_cap)][256 * sort_dpt(bits)], pass 0's words zero for the tiles
//          that hold keys (each pass clears the next pass's words of its tiles).
// ITEMS: keys per thread; NINE: whether `bits` may be 9 (the form of 9-bit digits exists).
template <int ITEMS, bool NINE>
inline cudaError_t radix_sort_pairs(const char *name, uint32_t *k0, uint32_t *v0, uint32_t *k1, uint32_t *v1,
                                    int64_t n_cap, const uint32_t *n_dev, int lo_bit, int bits,
                                    const uint32_t *hist, uint32_t *ticket, uint32_t *look,
                                    uint32_t *status, cudaStream_t stream, bool *result_in_1,
                                    LookBack lb = LookBack{}, int per_sm = 0) {
    SortPass ps[kMaxSortPasses];
    int np = plan_passes(lo_bit, bits, ps);
    *result_in_1 = (np & 1) != 0;
    if (np == 0 || n_cap == 0) return cudaSuccess;
    if (np > 4) return cudaErrorInvalidValue;
    const int dpt = sort_dpt(bits);
    static_assert(ITEMS == 4 || ITEMS == 8 || ITEMS == 16 || ITEMS == 32, "keys per thread of a radix pass");
    if (dpt == 2 && !NINE) return cudaErrorInvalidValue;
    const int64_t nb = sort_blocks(n_cap, ITEMS);
    const auto kern = dpt == 2 ? radix_onesweep_kernel<ITEMS, NINE ? 2 : 1> : radix_onesweep_kernel<ITEMS, 1>;
    static std::atomic<int> grids[2][kDeviceCache];  // per instance, by digit width and device
    const int grid_res = per_device(grids[dpt - 1], [kern] {
        return resident_grid((const void *)kern, kSortThreads, 0, int64_t(1) << 30);
    });
    const unsigned grid = (unsigned)std::min<int64_t>(grid_cap(grid_res, per_sm), nb);
    cudaError_t e;
    uint32_t *ki = k0, *vi = v0, *ko = k1, *vo = v1;
    for (int p = 0; p < np; ++p) {
        uint32_t *lk = look + (size_t)p * nb * kRadix * dpt;
        uint32_t *nl = p + 1 < np ? lk + (size_t)nb * kRadix * dpt : nullptr;
        const uint32_t *h = hist + p * kRadix * dpt;
        VPGS_LAUNCH(name, stream, launch_k(kern, grid, kSortThreads, 0, stream, ki, vi, ko, vo, n_cap, n_dev, ps[p], h,
                                           ticket + p, lk, nl, status, lb));
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        uint32_t *tk = ki, *tv = vi;
        ki = ko; vi = vo; ko = tk; vo = tv;
    }
    return cudaSuccess;
}

// Adds the digits of key k to block-shared histograms of every pass (s_h [passes][256 * dpt]).
VPGS_D void add_digits(uint32_t *s_h, const SortPass *ps, int np, uint32_t k, int dpt = 1) {
    for (int p = 0; p < np; ++p)
        atomicAdd(&s_h[p * kRadix * dpt + ((k >> ps[p].shift) & ((1u << ps[p].bits) - 1u))], 1u);
}

// Adds block-shared histograms into the global ones (non-zero bins only).
VPGS_D void flush_digits(const uint32_t *s_h, int n_bins, uint32_t *hist) {
    for (int i = threadIdx.x; i < n_bins; i += blockDim.x) {
        const uint32_t c = s_h[i];
        if (c) atomicAdd(hist + i, c);
    }
}

}  // namespace vpgs
