// Tile binning: which Gaussians touch which tile, in depth order.
//
//   1. scan of the visibility flags (tile count > 0) -> compacted (z bits, id)
//   2. stable radix sort of the visible pairs by the FP32 bit pattern of the
//      camera depth (positive floats order like their bits); ties keep index
//      order, i.e. (view, Gaussian) order
//   3. scan of the tile counts in depth order, then a block-cooperative emit
//      of each Gaussian's (global tile id, id) instances at its offset; the
//      tiles are those of the row-wise tile cover counted by the projection
//   4. stable radix sort of the instances by global tile id (only the bits a
//      tile id needs); instances stay in depth order inside each tile
//   5. [start, end) of every tile from the sorted keys
//   6. the compositing launch order: tiles by descending instance count
//
// Sorting the visible Gaussians once by depth and then the instances by tile
// id only moves 32-bit depth keys over N_visible items and a 12-14 bit tile key
// over the instances, instead of a 44+ bit (tile, depth) key over all instances.
#include "internal.h"
#include "prims.cuh"
#include "profiler.h"

namespace vpgs {

struct VisLoad {
    const uint32_t *tcount;
    __device__ uint32_t operator()(int64_t i) const { return tcount[i] > 0u ? 1u : 0u; }
};

struct VisStore {
    const Rec *rec;
    uint32_t *dkey, *dval, *vis_idx;
    int64_t cap;
    __device__ void operator()(int64_t i, uint32_t pos, uint32_t v) const {
        if (v && (int64_t)pos < cap) {
            dkey[pos] = __float_as_uint(rec[i].r2.y);  // camera z > near_z > 0
            dval[pos] = (uint32_t)i;
            vis_idx[pos] = (uint32_t)i;  // kept in index order (the sort reuses dval)
        }
    }
};

struct CountLoad {
    const uint32_t *tcount, *dval;
    __device__ uint32_t operator()(int64_t r) const { return tcount[dval[r]]; }
};

struct OffsetStore {
    uint32_t *inst_off;
    __device__ void operator()(int64_t r, uint32_t off, uint32_t) const { inst_off[r] = off; }
};

// Small calls.  Their binning is bound by the latency of its launches (7-15 us each by
// events, whatever they move), so the ten general ones become two that do more work:
//
// small_rank: compaction, depth sort and instance offsets.  The projection appends its
// visible pairs to a list in any order, and this kernel compares each with all of
// them: the pairs before it in (depth, index) order give its rank and its first
// instance; a bit per visible pair gives its place in index order.
//
// small_lists: a block per tile tests every visible pair, in depth order, against its
// tile and writes the tile's list, instead of emission, tile sort and tile ranges.  The
// lists lie in ws.ival in any order of tiles.
//
// Both are bound by the latency of their few loads and barriers below a few thousand
// pairs, then by their comparisons (bin_form says where they end).  Measured, general ->
// small: forward of 300 Gaussians in three 97x61 views 66 -> 30 us, tracking iteration
// of 10k Gaussians (5.3k visible) at 320x240 166 -> 101 us.
// The results are those of the general path.
constexpr int kRankThreads = 256;
constexpr int kRankOwn = 16;    // pairs a block ranks at a time; its half warps take alternate list entries
constexpr int kRankTile = 2048; // list entries staged at a time
constexpr int kRankWords = (int)(kSmallPairs / 32);
// kLists: for small_lists, each pair's tile rectangle (four bytes: first and last column
// and row) and (pair, view) by rank; else the pair and its first instance by rank
template <bool kLists>
__global__ void __launch_bounds__(kRankThreads)
small_rank_kernel(SmallList list, const uint32_t *__restrict__ tcount, const BinRec *__restrict__ bin, int n_pairs,
                  int N, uint32_t *__restrict__ vis_idx, uint32_t *__restrict__ by_rank_id,
                  uint32_t *__restrict__ by_rank, const uint32_t *n_vis, const uint32_t *status) {
    grid_dep_enter();
    if (*status != 0u) return;
    __shared__ __align__(16) unsigned long long s_e[kRankTile];  // depth key, pair index
    __shared__ __align__(8) uint32_t s_c[kLists ? 2 : kRankTile];  // tile count
    __shared__ uint32_t s_seen[kRankWords];                      // a bit per visible pair
    __shared__ uint32_t s_sum[3][kRankOwn];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = (int)*n_vis, own = lane & (kRankOwn - 1);
    if ((int)blockIdx.x * kRankOwn >= n) return;
    const int part = warp * 2 + (lane >> 4);  // this half warp's list entries: 2 part, 2 part + 1 of every kStep
    constexpr int kStep = 2 * kRankThreads / kRankOwn;
    constexpr int kUnroll = 8;
    // (loads in batches: a block's few warps do not hide the latency of one at a time)
    constexpr int kBatch = 8;
    for (int i0 = tid; i0 - lane < n_pairs; i0 += kBatch * kRankThreads) {  // warp-uniform
        uint32_t c[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const int i = i0 + u * kRankThreads;
            c[u] = i < n_pairs ? tcount[i] : 0u;
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const uint32_t m = __ballot_sync(0xffffffffu, c[u] > 0u);
            const int w = (i0 + u * kRankThreads) >> 5;
            if (lane == 0 && w < kRankWords) s_seen[w] = m;
        }
    }
    for (int i0 = (int)blockIdx.x * kRankOwn; i0 < n; i0 += (int)gridDim.x * kRankOwn) {  // block-uniform
        const int i = min(i0 + own, n - 1);
        const uint32_t id = list.pair[i];
        const unsigned long long me = (unsigned long long)list.key[i] << 32 | id;
        if (tid < 3 * kRankOwn) (&s_sum[0][0])[tid] = 0u;
        uint32_t rank = 0u, off = 0u, place = 0u;
        for (int t0 = 0; t0 < n; t0 += kRankTile) {
            // the tile, padded with entries that are before none
            const int nt = min(kRankTile, n - t0);
            const int np = (nt + kUnroll * kStep - 1) / (kUnroll * kStep) * (kUnroll * kStep);
            __syncthreads();
            {
                constexpr int kPer = kRankTile / kRankThreads;
                uint32_t ek[kPer], ep[kPer], ec[kPer];
#pragma unroll
                for (int u = 0; u < kPer; ++u) {
                    const int k = tid + u * kRankThreads;
                    const bool in = k < nt;
                    ek[u] = in ? list.key[t0 + k] : 0xffffffffu;
                    ep[u] = in ? list.pair[t0 + k] : 0xffffffffu;
                    if constexpr (!kLists) ec[u] = in ? list.cnt[t0 + k] : 0u;
                }
#pragma unroll
                for (int u = 0; u < kPer; ++u) {
                    const int k = tid + u * kRankThreads;
                    s_e[k] = (unsigned long long)ek[u] << 32 | ep[u];
                    if constexpr (!kLists) s_c[k] = ec[u];
                }
            }
            __syncthreads();
            for (int k = 2 * part; k < np; k += kUnroll * kStep) {
#pragma unroll
                for (int u = 0; u < kUnroll; ++u) {
                    const ulonglong2 e = *reinterpret_cast<const ulonglong2 *>(&s_e[k + u * kStep]);
                    rank += e.x < me;
                    rank += e.y < me;
                    if constexpr (!kLists) {
                        const uint2 c = *reinterpret_cast<const uint2 *>(&s_c[k + u * kStep]);
                        if (e.x < me) off += c.x;
                        if (e.y < me) off += c.y;
                    }
                }
            }
        }
        for (int w = part; w <= (int)(id >> 5); w += kStep / 2) {
            const uint32_t bits = s_seen[w];
            place += __popc(w < (int)(id >> 5) ? bits : bits & ((1u << (id & 31u)) - 1u));
        }
        atomicAdd(&s_sum[0][own], rank);
        if constexpr (!kLists) atomicAdd(&s_sum[1][own], off);
        atomicAdd(&s_sum[2][own], place);
        __syncthreads();
        if (tid < kRankOwn && i0 + tid < n) {
            const uint32_t r = s_sum[0][tid];
            vis_idx[s_sum[2][tid]] = id;
            if constexpr (kLists) {
                const uint2 rc = bin[id].rect;
                by_rank_id[r] = id | (id / (uint32_t)N) << 16;
                by_rank[r] = (rc.x & 0xffu) | (rc.x >> 16 & 0xffu) << 8 | (rc.y & 0xffu) << 16 | (rc.y >> 16 & 0xffu) << 24;
            } else {
                by_rank_id[r] = id;
                by_rank[r] = s_sum[1][tid];
            }
        }
        __syncthreads();
    }
}

constexpr int kListThreads = 256;
constexpr int kListWarps = kListThreads / 32;

__global__ void __launch_bounds__(kListThreads)
small_lists_kernel(const uint32_t *__restrict__ by_rank_id, const uint32_t *__restrict__ by_rank,
                   const BinRec *__restrict__ bin, const uint32_t *n_vis, const uint32_t *n_inst, int64_t M_cap,
                   CamParams cam, uint2 *__restrict__ ranges, uint32_t *__restrict__ ival, uint32_t *cursor,
                   uint32_t *status) {
    grid_dep_enter();
    if (__syncthreads_or(*status != 0u)) return;  // (this launch writes *status: see emit_kernel)
    if ((int64_t)*n_inst > M_cap) {
        if (threadIdx.x == 0) set_status(status, VPGS_ERR_CAPACITY);
        return;
    }
    __shared__ uint16_t s_cand[kSmallPairs + kListThreads];
    __shared__ uint32_t s_n[kListWarps], s_start;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t below = lanemask_lt();
    const int tile = (int)blockIdx.x;
    const uint32_t view = (uint32_t)(tile / cam.T);
    const int lt = tile - (int)view * cam.T, ty = lt / cam.tiles_x, tx = lt - ty * cam.tiles_x;
    // the warp's share of the depth order: consecutive ranks
    const int n = (int)*n_vis, share = (n + kListThreads - 1) / kListThreads * 32;
    const int first = warp * share, last = min(n, first + share);
    uint16_t *cand = s_cand + first;
    uint32_t c = 0u;  // candidates: pairs whose tile rectangle holds this tile
    constexpr int kBatch = 8;  // (loads in batches, as above)
    for (int r0 = first; r0 < last; r0 += 32 * kBatch) {
        uint32_t rc[kBatch], iv[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const int r = r0 + 32 * u + lane;
            rc[u] = r < last ? by_rank[r] : 0x00ff00ffu;  // (no column, no row)
            iv[u] = r < last ? by_rank_id[r] : 0u;
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const bool in = iv[u] >> 16 == view && tx >= (int)(rc[u] & 0xffu) && tx <= (int)(rc[u] >> 8 & 0xffu) &&
                            ty >= (int)(rc[u] >> 16 & 0xffu) && ty <= (int)(rc[u] >> 24);
            const uint32_t m = __ballot_sync(0xffffffffu, in);
            if (in) cand[c + __popc(m & below)] = (uint16_t)iv[u];
            c += __popc(m);
        }
    }
    __syncwarp();
    // those whose span of this tile row holds the tile, in place
    uint32_t hits = 0u;
    for (uint32_t k0 = 0u; k0 < c; k0 += 32u) {
        const bool live = k0 + lane < c;
        const uint32_t id = live ? cand[k0 + lane] : 0u;
        bool in = false;
        if (live) {
            const BinRec &b = bin[id];
            const uint2 rc = b.rect;
            const int ty_lo = (int)(rc.y & 0xffffu), rows = (int)(rc.y >> 16) - ty_lo + 1;
            if (rows <= kCoverRows) {
                const uint32_t pk = reinterpret_cast<const uint32_t *>(&b.cv)[ty - ty_lo];
                in = tx >= (int)(pk & 0xffffu) && tx <= (int)(pk >> 16);
            } else {
                const Cover cv = b.cv;
                const float4 uv = b.uv;
                const int2 sp = cover_row(cv, uv.x, uv.z, uv.y, uv.w, ty, (int)(rc.x & 0xffffu), (int)(rc.x >> 16),
                                          cam.tw_shift, cam.tile_h, cam.W, cam.H);
                in = tx >= sp.x && tx <= sp.y;
            }
        }
        const uint32_t m = __ballot_sync(0xffffffffu, in);
        if (in) cand[hits + __popc(m & below)] = (uint16_t)id;
        hits += __popc(m);
        __syncwarp();
    }
    if (lane == 0) s_n[warp] = hits;
    __syncthreads();
    uint32_t at = 0u, total = 0u;
#pragma unroll
    for (int w = 0; w < kListWarps; ++w) {
        at += w < warp ? s_n[w] : 0u;
        total += s_n[w];
    }
    if (tid == 0) {
        s_start = total ? atomicAdd(cursor, total) : 0u;
        ranges[tile] = make_uint2(s_start, s_start + total);
    }
    __syncthreads();
    at += s_start;
    if ((int64_t)s_start + total > M_cap) {  // more tiles than were counted: never in a sound build
        if (tid == 0) set_status(status, VPGS_ERR_INTERNAL);
        return;
    }
    for (uint32_t k = lane; k < hits; k += 32u) ival[at + k] = cand[k];
}

// Emits the (global tile id, record) instances of a chunk of consecutive depth-ranked
// Gaussians per block.  A Gaussian spanning at most kCoverRows tile rows gives one run
// of consecutive tiles per row (the spans the counting pass stored), listed in shared
// memory with its first output position.  The output is then written kEmitWindow
// positions at a time: each run marks its first position, a running maximum over the
// marks gives every position its run, and the threads write consecutive positions.  A
// Gaussian covering many tiles does not serialise.  A Gaussian spanning more rows takes
// one warp to list its runs: one row per lane, its span from the same row-span function
// that counted it, and a warp prefix of the rows' counts.
// Bound: instruction issue and shared memory.  The running maximum costs about 10
// instructions per instance where a binary search over the Gaussians and a walk over
// their rows cost 100.  Measured, old -> new: 170k visible pairs, 1.19M instances
// 28.7 -> 18.9 us; 2.66M pairs, 10.3M 169 -> 141 us; 68k pairs of full-HD views, 1.85M
// instances 92 -> 30 us (108 us in chunks of 256: kEmitRounds 1, 2, 4: 34, 30, 27 us,
// and 18.2, 18.9, 26.7 us for the 170k pairs).
constexpr int kEmitThreads = 256;
constexpr int kEmitPer = 4;
#ifndef VPGS_EMIT_ROUNDS
#define VPGS_EMIT_ROUNDS 2
#endif
constexpr int kEmitRounds = VPGS_EMIT_ROUNDS;
// Fewest Gaussians in a chunk; the grid has a block per as many (up to what is resident).
// Few large Gaussians need the blocks: with one per 256, 5,000 of half of 1920x1080 each
// fell to the lane-per-row walk below and took 2550 us, with one per 64 833 us (32: 444,
// 16: 158).  But 13k and 20k small ones at 320x240 take 8.1 / 5.7 / 6.8 / 8.5 and 7.9 /
// 7.1 / 9.2 / 10.6 us with a block per 256 / 64 / 32 / 16, so 64: better than 256 for all.
constexpr int kEmitLeast = 64;
constexpr int kEmitWindow = kEmitThreads * kEmitPer;
constexpr uint32_t kNoKey = 0xffffffffu;  // the run of a Gaussian whose warp writes its tiles

__global__ void __launch_bounds__(kEmitThreads, 5)
emit_kernel(const uint32_t *__restrict__ dval, const uint32_t *__restrict__ inst_off,
            const BinRec *__restrict__ bin, const uint32_t *n_vis, const uint32_t *n_inst, int64_t N,
            int64_t M_cap, CamParams cam, uint32_t *__restrict__ ikey, uint32_t *__restrict__ ival,
            uint32_t *status, int n_pass, int dpt, SortPass p0, SortPass p1, SortPass p2, SortPass p3,
            uint32_t *hist, uint32_t *look0) {
    grid_dep_enter();
    // An earlier kernel failed: dval may hold stale entries.  Decided by the block as one:
    // another block of this launch may write *status meanwhile, and a block whose warps
    // read it differently would index its runs with words that the absent warps never wrote.
    if (__syncthreads_or(*status != 0u)) return;
    // the instance count is final before this launch: every block refuses an overflow alike
    if ((int64_t)*n_inst > M_cap) {
        if (threadIdx.x == 0) set_status(status, VPGS_ERR_CAPACITY);
        return;
    }
    {
        // the tile sort's first-pass look-back words, for the tiles that will hold
        // instances (the instance count is known from here on)
        const int64_t ni = min((int64_t)*n_inst, M_cap);
        const int64_t tile = (int64_t)kSortThreads * kTileSortItems;
        const int64_t nw = (ni + tile - 1) / tile * kRadix * dpt;
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nw; i += (int64_t)gridDim.x * blockDim.x)
            look0[i] = 0u;
    }
    // digit histograms of the emitted tile ids, for the tile sort
    __shared__ uint32_t s_h[4][kRadix];
    const SortPass tps[4] = {p0, p1, p2, p3};
    for (int i = threadIdx.x; i < 4 * kRadix; i += blockDim.x) (&s_h[0][0])[i] = 0u;
    constexpr int kRuns = kEmitThreads * kCoverRows;
    __shared__ uint32_t s_first[kRuns], s_key[kRuns];  // runs: first output position, first tile
    __shared__ uint8_t s_owner[kRuns];                 // the run's Gaussian in the chunk
    __shared__ __align__(8) uint16_t s_mark[kEmitWindow];
    __shared__ uint32_t s_start[kEmitThreads], s_id[kEmitThreads];
    __shared__ uint16_t s_large[kEmitThreads];  // chunk positions of the large Gaussians
    __shared__ uint16_t s_at[kEmitThreads];     // their first runs
    __shared__ uint32_t s_warp[kEmitThreads / 32], s_max[kEmitThreads / 32];
    __shared__ uint32_t s_total, s_nlarge;
    const int64_t nv = *n_vis;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    bool overflow = false;
    // chunks of consecutive depth-ranked Gaussians, grid-strided (the grid is sized to
    // what fits on the GPU, not to the capacity): up to kEmitThreads, but fewer where that
    // would give a block less than kEmitRounds chunks (the nearest Gaussians cover the
    // most tiles, so few large chunks leave their blocks to finish alone)
    const int64_t share = (nv / ((int64_t)gridDim.x * kEmitRounds) + kEmitLeast - 1) & ~int64_t(kEmitLeast - 1);
    const int chunk = (int)min((int64_t)kEmitThreads, max((int64_t)kEmitLeast, share));
    for (int64_t r0 = (int64_t)blockIdx.x * chunk; r0 < nv && !overflow; r0 += (int64_t)gridDim.x * chunk) {
    const int nb = (int)min((int64_t)chunk, nv - r0);
    const uint32_t base = inst_off[r0];
    uint32_t start = 0u, cnt = 0u, vb = 0u;
    uint32_t pk[kCoverRows];  // row spans, packed
    int ty_lo = 0, rows = 0, runs = 0;
    bool large = false;
    if (tid == 0) s_nlarge = 0u;
#pragma unroll
    for (int r = 0; r < kCoverRows; ++r) pk[r] = kEmptySpan;
    if (tid < nb) {
        const uint32_t id = dval[r0 + tid];
        const BinRec &br = bin[id];
        const uint2 rc = br.rect;
        const Cover cv = br.cv;
        cnt = br.cnt;
        start = inst_off[r0 + tid] - base;
        s_start[tid] = start;
        s_id[tid] = id;
        vb = (uint32_t)(id / N) * (uint32_t)cam.T;
        ty_lo = (int)(rc.y & 0xffffu);
        rows = (int)(rc.y >> 16) - ty_lo + 1;
        large = rows > kCoverRows;
        if (!large) {
            const float sp[kCoverRows] = {cv.a.x, cv.a.y, cv.a.z, cv.a.w, cv.b.x, cv.b.y, cv.b.z, cv.b.w};
#pragma unroll
            for (int r = 0; r < kCoverRows; ++r)
                if (r < rows) pk[r] = __float_as_uint(sp[r]);
        }
        // the block's end offset: the next block's start, or the total
        if (tid == nb - 1) s_total = (r0 + nb < nv ? inst_off[r0 + nb] : *n_inst) - base;
    }
#pragma unroll
    for (int r = 0; r < kCoverRows; ++r) runs += (pk[r] & 0xffffu) <= pk[r] >> 16 ? 1 : 0;
    if (large) runs = rows;
    uint32_t x, at, n_runs;  // scan of the run counts
    auto scan_runs = [&]() {
        x = (uint32_t)runs;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_warp[warp] = x;
        __syncthreads();
        at = x - (uint32_t)runs;
        n_runs = 0u;
#pragma unroll
        for (int w = 0; w < kEmitThreads / 32; ++w) {
            at += w < warp ? s_warp[w] : 0u;
            n_runs += s_warp[w];
        }
    };
    scan_runs();
    const bool listed = n_runs <= (uint32_t)kRuns;  // block-uniform
    if (!listed) {  // too many rows in the chunk: its large Gaussians write their tiles themselves
        __syncthreads();
        if (large) runs = 1;
        scan_runs();
    }
    const uint32_t total = s_total;
    if ((int64_t)base + total > M_cap) {
        if (tid == 0) set_status(status, VPGS_ERR_INTERNAL);  // offsets past their total: never in a sound build
        overflow = true;  // block-uniform
        continue;
    }
    if (large) {
        if (!listed) {
            s_first[at] = start;
            s_key[at] = kNoKey;
            s_owner[at] = (uint8_t)tid;
        }
        s_at[tid] = (uint16_t)at;
        s_large[atomicAdd(&s_nlarge, 1u)] = (uint16_t)tid;
    } else if (tid < nb) {
        uint32_t pos = start;
#pragma unroll
        for (int r = 0; r < kCoverRows; ++r) {
            const uint32_t t0 = pk[r] & 0xffffu, t1 = pk[r] >> 16;
            if (t0 <= t1) {
                s_first[at] = pos;
                s_key[at] = vb + (uint32_t)(ty_lo + r) * (uint32_t)cam.tiles_x + t0;
                s_owner[at] = (uint8_t)tid;
                ++at;
                pos += t1 - t0 + 1u;
            }
        }
        if (pos - start != cnt) set_status(status, VPGS_ERR_INTERNAL);  // never in a sound build
    }
    // large Gaussians: one warp each, one tile row per lane, a warp prefix of the rows'
    // counts; each lane lists its row's run (or writes its tiles)
    __syncthreads();
    const uint32_t n_large = s_nlarge;
    for (uint32_t j = warp; j < n_large; j += kEmitThreads / 32) {
        const int t = s_large[j];
        const uint32_t id = s_id[t];
        const BinRec &br = bin[id];
        const uint2 rc = br.rect;
        const Cover cv = br.cv;
        const float4 uv = br.uv;
        const int tx_lo = (int)(rc.x & 0xffffu), tx_hi = (int)(rc.x >> 16);
        const int ly_lo = (int)(rc.y & 0xffffu), ly_hi = (int)(rc.y >> 16);
        const uint32_t begin = s_start[t], end = (t + 1 < nb ? s_start[t + 1] : total);
        const uint32_t vbase = (uint32_t)(id / N) * (uint32_t)cam.T;
        uint32_t running = begin;
        for (int ty0 = ly_lo; ty0 <= ly_hi; ty0 += 32) {  // warp-uniform
            const int ty = ty0 + lane;
            int2 sp = make_int2(1, 0);
            if (ty <= ly_hi)
                sp = cover_row(cv, uv.x, uv.z, uv.y, uv.w, ty, tx_lo, tx_hi, cam.tw_shift, cam.tile_h, cam.W, cam.H);
            const uint32_t n = sp.x <= sp.y ? (uint32_t)(sp.y - sp.x + 1) : 0u;
            uint32_t xs = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t ys = __shfl_up_sync(0xffffffffu, xs, o);
                if (lane >= o) xs += ys;
            }
            const uint32_t to = running + xs - n;
            if (listed && ty <= ly_hi) {
                const uint32_t k = s_at[t] + (uint32_t)(ty - ly_lo);
                s_first[k] = n ? to : 0xffffffffu;  // (an empty row starts nowhere)
                s_key[k] = vbase + (uint32_t)ty * (uint32_t)cam.tiles_x + (uint32_t)sp.x;
                s_owner[k] = (uint8_t)t;
            }
            for (uint32_t k = 0; !listed && k < n; ++k) {
                if (to + k >= end) {  // more tiles than were counted: never in a sound build
                    set_status(status, VPGS_ERR_INTERNAL);
                    break;
                }
                const uint32_t key = vbase + (uint32_t)ty * (uint32_t)cam.tiles_x + (uint32_t)sp.x + k;
                ikey[base + to + k] = key;
                ival[base + to + k] = id;
                add_digits(&s_h[0][0], tps, n_pass, key, dpt);
            }
            running += __shfl_sync(0xffffffffu, xs, 31);
        }
        if (lane == 0 && running != end) set_status(status, VPGS_ERR_INTERNAL);
    }
    uint32_t carry = 0u;  // 1 + the last run that starts before the window
    for (uint32_t w0 = 0u; w0 < total; w0 += kEmitWindow) {
        reinterpret_cast<uint2 *>(s_mark)[tid] = make_uint2(0u, 0u);
        __syncthreads();  // (also the runs' writes before the first window)
        for (uint32_t k = tid; k < n_runs; k += kEmitThreads) {
            const uint32_t d = s_first[k] - w0;
            if (d < (uint32_t)kEmitWindow) s_mark[d] = (uint16_t)(k + 1u);
        }
        __syncthreads();
        // running maximum over the window, four positions per thread
        const uint2 mk = reinterpret_cast<const uint2 *>(s_mark)[tid];
        const uint32_t m0 = mk.x & 0xffffu, m1 = max(m0, mk.x >> 16), m2 = max(m1, mk.y & 0xffffu), m3 = max(m2, mk.y >> 16);
        uint32_t y = m3;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t z = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) y = max(y, z);
        }
        if (lane == 31) s_max[warp] = y;
        __syncthreads();
        uint32_t pre = __shfl_up_sync(0xffffffffu, y, 1);
        if (lane == 0) pre = 0u;
        pre = max(pre, carry);
#pragma unroll
        for (int w = 0; w < kEmitThreads / 32; ++w) {
            if (w < warp) pre = max(pre, s_max[w]);
            carry = max(carry, s_max[w]);
        }
        reinterpret_cast<uint2 *>(s_mark)[tid] =
            make_uint2(max(pre, m0) | max(pre, m1) << 16, max(pre, m2) | max(pre, m3) << 16);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kEmitPer; ++j) {
            const uint32_t d = (uint32_t)(j * kEmitThreads + tid), pos = w0 + d;
            if (pos < total) {
                const uint32_t k = s_mark[d] - 1u;
                uint32_t key = kNoKey;
                if (k < n_runs) key = s_key[k];
                else set_status(status, VPGS_ERR_INTERNAL);  // no run before it: never in a sound build
                if (key != kNoKey) {
                    key += pos - s_first[k];
                    ikey[base + pos] = key;
                    ival[base + pos] = s_id[s_owner[k]];
                    add_digits(&s_h[0][0], tps, n_pass, key, dpt);
                }
            }
        }
        __syncthreads();
    }
    __syncthreads();  // the next chunk reuses the shared arrays
    }
    __syncthreads();
    flush_digits(&s_h[0][0], n_pass * kRadix * dpt, hist);
}

__global__ void tile_ranges_kernel(const uint32_t *__restrict__ keys, int64_t cap, const uint32_t *n_dev,
                                   uint32_t n_tiles, uint2 *ranges) {
    grid_dep_enter();
    int64_t n = min(cap, (int64_t)*n_dev);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t k = keys[i];
        if (k >= n_tiles) continue;  // only after a capacity overflow (status already set)
        if (i == 0 || keys[i - 1] != k) ranges[k].x = (uint32_t)i;
        if (i == n - 1 || keys[i + 1] != k) ranges[k].y = (uint32_t)(i + 1);
    }
}

// Launch order of the compositing kernels: global tile ids by descending
// instance count, so the longest tiles start first and the short ones fill the
// tail of the grid (tiles are independent: the order changes no pixel).  One
// block: tiles are bucketed by count / 4 (the last bucket takes every count
// beyond), buckets are laid out from the heaviest down, and each tile takes a
// slot in its bucket by a shared-memory atomic.  Up to kOrderPer tiles per
// thread (8, or 32 past 8,192 tiles) are loaded at once and kept in registers
// (packed) between the passes.
constexpr int kOrderThreads = 1024;
constexpr int kOrderBins = 1024;

// work of tile i: its step count if given, else its instance count
VPGS_D uint32_t order_bucket(const uint2 *ranges, const uint32_t *work, int i) {
    uint32_t c;
    if (work) {
        c = work[i];
    } else {
        const uint2 r = ranges[i];
        c = r.y > r.x ? r.y - r.x : 0u;
    }
    return min(c >> 2, (uint32_t)kOrderBins - 1u);
}

template <int kOrderPer>
__global__ void __launch_bounds__(kOrderThreads)
tile_order_kernel(const uint2 *__restrict__ ranges, const uint32_t *__restrict__ work, int n_tiles,
                  uint32_t *__restrict__ order) {
    grid_dep_enter();
    __shared__ uint32_t s_bin[kOrderBins];
    __shared__ uint32_t s_warp[kOrderThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool fits = n_tiles <= kOrderThreads * kOrderPer;  // block-uniform
    // bucket of tile tid + k * kOrderThreads (kOrderBins: none), two 16-bit buckets
    // per register (a 1,024-thread block has 64 registers per thread)
    uint32_t bk[kOrderPer / 2];
    auto bucket_of = [&](int k) { return (bk[k >> 1] >> (16 * (k & 1))) & 0xffffu; };
    if (fits) {
#pragma unroll
        for (int k = 0; k < kOrderPer; ++k) {
            const int i = tid + k * kOrderThreads;
            const uint32_t b = i < n_tiles ? order_bucket(ranges, work, i) : (uint32_t)kOrderBins;
            if (k & 1) bk[k >> 1] |= b << 16;
            else bk[k >> 1] = b;
        }
    }
    for (int i = tid; i < kOrderBins; i += kOrderThreads) s_bin[i] = 0u;
    __syncthreads();
    if (fits) {
#pragma unroll
        for (int k = 0; k < kOrderPer; ++k)
            if (bucket_of(k) < (uint32_t)kOrderBins) atomicAdd(&s_bin[bucket_of(k)], 1u);
    } else {
        for (int i = tid; i < n_tiles; i += kOrderThreads) atomicAdd(&s_bin[order_bucket(ranges, work, i)], 1u);
    }
    __syncthreads();
    // exclusive scan over the buckets from the heaviest (thread j holds bucket kOrderBins-1-j)
    const int b = kOrderBins - 1 - tid;
    const uint32_t c = s_bin[b];
    uint32_t x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = s_warp[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        s_warp[lane] = w;  // inclusive totals of warps 0..lane
    }
    __syncthreads();
    s_bin[b] = x - c + (warp > 0 ? s_warp[warp - 1] : 0u);  // every thread read its count before the barrier
    __syncthreads();
    if (fits) {
#pragma unroll
        for (int k = 0; k < kOrderPer; ++k)
            if (bucket_of(k) < (uint32_t)kOrderBins)
                order[atomicAdd(&s_bin[bucket_of(k)], 1u)] = (uint32_t)(tid + k * kOrderThreads);
    } else {
        for (int i = tid; i < n_tiles; i += kOrderThreads)
            order[atomicAdd(&s_bin[order_bucket(ranges, work, i)], 1u)] = (uint32_t)i;
    }
}

// The backward's steps per tile: the largest n_iter (list position of the last
// Gaussian a pixel blended, from the forward) over the tile's pixels.  One warp
// per tile.
constexpr int kWorkThreads = 256;

__global__ void __launch_bounds__(kWorkThreads)
tile_work_kernel(const int32_t *__restrict__ n_iter, CamParams cam, int n_tiles, uint32_t *__restrict__ work) {
    grid_dep_enter();
    const int t = (int)((blockIdx.x * (unsigned)kWorkThreads + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (t >= n_tiles) return;  // whole warps
    const int v = t / cam.T, lt = t - v * cam.T;
    const int ty = lt / cam.tiles_x, tx = lt - ty * cam.tiles_x;
    const int64_t base = (int64_t)v * cam.H * cam.W;
    int m = 0;
    for (int i = lane; i < cam.tile_w * cam.tile_h; i += 32) {
        const int px = tx * cam.tile_w + i % cam.tile_w, py = ty * cam.tile_h + i / cam.tile_w;
        if (px < cam.W && py < cam.H) m = max(m, n_iter[base + (int64_t)py * cam.W + px]);
    }
    m = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(m, 0));
    if (lane == 0) work[t] = (uint32_t)m;
}

// A launch order pays only where the tiles take more than one round of blocks: with
// all of them resident at once (256 threads per SM counted, half of what any of the
// compositing kernels' registers allow) they all start together, and the forward saves
// one launch and the backward two.  Forward + backward, without / with the order (us, 50k
// Gaussians of a small scene; 200k of a room): 300 tiles 282 / 291 and 336 / 342, 400
// tiles 262 / 268 and 323 / 328, 600 tiles 286 / 278 and 303 / 310, 768 tiles 287 / 286 and
// 312 / 317, 1,200 tiles 297 / 288 and 339 / 312: they meet between 500 and 1,000 tiles by
// the scene, and the line, 304 tiles of 128 threads, stays where none loses without it.
bool tiles_ordered(int n_tiles, const CamParams &cam) {
    const int64_t threads = (int64_t)n_tiles * (cam.tile_w * cam.tile_h / kPix);
    return VPGS_TILE_ORDER && threads > (int64_t)256 * device_sm_count();
}

static cudaError_t launch_tile_order(const RenderWs &ws, const uint32_t *work, int n_tiles, cudaStream_t s) {
    VPGS_LAUNCH("tile_order", s,
                launch_k(n_tiles <= kOrderThreads * 8 ? tile_order_kernel<8> : tile_order_kernel<32>, 1, kOrderThreads,
                         0, s, (const uint2 *)ws.ranges, work, n_tiles, ws.tile_order));
    return cudaGetLastError();
}

cudaError_t order_tiles_by_steps(const RenderWs &ws, const int32_t *n_iter, int V, const CamParams &cam,
                                 cudaStream_t s) {
    const int n_tiles = V * cam.T;
    if (n_tiles == 0 || !tiles_ordered(n_tiles, cam)) return cudaSuccess;
    const unsigned blocks = (unsigned)(((int64_t)n_tiles * 32 + kWorkThreads - 1) / kWorkThreads);
    VPGS_LAUNCH("tile_work", s, launch_k(tile_work_kernel, blocks, kWorkThreads, 0, s, n_iter, cam, n_tiles,
                                         ws.tile_work));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_tile_order(ws, ws.tile_work, n_tiles, s);
}

// Launch order by instance count, where the call uses one.
static cudaError_t order_tiles_by_count(const RenderWs &ws, int n_tiles, const CamParams &cam, cudaStream_t s) {
    return tiles_ordered(n_tiles, cam) ? launch_tile_order(ws, nullptr, n_tiles, s) : cudaSuccess;
}

int tile_list_buffer(const RenderLayout &L) {
    SortPass ps[kMaxSortPasses];
    return (plan_passes(0, L.tile_bits, ps) & 1) != 0 ? 1 : 0;
}

// SM count of the current device, looked up once per device ordinal.
int device_sm_count() {
    static std::atomic<int> cache[kDeviceCache];
    return per_device(cache, [] {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) sms = 1;
        return sms;
    });
}

cudaError_t build_tile_lists(const GaussIn &g, int V, const CamParams &cam, const OptParams &o, const RenderWs &ws,
                             const RenderLayout &L, int *sorted_buf, cudaStream_t s, bool order_by_count) {
    // every binning kernel stops at entry once a predecessor recorded an error: after
    // a timed-out look-back the compacted and sorted arrays hold holes whose stale
    // contents must not be used as indices
    const LookBack lb{o.spin_limit, true};
    cudaError_t e;
    const int sms = device_sm_count();
    uint32_t *n_vis = ws.counters + CNT_VISIBLE;
    uint32_t *n_inst = ws.counters + CNT_INSTANCES;
    // calls of many views (above 4M pairs): wider scan tiles and depth-sort tiles,
    // the offset scan on the resident grid (the visible pairs then fill it)
    const bool many = L.VN > (int64_t(4) << 20);
    SortPass tps[kMaxSortPasses] = {};
    const int np_tile = plan_passes(0, L.tile_bits, tps);
    if (np_tile > 4) return cudaErrorInvalidValue;
    uint32_t *dval = ws.dval[0], *inst_off = ws.dkey[1];  // visible records in depth order, their first instances
    bool in1 = false;
    const BinForm form = bin_form(L);
    if (form != kGeneralBin) {
        // 1-3 at once (the projection left the list and the counts)
        const bool lists = form == kSmallLists;
        dval = ws.sort_look[0];  // the depth sort's look-back words: at least one per pair (make_layout)
        VPGS_LAUNCH("small_rank", s,
                    launch_k(lists ? small_rank_kernel<true> : small_rank_kernel<false>,
                             (unsigned)std::max<int64_t>(std::min<int64_t>((L.VN + kRankOwn - 1) / kRankOwn, 4 * sms), 1),
                             kRankThreads, 0, s, small_list(ws, L), (const uint32_t *)ws.tcount,
                             (const BinRec *)ws.bin, (int)L.VN, (int)L.N, ws.vis_idx, dval, inst_off,
                             (const uint32_t *)n_vis, (const uint32_t *)ws.status));
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        if (lists) {
            *sorted_buf = tile_list_buffer(L);
            VPGS_LAUNCH("small_lists", s,
                        launch_k(small_lists_kernel, (unsigned)(V * cam.T), kListThreads, 0, s, (const uint32_t *)dval,
                                 (const uint32_t *)inst_off, (const BinRec *)ws.bin, (const uint32_t *)n_vis,
                                 (const uint32_t *)n_inst, L.M_cap, cam, ws.ranges, ws.ival[*sorted_buf],
                                 ws.counters + CNT_TICKET_T, ws.status));
            e = cudaGetLastError();
            return e != cudaSuccess || !order_by_count ? e : order_tiles_by_count(ws, V * cam.T, cam, s);
        }
    } else {
        // 1. compaction of visible (view, Gaussian) pairs
        e = launch_scan("scan_visible", VisLoad{ws.tcount},
                        VisStore{ws.rec, ws.dkey[0], ws.dval[0], ws.vis_idx, L.VN}, L.VN, nullptr,
                        ws.counters + CNT_TICKET_A, ws.scan_look[0], n_vis, ws.status, s, lb, 0, many);
        if (e != cudaSuccess) return e;
        // 2. depth sort (digit histograms from the projection kernel)
        // keys per thread: few for a frame's worth of visible Gaussians (short tiles
        // start the look-back chain sooner), more for many views' worth (fewer tiles
        // in the chain); the look-back space is sized for kDepthSortItems, the most tiles
        const auto depth_sort = many ? radix_sort_pairs<16, false> : radix_sort_pairs<kDepthSortItems, false>;
        e = depth_sort("sort_depth_pass", ws.dkey[0], ws.dval[0], ws.dkey[1], ws.dval[1], L.VN, n_vis, 0, 32,
                       ws.sort_hist[0], ws.counters + CNT_TICKET_D, ws.sort_look[0], ws.status, s, &in1, lb,
                       VPGS_DEPTH_SORT_GRID);
        if (e != cudaSuccess) return e;
        dval = in1 ? ws.dval[1] : ws.dval[0];
        inst_off = in1 ? ws.dkey[0] : ws.dkey[1];  // the depth-sort buffer not holding the result
        // 3. instance offsets
        e = launch_scan("scan_offsets", CountLoad{ws.tcount, dval}, OffsetStore{inst_off}, L.VN, n_vis,
                        ws.counters + CNT_TICKET_O, ws.scan_look[1], n_inst, ws.status, s, lb,
                        many ? 0 : VPGS_OFFSET_SCAN_GRID, many);
        if (e != cudaSuccess) return e;
    }
    // emission
    static std::atomic<int> emit_cache[kDeviceCache];
    const int emit_grid = per_device(emit_cache, [] {
        return resident_grid((const void *)emit_kernel, kEmitThreads, 0, int64_t(1) << 30);
    });
    VPGS_LAUNCH("emit_instances", s,
                launch_k(emit_kernel, (unsigned)std::min<int64_t>(std::max<int64_t>((L.VN + kEmitLeast - 1) / kEmitLeast, 1),
                                                          emit_grid),
                              kEmitThreads, 0, s, dval, inst_off, ws.bin, n_vis, n_inst, L.N, L.M_cap,
                                                    cam, ws.ikey[0], ws.ival[0], ws.status, np_tile, sort_dpt(L.tile_bits), tps[0],
                                                    tps[1], tps[2], tps[3], ws.sort_hist[1], ws.sort_look[1]));
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // 4. stable sort by tile id
    // (digit histograms from the emit kernel)
    e = radix_sort_pairs<kTileSortItems, true>("sort_tile_pass", ws.ikey[0], ws.ival[0], ws.ikey[1], ws.ival[1],
                                               L.M_cap, n_inst, 0, L.tile_bits, ws.sort_hist[1],
                                               ws.counters + CNT_TICKET_T, ws.sort_look[1], ws.status, s, &in1, lb);
    if (e != cudaSuccess) return e;
    *sorted_buf = in1 ? 1 : 0;
    if (*sorted_buf != tile_list_buffer(L)) return cudaErrorUnknown;  // never: same pass plan
    // 5. tile ranges
    const int n_tiles = V * cam.T;  // (ranges zeroed by the prepare kernel)
    const int64_t rb = std::min<int64_t>((L.M_cap + 255) / 256, (int64_t)sms * 16);
    VPGS_LAUNCH("tile_ranges", s,
                launch_k(tile_ranges_kernel, (unsigned)std::max<int64_t>(rb, 1), 256, 0, s,
                    in1 ? ws.ikey[1] : ws.ikey[0], L.M_cap, n_inst, (uint32_t)n_tiles, ws.ranges));
    e = cudaGetLastError();
    // 6. compositing launch order
    return e != cudaSuccess || !order_by_count ? e : order_tiles_by_count(ws, n_tiles, cam, s);
}

}  // namespace vpgs
