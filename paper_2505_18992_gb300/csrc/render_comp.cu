// Front-to-back alpha compositing per tile, and its backward pass.
//
// One CTA renders one tile (tile_w x tile_h / 2 threads, two rows of a column each),
// or, in persistent mode, a fixed number of CTAs per SM pull tiles from a work queue.
// The tile's depth-ordered Gaussian list is staged through shared memory in batches
// of one or two records per thread; each pixel walks the batch in order:
//   alpha = min(alpha_max, o 2^-((w1.d)^2 + (w2.d)^2)), d = pixel - mean, with
//           the whitening rows w scaled by sqrt(log2(e)/2) when the record is made
//   skip alpha < alpha_min; stop before T (1 - alpha) < t_min
// Each warp first compacts the staged batch into its own list of the Gaussians
// whose widened y extent reaches one of the warp's pixel rows (at the others
// alpha < alpha_min at every pixel of the warp), then walks only that list.
//   C += alpha T c, D += alpha T z, T *= 1 - alpha
// Means are made tile-local when staged ((u_hi - x0) + u_lo), so d keeps
// ~1e-7 px accuracy anywhere in the image.
//
// The backward pass walks the same list from the back, recovering T_i as
// T_{i+1} / (1 - alpha_i), and keeps the colour/depth "behind" each Gaussian,
//   B <- alpha c + (1 - alpha) B   (B starts at the background),
// giving dC/dalpha_i = T_i (c_i - B_i), dA/dalpha_i = T_final / (1 - alpha_i).
// Only g . B enters dL/dalpha (g the pixel's upstream gradient), so each pixel
// carries that scalar instead of B.
// Per-Gaussian 2D gradient sums of a warp are taken in the Gaussian's whitened frame
// t = W d: sum dpow t1, sum dpow t2, sum dpow t1^2, sum dpow t1 t2, sum dpow t2^2;
// then opacity, rgb, z.  The full backward collects its pixels' terms in shared memory
// and sums them one entry per lane; the geometric one (pose tracking) sums six of the
// ten by shuffles.  Each adds its sums with one atomic per value and warp.
// Near-degenerate records (negative y half extent) take the double-float pair
// evaluation (eval_pair_fine): one warp-uniform branch per list entry.
#include <type_traits>

#include "internal.h"
#include "profiler.h"

namespace vpgs {

struct TileCoord {
    int v, tx, ty;
};

VPGS_D TileCoord tile_coord(int t, const CamParams &cam) {
    TileCoord c;
    c.v = t / cam.T;
    const int lt = t - c.v * cam.T;
    c.ty = lt / cam.tiles_x;
    c.tx = lt - c.ty * cam.tiles_x;
    return c;
}

// Each thread owns kPix pixels of its tile column: rows kPix*ly .. kPix*ly + kPix - 1.
constexpr int kMaxThreads = 512 / kPix;  // tiles hold at most 512 pixels
#ifndef VPGS_FWD_BATCH
#define VPGS_FWD_BATCH 2  // records each forward thread stages per batch
#endif
constexpr int kFwdBatch = VPGS_FWD_BATCH;
#ifndef VPGS_BWD_BATCH
#define VPGS_BWD_BATCH 1  // records each thread of the full backward stages per batch (2: 20 KB more, 292 us)
#endif
constexpr int kBwdBatch = VPGS_BWD_BATCH;
#ifndef VPGS_GEO_BATCH
#define VPGS_GEO_BATCH 2  // the same of the geometric backward (1: 310 us, 2: 288 us)
#endif
constexpr int kGeoBatch = VPGS_GEO_BATCH;
// list entries whose alphas the forward evaluates before blending them (see VPGS_FWD_MAXREG)
#ifndef VPGS_FWD_WALK
#define VPGS_FWD_WALK 8
#endif
constexpr int kWalk = VPGS_FWD_WALK;

// Centre and half height of the band of tile-local pixel-centre rows held by
// this thread's warp (whole rows of the tile: its width divides 32).
VPGS_D float2 warp_rows(const CamParams &cam) {
    const int first = (int)(threadIdx.x & ~31u);
    const float lo = (float)(kPix * (first >> cam.tw_shift)) + 0.5f;
    const float hi = (float)(kPix * ((first + 31) >> cam.tw_shift) + kPix - 1) + 0.5f;
    return make_float2(0.5f * (lo + hi), 0.5f * (hi - lo));
}

// The tile of a block that renders one, loaded beside the status word and not after it:
// an empty tile costs little but the latency of its few loads, one after another.
// (Tile blockIdx.x of the order exists for every such block.)
VPGS_D int first_tile(const uint32_t *order, const uint32_t *work) {
    return order && !work ? (int)order[blockIdx.x] : (int)blockIdx.x;
}

// Whether a staged (plain) Gaussian can reach alpha_min at a pixel centre of
// the tile-local box [x0, x1] x [y0, y1]: the minimum over the box of the
// whitened square distance q = |W d|^2, d = p - mean, against log2(o /
// alpha_min) (alpha = o 2^-q).  The minimum of the convex q lies inside the box
// (then 0) or on an edge, where q is a quadratic in one variable.  The bound
// is widened by 0.1 % + 1e-3 so that every pixel the FP32 per-pixel evaluation
// would blend stays listed.
VPGS_D bool reaches_box(const float4 &a, const float4 &b, float x0, float x1, float y0, float y1,
                        float lg_amin) {
    const float A = fmaf(a.z, a.z, b.x * b.x), B = fmaf(a.z, a.w, b.x * b.y), C = fmaf(a.w, a.w, b.y * b.y);
    if (!(A > 0.f && C > 0.f)) return true;
    const float dx0 = x0 - a.x, dx1 = x1 - a.x, dy0 = y0 - a.y, dy1 = y1 - a.y;
    if (dx0 <= 0.f && dx1 >= 0.f && dy0 <= 0.f && dy1 >= 0.f) return true;
    auto q = [&](float dx, float dy) { return fmaf(A * dx, dx, fmaf(2.f * B * dx, dy, C * dy * dy)); };
    const float ra = -B / A, rc = -B / C;
    float m = q(fminf(fmaxf(ra * dy0, dx0), dx1), dy0);
    m = fminf(m, q(fminf(fmaxf(ra * dy1, dx0), dx1), dy1));
    m = fminf(m, q(dx0, fminf(fmaxf(rc * dx0, dy0), dy1)));
    m = fminf(m, q(dx1, fminf(fmaxf(rc * dx1, dy0), dy1)));
    const float level = __log2f(b.z) - lg_amin;
    return !(m > fmaf(1e-3f, fabsf(level), level) + 1e-3f);
}

// Compacts the batch positions [0, n) whose Gaussian reaches the warp's pixel rows
// into list, as byte offsets of the staged records (kRecStage float4 each), first
// record first or, with kBack, last record first; returns how many (warp-uniform).  A
// Gaussian is listed when its widened y extent reaches the rows and, with kExact (the
// backward) and a plain record, its alpha_min ellipse also meets the rows' pixel
// centres within the tile's columns [0.5, xmax].  Both forms list every Gaussian that
// blends into a pixel of the rows, so they may differ in what they skip but not in
// what they blend.  All 32 lanes take part.  `fine` tells (warp-uniform) whether a
// listed record is near-degenerate.
constexpr int kRecStage = 5;  // float4 per staged record: an odd number keeps 16-byte reads by lane conflict-free
// (the lists are 16-bit: a batch of the largest tile must not hold more records than they reach)
constexpr bool offsets_fit(int batch) { return (kMaxThreads * batch - 1) * kRecStage * 16 <= 65535; }
static_assert(offsets_fit(kFwdBatch) && offsets_fit(kBwdBatch) && offsets_fit(kGeoBatch),
              "the staged batch is larger than the lists' 16-bit offsets reach");
template <bool kExact, bool kBack>
VPGS_D int warp_offsets(const float4 *s_rec, int n, float2 band, uint16_t *list, int lane, bool &fine, float xmax,
                        float lg_amin) {
    const uint32_t below = (1u << lane) - 1u;
    int cnt = 0;
    bool any = false;
    for (int c0 = 0; c0 < n; c0 += 32) {
        const int k = kBack ? n - 1 - c0 - lane : c0 + lane;
        bool touch = false, f = false;
        if (kBack ? k >= 0 : k < n) {
            const float4 a = s_rec[kRecStage * k], b = s_rec[kRecStage * k + 1];
            touch = fabsf(a.y - band.x) <= fabsf(b.w) + band.y;
            f = touch && b.w < 0.f;
            if (kExact && touch && !f) touch = reaches_box(a, b, 0.5f, xmax, band.x - band.y, band.x + band.y, lg_amin);
        }
        const uint32_t m = __ballot_sync(0xffffffffu, touch);
        any |= __any_sync(0xffffffffu, f);
        if (touch) list[cnt + __popc(m & below)] = (uint16_t)(k * (kRecStage * 16));
        cnt += __popc(m);
    }
    __syncwarp();
    fine = any;
    return cnt;
}

// the staged record at a byte offset of such a list
VPGS_D const float4 *rec_at(const float4 *s_rec, int off) {
    return reinterpret_cast<const float4 *>(reinterpret_cast<const char *>(s_rec) + off);
}

// record -> shared staging: s0 = (u, v) tile-local, w1; s1 = w2, opacity, widened
// y half extent (negative: near-degenerate); s2 = colour, camera z.  The
// forward also stages fine_extra of a near-degenerate record; the backward
// kernels read it from the record in memory (a broadcast load, for such records only).
// what a near-degenerate record adds to its staged a = (ux, uy, ...): the
// rounding residual of the tile-local mean ((u_hi - ox) + u_lo = ux + residual,
// the subtraction split exactly) and the low parts of w2
VPGS_D float4 fine_extra(const Rec &r, float ox, float oy, float ux, float uy) {
    const df ex = two_sum(r.r0.x, -ox), ey = two_sum(r.r0.y, -oy);
    return make_float4(((ex.hi - ux) + r.r0.z) + ex.lo, ((ey.hi - uy) + r.r0.w) + ey.lo, r.r3.y, r.r3.w);
}

VPGS_D void stage(const Rec &r, float ox, float oy, float4 &a, float4 &b, float4 &c) {
    a = make_float4((r.r0.x - ox) + r.r0.z, (r.r0.y - oy) + r.r0.w, r.r1.x, r.r1.y);
    b = make_float4(r.r1.z, r.r1.w, r.r2.x, r.r3.z);
    c = make_float4(r.r2.z, r.r2.w, r.r3.x, r.r2.y);
}

// alpha of the thread's pixel q (tile-local (px, py)) for the staged Gaussian
// (a, b[, f]).  A thread's pixels are kPix consecutive rows of one column, so in
// the plain form the whitened coordinates of row q are those of its first row
// (t1_0, t2_0) plus q times the rows' y coefficients (w1y, w2y); the
// near-degenerate form evaluates each row in double-float.
template <bool kFine>
VPGS_D PairEval eval_staged(int q, float t1_0, float t2_0, float px, float py, const float4 &a, const float4 &b,
                            const float4 &f, float alpha_max) {
    if constexpr (kFine) {
        return eval_pair_fine(px, py, a.x, a.y, f.x, f.y, a.z, a.w, b.x, b.y, f.z, f.w, b.z, alpha_max);
    } else {
        PairEval e;
        e.t1 = fmaf((float)q, a.w, t1_0);
        e.t2 = fmaf((float)q, b.y, t2_0);
        e.G = ex2_approx(-fmaf(e.t1, e.t1, e.t2 * e.t2));
        e.alpha = fminf(alpha_max, b.z * e.G);
        return e;
    }
}

// whitened coordinates of the first of the thread's rows (plain form)
VPGS_D float2 first_row(float px, float py0, const float4 &a, const float4 &b) {
    const float dx = px - a.x, dy = py0 - a.y;
    return make_float2(fmaf(a.z, dx, a.w * dy), fmaf(b.x, dx, b.y * dy));
}

// register cap of the forward (0: only the launch bound of the largest tile).  96 with 8 entries
// per step: 140 us (room) and 163 us (a street frame whose longest tiles hold 3,600
// entries: there each warp's own latency counts, not the number of warps); 80 with 6:
// 144 / 181 us, 72 with 4: 150 / 200 us, 64 with 4: 150 / 230 us.
#ifndef VPGS_FWD_MAXREG
#define VPGS_FWD_MAXREG 96
#endif
#if VPGS_FWD_MAXREG > 0
#define VPGS_FWD_BOUNDS __maxnreg__(VPGS_FWD_MAXREG)
#else
#define VPGS_FWD_BOUNDS __launch_bounds__(kMaxThreads)
#endif

// One lane per column pair of pixels; the packed FP32 instructions work on the pair.
// A list step has no branch: a pixel that does not blend takes part with weight 0 and
// keeps its T by a select, which leaves every sum as it was (the rounding of each
// half is the scalar instructions').  The branches it replaces cost their exposed
// latency in long tiles and their issue slots in the others.  Measured, old -> new:
// 1M-Gaussian room 1200x680 192 -> 138 us, street frame 1241x376 of 316k visible
// Gaussians 524 -> 160 us, 8 keyframes of 2M 875 -> 646 us, four full-HD views 504 ->
// 391 us, 10k Gaussians 320x240 24 -> 12 us.  Frames of empty or nearly empty tiles pay
// for the fewer blocks per SM: 64 views of 640x480 with 150 Gaussians 173 -> 220 us.  The exact ellipse test of the backward's
// lists gains nothing here (room 144 us either way, street frame 181 -> 196 us).
__global__ void VPGS_FWD_BOUNDS
composite_fwd_kernel(const Rec *__restrict__ rec, const uint32_t *__restrict__ ival,
                     const uint2 *__restrict__ ranges, const uint32_t *__restrict__ order, int n_tiles,
                     CamParams cam, OptParams o,
                     vpgs_images out, const uint32_t *status, uint32_t *work) {
    grid_dep_enter();
    extern __shared__ float4 smem[];
    const int NT = blockDim.x * kFwdBatch;  // records per batch
    // records: mean and w1; w2, opacity, y half extent; (r, r, g, g); (b, b, z, z); fine_extra
    float4 *s_rec = smem;
    const int tid = threadIdx.x, lane = tid & 31;
    uint16_t *wl = reinterpret_cast<uint16_t *>(smem + kRecStage * NT) + (size_t)(tid >> 5) * NT;  // this warp's list
    __shared__ int s_tile;
    int tile = first_tile(order, work);
    if (*status != 0u) return;
    const int lx = tid & (cam.tile_w - 1), ly = tid >> cam.tw_shift;
    const float pxl = (float)lx + 0.5f;
    float pyl[kPix];
#pragma unroll
    for (int q = 0; q < kPix; ++q) pyl[q] = (float)(kPix * ly + q) + 0.5f;
    const float2 band = warp_rows(cam);
    const float lg_amin = __log2f(o.alpha_min);
    const f2 one2 = pack2(1.f, 1.f);
    int t = blockIdx.x;
    for (;;) {
        if (work) {
            if (tid == 0) s_tile = (int)atomicAdd(work, 1u);
            __syncthreads();
            t = s_tile;
            __syncthreads();
            if (t >= n_tiles) return;
            tile = order ? (int)order[t] : t;  // launch order -> global tile id
        }
        const TileCoord tc = tile_coord(tile, cam);
        const int px = tc.tx * cam.tile_w + lx;
        const float ox = (float)(tc.tx * cam.tile_w), oy = (float)(tc.ty * cam.tile_h);
        const float xmax = fminf((float)cam.tile_w, (float)cam.W - ox) - 0.5f;  // last pixel centre column
        const uint2 rg = ranges[tile];
        const int start = (int)rg.x, end = (int)rg.y;
        f2 T2 = one2, C0 = pack2(0.f, 0.f), C1 = C0, C2 = C0, D = C0;
        int cnt0 = 0, cnt1 = 0, last0 = 0, last1 = 0;
        const int py0 = tc.ty * cam.tile_h + kPix * ly;
        bool done0 = !(px < cam.W && py0 < cam.H), done1 = !(px < cam.W && py0 + 1 < cam.H);
        for (int b0 = start; b0 < end; b0 += NT) {
            if (__syncthreads_count(done0 && done1) == (int)blockDim.x) break;
#pragma unroll 1
            for (int u = 0; u < kFwdBatch; ++u) {
                const int k = tid + u * (int)blockDim.x;
                const int j = b0 + k;
                if (j < end) {
                    const Rec r = rec[ival[j]];
                    float4 a, b, c;
                    stage(r, ox, oy, a, b, c);
                    float4 *d = s_rec + kRecStage * k;
                    d[0] = a;
                    d[1] = b;
                    d[2] = make_float4(c.x, c.x, c.y, c.y);
                    d[3] = make_float4(c.z, c.z, c.w, c.w);
                    if (r.r3.z < 0.f) d[4] = fine_extra(r, ox, oy, a.x, a.y);
                }
            }
            __syncthreads();
            bool any_fine;
            const int nl = warp_offsets<false, false>(s_rec, min(NT, end - b0), band, wl, lane, any_fine, xmax, lg_amin);
            int lo0 = -1, lo1 = -1;  // offsets of the last records blended in this batch
            // blends one entry (alphas al) into the lane's pixels
            auto blend = [&](int off, f2 al, const float4 &c2, const float4 &c3) {
                const f2 nt = mul2(T2, add2(one2, neg2(al)));
                const bool act0 = lo2(al) >= o.alpha_min && !done0, act1 = hi2(al) >= o.alpha_min && !done1;
                const bool stop0 = lo2(nt) < o.t_min, stop1 = hi2(nt) < o.t_min;
                const bool bl0 = act0 && !stop0, bl1 = act1 && !stop1;
                const f2 w = mul2(al, T2);
                const f2 wm = pack2(bl0 ? lo2(w) : 0.f, bl1 ? hi2(w) : 0.f);
                C0 = fma2(wm, pack2(c2.x, c2.y), C0);
                C1 = fma2(wm, pack2(c2.z, c2.w), C1);
                C2 = fma2(wm, pack2(c3.x, c3.y), C2);
                D = fma2(wm, pack2(c3.z, c3.w), D);
                T2 = pack2(bl0 ? lo2(nt) : lo2(T2), bl1 ? hi2(nt) : hi2(T2));
                cnt0 += bl0;
                cnt1 += bl1;
                lo0 = bl0 ? off : lo0;
                lo1 = bl1 ? off : lo1;
                done0 |= act0 && stop0;
                done1 |= act1 && stop1;
            };
            auto alphas = [&](const float4 &a, const float4 &b) -> f2 {
                const float2 t0 = first_row(pxl, pyl[0], a, b);
                const f2 t12 = pack2(t0.x, t0.x + a.w), t22 = pack2(t0.y, t0.y + b.y);
                const f2 q = fma2(t12, t12, mul2(t22, t22));
                return pack2(fminf(o.alpha_max, b.z * ex2_approx(-lo2(q))),
                             fminf(o.alpha_max, b.z * ex2_approx(-hi2(q))));
            };
            if (!any_fine) {
                // kWalk entries at a time: their alphas, which do not depend on the
                // transmittance, before their blends
                int i = 0;
                for (; i + kWalk <= nl; i += kWalk) {
                    if (__all_sync(0xffffffffu, done0 && done1)) break;
                    int off[kWalk];
                    f2 al[kWalk];
#pragma unroll
                    for (int u = 0; u < kWalk; ++u) {
                        off[u] = wl[i + u];
                        const float4 *r = rec_at(s_rec, off[u]);
                        al[u] = alphas(r[0], r[1]);
                    }
#pragma unroll
                    for (int u = 0; u < kWalk; ++u) {
                        const float4 *r = rec_at(s_rec, off[u]);
                        blend(off[u], al[u], r[2], r[3]);
                    }
                }
                if (i + kWalk > nl)  // the last few (not after an early stop)
                    for (; i < nl; ++i) {
                        const float4 *r = rec_at(s_rec, wl[i]);
                        blend(wl[i], alphas(r[0], r[1]), r[2], r[3]);
                    }
            } else {
                // a batch with a near-degenerate record chooses the precision per entry
                for (int i = 0; i < nl; ++i) {
                    if (__all_sync(0xffffffffu, done0 && done1)) break;
                    const float4 *r = rec_at(s_rec, wl[i]);
                    const float4 a = r[0], b = r[1];
                    f2 al;
                    if (b.w < 0.f) {
                        const float4 f = r[4];
                        const PairEval e0 = eval_staged<true>(0, 0.f, 0.f, pxl, pyl[0], a, b, f, o.alpha_max);
                        const PairEval e1 = eval_staged<true>(1, 0.f, 0.f, pxl, pyl[1], a, b, f, o.alpha_max);
                        al = pack2(e0.alpha, e1.alpha);
                    } else {
                        al = alphas(a, b);
                    }
                    blend(wl[i], al, r[2], r[3]);
                }
            }
            if (lo0 >= 0) last0 = b0 - start + lo0 / (kRecStage * 16) + 1;
            if (lo1 >= 0) last1 = b0 - start + lo1 / (kRecStage * 16) + 1;
        }
        const int64_t HW = (int64_t)cam.H * cam.W;
#pragma unroll
        for (int q = 0; q < kPix; ++q) {
            const int py = py0 + q;
            if (!(px < cam.W && py < cam.H)) continue;
            const int64_t pix = (int64_t)tc.v * HW + (int64_t)py * cam.W + px;
            const float T = q ? hi2(T2) : lo2(T2);
            if (out.rgb) {
                float *rgb = out.rgb + (int64_t)tc.v * 3 * HW + (int64_t)py * cam.W + px;
                rgb[0] = fmaf(T, o.bg0, q ? hi2(C0) : lo2(C0));
                rgb[HW] = fmaf(T, o.bg1, q ? hi2(C1) : lo2(C1));
                rgb[2 * HW] = fmaf(T, o.bg2, q ? hi2(C2) : lo2(C2));
            }
            if (out.depth) out.depth[pix] = q ? hi2(D) : lo2(D);
            if (out.alpha) out.alpha[pix] = 1.f - T;
            out.t_final[pix] = T;
            if (out.n_contrib) out.n_contrib[pix] = q ? cnt1 : cnt0;
            out.n_iter[pix] = q ? last1 : last0;
        }
        if (!work) return;
        __syncthreads();
    }
}

// Transpose reduction of R values over a warp (R = 10: all 2D gradient slots;
// R = 6: the geometric ones).  Each halving step keeps ceil(R/2) live values
// per lane: one half of the lanes keeps the low slots, its partners the high
// slots, and each adds what the partner sent (5+3+2+1 shuffles for R = 10,
// 3+2+1 for R = 6), then the lane groups that hold the same slot are summed.
// Afterwards lane l holds the warp total of slot red_slot<R>(l) in v[0] (or
// nothing, red_slot = -1).
template <int R, int O, int N>
VPGS_D void half_step(float (&v)[N], int lane) {
    constexpr int S = (R + 1) / 2;
    const bool up = (lane & O) != 0;
#pragma unroll
    for (int i = 0; i < S; ++i) {
        const float lo = v[i];
        const float hi = (i + S < R) ? v[i + S] : 0.f;
        v[i] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, O);
    }
}

template <int R>
VPGS_D int red_slot(int lane) {
    int n = R, off = 0, r = R, bit = 16;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        if (r <= 1) break;
        const int S = (r + 1) / 2;
        if (lane & bit) {
            off += S;
            n = max(n - S, 0);
        } else {
            n = min(n, S);
        }
        r = S;
        bit >>= 1;
    }
    return (n >= 1 && (lane & (2 * bit - 1)) == 0) ? off : -1;
}

VPGS_D void warp_reduce(float (&a)[10], int lane) {
    half_step<10, 16>(a, lane);
    half_step<5, 8>(a, lane);
    half_step<3, 4>(a, lane);
    half_step<2, 2>(a, lane);
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
}

VPGS_D void warp_reduce(float (&a)[6], int lane) {
    half_step<6, 16>(a, lane);
    half_step<3, 8>(a, lane);
    half_step<2, 4>(a, lane);
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 2);
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
}

// 2D gradient slot [u, v, a, b, c, o, r, g, b, z] of accumulator q: the
// geometric form (NV = 6) keeps u, v, a, b, c and the depth z in q = 0..5
template <int NV>
VPGS_D int g2d_slot(int q) {
    return (NV == 6 && q == 5) ? 9 : q;
}

// per-pixel backward state
// beta = g . B: the upstream gradient (colour, depth) dotted with the colour /
// depth "behind" the current Gaussian, the only way B enters the gradient
struct PixState {
    float T, gAT, gC0, gC1, gC2, gD, beta;  // gAT = dL/dalpha_pixel * T_final
    int last;
};

// gradient of one pixel-Gaussian pair (Gaussian at list position jj), added to v;
// updates the pixel's transmittance and behind-colour; returns whether it blended.
// NV = 10: every 2D slot; NV = 6: only what the means, covariances and pose need
// (no opacity or colour sums), the form taken when no opacity or colour
// gradient is asked for
template <int NV>
VPGS_D bool pair_grad(PixState &p, int jj, const PairEval &e, const float4 &b, const float4 &c,
                      const OptParams &o, float (&v)[NV]) {
    if (jj >= p.last || e.alpha < o.alpha_min) return false;
    const float om = 1.f - e.alpha;
#if VPGS_BWD_RCP
    const float iom = __fdividef(1.f, om);  // om >= 1 - alpha_max > 0
    p.T *= iom;
    const float gat = p.gAT * iom;  // dA/dalpha_i = T_final / (1 - alpha_i)
#else
    p.T = p.T / om;
    const float gat = p.gAT / om;
#endif
    const float w = e.alpha * p.T;
    if constexpr (NV == 10) {
        v[6] = fmaf(w, p.gC0, v[6]);
        v[7] = fmaf(w, p.gC1, v[7]);
        v[8] = fmaf(w, p.gC2, v[8]);
        v[9] = fmaf(w, p.gD, v[9]);
    } else {
        v[5] = fmaf(w, p.gD, v[5]);
    }
    // dL/dalpha_i = T_i g . (c_i - B_i) + gat; behind this Gaussian
    // B <- B + alpha (c - B), so beta = g . B <- beta + alpha (g . c - beta)
    const float diff = fmaf(p.gC0, c.x, fmaf(p.gC1, c.y, fmaf(p.gC2, c.z, p.gD * c.w))) - p.beta;
    const float dA = fmaf(diff, p.T, gat);
    p.beta = fmaf(e.alpha, diff, p.beta);
    if (b.z * e.G <= o.alpha_max) {
        // slots 0-4 hold sums in the Gaussian's whitened frame t = W d, turned into
        // gradients once per Gaussian by the preprocess backward: sum dpow t1 and
        // sum dpow t2 for the mean (through the whitening rows and 2 ln 2), and
        // sum dpow t t^T (t1^2, t1 t2, t2^2) for the covariance (dL/dSigma' =
        // 2 ln^2 2 W^T S W).  t is O(1) where alpha matters, so these sums keep
        // their precision however elongated the Gaussian is.
        const float dpow = dA * e.alpha;
        if constexpr (NV == 10) v[5] = fmaf(dA, e.G, v[5]);
        const float pt1 = dpow * e.t1, pt2 = dpow * e.t2;
        v[0] += pt1;
        v[1] += pt2;
        v[2] = fmaf(pt1, e.t1, v[2]);
        v[3] = fmaf(pt1, e.t2, v[3]);
        v[4] = fmaf(pt2, e.t2, v[4]);
    }
    return true;
}

// ---------------------------------------------------------------------------
// Backward.  The ten 2D gradient sums of a Gaussian are linear in two numbers per
// pixel, its blend weight w and dpow (the gradient of the exponent):
//   sum w (g_r, g_g, g_b, g_z)   and   sum dpow (1, t1, t2, t1^2, t1 t2, t2^2)
// (sum dpow / o is the opacity's).  So a warp works in two phases:
//   1. one lane per column pair of pixels (two rows), as in the forward: walk the
//      list back to front, update T and beta, and leave (w, dpow) of both pixels in
//      a slot of shared memory.
//   2. after kSlots entries (or the list's end): kSlots x (32 / kSlots)
//      lanes, each summing one entry over its share of the warp's pixels in
//      registers, then log2(32 / kSlots) transpose steps and one global atomic per
//      (warp, Gaussian, slot).
// Both phases do their arithmetic on the two rows of a column at once with the
// packed FP32 instructions (fma.rn.f32x2), which round each half as the scalar
// ones do.  Lanes that do not blend take part with alpha = 0 (T and beta then keep
// their values exactly), so a step has no branch.
// Bound: the shared-memory pipe and latency (issue active 60 %, LSU data pipe 58 %, FMA
// pipe 42 %; 20 warps per SM).  103 warp instructions per listed entry, against 189 of
// the branching pair code and ten-value shuffle reduction it replaces.  Measured, old ->
// new: 1M-Gaussian room 1200x680 393 -> 280 us, 8 keyframes of 2M 1848 -> 1383 us, four
// full-HD views of 34k visible Gaussians 1111 -> 779 us, 10k Gaussians 320x240 41 -> 24 us.
// (16 entries halve the transpose steps but take 16 KB more per block: 322 us, room.)
// The shuffle form remains for near-degenerate records, entry by entry between the
// others, and for the batches with pixels or records whose magnitudes could turn 0 * x
// into a NaN (kOdd).  (With whole batches in it for one such record, 1920x1080, old -> so
// -> entry by entry: 100k flat discs 566 -> 618 -> 456 us, every 20th of 100k a disc
// 642 -> 494 -> 462, 100k elongated ones 450 -> 491 -> 366, 100k needles, whose long lists
// blend little, 260 -> 290 -> 312.)
//
// The geometric form (NV = 6: no opacity or colour gradient is asked, as in pose
// tracking) takes phase 1 without branches but sums each entry by shuffles, in the
// order and with the roundings it always had: 345 -> 289 us (room), 39 -> 29 us (10k
// Gaussians at 320x240).  Where a tile is one warp it gives the branching walk's bits;
// between warps only the order of the float32 atomics is open, as it was, and a tracking
// run feeds on its own roundings (the signs of the L1 loss near its minimum).  Ten tracked
// poses of the small scene differ from a run of the earlier kernel by 1.3e-10 in the median
// and 8.5e-7 at most, two runs of the earlier kernel by 1.2e-10 and 9.5e-7; of the room by
// 9.8e-9 and 1.7e-7, and 1.0e-8 and 1.8e-7.  The two-phase form took 250 us (room), but adds
// a warp's terms in another order: its runs leave that spread twice as often.
// ---------------------------------------------------------------------------
constexpr int kSlots = 8;
#ifndef VPGS_GEO_WALK
#define VPGS_GEO_WALK 2
#endif
constexpr int kGeoWalk = VPGS_GEO_WALK;  // entries whose alphas the geometric form evaluates at a time
#ifndef VPGS_BWD_DIRECT
#define VPGS_BWD_DIRECT 2
#endif
constexpr int kDirect = VPGS_BWD_DIRECT;  // at most this many active lanes: per-lane atomics, no reduction
#ifndef VPGS_BWD_UNROLL
#define VPGS_BWD_UNROLL 2
#endif
constexpr int kBwdUnroll = VPGS_BWD_UNROLL;
constexpr int kTermStride = 33;           // float4 per slot: 32 lanes, padded against bank conflicts
constexpr int kPixSize = 64 + 32 / kSlots;  // the lanes' gradients: 2 float4 each, one of padding per part of phase 2
// |upstream gradient| and |colour, depth| from which a pixel or record takes the
// branching walk: below it every product of the masked form stays finite
constexpr float kOdd = 1e15f;

static_assert(kPix == 2, "the packed forms hold two rows per lane");

// register cap (0: only the launch bound of the largest tile).  80: 6 blocks of 4 warps per
// SM, as many as the shared memory allows.  Room / 8 keyframes: 72 289 / 1437 us, 80 277 /
// 1379, 88 288 / 1450, 96 280 / 1412.  The full form spills 52 bytes a thread at 80 (-Xptxas
// -v; 36 loaded back) and 28 at 96, where one block less is resident.
#ifndef VPGS_BWD_MAXREG
#define VPGS_BWD_MAXREG 80
#endif
#if VPGS_BWD_MAXREG > 0
#define VPGS_BWD_BOUNDS __maxnreg__(VPGS_BWD_MAXREG)
#else
#define VPGS_BWD_BOUNDS __launch_bounds__(kMaxThreads)
#endif

template <int NV>
__global__ void VPGS_BWD_BOUNDS
composite_bwd_kernel(const Rec *__restrict__ rec, const uint32_t *__restrict__ ival,
                     const uint2 *__restrict__ ranges, const uint32_t *__restrict__ order, int n_tiles,
                     CamParams cam, OptParams o,
                     const float *__restrict__ t_final, const int32_t *__restrict__ n_iter,
                     const float *__restrict__ dL_drgb, const float *__restrict__ dL_ddepth,
                     const float *__restrict__ dL_dalpha, float *__restrict__ g2d,
                     const uint32_t *status, uint32_t *work) {
    grid_dep_enter();
    constexpr bool kGeo = NV == 6;
    constexpr int kTerm = kGeo ? 0 : kSlots * kTermStride, kPixN = kGeo ? 0 : kPixSize;  // float4 per warp
    extern __shared__ float4 smem[];
    constexpr int kBatch = NV == 6 ? kGeoBatch : kBwdBatch;
    const int NT = blockDim.x * kBatch;  // records per batch
    const int NW = blockDim.x >> 5;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // records: s0, s1 as in the forward, the colour and depth doubled (r, r, g, g), (b, b, z, z), the id
    float4 *s_rec = smem;
    float4 *s_term = smem + kRecStage * NT + warp * kTerm;              // this warp's (w, w, dpow, dpow)
    float4 *s_pix = smem + kRecStage * NT + NW * kTerm + warp * kPixN;  // this warp's -g
    uint16_t *wl = reinterpret_cast<uint16_t *>(smem + kRecStage * NT + NW * (kTerm + kPixN)) +
                   (size_t)warp * NT;  // this warp's list
    __shared__ int s_tile;
    __shared__ int s_max;
    __shared__ int s_odd;
    if (*status != 0u) return;
    const int lx = tid & (cam.tile_w - 1), ly = tid >> cam.tw_shift;
    const float pxl = (float)lx + 0.5f;
    float pyl[kPix];
#pragma unroll
    for (int q = 0; q < kPix; ++q) pyl[q] = (float)(kPix * ly + q) + 0.5f;
    const float2 band = warp_rows(cam);
    const float lg_amin = __log2f(o.alpha_min);
    const f2 one2 = pack2(1.f, 1.f);
    // adds the lanes' values of one entry to its slots: by a shuffle reduction, or where
    // few lanes blended by their own atomics
    const int red = red_slot<NV>(lane), slot = red >= 0 ? g2d_slot<NV>(red) : -1;
    auto add_sums = [&](uint32_t id, float (&v)[NV], bool act) {
        const uint32_t am = __ballot_sync(0xffffffffu, act);
        float *dst = g2d + 10 * (int64_t)id;
        if (am != 0u && __popc(am) <= kDirect) {
            if (act) {
#pragma unroll
                for (int q = 0; q < NV; ++q)
                    if (v[q] != 0.f) atomicAdd(dst + g2d_slot<NV>(q), v[q]);
            }
        } else if (am != 0u) {
            warp_reduce(v, lane);
            if (slot >= 0 && v[0] != 0.f) atomicAdd(dst + slot, v[0]);
        }
    };
    int t = blockIdx.x;
    for (;;) {
        if (work) {
            if (tid == 0) s_tile = (int)atomicAdd(work, 1u);
            __syncthreads();
            t = s_tile;
        }
        if (tid == 0) {
            s_max = 0;
            s_odd = 0;
        }
        __syncthreads();
        if (t >= n_tiles) return;
        const int tile = order ? (int)order[t] : t;  // launch order -> global tile id
        const uint2 rg = ranges[tile];
        // An empty list has no gradients, and its block leaves before the pixels' loads.  They
        // cost sparse calls 269 us (64 views of 640x480 with ten Gaussians, 76,800 tiles at six
        // blocks per SM); without them 97 us.  The forward's order load ahead of the status
        // (first_tile) took it from 187 to 179 us there, of which its images' bytes are 93 us.
        if (rg.y <= rg.x) {
            if (!work) return;
            continue;
        }
        const TileCoord tc = tile_coord(tile, cam);
        const int px = tc.tx * cam.tile_w + lx;
        const float ox = (float)(tc.tx * cam.tile_w), oy = (float)(tc.ty * cam.tile_h);
        const float xmax = fminf((float)cam.tile_w, (float)cam.W - ox) - 0.5f;  // last pixel centre column
        const int start = (int)rg.x;
        const int64_t HW = (int64_t)cam.H * cam.W;
        // per pixel: T, the negated upstream gradient ng, -dL/dalpha * T_final (ngat) and
        // beta = g . B, the upstream gradient dotted with the colour / depth behind the
        // current Gaussian (B starts at the background)
        float T[kPix], ng0[kPix], ng1[kPix], ng2[kPix], ngd[kPix], ngat[kPix], beta[kPix];
        int last[kPix];
        int my_max = 0;
        bool odd = false;
#pragma unroll
        for (int q = 0; q < kPix; ++q) {
            T[q] = 1.f;
            ng0[q] = ng1[q] = ng2[q] = ngd[q] = 0.f;
            last[q] = 0;
            float gA = 0.f;
            const int py = tc.ty * cam.tile_h + kPix * ly + q;
            if (px < cam.W && py < cam.H) {
                const int64_t pix = (int64_t)tc.v * HW + (int64_t)py * cam.W + px;
                T[q] = t_final[pix];
                last[q] = n_iter[pix];
                if (dL_drgb) {
                    const float *gp = dL_drgb + (int64_t)tc.v * 3 * HW + (int64_t)py * cam.W + px;
                    ng0[q] = -gp[0]; ng1[q] = -gp[HW]; ng2[q] = -gp[2 * HW];
                }
                if (dL_ddepth) ngd[q] = -dL_ddepth[pix];
                if (dL_dalpha) gA = dL_dalpha[pix];
            }
            ngat[q] = -(gA * T[q]);  // T holds T_final here
            beta[q] = -fmaf(ng0[q], o.bg0, fmaf(ng1[q], o.bg1, ng2[q] * o.bg2));
            odd |= !(fmaxf(fmaxf(fabsf(ng0[q]), fabsf(ng1[q])), fmaxf(fabsf(ng2[q]), fabsf(ngd[q]))) < kOdd) ||
                   !(fabsf(ngat[q]) < kOdd && fabsf(beta[q]) < kOdd) || ng0[q] != ng0[q] || ng1[q] != ng1[q] ||
                   ng2[q] != ng2[q] || ngd[q] != ngd[q];
            my_max = max(my_max, last[q]);
        }
        const bool warp_odd = __any_sync(0xffffffffu, odd);
        if constexpr (!kGeo) {
            s_pix[2 * lane + lane / kSlots] = make_float4(ng0[0], ng0[1], ng1[0], ng1[1]);
            s_pix[2 * lane + lane / kSlots + 1] = make_float4(ng2[0], ng2[1], ngd[0], ngd[1]);
        }
        f2 T2 = pack2(T[0], T[1]), beta2 = pack2(beta[0], beta[1]);
        const f2 ng02 = pack2(ng0[0], ng0[1]), ng12 = pack2(ng1[0], ng1[1]), ng22 = pack2(ng2[0], ng2[1]),
                 ngd2 = pack2(ngd[0], ngd[1]), ngat2 = pack2(ngat[0], ngat[1]);
        // the warp's own list length: warps whose pixels stop early skip the tail
        const int warp_max = (int)__reduce_max_sync(0xffffffffu, (unsigned)my_max);
        if (lane == 0 && warp_max > 0) atomicMax(&s_max, warp_max);
        __syncthreads();
        const int list_end = start + min(s_max, (int)rg.y - start);  // n_iter never exceeds the list
        for (int b1 = list_end; b1 > start; b1 -= NT) {
            const int b0 = max(start, b1 - NT);
            const int nb = b1 - b0;
            __syncthreads();
#pragma unroll 1
            for (int u = 0; u < kBatch; ++u) {
                const int k = tid + u * (int)blockDim.x;
                if (b0 + k < b1) {
                    const uint32_t id = ival[b0 + k];
                    float4 a, b, c;
                    stage(rec[id], ox, oy, a, b, c);
                    float4 *d = s_rec + kRecStage * k;
                    d[0] = a;
                    d[1] = b;
                    d[2] = make_float4(c.x, c.x, c.y, c.y);
                    d[3] = make_float4(c.z, c.z, c.w, c.w);
                    d[4].x = __uint_as_float(id);
                    if (!(fmaxf(fmaxf(fabsf(c.x), fabsf(c.y)), fmaxf(fabsf(c.z), fabsf(c.w))) < kOdd)) s_odd = 1;
                }
            }
            __syncthreads();
            const int k_end = min(nb, warp_max - (b0 - start));  // warp-uniform
            bool any_fine;
            const int nl = warp_offsets<true, true>(s_rec, k_end, band, wl, lane, any_fine, xmax, lg_amin);
            const int base = b0 - start;  // list position of the batch's first record
            const bool all_slow = warp_odd || s_odd != 0;
            // one entry in its precision form with branches, the warp's sums by shuffles
            auto branching = [&](int off) {
                const float4 *r = rec_at(s_rec, off);
                const int kk = off / (kRecStage * 16);
                const uint32_t id = __float_as_uint(r[4].x);
                const float4 a = r[0], b = r[1], c2 = r[2], c3 = r[3];
                const float4 c = make_float4(c2.x, c2.z, c3.x, c3.z);
                PixState ps[kPix];
#pragma unroll
                for (int q = 0; q < kPix; ++q) {
                    PixState &p = ps[q];
                    p.T = q ? hi2(T2) : lo2(T2);
                    p.beta = q ? hi2(beta2) : lo2(beta2);
                    p.gAT = -(q ? hi2(ngat2) : lo2(ngat2));
                    p.gC0 = -(q ? hi2(ng02) : lo2(ng02));
                    p.gC1 = -(q ? hi2(ng12) : lo2(ng12));
                    p.gC2 = -(q ? hi2(ng22) : lo2(ng22));
                    p.gD = -(q ? hi2(ngd2) : lo2(ngd2));
                    p.last = last[q];
                }
                float v[NV];
#pragma unroll
                for (int q = 0; q < NV; ++q) v[q] = 0.f;
                auto grads = [&](auto fine) -> bool {
                    constexpr bool kFine = decltype(fine)::value;
                    float4 f;
                    if constexpr (kFine) f = fine_extra(rec[id], ox, oy, a.x, a.y);
                    const float2 t0 = kFine ? make_float2(0.f, 0.f) : first_row(pxl, pyl[0], a, b);
                    bool any = false;
#pragma unroll
                    for (int q = 0; q < kPix; ++q) {
                        const PairEval e = eval_staged<kFine>(q, t0.x, t0.y, pxl, pyl[q], a, b, f, o.alpha_max);
                        any |= pair_grad(ps[q], base + kk, e, b, c, o, v);
                    }
                    return any;
                };
                const bool act = b.w < 0.f ? grads(std::true_type{}) : grads(std::false_type{});
                T2 = pack2(ps[0].T, ps[1].T);
                beta2 = pack2(ps[0].beta, ps[1].beta);
                add_sums(id, v, act);
            };
            if (all_slow || (kGeo && any_fine)) {  // warp-uniform
                for (int i = 0; i < nl; ++i) branching(wl[i]);
                continue;
            }
            // the offsets the pixels blend below (list positions clamped to the batch: a
            // position times the record size may not fit 32 bits)
            const int l0 = min(max(last[0] - base, 0), nb) * (kRecStage * 16),
                      l1 = min(max(last[1] - base, 0), nb) * (kRecStage * 16);
            // (blend weight, negated; dpow) of the lane's pixels for the record at off, zero
            // where a pixel does not blend; updates T and beta.  t12, t22: the whitened
            // coordinates of the two rows.  na: the negated alphas, masked; r: o G.
            auto alphas = [&](int off, const float4 &a, const float4 &b, f2 &t12, f2 &t22, f2 &r) -> f2 {
                const float2 t0 = first_row(pxl, pyl[0], a, b);
                t12 = pack2(t0.x, t0.x + a.w);
                t22 = pack2(t0.y, t0.y + b.y);
                const f2 q = fma2(t12, t12, mul2(t22, t22));
                r = pack2(b.z * ex2_approx(-lo2(q)), b.z * ex2_approx(-hi2(q)));
                const float al0 = fminf(o.alpha_max, lo2(r)), al1 = fminf(o.alpha_max, hi2(r));
                return pack2(al0 >= o.alpha_min && off < l0 ? -al0 : 0.f, al1 >= o.alpha_min && off < l1 ? -al1 : 0.f);
            };
            auto terms = [&](f2 na, f2 r, const float4 &c2, const float4 &c3, f2 &nw, f2 &dp) {
                const f2 om = add2(one2, na);  // 1 - alpha >= 1 - alpha_max > 0
#if VPGS_BWD_RCP
                const f2 iom = pack2(rcp_approx(lo2(om)), rcp_approx(hi2(om)));
                T2 = mul2(T2, iom);
                const f2 gat = mul2(ngat2, iom);
#else
                T2 = pack2(lo2(T2) / lo2(om), hi2(T2) / hi2(om));
                const f2 gat = pack2(lo2(ngat2) / lo2(om), hi2(ngat2) / hi2(om));
#endif
                // ed = g . (B - c); dL/dalpha_i = T_i g . (c_i - B_i) + dL/dalpha T_final / (1 - alpha_i)
                f2 ed = kGeo ? mul2(ngd2, pack2(c3.z, c3.w)) : fma2(ngd2, pack2(c3.z, c3.w), beta2);
                ed = fma2(ng02, pack2(c2.x, c2.y), fma2(ng12, pack2(c2.z, c2.w), fma2(ng22, pack2(c3.x, c3.y), ed)));
                if (kGeo) ed = add2(ed, beta2);
                const f2 ndA = fma2(ed, T2, gat);
                beta2 = fma2(na, ed, beta2);  // B <- B + alpha (c - B)
                nw = mul2(na, T2);
                const f2 d = mul2(ndA, na);
                // a clamped alpha has zero derivative
                dp = pack2(lo2(r) <= o.alpha_max ? lo2(d) : 0.f, hi2(r) <= o.alpha_max ? hi2(d) : 0.f);
            };
            if constexpr (kGeo) {
                // one entry after another: the six sums over the lane's two rows, then the warp's
                for (int i = 0; i < nl; i += kGeoWalk) {
                    f2 t12[kGeoWalk], t22[kGeoWalk], r[kGeoWalk], na[kGeoWalk];
                    int off[kGeoWalk];
#pragma unroll
                    for (int u = 0; u < kGeoWalk; ++u) {
                        off[u] = wl[min(i + u, nl - 1)];
                        const float4 *rc = rec_at(s_rec, off[u]);
                        na[u] = alphas(off[u], rc[0], rc[1], t12[u], t22[u], r[u]);
                    }
#pragma unroll
                    for (int u = 0; u < kGeoWalk; ++u) {
                        if (i + u >= nl) break;  // warp-uniform
                        const float4 *rc = rec_at(s_rec, off[u]);
                        f2 nw, dp;
                        terms(na[u], r[u], rc[2], rc[3], nw, dp);
                        const f2 pt1 = mul2(dp, t12[u]), pt2 = mul2(dp, t22[u]);
                        float v[NV];
                        v[0] = lo2(pt1) + hi2(pt1);
                        v[1] = lo2(pt2) + hi2(pt2);
                        v[2] = fmaf(hi2(pt1), hi2(t12[u]), lo2(pt1) * lo2(t12[u]));
                        v[3] = fmaf(hi2(pt1), hi2(t22[u]), lo2(pt1) * lo2(t22[u]));
                        v[4] = fmaf(hi2(pt2), hi2(t22[u]), lo2(pt2) * lo2(t22[u]));
                        v[5] = fmaf(hi2(nw), hi2(ngd2), lo2(nw) * lo2(ngd2));
                        add_sums(__float_as_uint(rc[4].x), v, lo2(na[u]) != 0.f || hi2(na[u]) != 0.f);
                    }
                }
                continue;
            } else {
            auto walk = [&](auto mix) {  // mix: the list holds near-degenerate records
            for (int g = 0; g < nl; g += kSlots) {
                const int n = min(kSlots, nl - g);  // warp-uniform
                // phase 1
                auto step = [&](int i) {
                    const int off = wl[g + i];
                    const float4 *rc = rec_at(s_rec, off);
                    f2 t12, t22, r, nw, dp;
                    const f2 na = alphas(off, rc[0], rc[1], t12, t22, r);
                    terms(na, r, rc[2], rc[3], nw, dp);
                    s_term[i * kTermStride + lane] = make_float4(lo2(nw), hi2(nw), lo2(dp), hi2(dp));
                };
                if constexpr (!decltype(mix)::value) {
#pragma unroll kBwdUnroll
                    for (int i = 0; i < n; ++i) step(i);
                } else {
                    // near-degenerate entries add their sums at once and leave no terms
#pragma unroll 1
                    for (int i = 0; i < n; ++i) {
                        const int off = wl[g + i];
                        if (rec_at(s_rec, off)[1].w < 0.f) {
                            s_term[i * kTermStride + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
                            branching(off);
                        } else {
                            step(i);
                        }
                    }
                }
                __syncwarp();
                // phase 2
                const int e = lane & (kSlots - 1), part = lane / kSlots;
                constexpr int kShare = kSlots;  // lanes (pixel pairs) of phase 1 per part: 32 / (32 / kSlots)
                const float4 *r = rec_at(s_rec, wl[g + (e < n ? e : 0)]);
                const float4 a = r[0], b = r[1];
                f2 v[NV];
#pragma unroll
                for (int q = 0; q < NV; ++q) v[q] = pack2(0.f, 0.f);
                const float4 *term = s_term + e * kTermStride + part * kShare;
                const float4 *pix = s_pix + (2 * kShare + 1) * part;
#pragma unroll
                for (int h = 0; h < kShare; h += 4) {
                    // four lanes in a row of the tile (tile_w is a multiple of 4)
                    const int j = part * kShare + h;
                    const float x0 = (float)(j & (cam.tile_w - 1)) + 0.5f;
                    const float dy = (float)(kPix * ((warp * 32 + j) >> cam.tw_shift)) + 0.5f - a.y;
                    const float y1 = a.w * dy, y2 = b.y * dy;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float4 tm = term[h + i];
                        const float dx = (x0 + (float)i) - a.x;
                        const float t1 = fmaf(a.z, dx, y1), t2 = fmaf(b.x, dx, y2);
                        const f2 t12 = pack2(t1, t1 + a.w), t22 = pack2(t2, t2 + b.y);
                        const f2 w = pack2(tm.x, tm.y), p = pack2(tm.z, tm.w);
                        const f2 pt1 = mul2(p, t12), pt2 = mul2(p, t22);
                        v[0] = add2(v[0], pt1);
                        v[1] = add2(v[1], pt2);
                        v[2] = fma2(pt1, t12, v[2]);
                        v[3] = fma2(pt1, t22, v[3]);
                        v[4] = fma2(pt2, t22, v[4]);
                        const float4 g0 = pix[2 * (h + i)], g1 = pix[2 * (h + i) + 1];
                        v[5] = add2(v[5], p);
                        v[6] = fma2(w, pack2(g0.x, g0.y), v[6]);
                        v[7] = fma2(w, pack2(g0.z, g0.w), v[7]);
                        v[8] = fma2(w, pack2(g1.x, g1.y), v[8]);
                        v[9] = fma2(w, pack2(g1.z, g1.w), v[9]);
                    }
                }
                // (rs[k] is slot kSlotOf[k]: the lanes that finish an entry then hold slots
                // 0 1 8 | 2 3 | 4 5 9 | 6 7)
                constexpr int kSlotOf[NV] = {0, 1, 8, 2, 3, 4, 5, 9, 6, 7};
                float rs[NV];
#pragma unroll
                for (int q = 0; q < NV; ++q) rs[q] = lo2(v[kSlotOf[q]]) + hi2(v[kSlotOf[q]]);
                rs[6] = __fdividef(rs[6], b.z);  // slot 5: dL/do = sum dpow / o
                // the parts' sums, the values spread over the lanes that held them
                constexpr int H = (NV + 1) / 2;
                static_assert(NV == 10 && kSlots == 8, "kSlotOf spreads ten slots over four lanes");
                half_step<NV, 16>(rs, lane);
                half_step<H, 8>(rs, lane);
                if (e < n) {
                    // A Gaussian's row in two instructions, of eight and of two slots: where every
                    // tile adds to the same few rows, the L2's work per 32-byte sector bounds the
                    // kernel.  One lane per three consecutive slots took three instructions of
                    // four scattered words: 500 Gaussians over all of 1920x1080 437 us, now 236
                    // (by a shuffle reduction per entry 234); room 276 -> 275 us.
                    const int p = (lane >> 4 & 1) * 2 + (lane >> 3 & 1);
                    float *row = g2d + 10 * (int64_t)__float_as_uint(r[4].x);
                    if (rs[0] != 0.f || rs[1] != 0.f)
                        atomicAdd(reinterpret_cast<float2 *>(row) + p, make_float2(rs[0], rs[1]));
                    if (!(p & 1) && rs[2] != 0.f) atomicAdd(row + 8 + (p >> 1), rs[2]);
                }
                __syncwarp();
            }
            };
            if (any_fine) walk(std::true_type{});
            else walk(std::false_type{});
            }
        }
        if (!work) return;
        __syncthreads();
    }
}

// dynamic shared memory of a compositing block of `threads` threads staging
// `records` per batch: the staged records (five float4 each) and the warps' lists; full
// backward also the warps' term slots and pixel gradients
static size_t list_bytes(int threads, int records) { return sizeof(uint16_t) * (size_t)(threads / 32) * records; }
static size_t fwd_smem(int threads, int records) {
    return sizeof(float4) * kRecStage * records + list_bytes(threads, records);
}
static size_t bwd_smem(int threads, int records, bool geometric_only) {
    const size_t per_warp = geometric_only ? 0 : kSlots * kTermStride + kPixSize;
    return sizeof(float4) * (kRecStage * (size_t)records + (size_t)(threads / 32) * per_warp) +
           list_bytes(threads, records);
}

static int persistent_grid(const void *kernel, int B, size_t smem, int per_sm, int n_tiles) {
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, B, smem);
    if (occ <= 0) occ = 1;
    const int g = device_sm_count() * std::min(occ, per_sm);
    return std::min(g, n_tiles);
}

cudaError_t launch_composite_fwd(const RenderWs &ws, const uint32_t *ival, int V,
                                 const CamParams &cam, const OptParams &o, const vpgs_images &out,
                                 int persistent_ctas, cudaStream_t s) {
    const int B = cam.tile_w * cam.tile_h / kPix;
    const int n_tiles = V * cam.T;
    const size_t sm = fwd_smem(B, B * kFwdBatch);
    uint32_t *work = nullptr;
    int grid = n_tiles;
    if (persistent_ctas > 0) {
        work = ws.counters + CNT_WORK;
        cudaError_t e = cudaMemsetAsync(work, 0, sizeof(uint32_t), s);
        if (e != cudaSuccess) return e;
        grid = persistent_grid((const void *)composite_fwd_kernel, B, sm, persistent_ctas, n_tiles);
    }
    if (grid == 0) return cudaSuccess;
    if (sm > 40 * 1024)
        cudaFuncSetAttribute((const void *)composite_fwd_kernel,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    VPGS_LAUNCH("composite_fwd", s,
                launch_k(composite_fwd_kernel, grid, B, sm, s, ws.rec, ival, ws.ranges,
                         tiles_ordered(n_tiles, cam) ? (const uint32_t *)ws.tile_order : nullptr, n_tiles, cam, o, out,
                         ws.status, work));
    return cudaGetLastError();
}

cudaError_t launch_composite_bwd(const RenderWs &ws, const uint32_t *ival, int V,
                                 const CamParams &cam, const OptParams &o, const vpgs_images &fwd,
                                 const float *dL_drgb, const float *dL_ddepth,
                                 const float *dL_dalpha, bool geometric_only, int persistent_ctas,
                                 cudaStream_t s) {
    const int B = cam.tile_w * cam.tile_h / kPix;
    const int n_tiles = V * cam.T;
    const auto kern = geometric_only ? composite_bwd_kernel<6> : composite_bwd_kernel<10>;
    const size_t sm = bwd_smem(B, B * (geometric_only ? kGeoBatch : kBwdBatch), geometric_only);
    // (the kernels' few static words count towards the default limit of 48 KB)
    if (sm > 40 * 1024)
        cudaFuncSetAttribute((const void *)kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    uint32_t *work = nullptr;
    int grid = n_tiles;
    if (persistent_ctas > 0) {
        work = ws.counters + CNT_WORK;
        cudaError_t e = cudaMemsetAsync(work, 0, sizeof(uint32_t), s);
        if (e != cudaSuccess) return e;
        grid = persistent_grid((const void *)kern, B, sm, persistent_ctas, n_tiles);
    }
    if (grid == 0) return cudaSuccess;
    VPGS_LAUNCH("composite_bwd", s,
                launch_k(kern, grid, B, sm, s, ws.rec, ival, ws.ranges,
                         tiles_ordered(n_tiles, cam) ? (const uint32_t *)ws.tile_order : nullptr, n_tiles, cam, o,
                         fwd.t_final, fwd.n_iter, dL_drgb, dL_ddepth, dL_dalpha, ws.g2d, ws.status, work));
    return cudaGetLastError();
}

}  // namespace vpgs
