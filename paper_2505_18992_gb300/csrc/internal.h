// Host-side declarations shared by the translation units of libvpgs.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "common.cuh"

namespace vpgs {

struct CamParams {
    int W, H;
    float fx, fy, cx, cy;
    int tile_w, tile_h, tiles_x, tiles_y, T;  // T = tiles per view
    int tw_shift;                             // log2(tile_w)
};

struct OptParams {
    float alpha_min, alpha_max, t_min, dilation, near_z;
    float bg0, bg1, bg2;
    int spin_limit;  // polls of a look-back wait before VPGS_ERR_TIMEOUT
};

struct GaussIn {
    const float *means, *scales, *quats, *opac, *colors;
    int64_t N;
    const int32_t *n_dev;
};

struct GaussGrad {
    float *means, *scales, *quats, *opac, *colors;
};

int device_sm_count();

// Which form the binning of a call takes (render_bin.cu): its general one, or for small
// calls the ranking by comparison, with tile lists by selection (kSmallLists) or by the
// general emission and sort (kSmallRank).  The small forms cost pairs^2 and pairs x tiles;
// the lines lie where their measured forward met the general one's with every pair
// visible (us, small / general): 12,288 pairs x 300 tiles 65 / 75, x 1,200 85 / 94,
// x 1,900 99 / 96; 5,000 pairs x 300 tiles 33 / 65, 1,000 22 / 52.  By rank alone (7,500
// tiles): 3,000 pairs 88 / 106, 6,000 107 / 121, 8,000 125 / 127, 10,000 142 / 136, 12,000
// 165 / 144, so the line stays below where they meet.
enum BinForm { kGeneralBin, kSmallRank, kSmallLists };
constexpr int64_t kSmallPairs = 12288;       // (below 2^14: a pair fits 16 bits beside its view)
constexpr int64_t kSmallRankPairs = 6144;
constexpr int64_t kSmallProduct = 15000000;  // pairs x tiles
inline BinForm bin_form(const RenderLayout &L) {
    const int64_t tiles = (int64_t)L.V * L.T;
    // (four bytes of a tile rectangle, 16 bits of a view)
    if (L.VN <= kSmallPairs && L.VN * tiles <= kSmallProduct && L.tiles_x <= 256 && L.tiles_y <= 256 && L.V <= 65535)
        return kSmallLists;
    return L.VN <= kSmallRankPairs ? kSmallRank : kGeneralBin;
}

// The visible (view, Gaussian) pairs of a small call, in any order, as the projection
// appends them: depth key, tile count, pair index.  They lie in the depth sort's
// buffers, which such a call does not use; NULL otherwise.
struct SmallList {
    uint32_t *key, *cnt, *pair;
};
inline SmallList small_list(const RenderWs &ws, const RenderLayout &L) {
    if (bin_form(L) == kGeneralBin) return SmallList{nullptr, nullptr, nullptr};
    return SmallList{ws.dkey[0], ws.dval[0], ws.dval[1]};
}

// render_pre.cu
// First launches of a render call: the prepare kernel (zeroes status, counters
// and the scratch later kernels expect at zero; converts the poses), the
// pre-cull and the exact projection.
cudaError_t launch_preprocess_fwd(const GaussIn &g, const double *T_cw, int V, const CamParams &cam,
                                  const OptParams &o, const RenderWs &ws, const RenderLayout &L,
                                  bool zero_g2d, cudaStream_t s);
cudaError_t launch_export_projection(const RenderWs &ws, int64_t VN, int32_t *tile_count,
                                     int32_t *tile_rect, float *mean2d, float *depth, float *conic,
                                     cudaStream_t s);
cudaError_t launch_preprocess_bwd(const GaussIn &g, const double *T_cw, int V, const CamParams &cam,
                                  const OptParams &o, const RenderWs &ws, const GaussGrad &gg,
                                  double *dpose, cudaStream_t s);

// render_bin.cu: visibility compaction, depth sort, instance emission, tile
// sort and tile ranges.  On return ws.ival[*sorted_buf] holds the tile lists.
cudaError_t build_tile_lists(const GaussIn &g, int V, const CamParams &cam, const OptParams &o, const RenderWs &ws,
                             const RenderLayout &L, int *sorted_buf, cudaStream_t s, bool order_by_count = true);
// Compositing launch order from the forward's n_iter: tiles by the backward's
// list steps, most first (ws.tile_work, ws.tile_order).
cudaError_t order_tiles_by_steps(const RenderWs &ws, const int32_t *n_iter, int V, const CamParams &cam,
                                 cudaStream_t s);
// Whether calls of n_tiles tiles use a launch order (ws.tile_order) at all.
bool tiles_ordered(int n_tiles, const CamParams &cam);
// Which ival buffer build_tile_lists leaves the tile lists in (host only, no launch).
int tile_list_buffer(const RenderLayout &L);

// render_comp.cu
cudaError_t launch_composite_fwd(const RenderWs &ws, const uint32_t *ival, int V,
                                 const CamParams &cam, const OptParams &o, const vpgs_images &out,
                                 int persistent_ctas, cudaStream_t s);
cudaError_t launch_composite_bwd(const RenderWs &ws, const uint32_t *ival, int V,
                                 const CamParams &cam, const OptParams &o, const vpgs_images &fwd,
                                 const float *dL_drgb, const float *dL_ddepth,
                                 const float *dL_dalpha, bool geometric_only, int persistent_ctas,
                                 cudaStream_t s);

// pose.cu
cudaError_t launch_pose_step(double *T_cw, double *dpose, double *adam, int V, double lr_rho,
                             double lr_phi, cudaStream_t s);

}  // namespace vpgs
