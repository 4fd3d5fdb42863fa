// features.cu -- the compositor with extra channels: the velocity, staticness
// and semantic maps (the adjoint is in features_bwd.cu).
//
// Each channel is a per-point value x_i composited with the colour's
// weights w_i = T_i alpha_i and no background:
//   v_bar = v exp(-rho / 2), rho = beta / l (Eq. 10)   velocity map, 3 ch.
//   min(rho, 2)                                         staticness map, 1 ch.
//   the point's semantic vector                         semantic map, n_sem ch.
// (Sec. 4: dynamic-element analysis and semantic rendering.)
//
// One pass composites colour, depth, opacity and the channels: the walk, the
// alphas and the weights are the colour pass's, the channels add one fused
// multiply-add per blend each.
#include "raster_fwd.cuh"

namespace pvg {

int feat_count(int mask, int n_sem) {
    return ((mask & kFeatVbar) ? 3 : 0) + ((mask & kFeatRho) ? 1 : 0) + ((mask & kFeatSem) ? n_sem : 0);
}

// Four pixels per lane from kFeatWide blocks of 128 pixels per SM, as far as
// their sums fit the registers (24 channels); two below, where the longest
// walk bounds the pass (23 channels, four / two: 1920x1280 with 1.5M
// Gaussians 708 / 1033 us, 1242x800 with 100k 169 / 209, 1242x375 with 300k
// 577 / 400, 640x480 with 200k 408 / 227; packed by channels since: 654, 158,
// 368 and 210).
constexpr int kFeatWide = 40, kFeatWideGroups = 6;

void launch_composite_feat(const Params &p, cudaStream_t s) {
    const int groups = (p.n_feat + 3) / 4, pixels = p.tile_w * p.tile_h;
    const bool wide = groups <= kFeatWideGroups && pixels >= 128 &&
                      (int64_t)p.total_tiles * pixels / 128 >= (int64_t)kFeatWide * device_sm_count();
    Params q = p;
    q.block_shift = wide && p.tile_h < 16 ? 4 : 3;
    q.blocks_per_tile = (uint32_t)(pixels / (wide ? 128 : 64));
    const uint32_t grid = p.total_tiles * q.blocks_per_tile;
    note_launch();
    if (wide) {
        switch (groups) {
            case 1: pdl_launch(k_composite<4, 1>, grid, 32, 0, s, q); break;
            case 2: pdl_launch(k_composite<4, 2>, grid, 32, 0, s, q); break;
            case 3: pdl_launch(k_composite<4, 3>, grid, 32, 0, s, q); break;
            case 4: pdl_launch(k_composite<4, 4>, grid, 32, 0, s, q); break;
            case 5: pdl_launch(k_composite<4, 5>, grid, 32, 0, s, q); break;
            default: pdl_launch(k_composite<4, 6>, grid, 32, 0, s, q); break;
        }
        return;
    }
    switch (groups) {
        case 1: pdl_launch(k_composite<2, 1>, grid, 32, 0, s, q); break;
        case 2: pdl_launch(k_composite<2, 2>, grid, 32, 0, s, q); break;
        case 3: pdl_launch(k_composite<2, 3>, grid, 32, 0, s, q); break;
        case 4: pdl_launch(k_composite<2, 4>, grid, 32, 0, s, q); break;
        case 5: pdl_launch(k_composite<2, 5>, grid, 32, 0, s, q); break;
        case 6: pdl_launch(k_composite<2, 6>, grid, 32, 0, s, q); break;
        case 7: pdl_launch(k_composite<2, 7>, grid, 32, 0, s, q); break;
        case 8: pdl_launch(k_composite<2, 8>, grid, 32, 0, s, q); break;
        default: pdl_launch(k_composite<2, 9>, grid, 32, 0, s, q); break;
    }
}

}  // namespace pvg
