// raster_bwd.cu -- adjoint of the per-tile compositing (stage d1).
//
// A warp walks its block's hits (raster_common.cuh) back to front from the
// last position any of its pixels takes part in, rebuilding T_i = T_{i+1} /
// (1 - alpha_i).  With X_i = gC.c_i + gD z_i + gO (the pixel's output
// gradients against entry i's channels) and the scalar suffix sum
//   S_i = sum_{j > i} X_j alpha_j T_j  (+ T_final gC.bg),
// the derivative of the pixel's loss with respect to alpha_i is
//   dL/dalpha_i = T_i X_i - S_i / (1 - alpha_i),
// so one scalar per pixel carries what the colour, depth and opacity
// suffix sums would.  The image-space gradient terms of an entry (moments of
// dL/dpower; r g b; z) are summed over a lane's pixels, then over the warp
// (flush_terms) and added to the Gaussian's row in global memory.  Alpha is the
// forward's expression (explicit roundings), so the blend decisions are the
// forward's; the rest of this file may contract a*b+c into fused multiply-adds.
#include "raster_bwd.cuh"

namespace pvg {

void launch_composite_bwd(const Params &p, cudaStream_t s) {
    if (p.total_tiles == 0) return;
    if (p.n_feat > 0) return launch_composite_feat_bwd(p, s);
    const WarpShape w = warp_shape(p, kBwdWide4, kBwdWide8);
    Params q = p;
    q.block_shift = w.shift;
    q.blocks_per_tile = w.blocks;
    const uint32_t grid = p.total_tiles * w.blocks;
    note_launch();
    if (w.px == 8) {
        if (p.aux) pdl_launch(k_composite_bwd<8, true, 0>, grid, 32, 0, s, q);
        else pdl_launch(k_composite_bwd<8, false, 0>, grid, 32, 0, s, q);
    } else if (w.px == 4) {
        if (p.aux) pdl_launch(k_composite_bwd<4, true, 0>, grid, 32, 0, s, q);
        else pdl_launch(k_composite_bwd<4, false, 0>, grid, 32, 0, s, q);
    } else {
        if (p.aux) pdl_launch(k_composite_bwd<2, true, 0>, grid, 32, 0, s, q);
        else pdl_launch(k_composite_bwd<2, false, 0>, grid, 32, 0, s, q);
    }
}

}  // namespace pvg
