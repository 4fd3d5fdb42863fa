// features_bwd.cu -- adjoint of the compositor with extra channels, and of
// the channel values.
//
// One walk serves colour and channels: X_i = gC.c_i + gD z_i + gO + gF.x_i
// carries the channels' effect on alpha, and dL/dx_i = sum gF w_i is
// accumulated per visible point.  k_feat_param_bwd then maps dL/dx to v,
// beta, l and the semantic vectors.
#include "raster_bwd.cuh"

namespace pvg {
namespace {

// dL/d(channel values) of each visible item -> v, beta, l, semantics
__global__ void k_feat_param_bwd(Params P) {
    pdl_enter();
    const uint32_t M = P.counters[0];
    for (uint32_t m = blockIdx.x * blockDim.x + threadIdx.x; m < M; m += gridDim.x * blockDim.x) {
        const uint32_t gid = P.sgid[m];
        const ViewDesc &V = P.views[view_of_item(P.views, P.n_views, gid)];
        const uint32_t i = gid - V.item_base;
        const float *gf = &P.gfeat[(size_t)m * P.n_feat];
        const float beta = V.beta[i], l = V.period[i];
        const float rho = __fdiv_rn(beta, l);
        float grho = 0.f;  // dL/drho
        int c = 0;
        if (P.feat_mask & kFeatVbar) {
            // v_bar = v exp(-rho / 2): d/dv = exp(-rho / 2), d/drho = -v_bar / 2
            const float w = expf(-0.5f * rho);
#pragma unroll
            for (int k = 0; k < 3; k++) {
                if (V.g_vel && gf[k] != 0.f) atomicAdd(V.g_vel + 3 * (size_t)i + k, gf[k] * w);
                grho -= 0.5f * gf[k] * V.vel[3 * (size_t)i + k] * w;
            }
            c = 3;
        }
        if (P.feat_mask & kFeatRho) {
            if (rho < 2.0f) grho += gf[c];
            c++;
        }
        if (grho != 0.f) {
            // rho = beta / l
            if (V.g_beta) atomicAdd(V.g_beta + i, grho / l);
            if (V.g_period) atomicAdd(V.g_period + i, -grho * beta / (l * l));
        }
        if ((P.feat_mask & kFeatSem) && V.g_sem)
            for (int k = 0; k < V.n_sem; k++)
                if (gf[c + k] != 0.f) atomicAdd(V.g_sem + (size_t)i * V.n_sem + k, gf[c + k]);
    }
}

}  // namespace

// Four pixels per lane from kFeatBwdWide blocks of 128 pixels per SM, as far
// as their output gradients fit the registers (32 channels); two below (23
// channels, four / two, before the arithmetic on channels was packed by them:
// 1920x1280 with 1.5M Gaussians 2.16 / 3.17 ms, 1242x800 with 100k 574 / 681
// us, 1242x375 with 300k 1,006 / 746 us; since then 1.83 ms, 451 and 706 us).
constexpr int kFeatBwdWide = 40, kFeatBwdWideGroups = 8;

void launch_composite_feat_bwd(const Params &p, cudaStream_t s) {
    const int groups = (p.n_feat + 3) / 4, pixels = p.tile_w * p.tile_h;
    const bool wide = groups <= kFeatBwdWideGroups && pixels >= 128 &&
                      (int64_t)p.total_tiles * pixels / 128 >= (int64_t)kFeatBwdWide * device_sm_count();
    Params q = p;
    q.block_shift = wide && p.tile_h < 16 ? 4 : 3;
    q.blocks_per_tile = (uint32_t)(pixels / (wide ? 128 : 64));
    const uint32_t grid = p.total_tiles * q.blocks_per_tile;
    note_launch();
    if (wide) {
        switch (groups) {
            case 1: pdl_launch(k_composite_bwd<4, true, 1>, grid, 32, 0, s, q); break;
            case 2: pdl_launch(k_composite_bwd<4, true, 2>, grid, 32, 0, s, q); break;
            case 3: pdl_launch(k_composite_bwd<4, true, 3>, grid, 32, 0, s, q); break;
            case 4: pdl_launch(k_composite_bwd<4, true, 4>, grid, 32, 0, s, q); break;
            case 5: pdl_launch(k_composite_bwd<4, true, 5>, grid, 32, 0, s, q); break;
            case 6: pdl_launch(k_composite_bwd<4, true, 6>, grid, 32, 0, s, q); break;
            case 7: pdl_launch(k_composite_bwd<4, true, 7>, grid, 32, 0, s, q); break;
            default: pdl_launch(k_composite_bwd<4, true, 8>, grid, 32, 0, s, q); break;
        }
        return;
    }
    switch (groups) {
        case 1: pdl_launch(k_composite_bwd<2, true, 1>, grid, 32, 0, s, q); break;
        case 2: pdl_launch(k_composite_bwd<2, true, 2>, grid, 32, 0, s, q); break;
        case 3: pdl_launch(k_composite_bwd<2, true, 3>, grid, 32, 0, s, q); break;
        case 4: pdl_launch(k_composite_bwd<2, true, 4>, grid, 32, 0, s, q); break;
        case 5: pdl_launch(k_composite_bwd<2, true, 5>, grid, 32, 0, s, q); break;
        case 6: pdl_launch(k_composite_bwd<2, true, 6>, grid, 32, 0, s, q); break;
        case 7: pdl_launch(k_composite_bwd<2, true, 7>, grid, 32, 0, s, q); break;
        case 8: pdl_launch(k_composite_bwd<2, true, 8>, grid, 32, 0, s, q); break;
        default: pdl_launch(k_composite_bwd<2, true, 9>, grid, 32, 0, s, q); break;
    }
}

void launch_feat_param_bwd(const Params &p, cudaStream_t s) {
    if (p.n_items == 0 || p.n_feat <= 0) return;
    note_launch();
    pdl_launch(k_feat_param_bwd, 4 * device_sm_count(), 256, 0, s, p);
}

}  // namespace pvg
