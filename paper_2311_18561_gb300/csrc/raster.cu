// raster.cu -- per-tile compositing (stage c).
//
// Sec. 3.1, Eq. 3 with the depth and opacity channels Sec. 3.1 renders
// beside colour: one warp per block of 32 PX pixels (raster_common.cuh),
// which walks its tile's sorted list front to back.  A pixel's weight is one
// SFU ex2,
//   alpha = min(0.99, o~ 2^(a' dx^2 + b' dx dy + c' dy^2)),
// with the conic pre-scaled by -log2(e).  A pixel skips alpha < 1/255, stops
// before a blend that would leave T < 1e-4, and accumulates C += c alpha T,
// D += z alpha T, O += alpha T.  Every pixel's arithmetic is the same
// expression whatever the tile and block shapes, so images are bit-identical
// across them.
#include <algorithm>
#include <climits>

#include "raster_fwd.cuh"

namespace pvg {
namespace {

// Work counts of the last forward: the number of list entries whose footprint
// box contains the pixel, up to and including the one that stopped it (the
// compositing work E), and the number of those with alpha >= 1/255 (blended,
// or stopping the pixel).  Every entry counts, so none is culled; a warp's
// records pass through shared memory, four pixels per lane share them (read by
// every lane for one pixel, 1920x1280 with 1.5M Gaussians: the whole call 665
// us, so 404 us).
template <int PX>
__global__ void __launch_bounds__(32) k_composite_stats(Params P) {
    pdl_enter();
    __shared__ RawRecords raw;
    __shared__ float4 s_a[32], s_b[32];  // (u, v, a', b'), (c', o~, half widths)
    const BlockGeom G = block_geom<PX>(P);
    const ViewDesc &V = *G.V;
    const int lane = threadIdx.x;
    const uint32_t len = G.r.y - G.r.x;
    const float fx = (float)G.px + 0.5f;
    float T[PX];
    uint32_t neval[PX], nblend[PX];
    bool done[PX], all = true;
#pragma unroll
    for (int p = 0; p < PX; p++) {
        T[p] = 1.0f;
        neval[p] = nblend[p] = 0;
        done[p] = !(G.px < V.W && G.py0 + p < V.H);
        all &= done[p];
    }
    uint32_t m = (uint32_t)lane < len ? P.pair_vals[G.r.x + lane] : kNoRecord;
    fetch_record(P, raw, m, lane);
    for (uint32_t base = 0; base < len && !__all_sync(0xffffffffu, all); base += 32) {
        wait_records();
        if (m != kNoRecord) {
            const float4 q[3] = {raw.q[0][lane], raw.q[1][lane], raw.q[2][lane]};
            float4 g, col;
            float2 c;
            record_terms(q, 0, g, c, col);
            s_a[lane] = g;
            s_b[lane] = make_float4(c.x, c.y, q[1].w, q[2].w);
        }
        __syncwarp();
        m = base + 32u + lane < len ? P.pair_vals[G.r.x + base + 32u + lane] : kNoRecord;
        fetch_record(P, raw, m, lane);
        const int cnt = (int)min(32u, len - base);
        for (int k = 0; k < cnt && !all; k++) {
            const float4 a = s_a[k], b = s_b[k];
            const float dx = __fsub_rn(fx, a.x);
            const FalloffColumn fc = falloff_column(a.z, a.w, dx);
            all = true;
#pragma unroll
            for (int p = 0; p < PX; p++) {
                if (done[p]) continue;
                const float dy = __fsub_rn((float)(G.py0 + p) + 0.5f, a.y);
                if (fabsf(dx) <= b.z && fabsf(dy) <= b.w) neval[p]++;
                const float al = __fmul_rn(b.y, ex2_approx(falloff_exp2(fc, b.x, dy)));
                if (al >= kAlphaMin) {
                    nblend[p]++;
                    const float Tn = __fsub_rn(T[p], __fmul_rn(fminf(kAlphaCap, al), T[p]));
                    done[p] = Tn < kTStop;
                    T[p] = Tn;
                }
                all &= done[p];
            }
        }
        __syncwarp();  // the next group restages
    }
    wait_records();  // a copy may still be under way when the walk ended early
    if (G.px >= V.W) return;
#pragma unroll
    for (int p = 0; p < PX; p++) {
        if (G.py0 + p >= V.H) break;
        const size_t pix = (size_t)(G.py0 + p) * V.W + G.px;
        P.pix_neval[V.pix_base + pix] = neval[p];
        P.pix_neval[P.total_pix + V.pix_base + pix] = nblend[p];
    }
}

}  // namespace

bool composite_supported(int tw, int th, int px) {
#define PVG_CHECK(W, H, X) if (tw == W && th == H && px == X) return true;
    PVG_TILE_CONFIGS(PVG_CHECK)
#undef PVG_CHECK
    return false;
}

// Pixels per lane and block shape of the compositing kernels.  More pixels
// per lane share an entry's work among more pixels; fewer make more and
// shorter walks, which a frame that cannot fill the SMs with wide blocks (or
// a tile of 64 pixels) needs.
WarpShape warp_shape(const Params &p, int wide4, int wide8) {
    const int pixels = p.tile_w * p.tile_h;
    const int64_t all = (int64_t)p.total_tiles * pixels, sms = device_sm_count();
    WarpShape w;
    w.px = p.tile_w >= 16 && p.tile_h >= 16 && all / 256 >= wide8 * sms ? 8
           : pixels >= 128 && all / 128 >= wide4 * sms                  ? 4
                                                                        : 2;
    w.shift = w.px == 8 || (w.px == 4 && p.tile_h < 16) ? 4 : 3;
    w.blocks = (uint32_t)(pixels / (32 * w.px));
    return w;
}

static Params with_shape(const Params &p, const WarpShape &w) {
    Params q = p;
    q.block_shift = w.shift;
    q.blocks_per_tile = w.blocks;
    return q;
}

// One pixel per lane: where four would not fill the SMs (warp_shape gives
// two), and the lists are short.  With long lists the instructions of all blocks
// bound the pass, the sooner the more blocks the SMs have; with hardly any
// entries the blocks themselves do.  Measured with two / one pixel per lane, by items per
// block of 128 pixels, at 16 blocks per SM (641x479): 8: 23 / 20 us, 104: 95 /
// 84, 416: 54 / 56; at 24 (1242x375): 16: 47 / 43, 69: 122 / 93, 137: 67 / 70,
// 275: 71 / 80; at 46 (1000x900): 3: 25 / 29, 8: 43 / 41, 36: 86 / 78, 71: 78
// / 95.  The line lies below the smallest loss: where few entries stop the
// pixels, more items would still gain (four 640x480 views, 60 blocks per SM,
// 110 items per block: 186 / 156), but their number does not tell.
static bool one_pixel(const Params &p) {
    const int64_t blocks = (int64_t)p.total_tiles * p.tile_w * p.tile_h / 128, sms = device_sm_count();
    const int64_t items = p.n_items, full = 32 * sms;
    return items >= 8 * blocks && items * std::max(blocks, full) <= 96 * blocks * full;
}

void launch_composite(const Params &p, cudaStream_t s) {
    if (p.total_tiles == 0) return;
    if (p.n_feat > 0) return launch_composite_feat(p, s);
    WarpShape w = warp_shape(p, kFwdWide, INT_MAX);
    if (w.px == 2 && one_pixel(p)) w = WarpShape{1, 3, (uint32_t)(p.tile_w * p.tile_h / 32)};
    const Params q = with_shape(p, w);
    note_launch();
    if (w.px == 1) pdl_launch(k_composite1<kFwdUnroll1>, p.total_tiles * w.blocks, 32, 0, s, q);
    else if (w.px == 4) pdl_launch(k_composite<4, 0>, p.total_tiles * w.blocks, 32, 0, s, q);
    else pdl_launch(k_composite<2, 0>, p.total_tiles * w.blocks, 32, 0, s, q);
}

void launch_composite_stats(const Params &p, cudaStream_t s) {
    if (p.total_tiles == 0) return;
    const WarpShape w = warp_shape(p, 0, INT_MAX);  // four pixels per lane, two in a tile of 64
    const Params q = with_shape(p, w);
    note_launch();
    if (w.px == 4) pdl_launch(k_composite_stats<4>, p.total_tiles * w.blocks, 32, 0, s, q);
    else pdl_launch(k_composite_stats<2>, p.total_tiles * w.blocks, 32, 0, s, q);
}

}  // namespace pvg
