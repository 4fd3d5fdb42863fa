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
#include <climits>

#include "raster_common.cuh"

namespace pvg {
namespace {

// Entries whose alphas are evaluated together, before the chain of their
// transmittances: a lone warp (the longest walk of a frame, the small
// frames) waits on latencies, which four independent evaluations overlap
// (two 641x479-sized views of 250k Gaussians: 350 us with 2, 280 us with 4).
constexpr int kFwdUnroll = 4;
// Resident warps per SM that the registers are held to, by pixels per lane:
// without spills (16 warps of 128 registers against 20 of 96: 280 and 310 us
// on those views, 193 and 195 us on the 1.5M-Gaussian 1920x1280 frame).
constexpr int kFwdWarps4 = 16, kFwdWarps2 = 20;
// Blocks of 128 pixels per SM from which a lane takes four pixels and not
// two: below it the longest walk bounds the pass and two pixels per lane
// shorten it (9,100 blocks: 186 us with two, 280 us with four); above it the
// issue slots do (19,200 blocks: 243 and 193 us).
constexpr int kFwdWide = 64;

// Writes the images (and the saved per-pixel state) of a thread's PX pixels.
template <int PX>
__device__ __forceinline__ void composite_epilogue(const Params &P, const ViewDesc &V, const BlockGeom &G,
                                                   const float (&T)[PX], const float (&C0)[PX],
                                                   const float (&C1)[PX], const float (&C2)[PX],
                                                   const float (&D)[PX], const float (&O)[PX],
                                                   const uint32_t (&last)[PX]) {
    if (G.px >= V.W) return;
    const size_t HW = (size_t)V.W * V.H;
#pragma unroll
    for (int p = 0; p < PX; p++) {
        const int py = G.py0 + p;
        if (py >= V.H) break;
        const size_t pix = (size_t)py * V.W + G.px;
        if (V.sky) {  // C + (1 - O) f_sky(d)
            size_t ti[4];
            float tw[4];
            sky_texels(V, G.px, py, ti, tw);
            float f[3];
#pragma unroll
            for (int c = 0; c < 3; c++)
                f[c] = tw[0] * V.sky[ti[0] + c] + tw[1] * V.sky[ti[1] + c] + tw[2] * V.sky[ti[2] + c] +
                       tw[3] * V.sky[ti[3] + c];
            const float wo = 1.0f - O[p];
            V.out_rgb[pix] = C0[p] + wo * f[0];
            V.out_rgb[HW + pix] = C1[p] + wo * f[1];
            V.out_rgb[2 * HW + pix] = C2[p] + wo * f[2];
        } else {
            V.out_rgb[pix] = C0[p] + T[p] * V.bg[0];
            V.out_rgb[HW + pix] = C1[p] + T[p] * V.bg[1];
            V.out_rgb[2 * HW + pix] = C2[p] + T[p] * V.bg[2];
        }
        if (V.out_depth) V.out_depth[pix] = D[p];
        if (V.out_alpha) V.out_alpha[pix] = O[p];
        if (P.pix_T) {
            P.pix_T[V.pix_base + pix] = T[p];
            P.pix_last[V.pix_base + pix] = last[p];
        }
    }
}

// The compositor: a warp walks its block's hits front to back, its pixels as
// packed pairs of vertically adjacent ones (the falloff, alpha,
// transmittance and accumulation of both take one .f32x2 instruction each).
// A pixel that does not blend (alpha < 1/255, stopped, outside the image)
// has its alpha zeroed: its weight is then 0 and its T and sums keep their
// bits, so a warp takes no branch per pixel; entries with non-finite terms,
// for which 0 weights would not do, take the one-pixel-at-a-time path.  The
// sums are kept negated (the weight is -alpha T), which packed arithmetic
// needs no negation for.
template <int PX>
__global__ void __launch_bounds__(32, PX == 4 ? kFwdWarps4 : kFwdWarps2) k_composite(Params P) {
    pdl_enter();
    static_assert(PX % 2 == 0, "pairs of pixels");
    constexpr int NP = PX / 2, U = kFwdUnroll;
    constexpr uint32_t ALL = (1u << PX) - 1u;
    __shared__ RawRecords raw;
    __shared__ Staged S;
    const int lane = threadIdx.x;
    const BlockGeom G = block_geom<PX>(P);
    const ViewDesc &V = *G.V;
    const uint2 r = G.r;
    const float fx = (float)G.px + 0.5f;
    const float2 nzero2 = make_float2(-0.0f, -0.0f);
    float2 fy[NP], T[NP], C0[NP], C1[NP], C2[NP], D[NP], O[NP];
    uint32_t last[PX];  // list position where the pixel stopped (else the list's length)
    uint32_t done = 0;
#pragma unroll
    for (int q = 0; q < NP; q++) {
        fy[q] = make_float2((float)(G.py0 + 2 * q) + 0.5f, (float)(G.py0 + 2 * q + 1) + 0.5f);
        T[q] = make_float2(1.0f, 1.0f);
        C0[q] = C1[q] = C2[q] = D[q] = O[q] = nzero2;
    }
    const uint32_t len = r.y - r.x;
#pragma unroll
    for (int p = 0; p < PX; p++) {
        last[p] = len;
        if (!(G.px < V.W && G.py0 + p < V.H)) {
            last[p] = 0;
            done |= 1u << p;
        }
    }
    // A pixel that is done (stopped, or outside the image) gets a row
    // coordinate far away: its falloff exponent is then -inf or NaN, its
    // alpha 0 or NaN, and the alpha test (false for NaN) never passes again.
    auto far_rows = [&]() {
#pragma unroll
        for (int q = 0; q < NP; q++) {
            if (done & (1u << (2 * q))) fy[q].x = kFarRow;
            if (done & (2u << (2 * q))) fy[q].y = kFarRow;
        }
    };
    far_rows();
    uint32_t m0 = lane < len ? P.pair_vals[r.x + lane] : kNoRecord;
    fetch_record(P, raw, m0, lane);
    uint32_t m1 = lane + 32u < len ? P.pair_vals[r.x + 32u + lane] : kNoRecord;
    bool finished = __all_sync(0xffffffffu, done == ALL);
    for (uint32_t base = 0; base < len && !finished; base += 32) {
        wait_records();
        const int hits = stage_hits<U>(raw, S, m0 != kNoRecord, m0, base + lane, G, lane);
        m0 = m1;
        fetch_record(P, raw, m0, lane);
        m1 = base + 64u + lane < len ? P.pair_vals[r.x + base + 64u + lane] : kNoRecord;
        for (int k = 0; k < hits; k += U) {
            // alphas of U entries (negated, -0 where a pixel does not blend)
            float2 na[U][NP];
            uint32_t pos[U];
#pragma unroll
            for (int u = 0; u < U; u++) {
                const float4 A = S.a[k + u], B = S.b[k + u];
                const float2 no2 = reinterpret_cast<const float2 *>(&S.c[k + u])[0];
                pos[u] = __float_as_uint(A.w);
                const float dx = __fsub_rn(fx, A.x);
                const FalloffColumn fc = falloff_column(A.y, A.z, dx);
                const float2 A2 = make_float2(fc.A, fc.A), B2 = make_float2(fc.B, fc.B);
                const float2 v2 = make_float2(B.x, B.y), cp2 = make_float2(B.z, B.w);
#pragma unroll
                for (int q = 0; q < NP; q++) {
                    const float2 e = falloff_exp2_x2(A2, B2, cp2, sub2(fy[q], v2));
                    const float2 nr = mul2(no2, make_float2(ex2_approx(e.x), ex2_approx(e.y)));
                    na[u][q] = make_float2(nr.x <= -kAlphaMin ? nr.x : -0.0f, nr.y <= -kAlphaMin ? nr.y : -0.0f);
                }
            }
            uint32_t flags = pos[0];
#pragma unroll
            for (int u = 1; u < U; u++) flags |= pos[u];
            if (flags > kPosMask) {
                // o~ may exceed the cap (one that cannot is left as it is)
#pragma unroll
                for (int u = 0; u < U; u++)
#pragma unroll
                    for (int q = 0; q < NP; q++)
                        na[u][q] = make_float2(fmaxf(na[u][q].x, -kAlphaCap), fmaxf(na[u][q].y, -kAlphaCap));
                if (flags & kOddEntry) {  // non-finite terms: one pixel at a time
#pragma unroll
                    for (int u = 0; u < U; u++) {
                        const float col[4] = {S.c[k + u].z, S.d[k + u].x, S.d[k + u].z, S.e[k + u].x};
                        auto one = [&](float nal, float &t, float &c0, float &c1, float &c2, float &d, float &o, int p) {
                            if (!(nal < 0.0f) || (done & (1u << p))) return;
                            const float nw = __fmul_rn(nal, t), tn = __fadd_rn(t, nw);
                            if (tn < kTStop) {
                                done |= 1u << p;
                                last[p] = pos[u] & kPosMask;
                                return;
                            }
                            c0 = __fmaf_rn(col[0], nw, c0);
                            c1 = __fmaf_rn(col[1], nw, c1);
                            c2 = __fmaf_rn(col[2], nw, c2);
                            d = __fmaf_rn(col[3], nw, d);
                            o = __fadd_rn(o, nw);
                            t = tn;
                        };
#pragma unroll
                        for (int q = 0; q < NP; q++) {
                            one(na[u][q].x, T[q].x, C0[q].x, C1[q].x, C2[q].x, D[q].x, O[q].x, 2 * q);
                            one(na[u][q].y, T[q].y, C0[q].y, C1[q].y, C2[q].y, D[q].y, O[q].y, 2 * q + 1);
                        }
                    }
                    far_rows();
                    if (__all_sync(0xffffffffu, done == ALL)) {
                        finished = true;
                        break;
                    }
                    continue;
                }
            }
            // weights; T only falls, so a pixel stops in these entries exactly
            // if its T after the last of them is below the stop
            float2 nw[U][NP], Tn[NP];
            bool stop = false;
#pragma unroll
            for (int q = 0; q < NP; q++) {
                Tn[q] = T[q];
#pragma unroll
                for (int u = 0; u < U; u++) {
                    nw[u][q] = mul2(na[u][q], Tn[q]);
                    Tn[q] = add2(Tn[q], nw[u][q]);
                }
                stop |= Tn[q].x < kTStop || Tn[q].y < kTStop;
            }
            const bool any_stop = __any_sync(0xffffffffu, stop);
            if (any_stop) {
                // a pixel takes no part from the entry that would stop it on
                auto stopping = [&](float t, float &tn, auto weight, int p) {
                    if (!(tn < kTStop)) return;
                    bool off = false;
#pragma unroll
                    for (int u = 0; u < U; u++) {
                        float &w = weight(u);
                        if (!off && __fadd_rn(t, w) < kTStop) {
                            off = true;
                            done |= 1u << p;
                            last[p] = pos[u] & kPosMask;
                        }
                        if (off) w = -0.0f;
                        t = __fadd_rn(t, w);
                    }
                    tn = t;
                };
#pragma unroll
                for (int q = 0; q < NP; q++) {
                    stopping(T[q].x, Tn[q].x, [&](int u) -> float & { return nw[u][q].x; }, 2 * q);
                    stopping(T[q].y, Tn[q].y, [&](int u) -> float & { return nw[u][q].y; }, 2 * q + 1);
                }
                far_rows();
            }
#pragma unroll
            for (int u = 0; u < U; u++) {
                const float2 r2 = reinterpret_cast<const float2 *>(&S.c[k + u])[1], z2 = S.e[k + u];
                const float4 Dq = S.d[k + u];
                const float2 g2 = make_float2(Dq.x, Dq.y), b2 = make_float2(Dq.z, Dq.w);
#pragma unroll
                for (int q = 0; q < NP; q++) {
                    C0[q] = fma2(r2, nw[u][q], C0[q]);
                    C1[q] = fma2(g2, nw[u][q], C1[q]);
                    C2[q] = fma2(b2, nw[u][q], C2[q]);
                    D[q] = fma2(z2, nw[u][q], D[q]);
                    O[q] = add2(O[q], nw[u][q]);
                }
            }
#pragma unroll
            for (int q = 0; q < NP; q++) T[q] = Tn[q];
            if (any_stop && __all_sync(0xffffffffu, done == ALL)) {
                finished = true;
                break;
            }
        }
        __syncwarp();  // the next group restages
    }
    wait_records();  // a copy may still be under way when the walk ended early
    float Ts[PX], C0s[PX], C1s[PX], C2s[PX], Ds[PX], Os[PX];
#pragma unroll
    for (int q = 0; q < NP; q++) {
        Ts[2 * q] = T[q].x; Ts[2 * q + 1] = T[q].y;
        C0s[2 * q] = -C0[q].x; C0s[2 * q + 1] = -C0[q].y;
        C1s[2 * q] = -C1[q].x; C1s[2 * q + 1] = -C1[q].y;
        C2s[2 * q] = -C2[q].x; C2s[2 * q + 1] = -C2[q].y;
        Ds[2 * q] = -D[q].x; Ds[2 * q + 1] = -D[q].y;
        Os[2 * q] = -O[q].x; Os[2 * q + 1] = -O[q].y;
    }
    composite_epilogue<PX>(P, V, G, Ts, C0s, C1s, C2s, Ds, Os, last);
    if (P.tile_walk) {  // how far the tile's adjoint walks, for its launch order
        uint32_t w = last[0];
#pragma unroll
        for (int p = 1; p < PX; p++) w = max(w, last[p]);
        w = __reduce_max_sync(0xffffffffu, w);
        if (lane == 0 && w) atomicMax(&P.tile_walk[G.tile], w);
    }
}

// Work counts of the last forward, one pixel per thread: the number of list
// entries whose footprint box contains the pixel, up to and including the
// one that stopped it (the compositing work E), and the number of those with
// alpha >= 1/255 (blended, or stopping the pixel).
__global__ void __launch_bounds__(32) k_composite_stats(Params P) {
    pdl_enter();
    const BlockGeom G = block_geom<1>(P);
    const ViewDesc &V = *G.V;
    if (!(G.px < V.W && G.py0 < V.H)) return;
    const float fx = (float)G.px + 0.5f, fy = (float)G.py0 + 0.5f;
    float T = 1.0f;
    uint32_t neval = 0, nblend = 0;
    for (uint32_t j = G.r.x; j < G.r.y; j++) {
        const uint32_t m = P.pair_vals[j];
        float4 g, col;
        float2 q;
        record_terms(P.rec, m, g, q, col);
        const float dx = __fsub_rn(fx, g.x), dy = __fsub_rn(fy, g.y);
        if (fabsf(dx) <= P.rec[3 * (size_t)m + 1].w && fabsf(dy) <= P.rec[3 * (size_t)m + 2].w) neval++;
        const float raw = __fmul_rn(q.y, ex2_approx(falloff_exp2(falloff_column(g.z, g.w, dx), q.x, dy)));
        if (!(raw >= kAlphaMin)) continue;
        nblend++;
        const float Tn = __fsub_rn(T, __fmul_rn(fminf(kAlphaCap, raw), T));
        if (Tn < kTStop) break;
        T = Tn;
    }
    const size_t pix = (size_t)G.py0 * V.W + G.px;
    P.pix_neval[V.pix_base + pix] = neval;
    P.pix_neval[P.total_pix + V.pix_base + pix] = nblend;
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

void launch_composite(const Params &p, cudaStream_t s) {
    if (p.total_tiles == 0) return;
    const WarpShape w = warp_shape(p, kFwdWide, INT_MAX);
    const Params q = with_shape(p, w);
    note_launch();
    if (w.px == 4) pdl_launch(k_composite<4>, p.total_tiles * w.blocks, 32, 0, s, q);
    else pdl_launch(k_composite<2>, p.total_tiles * w.blocks, 32, 0, s, q);
}

void launch_composite_stats(const Params &p, cudaStream_t s) {
    if (p.total_tiles == 0) return;
    const Params q = with_shape(p, WarpShape{1, 3, (uint32_t)(p.tile_w * p.tile_h / 32)});
    note_launch();
    pdl_launch(k_composite_stats, p.total_tiles * q.blocks_per_tile, 32, 0, s, q);
}

}  // namespace pvg
