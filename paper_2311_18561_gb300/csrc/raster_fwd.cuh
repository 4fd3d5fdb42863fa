// raster_fwd.cuh -- the compositor, for colour alone (raster.cu) and with
// extra channels (features.cu).
#pragma once
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
// Blocks of 128 pixels per SM from which a lane takes four pixels: below it
// the longest walk bounds the pass and fewer pixels per lane shorten it
// (four 640x480 views of 250k Gaussians, 9,100 blocks: 280 us with four, 186
// us with two, 156 us with one); above it the instructions of all blocks do
// (1920x1280, 19,200 blocks: 193, 243 and 313 us).
constexpr int kFwdWide = 64;
// With one pixel per lane (four entries together: 156 us on those views,
// eight 164 us).
constexpr int kFwdWarps1 = 24, kFwdUnroll1 = 4;
// With extra channels (two or four pixels per lane; their sums, packed by
// pairs of channels, fill the registers).  The longest walk bounds the pass
// here too (23 channels, 1242x375, 200k Gaussians: 330 us with two entries
// together, 282 us with four).
constexpr int kFwdWarpsFeat = 8, kFwdUnrollFeat = 4;

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
template <int PX, int NG>
__global__ void __launch_bounds__(32, NG > 0 ? kFwdWarpsFeat : PX == 4 ? kFwdWarps4 : kFwdWarps2) k_composite(Params P) {
    pdl_enter();
    static_assert(PX % 2 == 0, "pairs of pixels");
    constexpr int NP = PX / 2, U = NG > 0 ? kFwdUnrollFeat : kFwdUnroll;
    constexpr uint32_t ALL = (1u << PX) - 1u;
    __shared__ RawRecords raw;
    __shared__ Staged S;
    __shared__ StagedFeats<NG> F;
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
    float2 fa[PX][NG > 0 ? 2 * NG : 1];  // extra channels' sums (negated), pairs of channels
    if constexpr (NG > 0) {
#pragma unroll
        for (int p = 0; p < PX; p++)
#pragma unroll
            for (int c = 0; c < 2 * NG; c++) fa[p][c] = nzero2;
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
    if constexpr (NG > 0) clear_feats(F, lane);
    uint32_t i0 = 0;  // the lane's Gaussian
    if constexpr (NG > 0) i0 = m0 != kNoRecord ? P.sgid[m0] - V.item_base : 0u;
    uint32_t m1 = lane + 32u < len ? P.pair_vals[r.x + 32u + lane] : kNoRecord;
    bool finished = __all_sync(0xffffffffu, done == ALL);
    for (uint32_t base = 0; base < len && !finished; base += 32) {
        wait_records();
        int hits;
        if constexpr (NG > 0) hits = stage_hits<U>(raw, S, m0 != kNoRecord, m0, base + lane, G, lane, i0, F.item);
        else hits = stage_hits<U>(raw, S, m0 != kNoRecord, m0, base + lane, G, lane);
        m0 = m1;
        fetch_record(P, raw, m0, lane);
        m1 = base + 64u + lane < len ? P.pair_vals[r.x + base + 64u + lane] : kNoRecord;
        if constexpr (NG > 0) {
            if (m0 != kNoRecord) i0 = P.sgid[m0] - V.item_base;
            stage_feats<NG, U>(P, V, S, F, hits, lane);
        }
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
                        auto one = [&](float nal, float &t, float &c0, float &c1, float &c2, float &d, float &o, const int p) {
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
                            if constexpr (NG > 0) {
#pragma unroll
                                for (int c = 0; c < 4 * NG; c++) {
                                    float &a = c & 1 ? fa[p][c / 2].y : fa[p][c / 2].x;
                                    a = __fmaf_rn(F.f[k + u][c], nw, a);
                                }
                            }
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
                if constexpr (NG > 0) {
#pragma unroll
                    for (int g = 0; g < NG; g++) {  // (packed by pixels, every value staged twice: 8 % more)
                        const float4 f = reinterpret_cast<const float4 *>(&F.f[k + u][0])[g];
#pragma unroll
                        for (int p = 0; p < PX; p++) {
                            const float w = p & 1 ? nw[u][p / 2].y : nw[u][p / 2].x;
                            fa[p][2 * g] = fma2(make_float2(f.x, f.y), make_float2(w, w), fa[p][2 * g]);
                            fa[p][2 * g + 1] = fma2(make_float2(f.z, f.w), make_float2(w, w), fa[p][2 * g + 1]);
                        }
                    }
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
    if constexpr (NG > 0) {
        const size_t HW = (size_t)V.W * V.H;
#pragma unroll
        for (int p = 0; p < PX; p++) {
            if (!(G.px < V.W && G.py0 + p < V.H)) continue;
            float *out = V.out_feat + (size_t)(G.py0 + p) * V.W + G.px;
#pragma unroll
            for (int c = 0; c < 4 * NG; c++)
                if (c < P.n_feat) out[c * HW] = -(c & 1 ? fa[p][c / 2].y : fa[p][c / 2].x);
        }
    }
    if (P.tile_walk) {  // how far the tile's adjoint walks, for its launch order
        uint32_t w = last[0];
#pragma unroll
        for (int p = 1; p < PX; p++) w = max(w, last[p]);
        w = __reduce_max_sync(0xffffffffu, w);
        if (lane == 0 && w) atomicMax(&P.tile_walk[G.tile], w);
    }
}

// The compositor with one pixel per lane: a block of 32 pixels has fewer
// hits and its walk is the shortest, which frames need whose longest walks
// bound the pass.  The packed arithmetic takes two neighbouring entries of
// the pixel instead of two pixels: the same operations per pixel and entry,
// half the issue slots, and nothing staged twice (961x641 with 300k
// Gaussians: 104 us with two pixels per lane, 80 us with one).
template <int U>
__global__ void __launch_bounds__(32, kFwdWarps1) k_composite1(Params P) {
    pdl_enter();
    static_assert(U % 4 == 0 && kStagedPlaces % U == 0, "whole groups of four entries");
    __shared__ RawRecords raw;
    __shared__ __align__(16) StagedEntries S;
    const int lane = threadIdx.x;
    const BlockGeom G = block_geom<1>(P);
    const ViewDesc &V = *G.V;
    const uint2 r = G.r;
    const uint32_t len = r.y - r.x;
    const bool inside = G.px < V.W && G.py0 < V.H;
    const float2 fx2 = make_float2((float)G.px + 0.5f, (float)G.px + 0.5f);
    bool done = !inside;
    float fy = done ? kFarRow : (float)G.py0 + 0.5f;  // (far away once done: blends nothing)
    float T[1] = {1.0f}, C0[1] = {-0.0f}, C1[1] = {-0.0f}, C2[1] = {-0.0f}, D[1] = {-0.0f}, O[1] = {-0.0f};  // sums negated
    uint32_t last[1] = {inside ? len : 0u};
    uint32_t m0 = lane < len ? P.pair_vals[r.x + lane] : kNoRecord;
    fetch_record(P, raw, m0, lane);
    uint32_t m1 = lane + 32u < len ? P.pair_vals[r.x + 32u + lane] : kNoRecord;
    bool finished = __all_sync(0xffffffffu, done);
    for (uint32_t base = 0; base < len && !finished; base += 32) {
        wait_records();
        const int hits = stage_hits<U>(raw, S, m0 != kNoRecord, m0, base + lane, G, lane);
        m0 = m1;
        fetch_record(P, raw, m0, lane);
        m1 = base + 64u + lane < len ? P.pair_vals[r.x + base + 64u + lane] : kNoRecord;
        for (int k = 0; k < hits; k += U) {
            const float2 fy2 = make_float2(fy, fy);
            float na[U];  // -alpha, -0 where the pixel does not blend
            uint32_t flags = 0;
#pragma unroll
            for (int g = 0; g < U / 4; g++) {
                auto four = [&](const float *f) { return reinterpret_cast<const float4 *>(f + k)[g]; };
                const float4 u = four(S.u), v = four(S.v), a = four(S.a), b = four(S.b), c = four(S.c), no = four(S.no);
                const uint4 p = reinterpret_cast<const uint4 *>(S.pos + k)[g];
                flags |= p.x | p.y | p.z | p.w;
                auto two = [&](float2 u2, float2 v2, float2 a2, float2 b2, float2 c2, float2 no2, float *out) {
                    const float2 dx = sub2(fx2, u2), dy = sub2(fy2, v2);
                    const float2 e = falloff_exp2_x2(mul2(mul2(a2, dx), dx), mul2(b2, dx), c2, dy);
                    const float2 nr = mul2(no2, make_float2(ex2_approx(e.x), ex2_approx(e.y)));
                    out[0] = nr.x <= -kAlphaMin ? nr.x : -0.0f;
                    out[1] = nr.y <= -kAlphaMin ? nr.y : -0.0f;
                };
                two(make_float2(u.x, u.y), make_float2(v.x, v.y), make_float2(a.x, a.y), make_float2(b.x, b.y),
                    make_float2(c.x, c.y), make_float2(no.x, no.y), na + 4 * g);
                two(make_float2(u.z, u.w), make_float2(v.z, v.w), make_float2(a.z, a.w), make_float2(b.z, b.w),
                    make_float2(c.z, c.w), make_float2(no.z, no.w), na + 4 * g + 2);
            }
            if (flags > kPosMask) {  // o~ may exceed the cap (one that cannot is left as it is)
#pragma unroll
                for (int u = 0; u < U; u++) na[u] = fmaxf(na[u], -kAlphaCap);
            }
            float nw[U], t = T[0];
#pragma unroll
            for (int u = 0; u < U; u++) {
                nw[u] = __fmul_rn(na[u], t);
                t = __fadd_rn(t, nw[u]);
            }
            // T only falls, so the pixel stops in these entries exactly if its
            // T after the last of them is below the stop
            const bool any_stop = __any_sync(0xffffffffu, t < kTStop);
            if (any_stop && t < kTStop) {  // no part from the entry that would stop it on
                t = T[0];
#pragma unroll
                for (int u = 0; u < U; u++) {
                    if (!done && __fadd_rn(t, nw[u]) < kTStop) {
                        done = true;
                        last[0] = S.pos[k + u] & kPosMask;
                        fy = kFarRow;
                    }
                    if (done) nw[u] = -0.0f;
                    t = __fadd_rn(t, nw[u]);
                }
            }
            T[0] = t;
            const bool odd = flags & kOddEntry;
#pragma unroll
            for (int u = 0; u < U; u++) {
                const float4 col = S.col[k + u];
                if (odd && nw[u] == 0.0f) continue;  // non-finite terms: a zero weight must not meet them
                C0[0] = __fmaf_rn(col.x, nw[u], C0[0]);
                C1[0] = __fmaf_rn(col.y, nw[u], C1[0]);
                C2[0] = __fmaf_rn(col.z, nw[u], C2[0]);
                D[0] = __fmaf_rn(col.w, nw[u], D[0]);
                O[0] = __fadd_rn(O[0], nw[u]);
            }
            if (any_stop && __all_sync(0xffffffffu, done)) {
                finished = true;
                break;
            }
        }
        __syncwarp();  // the next group restages
    }
    wait_records();  // a copy may still be under way when the walk ended early
    C0[0] = -C0[0]; C1[0] = -C1[0]; C2[0] = -C2[0]; D[0] = -D[0]; O[0] = -O[0];
    composite_epilogue<1>(P, V, G, T, C0, C1, C2, D, O, last);
    if (P.tile_walk) {
        const uint32_t w = __reduce_max_sync(0xffffffffu, last[0]);
        if (lane == 0 && w) atomicMax(&P.tile_walk[G.tile], w);
    }
}

}  // namespace
}  // namespace pvg
