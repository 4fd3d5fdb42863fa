// raster_bwd.cuh -- the compositor's adjoint, for colour alone
// (raster_bwd.cu) and with extra channels (features_bwd.cu).
#pragma once

#include "raster_common.cuh"

namespace pvg {
namespace {

// Resident warps per SM that the registers are held to (16 warps of 126
// registers with eight pixels per lane), and entries whose alphas are
// evaluated together, by pixels per lane: with two or four pixels a lane the
// longest walk bounds the frame and four evaluations overlap its latencies
// (1242x375, four pixels: 162 us one by one, 147 us by twos, 139 us by
// fours), with eight the pixels are parallel enough.
template <int PX>
struct BwdTune {
    static constexpr int kWarps = PX == 2 ? 20 : 16;
    static constexpr int kUnroll = PX == 8 ? 1 : 4;
};
// Blocks of 256 (128) pixels per SM from which a lane takes eight (four)
// pixels.  Eight make an entry's fixed work (its staged loads, the warp sum,
// the atomics) a quarter of that of two: 362 us against 405 us with four on
// the 1.5M-Gaussian 1920x1280 frame (9,600 blocks), 2.15 against 2.38 ms on
// 12 mixed views (14,900 blocks); a 961x641 frame of 300k Gaussians (2,501
// blocks), which its longest walks bound, takes 535 us with eight, 291 us
// with four.  Two only for frames too small for four (1242x375: 178 us with
// two, 133 us with four).
constexpr int kBwdWide8 = 48, kBwdWide4 = 16;
// With extra channels (two or four pixels per lane): two entries' channel sums
// taken together (23 channels, 1242x375, 200k Gaussians: 723 us one by one,
// 638 us by twos, 641 us by fours).
constexpr int kBwdWarpsFeat = 8, kBwdUnrollFeat = 2;

// Warp sums of an entry's NT terms (9, or 10 with the depth term) over the
// lanes, four entries at a time, by a transposition through shared memory:
// every lane stores its terms of an entry (two float4 and one or two
// floats), and once four entries are stored lane r sums eight lanes' float4
// of entry r >> 3, half (r >> 2) & 1, and folds the four partial sums that
// the lanes r & 3 of a half hold with three shuffles.  About 14 instructions
// per entry; a shuffle butterfly over 9 terms takes 44.  The halves are 36
// float4 apart so that the eight lanes of a load phase (two halves, four
// lanes each) read distinct banks.
constexpr int kSlots = 4;
constexpr int kHalfStride = 36;

template <int NT>
struct TermBuffer {
    float4 h[kSlots][2][kHalfStride];
    float e[NT - 8][kSlots][32];
};

// Adds the totals of the stored entries (bit i of `valid`: slot i, staged
// entry base + i) to their Gaussians' rows.
template <int NT>
__device__ __forceinline__ void flush_terms(const TermBuffer<NT> &buf, const Staged &S, int base, uint32_t valid,
                                            int lane, const Params &P) {
    const int slot = lane >> 3, half = (lane >> 2) & 1, sub = lane & 3;
    // the slot's entry: loaded ahead of the sums
    const size_t m = S.m[base + slot];
    const float4 ab = S.a[base + slot], gb = S.d[base + slot];  // (u, a', b', -), (g, g, b, b)
    const float cc = S.b[base + slot].z, red = S.c[base + slot].z;
    __syncwarp();
    const float4 *h = &buf.h[slot][half][sub];
    float2 a, b;
#pragma unroll
    for (int j = 0; j < 8; j++) {
        const float4 v = h[4 * j];
        a = j ? add2(a, make_float2(v.x, v.y)) : make_float2(v.x, v.y);
        b = j ? add2(b, make_float2(v.z, v.w)) : make_float2(v.z, v.w);
    }
    float s[NT - 8];
#pragma unroll
    for (int t = 0; t < NT - 8; t++) {
        const float4 v = reinterpret_cast<const float4 *>(&buf.e[t][0][0])[lane];
        s[t] = (v.x + v.y) + (v.z + v.w);
    }
    const bool hi2 = sub & 2, hi1 = sub & 1;
    const float c0 = (hi2 ? b.x : a.x) + __shfl_xor_sync(0xffffffffu, hi2 ? a.x : b.x, 2);
    const float c1 = (hi2 ? b.y : a.y) + __shfl_xor_sync(0xffffffffu, hi2 ? a.y : b.y, 2);
#pragma unroll
    for (int o = 1; o < 8; o <<= 1)
#pragma unroll
        for (int t = 0; t < NT - 8; t++) s[t] += __shfl_xor_sync(0xffffffffu, s[t], o);
    const float d = (hi1 ? c1 : c0) + __shfl_xor_sync(0xffffffffu, hi1 ? c0 : c1, 1);
    const float q = __shfl_xor_sync(0xffffffffu, d, 1);
    __syncwarp();  // the buffer is free
    // Half 0 holds m_xx, m_xy, m_yy, m_0, half 1 m_x, m_y, r, g; every lane
    // but one adds one float (a lane of the second moments the colour b or
    // the depth), three lanes a moment in 64 bits: the per-item adjoint's
    // products with the conic cancel and amplify the rounding of their sums.
    // The gradients of u and v (conic a = -2 ln 2 a', b = -ln 2 b') are taken
    // here and not from the moments' totals, since a m_x + b m_y cancels too.
    // No colour term where the forward clamped.  (Two atomics for the whole
    // warp: one per kind of term in branches of their own took 7 us more
    // on the 1242x375 frame and 33 us on a sparse 961x641 one.)
    const float uv = -0.6931471805599453f * (2.0f * (sub == 0 ? ab.y : cc) * d + ab.z * q);
    const float gate = half == 0 ? (sub == 0 ? gb.z : 1.0f) : sub == 2 ? red : sub == 3 ? gb.x : 1.0f;
    const float v = half == 0 ? (sub == 0 ? s[0] : sub == 3 ? d : NT == 10 && sub == 1 ? s[NT - 9] : 0.0f)
                              : (sub < 2 ? uv : d);
    const int t = half == 0 ? (sub == 0 ? kG2dColour + 2 : sub == 1 ? kG2dDepth : kG2dPower)
                            : (sub < 2 ? sub : kG2dColour + sub - 2);
    const bool on = (valid >> slot) & 1u;
    if (on && v != 0.f && gate > 0.f) atomicAdd(P.g2d + kG2dRow * m + t, v);
    if (on && half == 0 && sub < 3 && d != 0.f) atomicAdd(P.g2m + 3 * m + sub, (double)d);
}

// The channels' gradients of up to U entries, summed over the warp and added
// to their Gaussians' rows of gfeat: the transposition of flush_terms with a
// float4 group of channels in the place of a half (eight groups at a time;
// lanes 4 g .. 4 g + 3 end with the totals of group g).
template <int NG, int U>
struct FeatBuffer {
    float4 h[U][NG][kHalfStride];
};
template <int U>
struct FeatBuffer<0, U> {};

template <int NG, int U>
__device__ __forceinline__ void store_feats(FeatBuffer<NG, U> &buf, int u, const float2 (&gf)[2 * NG], int lane) {
#pragma unroll
    for (int g = 0; g < NG; g++) buf.h[u][g][lane] = make_float4(gf[2 * g].x, gf[2 * g].y, gf[2 * g + 1].x, gf[2 * g + 1].y);
}

// bit u of valid: the u-th stored entry, staged entry k0 + u
template <int NG, int U>
__device__ __forceinline__ void flush_feats(const FeatBuffer<NG, U> &buf, const Staged &S, int k0, uint32_t valid,
                                            int lane, const Params &P) {
    __syncwarp();
    const int sub = lane & 3;
    const bool hi2 = sub & 2, hi1 = sub & 1;
#pragma unroll
    for (int g0 = 0; g0 < NG; g0 += 8) {
        const int g = min(g0 + (lane >> 2), NG - 1), c = 4 * g0 + lane;
#pragma unroll
        for (int u = 0; u < U; u++) {
            const float4 *h = &buf.h[u][g][sub];
            float2 a, b;
#pragma unroll
            for (int j = 0; j < 8; j++) {
                const float4 v = h[4 * j];
                a = j ? add2(a, make_float2(v.x, v.y)) : make_float2(v.x, v.y);
                b = j ? add2(b, make_float2(v.z, v.w)) : make_float2(v.z, v.w);
            }
            const float c0 = (hi2 ? b.x : a.x) + __shfl_xor_sync(0xffffffffu, hi2 ? a.x : b.x, 2);
            const float c1 = (hi2 ? b.y : a.y) + __shfl_xor_sync(0xffffffffu, hi2 ? a.y : b.y, 2);
            const float d = (hi1 ? c1 : c0) + __shfl_xor_sync(0xffffffffu, hi1 ? c0 : c1, 1);
            if (((valid >> u) & 1u) && c < P.n_feat && d != 0.f)
                atomicAdd(P.gfeat + (size_t)S.m[k0 + u] * P.n_feat + c, d);
        }
    }
    __syncwarp();
}

// Per-pixel state of the adjoint walk: final transmittance, stop
// position, output gradients and the initial suffix sum (the background's
// share); with a sky map, its gradient is scattered here and its effect on
// dL/dO folded into gO.
struct PixelAdjoint {
    float T, gC0, gC1, gC2, gD, gO, S;
    uint32_t last;
};

// dL/d(sky texels) of a lane's pixels, one after another: vertically adjacent
// pixels mostly sample the same four texels, whose shares are added up here
// and reach memory once (a 961 pixels wide 50 degree view of a 256-texel face
// has seven pixels to a texel)
struct SkyScatter {
    size_t first = ~(size_t)0, last = 0;  // indices of the corners (0, 0) and (1, 1), which fix the other two
    size_t idx[4];
    float acc[4][3];

    __device__ __forceinline__ void add(const ViewDesc &V, const size_t (&ti)[4], const float (&tw)[4], float wo,
                                        const float (&gc)[3]) {
        if (ti[0] != first || ti[3] != last) {
            flush(V);
            first = ti[0];
            last = ti[3];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                idx[q] = ti[q];
#pragma unroll
                for (int c = 0; c < 3; c++) acc[q][c] = 0.f;
            }
        }
#pragma unroll
        for (int q = 0; q < 4; q++)
#pragma unroll
            for (int c = 0; c < 3; c++)
                if (tw[q] != 0.f && gc[c] != 0.f) acc[q][c] += tw[q] * wo * gc[c];
    }
    __device__ __forceinline__ void flush(const ViewDesc &V) {
        if (first == ~(size_t)0) return;
#pragma unroll
        for (int q = 0; q < 4; q++)
#pragma unroll
            for (int c = 0; c < 3; c++)
                if (acc[q][c] != 0.f) atomicAdd(V.g_sky + idx[q] + c, acc[q][c]);
        first = ~(size_t)0;
    }
};

__device__ __forceinline__ PixelAdjoint pixel_adjoint(const Params &P, const ViewDesc &V, int px, int py,
                                                      SkyScatter &sky) {
    PixelAdjoint a;
    a.T = 1.0f;
    a.gC0 = a.gC1 = a.gC2 = a.gD = a.gO = 0.f;
    a.last = 0;
    const bool inside = px < V.W && py < V.H;
    if (inside) {
        const size_t HW = (size_t)V.W * V.H, pix = (size_t)py * V.W + px;
        a.T = P.pix_T[V.pix_base + pix];
        a.last = P.pix_last[V.pix_base + pix];
        if (V.dl_rgb) {
            a.gC0 = V.dl_rgb[pix];
            a.gC1 = V.dl_rgb[HW + pix];
            a.gC2 = V.dl_rgb[2 * HW + pix];
        }
        if (V.dl_depth) a.gD = V.dl_depth[pix];
        if (V.dl_alpha) a.gO = V.dl_alpha[pix];
    }
    a.S = a.T * (a.gC0 * V.bg[0] + a.gC1 * V.bg[1] + a.gC2 * V.bg[2]);
    if (V.sky && inside) {
        // colour = C + (1 - O) f: no constant background, dL/dO -= gC.f,
        // dL/df = (1 - O) gC scattered to the four texels
        size_t ti[4];
        float tw[4];
        sky_texels(V, px, py, ti, tw);
        const float gc[3] = {a.gC0, a.gC1, a.gC2};
        const float wo = a.T;  // 1 - O = T_final
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const float f = tw[0] * V.sky[ti[0] + c] + tw[1] * V.sky[ti[1] + c] + tw[2] * V.sky[ti[2] + c] +
                            tw[3] * V.sky[ti[3] + c];
            a.gO -= gc[c] * f;
        }
        if (V.g_sky) sky.add(V, ti, tw, wo, gc);
        a.S = 0.f;
    }
    return a;
}

// kAux: the call has depth or opacity-map gradients or a sky map (dL/dO
// and the depth term of X can be non-zero); without them X = gC.c and the
// depth term is not reduced (9 terms).  The output gradients and the blend
// weights are kept negated, which leaves the packed arithmetic no negation.
template <int PX, bool kAux, int NG>
__global__ void __launch_bounds__(32, NG > 0 ? kBwdWarpsFeat : BwdTune<PX>::kWarps) k_composite_bwd(Params P) {
    pdl_enter();
    constexpr int NT = kAux ? 10 : 9, NP = PX / 2, U = NG > 0 ? kBwdUnrollFeat : BwdTune<PX>::kUnroll;
    __shared__ RawRecords raw;
    __shared__ Staged Sg;
    __shared__ TermBuffer<NT> buf;
    __shared__ StagedFeats<NG> F;
    __shared__ FeatBuffer<NG, (NG > 0 ? kBwdUnrollFeat : 1)> fbuf;
    const int lane = threadIdx.x;
    const BlockGeom G = block_geom<PX>(P);
    const ViewDesc &V = *G.V;
    const uint2 r = G.r;
    const float fx = (float)G.px + 0.5f;
    const float2 one2 = make_float2(1.0f, 1.0f);
    float2 fy[NP], T[NP], nC0[NP], nC1[NP], nC2[NP], nD[NP], nO[NP];
    float2 S[NP];  // suffix sum of X_j alpha_j T_j
    uint32_t last[PX];
    uint32_t walk = 0;
    SkyScatter sky;
    // pixels one at a time: non-finite or huge output gradients, and from the
    // first 32 entries on that hold such a term, behind which a pixel's suffix
    // sum may be infinite (carried by entry it costs the adjoint 1 %)
    bool odd = false;
#pragma unroll
    for (int q = 0; q < NP; q++) {
        fy[q] = make_float2((float)(G.py0 + 2 * q) + 0.5f, (float)(G.py0 + 2 * q + 1) + 0.5f);
        const PixelAdjoint a = pixel_adjoint(P, V, G.px, G.py0 + 2 * q, sky);
        const PixelAdjoint b = pixel_adjoint(P, V, G.px, G.py0 + 2 * q + 1, sky);
        T[q] = make_float2(a.T, b.T);
        S[q] = make_float2(a.S, b.S);
        nC0[q] = make_float2(-a.gC0, -b.gC0);
        nC1[q] = make_float2(-a.gC1, -b.gC1);
        nC2[q] = make_float2(-a.gC2, -b.gC2);
        nD[q] = make_float2(-a.gD, -b.gD);
        nO[q] = make_float2(-a.gO, -b.gO);
        last[2 * q] = a.last;
        last[2 * q + 1] = b.last;
        walk = max(walk, max(a.last, b.last));
        for (const PixelAdjoint &e : {a, b})
            odd |= !(fabsf(e.gC0) + fabsf(e.gC1) + fabsf(e.gC2) + fabsf(e.gD) + fabsf(e.gO) + fabsf(e.S) < kGradBound);
    }
    sky.flush(V);
    // output gradients of the extra channels (negated), pairs of channels: packed
    // by pixels instead, every channel's two halves have to be added up
    // (1242x1242 with 300k Gaussians, 23 channels: 1025 us, by channels 838)
    float2 nF[PX][NG > 0 ? 2 * NG : 1];
    if constexpr (NG > 0) {
        const size_t HW = (size_t)V.W * V.H;
#pragma unroll
        for (int p = 0; p < PX; p++) {
            const bool in = V.dl_feat && G.px < V.W && G.py0 + p < V.H;
            const float *src = V.dl_feat + (size_t)(G.py0 + p) * V.W + G.px;
#pragma unroll
            for (int c = 0; c < 2 * NG; c++) {
                nF[p][c].x = in && 2 * c < P.n_feat ? -src[2 * c * HW] : 0.f;
                nF[p][c].y = in && 2 * c + 1 < P.n_feat ? -src[(2 * c + 1) * HW] : 0.f;
                odd |= !(fabsf(nF[p][c].x) + fabsf(nF[p][c].y) < kGradBound);
            }
        }
    }
    odd = __any_sync(0xffffffffu, odd);
    walk = __reduce_max_sync(0xffffffffu, walk);
    // groups of 32 entries from the walk's end; lane i of a group holds entry start + i
    auto load_index = [&](int start) { return start + lane >= 0 && start + lane < (int)walk ? P.pair_vals[r.x + start + lane] : kNoRecord; };
    int start = (int)walk - 32;
    uint32_t m0 = load_index(start);
    fetch_record(P, raw, m0, lane);
    if constexpr (NG > 0) clear_feats(F, lane);
    uint32_t i0 = 0;  // the lane's Gaussian
    if constexpr (NG > 0) i0 = m0 != kNoRecord ? P.sgid[m0] - V.item_base : 0u;
    uint32_t m1 = load_index(start - 32);
    for (; start > -32; start -= 32) {
        wait_records();
        int hits;
        if constexpr (NG > 0)
            hits = stage_hits<kSlots>(raw, Sg, m0 != kNoRecord, m0, (uint32_t)(start + lane), G, lane, i0, F.item);
        else hits = stage_hits<kSlots>(raw, Sg, m0 != kNoRecord, m0, (uint32_t)(start + lane), G, lane);
        m0 = m1;
        fetch_record(P, raw, m0, lane);
        m1 = load_index(start - 64);
        if constexpr (NG > 0) {
            if (m0 != kNoRecord) i0 = P.sgid[m0] - V.item_base;
            stage_feats<NG, kSlots>(P, V, Sg, F, hits, lane);
        }
        odd |= __any_sync(0xffffffffu, lane < hits && (__float_as_uint(Sg.a[lane].w) & kOddEntry));
        for (int base = (hits - 1) & ~(kSlots - 1); base >= 0; base -= kSlots) {
            uint32_t valid = 0;  // slots that hold an entry's terms
#pragma unroll 1
            for (int k0 = kSlots - U; k0 >= 0; k0 -= U) {
                // alphas of U entries, the later first (negated, 0 where a pixel does not blend)
                float2 dy[U][NP], na[U][NP];
                float dx[U];
                uint32_t pf[U];
                uint32_t any = 0;
#pragma unroll
                for (int u = U - 1; u >= 0; u--) {
                    const int k = base + k0 + u;
                    const float4 A = Sg.a[k], B = Sg.b[k];
                    const float2 no2 = reinterpret_cast<const float2 *>(&Sg.c[k])[0];
                    pf[u] = __float_as_uint(A.w);
                    const uint32_t pos = pf[u] & kPosMask;
                    dx[u] = __fsub_rn(fx, A.x);
                    const FalloffColumn fc = falloff_column(A.y, A.z, dx[u]);
                    const float2 A2 = make_float2(fc.A, fc.A), B2 = make_float2(fc.B, fc.B);
                    const float2 v2 = make_float2(B.x, B.y), cp2 = make_float2(B.z, B.w);
                    bool hit = false;
#pragma unroll
                    for (int q = 0; q < NP; q++) {
                        dy[u][q] = sub2(fy[q], v2);
                        const float2 e = falloff_exp2_x2(A2, B2, cp2, dy[u][q]);
                        const float2 nr = mul2(no2, make_float2(ex2_approx(e.x), ex2_approx(e.y)));
                        const bool bx = pos < last[2 * q] && nr.x <= -kAlphaMin;
                        const bool by = pos < last[2 * q + 1] && nr.y <= -kAlphaMin;
                        hit |= bx || by;
                        na[u][q] = make_float2(bx ? nr.x : 0.f, by ? nr.y : 0.f);
                    }
                    any |= __any_sync(0xffffffffu, hit) ? 1u << u : 0u;
                }
#pragma unroll
                for (int u = U - 1; u >= 0; u--) {
                    if (!((any >> u) & 1u)) continue;
                    const int k = base + k0 + u;
                    const float2 r2 = reinterpret_cast<const float2 *>(&Sg.c[k])[1];
                    const float4 Dq = Sg.d[k];
                    const float2 g2 = make_float2(Dq.x, Dq.y), b2 = make_float2(Dq.z, Dq.w);
                    float2 z2;
                    if constexpr (kAux) z2 = Sg.e[k];
                    float A0, M1, M2, c0, c1, c2, zs = 0.f;
                    float2 nwf[NP];  // the pixels' weights (negated)
                    if (!odd) {
                        float2 A0v, M1v, M2v, c0v, c1v, c2v, zv;
                        auto pairs = [&](auto capped) {
                            constexpr bool kCap = decltype(capped)::value;
#pragma unroll
                            for (int q = 0; q < NP; q++) {
                                float2 nq = na[u][q];
                                bool ox = false, oy = false;  // over the cap: alpha does not depend on the power
                                if constexpr (kCap) {
                                    ox = nq.x < -kAlphaCap;
                                    oy = nq.y < -kAlphaCap;
                                    nq = make_float2(fmaxf(nq.x, -kAlphaCap), fmaxf(nq.y, -kAlphaCap));
                                }
                                const float2 om = add2(one2, nq);
                                // (rcp.approx(1) = 1: a pixel that does not blend keeps its T)
                                const float2 inv = make_float2(rcp_approx(om.x), rcp_approx(om.y));
                                const float2 Ti = mul2(T[q], inv);
                                const float2 nw = mul2(nq, Ti);
                                float2 nX;
                                if constexpr (kAux) {
                                    nX = add2(fma2(nC2[q], b2, fma2(nC1[q], g2, mul2(nC0[q], r2))), fma2(nD[q], z2, nO[q]));
                                    zv = q ? fma2(nD[q], nw, zv) : mul2(nD[q], nw);
                                } else {
                                    nX = fma2(nC2[q], b2, fma2(nC1[q], g2, mul2(nC0[q], r2)));
                                }
                                if constexpr (NG > 0) {
                                    float2 ex, ey;  // the two pixels' sums
#pragma unroll
                                    for (int g = 0; g < NG; g++) {
                                        const float4 f = reinterpret_cast<const float4 *>(&F.f[k][0])[g];
                                        const float2 fa = make_float2(f.x, f.y), fb = make_float2(f.z, f.w);
                                        ex = g ? fma2(nF[2 * q][2 * g], fa, ex) : mul2(nF[2 * q][2 * g], fa);
                                        ey = g ? fma2(nF[2 * q + 1][2 * g], fa, ey) : mul2(nF[2 * q + 1][2 * g], fa);
                                        ex = fma2(nF[2 * q][2 * g + 1], fb, ex);
                                        ey = fma2(nF[2 * q + 1][2 * g + 1], fb, ey);
                                    }
                                    nX = add2(nX, make_float2(ex.x + ex.y, ey.x + ey.y));
                                    nwf[q] = nw;
                                }
                                // -dL/dalpha, then dL/dpower = dL/dalpha alpha
                                float2 gp = mul2(fma2(Ti, nX, mul2(inv, S[q])), nq);
                                if constexpr (kCap) gp = make_float2(ox ? 0.f : gp.x, oy ? 0.f : gp.y);
                                S[q] = fma2(nX, nw, S[q]);
                                T[q] = Ti;
                                const float2 my = mul2(gp, dy[u][q]);
                                c0v = q ? fma2(nC0[q], nw, c0v) : mul2(nC0[q], nw);
                                c1v = q ? fma2(nC1[q], nw, c1v) : mul2(nC1[q], nw);
                                c2v = q ? fma2(nC2[q], nw, c2v) : mul2(nC2[q], nw);
                                A0v = q ? add2(A0v, gp) : gp;
                                M1v = q ? add2(M1v, my) : my;
                                M2v = q ? fma2(my, dy[u][q], M2v) : mul2(my, dy[u][q]);
                            }
                        };
                        if (pf[u] & kCappedEntry) pairs(std::true_type{});
                        else pairs(std::false_type{});
                        A0 = A0v.x + A0v.y; M1 = M1v.x + M1v.y; M2 = M2v.x + M2v.y;
                        c0 = c0v.x + c0v.y; c1 = c1v.x + c1v.y; c2 = c2v.x + c2v.y;
                        if constexpr (kAux) zs = zv.x + zv.y;
                    } else {
                        A0 = M1 = M2 = c0 = c1 = c2 = 0.f;
                        auto one = [&](float nr, float dyp, float &t, float &Sp, float h0, float h1, float h2, float hd,
                                       float ho, float &wf, const int p) {
                            wf = 0.f;
                            if (!(nr < 0.f)) return;
                            const float nal = fmaxf(nr, -kAlphaCap);
                            const float inv = rcp_approx(1.0f + nal);
                            const float Ti = t * inv, nw = nal * Ti;
                            float nX = h0 * r2.x + h1 * g2.x + h2 * b2.x;
                            if constexpr (kAux) {
                                nX += hd * z2.x + ho;
                                zs += hd * nw;
                            }
                            if constexpr (NG > 0) {
                                wf = nw;
#pragma unroll
                                for (int c = 0; c < 4 * NG; c++)
                                    nX += (c & 1 ? nF[p][c / 2].y : nF[p][c / 2].x) * F.f[k][c];
                            }
                            c0 += h0 * nw;
                            c1 += h1 * nw;
                            c2 += h2 * nw;
                            if (nr >= -kAlphaCap) {
                                const float gp = (inv * Sp + Ti * nX) * nal, my = gp * dyp;
                                A0 += gp;
                                M1 += my;
                                M2 += my * dyp;
                            }
                            Sp += nX * nw;
                            t = Ti;
                        };
#pragma unroll
                        for (int q = 0; q < NP; q++) {
                            one(na[u][q].x, dy[u][q].x, T[q].x, S[q].x, nC0[q].x, nC1[q].x, nC2[q].x, nD[q].x, nO[q].x,
                                nwf[q].x, 2 * q);
                            one(na[u][q].y, dy[u][q].y, T[q].y, S[q].y, nC0[q].y, nC1[q].y, nC2[q].y, nD[q].y, nO[q].y,
                                nwf[q].y, 2 * q + 1);
                        }
                    }
                    if constexpr (NG > 0) {
                        float2 gf[2 * NG];
                        if (!odd) {
#pragma unroll
                            for (int p = 0; p < PX; p++) {
                                const float w = p & 1 ? nwf[p / 2].y : nwf[p / 2].x;
                                const float2 w2 = make_float2(w, w);
#pragma unroll
                                for (int c = 0; c < 2 * NG; c++)
                                    gf[c] = p ? fma2(nF[p][c], w2, gf[c]) : mul2(nF[p][c], w2);
                            }
                        } else {  // a pixel that does not blend has no share, whatever its gradients
#pragma unroll
                            for (int c = 0; c < 2 * NG; c++) gf[c] = make_float2(0.f, 0.f);
#pragma unroll
                            for (int p = 0; p < PX; p++) {
                                const float w = p & 1 ? nwf[p / 2].y : nwf[p / 2].x;
                                if (w == 0.f) continue;
#pragma unroll
                                for (int c = 0; c < 2 * NG; c++) gf[c] = fma2(nF[p][c], make_float2(w, w), gf[c]);
                            }
                        }
                        store_feats<NG, U>(fbuf, u, gf, lane);
                    }
                    // the pixels share dx: m_x = dx m_0, m_xx = dx m_x, m_xy = dx m_y
                    const float mx = dx[u] * A0;
                    buf.h[k0 + u][0][lane] = make_float4(dx[u] * mx, dx[u] * M1, M2, A0);
                    buf.h[k0 + u][1][lane] = make_float4(mx, M1, c0, c1);
                    buf.e[0][k0 + u][lane] = c2;
                    if constexpr (kAux) buf.e[1][k0 + u][lane] = zs;
                }
                if constexpr (NG > 0) {
                    if (any) flush_feats<NG, U>(fbuf, Sg, base + k0, any, lane, P);
                }
                valid |= any << k0;
            }
            if (valid) flush_terms<NT>(buf, Sg, base, valid, lane, P);
        }
        __syncwarp();  // the next group restages
    }
}

}  // namespace
}  // namespace pvg
