// raster_common.cuh -- the warp's walk over its tile's list, shared by the
// compositor (raster.cu) and its adjoint (raster_bwd.cu).
//
// One warp per CTA owns a block of 32 PX pixels of a tile: lanes in 8
// columns x 4 rows (16 x 2 for tiles of 8 rows with PX = 4, and for PX = 8),
// each lane PX vertically adjacent pixels.  It takes the tile's sorted list 32
// entries at a time, one per lane: the lane tests whether the entry's footprint can
// reach the block at all (block_hit) and the hits are compacted into shared
// memory, so that the loop over entries only sees those.  No warp waits for
// another: a block whose pixels have all stopped ends at once, the blocks of
// a long list run on different SMs, and no barrier separates the batches.
#pragma once
#include <type_traits>

#include "pvg_internal.cuh"

namespace pvg {
namespace {

struct BlockGeom {
    const ViewDesc *V;
    uint32_t tile;
    int px, py0;          // this lane's first pixel (column px, rows py0 .. py0 + PX - 1)
    float x0, x1, y0, y1; // centres of the block's outermost pixels
    uint2 r;              // list range
};

template <int PX>
__device__ __forceinline__ BlockGeom block_geom(const Params &P) {
    BlockGeom g;
    const uint32_t t = blockIdx.x / P.blocks_per_tile, sub = blockIdx.x % P.blocks_per_tile;
    g.tile = P.tile_order ? P.tile_order[t] : t;
    g.V = &P.views[view_of_tile(P.views, P.n_views, g.tile)];
    const uint32_t lt = g.tile - g.V->tile_base;
    const int bw = 1 << P.block_shift, bh = (32 >> P.block_shift) * PX;
    const uint32_t nbx = (uint32_t)P.tile_w >> P.block_shift;
    const int bx = (int)(lt % (uint32_t)g.V->tiles_x) * P.tile_w + (int)(sub % nbx) * bw;
    const int by = (int)(lt / (uint32_t)g.V->tiles_x) * P.tile_h + (int)(sub / nbx) * bh;
    const int lane = threadIdx.x;
    g.px = bx + (lane & (bw - 1));
    g.py0 = by + (lane >> P.block_shift) * PX;
    g.x0 = (float)bx + 0.5f;
    g.x1 = (float)(bx + bw) - 0.5f;
    g.y0 = (float)by + 0.5f;
    g.y1 = (float)(by + bh) - 0.5f;
    g.r = P.ranges[g.tile];
    return g;
}

// Whether an entry can blend at a pixel centre of [x0, x1] x [y0, y1]:
// false only when the largest exponent a' dx^2 + b' dx dy + c' dy^2 over the
// rectangle is below -log2(255 o~), so that alpha < 1/255 everywhere on it.
// The form is concave: its maximum over a rectangle that does not hold the
// centre lies on the edge nearest in x or the one nearest in y, at that
// edge's own maximum clamped into it.  The level is widened by 1 % + 1e-4
// against the rounding of the compositor's own evaluation, and needle
// footprints ((a + c)^2 > 1e4 (ac - b^2), where that rounding may exceed it)
// and conics that are not finite always count as hits; an entry whose position
// or opacity is NaN may be culled, since its alpha test is false at every
// pixel.  So culling changes no image.
__device__ __forceinline__ bool block_hit(float u, float v, float ap, float bp, float cp, float ot, float x0,
                                          float x1, float y0, float y1) {
    const float hb = 0.5f * bp, tr = ap + cp;
    const bool well = tr * tr <= 1e4f * diff_of_products(ap, cp, hb, hb);
    const float level = -(1.01f * fmaxf(lg2_approx(255.0f * ot), 0.0f) + 1e-4f);
    const float ax = x0 - u, bx = x1 - u, ay = y0 - v, by = y1 - v;
    const float xe = fminf(fmaxf(0.0f, ax), bx), ye = fminf(fmaxf(0.0f, ay), by);
    const float ys = fminf(fmaxf(-hb * xe * rcp_approx(cp), ay), by);
    const float xs = fminf(fmaxf(-hb * ye * rcp_approx(ap), ax), bx);
    const float p1 = ap * xe * xe + ys * (bp * xe + cp * ys), p2 = cp * ye * ye + xs * (bp * ye + ap * xs);
    return !(well && p1 < level && p2 < level);
}

// flags beside an entry's list position
constexpr uint32_t kOddEntry = 0x80000000u;     // non-finite or huge terms: pixels one at a time
constexpr uint32_t kCappedEntry = 0x40000000u;  // o~ may exceed the alpha cap
constexpr uint32_t kPosMask = 0x3fffffffu;      // a list of 2^30 entries does not fit the device memory

// Below these bounds of an entry's terms and channel values and of a pixel's
// output gradients, the arithmetic that gives a pixel without a blend the
// weight zero meets finite values only: X, a sum of at most 41 products of one
// with the other, and the adjoint's suffix sum, a weighted mean of such X.
// Whatever lies above takes pixels one at a time.
constexpr float kTermBound = 1e18f, kGradBound = 1e15f;
static_assert(41.0 * kTermBound * kGradBound < 1e36, "two orders below the largest float");

constexpr int kStagedPlaces = 32;

// The hits of 32 list entries, operands of the packed arithmetic in pairs.
struct Staged {
    float4 a[kStagedPlaces];  // (u, a', b', list position | flags)
    float4 b[kStagedPlaces];  // (v, v, c', c')
    float4 c[kStagedPlaces];  // (-o~, -o~, r, r)
    float4 d[kStagedPlaces];  // (g, g, b, b)
    float2 e[kStagedPlaces];  // (z, z)
    uint32_t m[kStagedPlaces];

    __device__ __forceinline__ void put(int k, const float4 &g, const float2 &q, const float4 &col, uint32_t pos,
                                        uint32_t rec) {
        a[k] = make_float4(g.x, g.z, g.w, __uint_as_float(pos));
        b[k] = make_float4(g.y, g.y, q.x, q.x);
        c[k] = make_float4(-q.y, -q.y, col.x, col.x);
        d[k] = make_float4(col.y, col.y, col.z, col.z);
        e[k] = make_float2(col.w, col.w);
        m[k] = rec;
    }
};

// The hits for one pixel per lane, whose packed arithmetic takes two
// neighbouring entries.
struct StagedEntries {
    float u[kStagedPlaces], v[kStagedPlaces], a[kStagedPlaces], b[kStagedPlaces], c[kStagedPlaces];
    float no[kStagedPlaces];       // -o~
    uint32_t pos[kStagedPlaces];   // list position | flags
    float4 col[kStagedPlaces];     // (r, g, b, z)

    __device__ __forceinline__ void put(int k, const float4 &g, const float2 &q, const float4 &cl, uint32_t p, uint32_t) {
        u[k] = g.x;
        v[k] = g.y;
        a[k] = g.z;
        b[k] = g.w;
        c[k] = q.x;
        no[k] = -q.y;
        pos[k] = p;
        col[k] = cl;
    }
};

// 32 records on their way to shared memory, one per lane
struct RawRecords {
    float4 q[3][32];
};

constexpr uint32_t kNoRecord = 0xffffffffu;

// starts the copy of record m into the lane's place
__device__ __forceinline__ void fetch_record(const Params &P, RawRecords &raw, uint32_t m, int lane) {
    if (m == kNoRecord) return;
    const float4 *src = P.rec + 3 * (size_t)m;
#pragma unroll
    for (int k = 0; k < 3; k++)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(&raw.q[k][lane])),
                     "l"(src + k)
                     : "memory");
}

__device__ __forceinline__ void wait_records() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The lane's record (arrived), tested and, if it can reach the block,
// written to the next free place of S; returns the number of hits.  pos: the
// record's list position.  The places up to the next multiple of U get an
// entry that blends nowhere.
// items (optional): the hits' values of `item`, in their places.
template <int U, class Stage>
__device__ __forceinline__ int stage_hits(const RawRecords &raw, Stage &S, bool have, uint32_t m, uint32_t pos,
                                          const BlockGeom &G, int lane, uint32_t item = 0,
                                          uint32_t *items = nullptr) {
    bool hit = false;
    float4 a, c;
    float2 b;
    if (have) {
        const float4 q[3] = {raw.q[0][lane], raw.q[1][lane], raw.q[2][lane]};
        record_terms(q, 0, a, b, c);
        hit = block_hit(a.x, a.y, a.z, a.w, b.x, b.y, G.x0, G.x1, G.y0, G.y1);
    }
    const uint32_t mask = __ballot_sync(0xffffffffu, hit);
    if (hit) {
        const int k = __popc(mask & ((1u << lane) - 1u));
        const float s = fabsf(a.x) + fabsf(a.y) + fabsf(a.z) + fabsf(a.w) + fabsf(b.x) + fabsf(b.y) + fabsf(c.x) +
                        fabsf(c.y) + fabsf(c.z) + fabsf(c.w);
        pos |= (s < kTermBound ? 0u : kOddEntry) | (b.y <= kUncappedOpacity ? 0u : kCappedEntry);
        S.put(k, a, b, c, pos, m);
        if (items) items[k] = item;
    }
    const int hits = __popc(mask);
    if (U > 1 && lane < (U - hits % U) % U) {
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        S.put(hits + lane, zero, make_float2(-kMinRowCoef, 0.f), zero, 0u, 0u);
    }
    __syncwarp();
    return hits;
}

// Extra channels of the staged entries, zeros beyond the call's channels.  The
// arithmetic on channels is packed by pairs of channels, which needs no value
// twice.
template <int NG>
struct StagedFeats {
    alignas(16) float f[kStagedPlaces][4 * NG];
    uint32_t item[kStagedPlaces];  // Gaussian of the entry's scene
};
template <>
struct StagedFeats<0> {};

// Zeroes the channel values once: those beyond the call's channels stay zero.
template <int NG>
__device__ __forceinline__ void clear_feats(StagedFeats<NG> &F, int lane) {
    for (int k = lane; k < kStagedPlaces * NG; k += 32)
        reinterpret_cast<float4 *>(&F.f[0][0])[k] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// The channel values of the `hits` staged entries (their Gaussians in
// F.item; places up to the next multiple of U zeroed): every semantic row by
// the whole warp, all rows' copies in flight together and behind them v_bar
// and rho by the entries' lanes; then one pass looks for semantic values that
// are not finite.
// Entries with non-finite values are flagged in S.
template <int NG, int U>
__device__ __forceinline__ void stage_feats(const Params &P, const ViewDesc &V, Staged &S, StagedFeats<NG> &F,
                                            int hits, int lane) {
    const int places = (hits + U - 1) / U * U;
    const int c0 = ((P.feat_mask & kFeatVbar) ? 3 : 0) + ((P.feat_mask & kFeatRho) ? 1 : 0);
    const int n_sem = (P.feat_mask & kFeatSem) ? V.n_sem : 0;
    if (lane < n_sem) {
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&F.f[0][c0 + lane]);
        for (int k = 0; k < hits; k++)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + k * (uint32_t)sizeof(F.f[0])),
                         "l"(V.sem + (size_t)F.item[k] * n_sem + lane)
                         : "memory");
    }
    if (c0 && lane < hits) {
        const uint32_t i = F.item[lane];
        const float rho = __fdiv_rn(V.beta[i], V.period[i]);
        float bad = 0.f;
        int c = 0;
        auto put = [&](float v) {
            F.f[lane][c++] = v;
            bad += fabsf(v);
        };
        if (P.feat_mask & kFeatVbar) {
            const float w = expf(-0.5f * rho);
            const float3 vel = make_float3(V.vel[3 * (size_t)i], V.vel[3 * (size_t)i + 1], V.vel[3 * (size_t)i + 2]);
            put(vel.x * w);
            put(vel.y * w);
            put(vel.z * w);
        }
        if (P.feat_mask & kFeatRho) put(fminf(rho, 2.0f));
        if (!(bad < kTermBound)) S.a[lane].w = __uint_as_float(__float_as_uint(S.a[lane].w) | kOddEntry);
    }
    for (int k = hits; k < places; k++)
        for (int c = lane; c < 4 * NG; c += 32) F.f[k][c] = 0.f;
    if (n_sem) {
        wait_records();
        uint32_t bad = 0;  // entries with a non-finite value of this lane's class
        if (lane < n_sem)
#pragma unroll 4
            for (int k = 0; k < hits; k++) {
                bad |= fabsf(F.f[k][c0 + lane]) < kTermBound ? 0u : 1u << k;
            }
        bad = __reduce_or_sync(0xffffffffu, bad);
        if ((bad >> lane) & 1u) S.a[lane].w = __uint_as_float(__float_as_uint(S.a[lane].w) | kOddEntry);
    }
    __syncwarp();
}

}  // namespace

// Pixels per lane of the compositing kernels and the block's shape in a
// tile.  A lane takes eight (four) pixels when the frame has wide8 blocks of
// 256 (wide4 of 128) pixels per SM, else two.
struct WarpShape {
    int px, shift;
    uint32_t blocks;  // per tile
};
WarpShape warp_shape(const Params &p, int wide4, int wide8);

}  // namespace pvg

// Supported (tile width, tile height, pixels per thread) combinations.
#define PVG_TILE_CONFIGS(X)                                                                               \
    X(16, 16, 1) X(16, 16, 2) X(16, 16, 4) X(8, 8, 1) X(8, 8, 2) X(16, 8, 1) X(16, 8, 2) X(32, 8, 1)    \
    X(32, 16, 1) X(32, 16, 2) X(32, 16, 4) X(32, 32, 4) X(16, 32, 4)
