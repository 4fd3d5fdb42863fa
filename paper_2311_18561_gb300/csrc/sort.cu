// sort.cu -- device-wide scans, stream compaction, pair emission and a
// stable LSD radix sort of (u32 key, u32 value) pairs, all with the element
// count read from device memory so that no host round trip is needed.
//
// Role in the method: the camera-space depth order of the Gaussians
// (Sec. 3.1) within every tile of the tile-based rasterizer.
// The sort is done in two stages:
//   1. the visible (view, Gaussian) items are sorted by the float32 bits of
//      their camera depth (4 digit passes over M items; the items start in
//      gid order and the sort is stable, so equal depths keep gid order);
//   2. each item, in that depth order, emits one (tile id, depth position)
//      pair per tile its footprint ellipse meets, and the K pairs are
//      sorted stably by tile id
//      alone (ceil(log2 tiles) bits, 2-3 passes).
// The result is ordered by (tile, depth, gid) -- the per-tile front-to-back
// lists -- while the wide K-sized sort only moves the tile bits.
//
// Partitioning: a fixed grid of G blocks (one wave: G is the SM count times
// the CTAs of the pass that fit on an SM, at most 4); block b owns the
// contiguous segment [b*seg, (b+1)*seg) with seg = ceil(n / G) rounded up
// to the tile size, so a block's output for a digit always precedes block
// b+1's (stability across blocks); inside a block, tiles are taken in order
// and each key is ranked stably within its warp by one ballot per digit
// bit (the lanes holding the same digit, then those before it).  The first
// digit pass's histogram can be counted by the kernel that writes the keys
// (compaction, pair expansion), which saves that pass's upsweep.
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>
#include <type_traits>
#include "pvg_internal.cuh"

namespace pvg {
namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 4;
constexpr int kScanChunk = kScanThreads * kScanItems;  // 1024

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
// keys per thread of the radix passes: 16 for large sorts (fewer tiles,
// fewer barriers per key), 4 when the capacity is at most
// kSmallSort (a block's chain of dependent steps is shorter)
constexpr int kSortItems = 16;
constexpr int kSmallItems = 4;
constexpr uint32_t kSmallSort = 4u << 20;
constexpr uint32_t kLateSortKeys = 12u << 20;  // capacity from which the wide sort reads values late
constexpr int kRadix = kSortRadix;

constexpr uint32_t kEmitChunk = 2048;      // pair outputs per expansion chunk
constexpr uint32_t kEmitChunkSmall = 512;  // of the small frames
constexpr int kEmitThreads = 256;
static_assert(kEmitChunk % kEmitThreads == 0 && kEmitChunkSmall % kEmitThreads == 0, "whole warps per expansion pass");
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// inclusive warp scan
__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

// exclusive block scan over blockDim.x (multiple of 32, <= 1024) values;
// returns the exclusive prefix, *total receives the block sum.  Uses
// 33 words of shared memory.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t *smem, uint32_t *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const uint32_t incl = warp_incl_scan(v);
    if (lane == 31) smem[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < nw ? smem[lane] : 0;
        const uint32_t wi = warp_incl_scan(w);
        if (lane < nw) smem[lane] = wi - w;
        if (lane == 31) smem[32] = wi;
    }
    __syncthreads();
    const uint32_t r = smem[warp] + incl - v;
    *total = smem[32];
    __syncthreads();
    return r;
}

__device__ __forceinline__ void segment_of(uint32_t n, int G, int align, uint32_t *b0, uint32_t *b1) {
    uint32_t seg = (n + G - 1) / G;
    seg = (seg + align - 1) / align * align;
    const uint64_t s = (uint64_t)blockIdx.x * seg;
    *b0 = (uint32_t)(s < n ? s : n);
    const uint64_t e = s + seg;
    *b1 = (uint32_t)(e < n ? e : n);
}

// ---------------------------------------------------------------- scans

// Functor protocol: n() element count, value(i) item's count,
// apply(i, offset) consumes the exclusive prefix.
// inv: set to 0xffffffff for the invisible items (the depth sort's last
// pass writes the visible ones' positions)
struct CompactF {
    const uint32_t *cnt, *zkey;
    uint32_t *keys_out, *vals_out, *inv;
    uint32_t n_items;
    __device__ uint32_t n() const { return n_items; }
    __device__ uint32_t value(uint32_t i) const { return cnt[i] > 0u ? 1u : 0u; }
    __device__ void apply(uint32_t i, uint32_t off, uint32_t v) const {
        if (v) {
            keys_out[off] = zkey[i];
            vals_out[off] = i;
        } else {
            inv[i] = 0xffffffffu;
        }
    }
};

// Count scan of the per-visible-item tile counts.  apply() stores the
// item's first output position and, for every chunk of kEmitChunk outputs
// that starts inside the item's outputs, the item index, so the expansion
// kernel can find each chunk's items without a global search.
struct EmitF {
    const uint32_t *d_m;
    const uint32_t *vis_cnt;
    uint32_t *vis_off;
    uint32_t *chunk_start;
    uint32_t capacity;
    __device__ uint32_t n() const { return *d_m; }
    __device__ uint32_t value(uint32_t m) const { return vis_cnt[m]; }
    __device__ void apply(uint32_t m, uint32_t off, uint32_t v) const {
        vis_off[m] = off;
        if (v == 0) return;
        const uint32_t end = min(off + v, capacity);
        for (uint32_t c = (off + kEmitChunk - 1) / kEmitChunk; c * kEmitChunk < end; c++) chunk_start[c] = m;
    }
};

// zero (optional): nzero words that a later kernel of the sequence
// accumulates into or fills sparsely, zeroed here grid-wide (saving a
// memset node between kernel launches)
template <class F>
__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(F f, uint32_t *partials, uint32_t *zero,
                                                              uint32_t nzero) {
    pdl_enter();
    __shared__ uint32_t smem[33];
    if (zero)
        for (uint32_t i = blockIdx.x * kScanThreads + threadIdx.x; i < nzero; i += gridDim.x * kScanThreads)
            zero[i] = 0u;
    uint32_t b0, b1;
    segment_of(f.n(), gridDim.x, kScanChunk, &b0, &b1);
    uint32_t acc = 0;
    for (uint32_t i = b0 + threadIdx.x; i < b1; i += kScanThreads) acc += f.value(i);
    uint32_t total;
    block_excl_scan(acc, smem, &total);
    if (threadIdx.x == 0) partials[blockIdx.x] = total;
}

// exclusive scan of G partials in place (one block of 1024 threads);
// *total = sum; if cap_flag != NULL and total > capacity, set *cap_flag.
__global__ void __launch_bounds__(1024) k_scan_partials(uint32_t *partials, int G, uint32_t *total,
                                                        uint32_t capacity, uint32_t *cap_flag) {
    pdl_enter();
    __shared__ uint32_t smem[33];
    const uint32_t v = threadIdx.x < (unsigned)G ? partials[threadIdx.x] : 0u;
    uint32_t tot;
    const uint32_t ex = block_excl_scan(v, smem, &tot);
    if (threadIdx.x < (unsigned)G) partials[threadIdx.x] = ex;
    if (threadIdx.x == 0) {
        *total = tot;
        if (cap_flag && tot > capacity) *cap_flag = 1u;
    }
}

template <class F>
__global__ void __launch_bounds__(kScanThreads) k_scan_apply(F f, const uint32_t *partials, uint32_t *zero,
                                                             uint32_t nzero) {
    pdl_enter();
    __shared__ uint32_t smem[33];
    if (zero)
        for (uint32_t i = blockIdx.x * kScanThreads + threadIdx.x; i < nzero; i += gridDim.x * kScanThreads)
            zero[i] = 0u;
    uint32_t b0, b1;
    segment_of(f.n(), gridDim.x, kScanChunk, &b0, &b1);
    uint32_t base = partials[blockIdx.x];
    for (uint32_t c0 = b0; c0 < b1; c0 += kScanChunk) {
        // blocked arrangement: thread t owns items c0 + t*4 .. +3
        uint32_t v[kScanItems];
        uint32_t sum = 0;
        const uint32_t first = c0 + threadIdx.x * kScanItems;
#pragma unroll
        for (int k = 0; k < kScanItems; k++) {
            const uint32_t i = first + k;
            v[k] = i < b1 ? f.value(i) : 0u;
            sum += v[k];
        }
        uint32_t total;
        uint32_t off = base + block_excl_scan(sum, smem, &total);
#pragma unroll
        for (int k = 0; k < kScanItems; k++) {
            const uint32_t i = first + k;
            if (i < b1) f.apply(i, off, v[k]);
            off += v[k];
        }
        base += total;
    }
}

// k_scan_apply for the compaction of the visible items, which also writes
// inv[i] = 0xffffffff for the invisible items and counts the first digit
// pass of the depth sort that follows: hist[d * sort_G + b] = keys with
// low byte d in the sort block b that owns their output position (the
// sort's partition of M keys into sort_G segments of whole tiles of
// sort_tile keys).  A block's outputs are contiguous, so its counts are
// summed in shared memory and added with at most 256 atomics per sort
// block they touch.  hist is zeroed by the compaction's reduce kernel.
constexpr int kCompactSpan = 4;  // sort blocks one apply block's outputs can touch (checked; else direct atomics)
__global__ void __launch_bounds__(kScanThreads) k_compact_apply(CompactF f, const uint32_t *partials,
                                                               const uint32_t *d_m, uint32_t *hist, int sort_G,
                                                               uint32_t sort_tile) {
    pdl_enter();
    __shared__ uint32_t smem[33];
    __shared__ uint32_t s_hist[kCompactSpan][kRadix];
    for (int k = threadIdx.x; k < kCompactSpan * kRadix; k += kScanThreads) (&s_hist[0][0])[k] = 0u;
    uint32_t b0, b1;
    segment_of(f.n(), gridDim.x, kScanChunk, &b0, &b1);
    const uint32_t M = *d_m;
    const uint32_t seg = ((M + sort_G - 1) / sort_G + sort_tile - 1) / sort_tile * sort_tile;
    const uint32_t block_base = partials[blockIdx.x];
    const uint32_t sb0 = block_base / max(seg, 1u);  // first sort block of this block's outputs
    uint32_t base = block_base;
    __syncthreads();
    for (uint32_t c0 = b0; c0 < b1; c0 += kScanChunk) {
        uint32_t v[kScanItems];
        uint32_t sum = 0;
        const uint32_t first = c0 + threadIdx.x * kScanItems;
#pragma unroll
        for (int k = 0; k < kScanItems; k++) {
            const uint32_t i = first + k;
            v[k] = i < b1 ? f.value(i) : 0u;
            sum += v[k];
        }
        uint32_t total;
        uint32_t off = base + block_excl_scan(sum, smem, &total);
#pragma unroll
        for (int k = 0; k < kScanItems; k++) {
            const uint32_t i = first + k;
            if (i < b1) {
                f.apply(i, off, v[k]);
                if (v[k]) {
                    const uint32_t d = f.zkey[i] & (kRadix - 1u);
                    const uint32_t sb = off / seg - sb0;
                    if (sb < (uint32_t)kCompactSpan) atomicAdd(&s_hist[sb][d], 1u);
                    else atomicAdd(&hist[(size_t)d * sort_G + sb0 + sb], 1u);
                }
            }
            off += v[k];
        }
        base += total;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < kCompactSpan * kRadix; k += kScanThreads) {
        const uint32_t c = (&s_hist[0][0])[k];
        const uint32_t sb = sb0 + (uint32_t)(k / kRadix), d = (uint32_t)(k % kRadix);
        if (c) atomicAdd(&hist[(size_t)d * sort_G + sb], c);
    }
}

int scan_blocks(uint32_t capacity) {
    uint32_t g = (capacity + kScanChunk - 1) / kScanChunk;
    if (g < 1) g = 1;
    if (g > kMaxScanBlocks) g = kMaxScanBlocks;
    return (int)g;
}

// CTAs of the 16-keys-per-thread downsweep (late: the variant with late
// value reads) that fit on one SM (its registers and 43 KB of shared
// memory), at most 4: the grid of the wide sorts stays one wave, since a
// block's tiles run one after another and a second wave of blocks would
// double the pass.  Read once.
int wide_sort_blocks_per_sm(bool late);

int sort_blocks(uint32_t capacity, int tile) {
    uint32_t g = (capacity + tile - 1) / tile;
    const int per_sm = tile == kSortThreads * kSortItems ? wide_sort_blocks_per_sm(capacity >= kLateSortKeys) : 4;
    const uint32_t cap = (uint32_t)std::min(kMaxSortBlocks, per_sm * device_sm_count());
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

// ---------------------------------------------------------------- radix

template <int ITEMS>
__global__ void __launch_bounds__(kSortThreads) k_radix_upsweep(const uint32_t *keys, const uint32_t *d_n,
                                                                uint32_t cap, int shift, uint32_t mask,
                                                                uint32_t *hist) {
    pdl_enter();
    __shared__ uint32_t sh[kRadix];
    for (int d = threadIdx.x; d < kRadix; d += kSortThreads) sh[d] = 0;
    __syncthreads();
    uint32_t b0, b1;
    segment_of(min(*d_n, cap), gridDim.x, kSortThreads * ITEMS, &b0, &b1);
    for (uint32_t i = b0 + threadIdx.x; i < b1; i += kSortThreads) atomicAdd(&sh[(keys[i] >> shift) & mask], 1u);
    __syncthreads();
    for (int d = threadIdx.x; d < kRadix; d += kSortThreads) hist[d * gridDim.x + blockIdx.x] = sh[d];
}

// Row scan of the digit-major histogram hist[d * G + b], one block per
// digit d: exclusive prefix over the G blocks in place, row total to
// totals[d].  The downsweep adds the exclusive prefix of the totals over
// the digits.  G <= 1024.
__global__ void __launch_bounds__(1024) k_radix_scan(uint32_t *hist, uint32_t *totals, int G) {
    pdl_enter();
    __shared__ uint32_t smem[33];
    uint32_t *row = hist + (size_t)blockIdx.x * G;
    const uint32_t v = (int)threadIdx.x < G ? row[threadIdx.x] : 0u;
    uint32_t tot;
    const uint32_t ex = block_excl_scan(v, smem, &tot);
    if ((int)threadIdx.x < G) row[threadIdx.x] = ex;
    if (threadIdx.x == 0) totals[blockIdx.x] = tot;
}

// Expansion of the sorted visible items into (tile id, depth position)
// pairs, one chunk of kEmitChunk outputs at a time.  The item of every
// output comes from a block max-scan of start markers (each item whose
// first output falls in the chunk marks that slot with its m; the scan
// carries the last mark forward).  Its r-th pair is the r-th tile, row by
// row, of the rectangle tiles that its footprint ellipse meets: read from
// the item's packed row table when it has one (at most kTabRows rows).  The
// chunk's items without a table are listed and taken one after another by
// whole warps, which evaluate 32 rows of the stored ellipse at once and then
// write all of the item's outputs in those rows (evaluating the rows for
// every 32 outputs made the batched views' expansion 292 M warp instructions
// for 40 M pairs).  The kernel also counts the first digit pass of the tile
// sort that follows (hist, zeroed by the scan before it; NULL: none): each
// chunk's outputs are contiguous, so their counts are summed in shared
// memory per sort block and added with atomics.
template <uint32_t kEmitChunk>
__global__ void __launch_bounds__(kEmitThreads, 4) k_expand_pairs(const uint32_t *__restrict__ vis_off,
                                                              const uint32_t *__restrict__ vis_cnt,
                                                              const uint32_t *__restrict__ chunk_start,
                                                              const uint2 *__restrict__ rect,
                                                              const uint4 *__restrict__ rowtab,
                                                              const float4 *__restrict__ ell, int tile_w,
                                                              int tile_h, const uint32_t *__restrict__ vis_tile,
                                                              const uint32_t *__restrict__ vis_stride,
                                                              const ViewDesc *views, int nv, const uint32_t *d_m,
                                                              const uint32_t *d_k, uint32_t capacity,
                                                              uint32_t *__restrict__ keys, uint32_t *__restrict__ vals,
                                                              uint32_t *__restrict__ hist, int sort_G,
                                                              uint32_t sort_tile) {
    pdl_enter();
    constexpr int kPer = kEmitChunk / kEmitThreads;  // slots per thread in the scan
    __shared__ uint32_t s_item[kEmitChunk];
    __shared__ uint32_t s_big[kEmitChunk];  // the chunk's items without a table
    __shared__ uint32_t s_nbig;
    __shared__ uint32_t s_warp[kEmitThreads / 32];
    __shared__ uint32_t s_hist[kCompactSpan][kRadix];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t M = *d_m;
    const uint32_t K = min(*d_k, capacity);
    const uint32_t nchunks = (K + kEmitChunk - 1) / kEmitChunk;
    // the tile sort's partition of the K pairs (its segment of whole tiles)
    const uint32_t seg = max(((K + sort_G - 1) / sort_G + sort_tile - 1) / sort_tile * sort_tile, 1u);
    for (uint32_t c = blockIdx.x; c < nchunks; c += gridDim.x) {
        const uint32_t j0 = c * kEmitChunk;
        const uint32_t m_lo = chunk_start[c];
        const uint32_t m_hi = (c + 1 < nchunks) ? chunk_start[c + 1] : M - 1;
        // sort blocks of the chunk's outputs: sb0 .. sb0 + nsb - 1 counted in
        // shared memory (any beyond kCompactSpan straight into hist)
        const uint32_t sb0 = j0 / seg;
        const int nsb = !hist ? 0 : (int)min((min(j0 + kEmitChunk, K) - 1) / seg - sb0 + 1, (uint32_t)kCompactSpan);
        __syncthreads();
        if (threadIdx.x == 0) s_nbig = 0u;
        for (int q = threadIdx.x; q < (int)kEmitChunk; q += kEmitThreads) s_item[q] = 0u;
        for (int q = threadIdx.x; q < nsb * kRadix; q += kEmitThreads) (&s_hist[0][0])[q] = 0u;
        __syncthreads();
        // marks: slot 0 holds the item containing j0 (chunk_start); a
        // non-empty item starting inside the chunk marks its first slot
        // (distinct slots: non-empty items start at distinct offsets)
        if (threadIdx.x == 0) s_item[0] = m_lo;
        for (uint32_t m = m_lo + threadIdx.x; m <= m_hi; m += kEmitThreads) {
            const uint32_t o = vis_off[m];
            const uint2 rc = rect[m];
            const bool starts = o >= j0 && o - j0 < kEmitChunk && vis_cnt[m] > 0u;
            if (starts) s_item[o - j0] = m;
            if ((starts || m == m_lo) &&
                !has_row_table(rc.x & 0xffffu, rc.x >> 16, rc.y & 0xffffu, rc.y >> 16))
                s_big[atomicAdd(&s_nbig, 1u)] = m;
        }
        __syncthreads();
        // inclusive max-scan of the marks: kPer consecutive slots per
        // thread, then across the warp, then across the warps
        uint32_t loc[kPer];
        uint32_t run = 0;
#pragma unroll
        for (int i = 0; i < kPer; i++) {
            run = max(run, s_item[threadIdx.x * kPer + i]);
            loc[i] = run;
        }
        uint32_t wrun = run;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, wrun, o);
            if (lane >= o) wrun = max(wrun, y);
        }
        if (lane == 31) s_warp[warp] = wrun;
        uint32_t before = __shfl_up_sync(kFull, wrun, 1);
        if (lane == 0) before = 0;
        __syncthreads();
        for (int w = 0; w < warp; w++) before = max(before, s_warp[w]);
#pragma unroll
        for (int i = 0; i < kPer; i++) s_item[threadIdx.x * kPer + i] = max(loc[i], before);
        __syncthreads();
        // output j of item m: its tile's id, and its digit counted
        auto emit = [&](uint32_t j, uint32_t m, uint32_t key) {
            keys[j] = key;
            vals[j] = m;
            if (!hist) return;
            const uint32_t d = key & (kRadix - 1u), sb = j / seg - sb0;
            if (sb < (uint32_t)nsb) atomicAdd(&s_hist[sb][d], 1u);
            else atomicAdd(&hist[(size_t)d * sort_G + sb0 + sb], 1u);
        };
        const uint32_t tile0 = nv > 1 ? 0u : views[0].tile_base, stride0 = nv > 1 ? 0u : (uint32_t)views[0].tiles_x;
        // items with a table, an output per thread; four outputs of a thread
        // at a time, their items' data loaded together: the loads' latency
        // bounds the expansion, not its bytes
        constexpr int kAhead = kPer < 4 ? kPer : 4;
        static_assert(kPer % kAhead == 0, "whole batches of outputs");
        for (uint32_t q0 = threadIdx.x; q0 < kEmitChunk && j0 + q0 < K; q0 += kAhead * kEmitThreads) {
            uint32_t am[kAhead], aoff[kAhead], atile[kAhead], astride[kAhead];
            uint2 arc[kAhead];
            uint4 atab[kAhead];
#pragma unroll
            for (int i = 0; i < kAhead; i++) am[i] = j0 + q0 + i * kEmitThreads < K ? s_item[q0 + i * kEmitThreads] : m_lo;
#pragma unroll
            for (int i = 0; i < kAhead; i++) {
                aoff[i] = vis_off[am[i]];
                arc[i] = rect[am[i]];
                atab[i] = rowtab[am[i]];  // (not written for items without a table, and not used then)
                atile[i] = nv > 1 ? vis_tile[am[i]] : 0u;
                astride[i] = nv > 1 ? vis_stride[am[i]] : stride0;
            }
#pragma unroll
            for (int i = 0; i < kAhead; i++) {
                const uint32_t j = j0 + q0 + i * kEmitThreads;
                const uint32_t tx0 = arc[i].x & 0xffffu, ty0 = arc[i].x >> 16, tx1 = arc[i].y & 0xffffu, ty1 = arc[i].y >> 16;
                if (j >= K || !has_row_table(tx0, ty0, tx1, ty1)) continue;
                const uint32_t w[4] = {atab[i].x, atab[i].y, atab[i].z, atab[i].w};
                uint32_t r = j - aoff[i], col = 0, row = 0;  // the rows sum to the item's count
#pragma unroll
                for (int t = 0; t < (int)kTabRows; t++) {
                    if (ty0 + t >= ty1) break;
                    const uint32_t v = (w[t >> 1] >> (16 * (t & 1))) & 0xffffu;
                    const uint32_t sp = v >> 8;
                    if (r < sp) {
                        col = (v & 0xffu) + r;
                        row = t;
                        break;
                    }
                    r -= sp;
                }
                const uint32_t first = nv > 1 ? atile[i] : tile0 + ty0 * stride0 + tx0;
                emit(j, am[i], first + row * astride[i] + col);
            }
        }
        // items without a table: one with more than kEmitThreads outputs in
        // the chunk by all warps, 32 outputs each in turn, the others by one
        // warp each
        const uint32_t jend = min(j0 + kEmitChunk, K), nbig = s_nbig;
        for (uint32_t b = 0; b < nbig; b++) {
            const uint32_t m = s_big[b], off = vis_off[m], lo = max(off, j0), hi = min(off + vis_cnt[m], jend);
            if (lo >= hi) continue;
            const bool shared = hi - lo > (uint32_t)kEmitThreads;
            if (!shared && (int)(b % (kEmitThreads / 32)) != warp) continue;
            const uint32_t mine = lo + (shared ? 32u * warp : 0u) + lane, step = shared ? (uint32_t)kEmitThreads : 32u;
            const FootprintEllipse E = load_ellipse(ell, m);
            const uint2 rc = rect[m];
            const uint32_t tx0 = rc.x & 0xffffu, ty0 = rc.x >> 16, tx1 = rc.y & 0xffffu, ty1 = rc.y >> 16;
            const uint32_t stride = nv > 1 ? vis_stride[m] : stride0;
            const uint32_t first = nv > 1 ? vis_tile[m] : tile0 + ty0 * stride0 + tx0;
            uint32_t base = off;  // first output of the 32 rows
            uint32_t j = mine;
            for (uint32_t row0 = ty0; row0 < ty1 && base < hi; row0 += 32) {
                const uint32_t row = row0 + lane;
                uint32_t cx = 0, sp = 0;
                if (row < ty1) {
                    const uint2 cc = footprint_cols(E, row, tile_w, tile_h, tx0, tx1);
                    cx = cc.x;
                    sp = cc.y - cc.x;
                }
                const uint32_t inc = warp_incl_scan(sp);
                const uint32_t end = base + __shfl_sync(kFull, inc, 31);
                while (__any_sync(kFull, j < min(end, hi))) {
                    const bool on = j < min(end, hi);
                    const uint32_t rr = on ? j - base : 0u;
                    uint32_t k = 0;  // first lane whose inclusive sum exceeds rr
#pragma unroll
                    for (int s = 16; s; s >>= 1) {
                        const uint32_t v = __shfl_sync(kFull, inc, k + s - 1);
                        if (v <= rr) k += s;
                    }
                    const uint32_t inc_k = __shfl_sync(kFull, inc, k & 31), sp_k = __shfl_sync(kFull, sp, k & 31);
                    const uint32_t cx_k = __shfl_sync(kFull, cx, k & 31);
                    if (on) {
                        emit(j, m, first + (row0 + k - ty0) * stride + (cx_k - tx0) + rr - (inc_k - sp_k));
                        j += step;
                    }
                }
                base = end;
            }
        }
        __syncthreads();
        for (int q = threadIdx.x; q < nsb * kRadix; q += kEmitThreads) {
            const uint32_t cnt = (&s_hist[0][0])[q];
            if (cnt) atomicAdd(&hist[(size_t)(q % kRadix) * sort_G + sb0 + (uint32_t)(q / kRadix)], cnt);
        }
    }
}

static_assert(kSortThreads == kRadix, "one thread per digit in the downsweep");

template <int TILE>
struct SortSmem {
    uint32_t warp_hist[kSortWarps][kRadix];
    uint32_t off[kRadix];                 // global position of a digit's run, less its place in the tile
    uint32_t keys[TILE];
    uint32_t vals[TILE];
    uint32_t scan[33];
};

// exclusive scan over the block's kSortThreads values, one barrier; smem: a
// word per warp, not written again before the caller's next barrier
__device__ __forceinline__ uint32_t sort_excl_scan(uint32_t v, uint32_t *smem) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t incl = warp_incl_scan(v);
    if (lane == 31) smem[warp] = incl;
    __syncthreads();
    uint32_t before = 0;
#pragma unroll
    for (int w = 0; w < kSortWarps; w++) before += w < warp ? smem[w] : 0u;
    return before + incl - v;
}

// NB: ballots per key in the ranking (the pass's digit width, or 8).  A
// block's tiles follow one another, so a tile's global loads are started as
// soon as the previous tile's keys have left the registers, and complete
// behind its write-out; four barriers per tile.  The ALU pipe is the busiest
// (the ballots; half of its slots), so whole tiles skip the tests of the end
// and a key's place takes one shared load (8M 32-bit pairs, four passes: 311
// -> 297 us; a step of twelve views, 40M pairs: 6,242 -> 6,206 us).
template <int ITEMS, int NB, bool kLateVals>
__device__ __forceinline__ void radix_downsweep(const uint32_t *__restrict__ keys_in,
                                                const uint32_t *__restrict__ vals_in, uint32_t *__restrict__ keys_out,
                                                uint32_t *__restrict__ vals_out, const uint32_t *d_n, uint32_t cap,
                                                int shift, uint32_t mask, const uint32_t *hist,
                                                const uint32_t *totals, uint32_t *__restrict__ inv_out) {
    constexpr int kSortTile = kSortThreads * ITEMS;
    __shared__ SortSmem<kSortTile> S;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t b0, b1;
    segment_of(min(*d_n, cap), gridDim.x, kSortTile, &b0, &b1);
    // kLateVals: the values are read only when they are placed (below),
    // so that a thread holds its keys and ranks but not its values
    // meanwhile (64 registers: four CTAs per SM)
    uint32_t key[ITEMS], val[kLateVals ? 1 : ITEMS];
    const uint32_t mine = warp * (32 * ITEMS) + lane;  // the thread's first place in a tile
    auto load = [&](uint32_t t0) {
#pragma unroll
        for (int j = 0; j < ITEMS; j++) {
            const uint32_t pos = t0 + mine + j * 32;
            key[j] = pos < b1 ? keys_in[pos] : 0u;
            if constexpr (!kLateVals) val[j] = pos < b1 ? vals_in[pos] : 0u;
        }
    };
    if (b0 < b1) load(b0);
    // digit bases: exclusive prefix of the per-digit totals (one thread per
    // digit); thread d keeps digit d's running global offset
    uint32_t base = sort_excl_scan(totals[tid], S.scan) + hist[tid * gridDim.x + blockIdx.x];
    __syncthreads();
    const uint32_t lt = lanemask_lt();
    for (uint32_t t0 = b0; t0 < b1; t0 += kSortTile) {
        const uint32_t n = min(b1 - t0, (uint32_t)kSortTile);
        for (int k = lane; k < kRadix; k += 32) S.warp_hist[warp][k] = 0;
        __syncwarp();
        // place in the tile: first among the warp's keys of its digit; whole
        // tiles need no test of the end
        const bool whole = n == (uint32_t)kSortTile;
        uint32_t rank[ITEMS];
        auto rank_keys = [&](auto all) {
            constexpr bool kWhole = decltype(all)::value;
#pragma unroll
            for (int j = 0; j < ITEMS; j++) {
                const bool valid = kWhole || mine + j * 32 < n;
                const uint32_t d = (key[j] >> shift) & mask;
                uint32_t peers = kWhole ? 0xffffffffu : __ballot_sync(0xffffffffu, valid);
#pragma unroll
                for (int bit = 0; bit < NB; bit++) {
                    const bool on = (d >> bit) & 1u;
                    const uint32_t b = __ballot_sync(0xffffffffu, on);
                    peers &= on ? b : ~b;
                }
                uint32_t before = 0;
                if (valid) before = S.warp_hist[warp][d];
                __syncwarp();
                if (valid && (peers & lt) == 0) S.warp_hist[warp][d] = before + __popc(peers);
                __syncwarp();
                rank[j] = before + __popc(peers & lt);
            }
        };
        if (whole) rank_keys(std::true_type());
        else rank_keys(std::false_type());
        __syncthreads();
        // per digit: the tile's count, its start, the warps' starts
        {
            const int d = tid;  // kSortThreads == kRadix
            uint32_t cnt[kSortWarps], tile_cnt = 0;
#pragma unroll
            for (int w = 0; w < kSortWarps; w++) {
                cnt[w] = S.warp_hist[w][d];
                tile_cnt += cnt[w];
            }
            uint32_t start = sort_excl_scan(tile_cnt, S.scan);
            S.off[d] = base - start;
            base += tile_cnt;
#pragma unroll
            for (int w = 0; w < kSortWarps; w++) {
                S.warp_hist[w][d] = start;
                start += cnt[w];
            }
        }
        __syncthreads();
        auto place = [&](auto all) {
#pragma unroll
            for (int j = 0; j < ITEMS; j++) {
                if (!decltype(all)::value && mine + j * 32 >= n) continue;
                const uint32_t p = S.warp_hist[warp][(key[j] >> shift) & mask] + rank[j];
                S.keys[p] = key[j];
                if constexpr (kLateVals) S.vals[p] = vals_in[t0 + mine + j * 32];
                else S.vals[p] = val[j];
            }
        };
        if (whole) place(std::true_type());
        else place(std::false_type());
        if (t0 + kSortTile < b1) load(t0 + kSortTile);
        __syncthreads();
        // (the next tile's writes to keys, vals, off lie behind its barriers)
#pragma unroll 4
        for (uint32_t p = tid; p < n; p += kSortThreads) {
            const uint32_t k = S.keys[p], v = S.vals[p];
            const uint32_t dst = S.off[(k >> shift) & mask] + p;
            keys_out[dst] = k;
            vals_out[dst] = v;
            if (inv_out) inv_out[v] = dst;
        }
    }
}

// The downsweep for ITEMS keys per thread, values read with the keys; and
// the wide one for long sorts (kLateSortKeys and more), with late value
// reads, held to 64 registers: four CTAs of 43 KB per SM instead of three.
// A block of a long sort walks tens of tiles, where the extra CTA per SM
// pays (64M random keys: 2.09 vs 2.40 ms); with a few tiles per block the
// late reads' latency shows instead (a 3.3M-pair tile sort: 0.070 vs 0.061
// ms).
template <int ITEMS, int NB>
__global__ void __launch_bounds__(kSortThreads, ITEMS == kSortItems ? 3 : 4) k_radix_downsweep(const uint32_t *__restrict__ keys_in,
                                                                  const uint32_t *__restrict__ vals_in,
                                                                  uint32_t *__restrict__ keys_out,
                                                                  uint32_t *__restrict__ vals_out,
                                                                  const uint32_t *d_n, uint32_t cap, int shift,
                                                                  uint32_t mask, const uint32_t *hist,
                                                                  const uint32_t *totals,
                                                                  uint32_t *__restrict__ inv_out) {
    pdl_enter();
    radix_downsweep<ITEMS, NB, false>(keys_in, vals_in, keys_out, vals_out, d_n, cap, shift, mask, hist, totals,
                                      inv_out);
}

template <int NB>
__global__ void __launch_bounds__(kSortThreads, 4) k_radix_downsweep_wide(const uint32_t *__restrict__ keys_in,
                                                                           const uint32_t *__restrict__ vals_in,
                                                                           uint32_t *__restrict__ keys_out,
                                                                           uint32_t *__restrict__ vals_out,
                                                                           const uint32_t *d_n, uint32_t cap,
                                                                           int shift, uint32_t mask,
                                                                           const uint32_t *hist,
                                                                           const uint32_t *totals,
                                                                           uint32_t *__restrict__ inv_out) {
    pdl_enter();
    radix_downsweep<kSortItems, NB, true>(keys_in, vals_in, keys_out, vals_out, d_n, cap, shift, mask, hist, totals,
                                          inv_out);
}

// [start, end) of every tile's run in the sorted keys.  Eight keys per
// thread per sweep (two 16-byte loads and the two neighbours), so that
// few dependent sweeps remain.
__global__ void __launch_bounds__(256) k_ranges(const uint32_t *__restrict__ keys, const uint32_t *d_k,
                                                uint32_t capacity, uint2 *__restrict__ ranges) {
    pdl_enter();
    constexpr uint32_t kNone = 0xffffffffu;  // no tile has this id
    const uint32_t K = min(*d_k, capacity);
    const uint32_t stride = gridDim.x * blockDim.x * 8u;
    for (uint32_t j0 = (blockIdx.x * blockDim.x + threadIdx.x) * 8u; j0 < K; j0 += stride) {
        uint32_t k[10];  // keys[j0 - 1 .. j0 + 8]
        k[0] = j0 > 0 ? keys[j0 - 1] : kNone;
        if (j0 + 8 <= K) {
            const uint4 a = reinterpret_cast<const uint4 *>(keys + j0)[0];
            const uint4 b = reinterpret_cast<const uint4 *>(keys + j0)[1];
            k[1] = a.x; k[2] = a.y; k[3] = a.z; k[4] = a.w;
            k[5] = b.x; k[6] = b.y; k[7] = b.z; k[8] = b.w;
        } else {
#pragma unroll
            for (int i = 0; i < 8; i++) k[1 + i] = j0 + i < K ? keys[j0 + i] : kNone;
        }
        k[9] = j0 + 8 < K ? keys[j0 + 8] : kNone;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const uint32_t t = k[1 + i];
            if (t == kNone) break;
            if (k[i] != t) ranges[t].x = j0 + i;
            if (k[2 + i] != t) ranges[t].y = j0 + i + 1;
        }
    }
}

int wide_sort_blocks_per_sm(bool late) {
    static std::atomic<int> cached[2] = {{0}, {0}};
    int n = cached[late].load(std::memory_order_relaxed);
    if (n > 0) return n;
    int occ = 0;
    const cudaError_t e =
        late ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_radix_downsweep_wide<8>, kSortThreads, 0)
             : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_radix_downsweep<kSortItems, 8>, kSortThreads, 0);
    if (e != cudaSuccess) {
        cudaGetLastError();
        occ = 3;
    }
    n = std::max(1, std::min(occ, 4));
    cached[late].store(n, std::memory_order_relaxed);
    return n;
}

struct TempLayout {
    uint32_t *hist;      // kRadix * kMaxSortBlocks
    uint32_t *partials;  // kMaxScanBlocks
    uint32_t *totals;    // kRadix (shares the partials' space: never live together)
};

TempLayout temp_layout(void *temp) {
    TempLayout t;
    t.hist = (uint32_t *)temp;
    t.partials = t.hist + kRadix * kMaxSortBlocks;
    t.totals = t.partials;
    return t;
}

}  // namespace

static_assert(kSortTempBytes >= sizeof(uint32_t) * ((size_t)kRadix * kMaxSortBlocks + kMaxScanBlocks),
              "sort scratch layout");
size_t sort_temp_bytes() { return kSortTempBytes; }

void compact_visible(const Params &p, uint32_t *keys_out, uint32_t *vals_out, uint32_t *inv, void *temp,
                     cudaStream_t s) {
    TempLayout t = temp_layout(temp);
    CompactF f{p.item_cnt, p.item_zkey, keys_out, vals_out, inv, p.n_items};
    const int G = scan_blocks(p.n_items);
    // the depth sort's partition (radix_sort_pairs with capacity n_items)
    const int sort_items = p.n_items <= kSmallSort ? kSmallItems : kSortItems;
    const int sort_G = sort_blocks(p.n_items, kSortThreads * sort_items);
    note_launch();
    pdl_launch(k_scan_reduce<CompactF>, G, kScanThreads, 0, s, f, t.partials, t.hist, (uint32_t)(kRadix * sort_G));
    note_launch();
    pdl_launch(k_scan_partials, 1, 1024, 0, s, t.partials, G, &p.counters[0], 0xffffffffu, nullptr);
    note_launch();
    pdl_launch(k_compact_apply, G, kScanThreads, 0, s, f, (const uint32_t *)t.partials,
               (const uint32_t *)&p.counters[0], t.hist, sort_G, (uint32_t)(kSortThreads * sort_items));
}

template <int ITEMS>
void radix_passes(uint32_t *keys, uint32_t *vals, uint32_t *keys_alt, uint32_t *vals_alt, const uint32_t *d_count,
                  uint32_t capacity, int begin_bit, int end_bit, void *temp, cudaStream_t s, bool *result_in_alt,
                  uint32_t *inv_out, bool first_hist);

void radix_sort_pairs(uint32_t *keys, uint32_t *vals, uint32_t *keys_alt, uint32_t *vals_alt,
                      const uint32_t *d_count, uint32_t capacity, int begin_bit, int end_bit, void *temp,
                      cudaStream_t s, bool *result_in_alt, uint32_t *inv_out, bool first_hist) {
    if (capacity <= kSmallSort)
        radix_passes<kSmallItems>(keys, vals, keys_alt, vals_alt, d_count, capacity, begin_bit, end_bit, temp, s,
                                  result_in_alt, inv_out, first_hist);
    else
        radix_passes<kSortItems>(keys, vals, keys_alt, vals_alt, d_count, capacity, begin_bit, end_bit, temp, s,
                                 result_in_alt, inv_out, first_hist);
}

template <int ITEMS>
void radix_passes(uint32_t *keys, uint32_t *vals, uint32_t *keys_alt, uint32_t *vals_alt, const uint32_t *d_count,
                  uint32_t capacity, int begin_bit, int end_bit, void *temp, cudaStream_t s, bool *result_in_alt,
                  uint32_t *inv_out, bool first_hist) {
    TempLayout t = temp_layout(temp);
    const int G = sort_blocks(capacity, kSortThreads * ITEMS);
    bool alt = false;
    for (int b = begin_bit; b < end_bit;) {
        const int nb = (end_bit - b) >= 8 ? 8 : (end_bit - b);
        const uint32_t mask = (1u << nb) - 1u;
        const uint32_t *ki = alt ? keys_alt : keys;
        const uint32_t *vi = alt ? vals_alt : vals;
        uint32_t *ko = alt ? keys : keys_alt;
        uint32_t *vo = alt ? vals : vals_alt;
        if (!(first_hist && b == begin_bit)) {  // else counted by the producer of the keys
            note_launch();
            pdl_launch(k_radix_upsweep<ITEMS>, G, kSortThreads, 0, s, ki, d_count, capacity, b, mask, t.hist);
        }
        note_launch();
        pdl_launch(k_radix_scan, kRadix, 1024, 0, s, t.hist, t.totals, G);
        note_launch();
        uint32_t *inv_pass = b + nb >= end_bit ? inv_out : nullptr;  // the last pass only
        // one ballot per digit bit: the last pass of a sort by fewer than a
        // multiple of 8 bits ranks with fewer ballots
#define PVG_DOWNSWEEP(NBITS)                                                                                    \
    case NBITS:                                                                                                 \
        if (ITEMS == kSortItems && capacity >= kLateSortKeys)                                                  \
            pdl_launch(k_radix_downsweep_wide<NBITS>, G, kSortThreads, 0, s, ki, vi, ko, vo, d_count, capacity, b, \
                       mask, t.hist, t.totals, inv_pass);                                                       \
        else                                                                                                    \
            pdl_launch(k_radix_downsweep<ITEMS, NBITS>, G, kSortThreads, 0, s, ki, vi, ko, vo, d_count, capacity, b, \
                       mask, t.hist, t.totals, inv_pass);                                                       \
        break;
        switch (nb) {
            PVG_DOWNSWEEP(1) PVG_DOWNSWEEP(2) PVG_DOWNSWEEP(3) PVG_DOWNSWEEP(4)
            PVG_DOWNSWEEP(5) PVG_DOWNSWEEP(6) PVG_DOWNSWEEP(7)
            default: PVG_DOWNSWEEP(8)
        }
#undef PVG_DOWNSWEEP
        alt = !alt;
        b += nb;
    }
    *result_in_alt = alt;
}

// scan of the per-visible tile counts: K -> counters[1], overflow flag ->
// counters[2]; then emission of the (tile, m) pairs in depth order.
void scan_count_pairs(const Params &p, void *temp, cudaStream_t s) {
    TempLayout t = temp_layout(temp);
    EmitF f{&p.counters[0], p.vis_cnt, p.vis_off, p.chunk_start, p.pair_capacity};
    const int G = scan_blocks(p.n_items);
    // the tile ranges are zeroed here for k_ranges, which writes only the
    // non-empty tiles' (no memset node in the launch sequence)
    note_launch();
    pdl_launch(k_scan_reduce<EmitF>, G, kScanThreads, 0, s, f, t.partials, reinterpret_cast<uint32_t *>(p.ranges),
               (uint32_t)(2 * p.total_tiles));
    note_launch();
    pdl_launch(k_scan_partials, 1, 1024, 0, s, t.partials, G, &p.counters[1], p.pair_capacity, &p.counters[2]);
}

// the small frames' chunks are the shorter ones
static_assert(kEmitChunkSmall <= kEmitChunk, "entries for either chunk length");
size_t emit_chunks(uint32_t capacity) { return capacity / kEmitChunkSmall + 2; }

void scan_emit_pairs(const Params &p, void *temp, cudaStream_t s) {
    TempLayout t = temp_layout(temp);
    EmitF f{&p.counters[0], p.vis_cnt, p.vis_off, p.chunk_start, p.pair_capacity};
    const int G = scan_blocks(p.n_items);
    // the tile sort's partition (radix_sort_pairs with capacity pair_capacity);
    // its first histogram is zeroed here and counted by the expansion
    const int sort_items = p.pair_capacity <= kSmallSort ? kSmallItems : kSortItems;
    const int sort_G = sort_blocks(p.pair_capacity, kSortThreads * sort_items);
    note_launch();
    pdl_launch(k_scan_apply<EmitF>, G, kScanThreads, 0, s, f, (const uint32_t *)t.partials, t.hist,
               (uint32_t)(kRadix * sort_G));
    uint32_t grid = (uint32_t)((p.pair_capacity + kEmitChunk - 1) / kEmitChunk);
    if (grid < 1) grid = 1;
    if (grid > (uint32_t)(8 * device_sm_count())) grid = 8 * device_sm_count();
    note_launch();
    pdl_launch(k_expand_pairs<kEmitChunk>, grid, kEmitThreads, 0, s, p.vis_off, p.vis_cnt, p.chunk_start, p.rect, p.rowtab, p.ell,
                                                 p.tile_w, p.tile_h,
                                                 p.vis_tile, p.vis_stride, p.views, p.n_views,
                                                 &p.counters[0], &p.counters[1], p.pair_capacity, p.pair_keys,
                                                 p.pair_vals, t.hist, sort_G, (uint32_t)(kSortThreads * sort_items));
}

// Tile order for the compositor: heaviest lists first (64 log-spaced
// length buckets, longest bucket first), so the long tiles start at once
// and the short ones fill in behind them.  Order within a bucket is left
// to the atomics (each tile's result does not depend on when it runs).
// walk (optional): order by the tiles' walk lengths instead (the adjoint:
// each tile's largest stop position, which the forward recorded).
// One cluster of kOrderCtas CTAs (rank: this one's), which count their
// shares of the tiles and read one another's counts; a warp adds once per
// bucket it meets (with 55,000 tiles one CTA with an atomic per tile took 60
// us, most tiles being in a few buckets).  Every CTA of the cluster calls.
// CTAS = 1: one CTA without a cluster.
constexpr int kOrderCtas = 8;

template <int CTAS>
__device__ __forceinline__ void tile_order(uint32_t rank, const uint2 *__restrict__ ranges,
                                                   const uint32_t *walk, uint32_t n_tiles,
                                                   uint32_t *__restrict__ order) {
    __shared__ uint32_t cnt[64], place[64];
    __shared__ uint32_t smem[33];
    if (threadIdx.x < 64) cnt[threadIdx.x] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const uint32_t stride = CTAS * blockDim.x, first = rank * blockDim.x + threadIdx.x;
    // the lane's tile's bucket (64: none), and the lanes of its bucket
    auto bucket = [&](uint32_t t) {
        if (t >= n_tiles) return 64;
        const uint32_t len = walk ? walk[t] : ranges[t].y - ranges[t].x;
        return 63 - min(63, (int)(lg2_approx((float)len + 1.0f) * 3.0f));  // longest first
    };
    auto take = [&](uint32_t *counts, int b, uint32_t peers) {
        uint32_t base = 0;
        if (b < 64 && lane == __ffs(peers) - 1) base = atomicAdd(&counts[b], __popc(peers));
        return __shfl_sync(0xffffffffu, base, __ffs(peers) - 1) + __popc(peers & lanemask_lt());
    };
    const uint32_t rounds = (n_tiles + stride - 1) / stride;
    for (uint32_t k = 0; k < rounds; k++) {
        const int b = bucket(first + k * stride);
        take(cnt, b, __match_any_sync(0xffffffffu, b));
    }
    if constexpr (CTAS > 1) cooperative_groups::this_cluster().sync();
    else __syncthreads();
    // places: the longer buckets of all CTAs, then this bucket's of the CTAs before
    uint32_t all = 0, before = 0;
    if (threadIdx.x < 64) {
        if constexpr (CTAS > 1) {
            for (uint32_t c = 0; c < CTAS; c++) {
                const uint32_t v = cooperative_groups::this_cluster().map_shared_rank(cnt, c)[threadIdx.x];
                all += v;
                before += c < rank ? v : 0u;
            }
        } else {
            all = cnt[threadIdx.x];
        }
    }
    uint32_t tot;
    const uint32_t ex = block_excl_scan(all, smem, &tot);
    if (threadIdx.x < 64) place[threadIdx.x] = ex + before;
    // no CTA leaves, or counts again, while another reads its counts
    if constexpr (CTAS > 1) cooperative_groups::this_cluster().sync();
    else __syncthreads();
    for (uint32_t k = 0; k < rounds; k++) {
        const uint32_t t = first + k * stride;
        const int b = bucket(t);
        const uint32_t at = take(place, b, __match_any_sync(0xffffffffu, b));
        if (b < 64) order[at] = t;
    }
}

__global__ void __cluster_dims__(kOrderCtas, 1, 1) __launch_bounds__(1024)
    k_tile_order(const uint2 *__restrict__ ranges, uint32_t n_tiles, uint32_t *__restrict__ order,
                 uint32_t *__restrict__ walk) {
    pdl_enter();
    if (walk)
        for (uint32_t t = blockIdx.x * 1024u + threadIdx.x; t < n_tiles; t += kOrderCtas * 1024u) walk[t] = 0u;
    tile_order<kOrderCtas>(blockIdx.x, ranges, nullptr, n_tiles, order);
}

// The adjoint's first kernel: rows [0, *d_m) of the image-space gradients
// zeroed (the visible items', which the adjoint accumulates) by all clusters
// but the last, which orders the tiles by their walk lengths and resets the
// per-item adjoint's chunk ticket (counters[3]).
__global__ void __cluster_dims__(kOrderCtas, 1, 1) __launch_bounds__(1024) k_bwd_prep(double *__restrict__ g2m, float *__restrict__ g2d,
                                                  const uint32_t *d_m, const uint32_t *walk, uint32_t n_tiles,
                                                  uint32_t *__restrict__ order, uint32_t *ticket) {
    pdl_enter();
    if (blockIdx.x + kOrderCtas >= gridDim.x) {
        const uint32_t rank = blockIdx.x + kOrderCtas - gridDim.x;
        if (rank == 0 && threadIdx.x == 0) *ticket = 0u;  // the per-item adjoint's chunk ticket
        tile_order<kOrderCtas>(rank, nullptr, walk, n_tiles, order);
        return;
    }
    const size_t M = *d_m, stride = (size_t)(gridDim.x - kOrderCtas) * blockDim.x;
    const size_t first = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    for (size_t k = first; k < 3 * M; k += stride) g2m[k] = 0.0;
    float4 *rows = reinterpret_cast<float4 *>(g2d);
    for (size_t k = first; k < kG2dRow / 4 * M; k += stride) rows[k] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// ---------------------------------------------------------------- small frames
//
// With at most kSmallFrameItems items (and pairs) the general passes are a
// chain of some twenty launches of a few microseconds each that leave the
// chip idle; one CTA does each stage's work in shared memory instead: the
// compaction and depth sort (14 launches), the pair count scan (3), the tile
// sort with ranges and launch order (4 to 7).  Same order: stable passes over
// items in gid order, pairs in depth order.
namespace {

constexpr int kOneThreads = 1024, kOneWarps = kOneThreads / 32;
constexpr int kOneItems = (int)kSmallFrameItems / kOneThreads;  // keys per thread at most
static_assert(kOneItems * kOneThreads == (int)kSmallFrameItems && kSmallFrameItems <= 65536, "16-bit values");

struct OneSmem {
    uint32_t keys[kSmallFrameItems];
    uint16_t vals[kSmallFrameItems];
    uint16_t hist[kOneWarps][kRadix];
    uint32_t start[kRadix];
    uint32_t scan[33];
};

// Stable LSD sort of S.keys / S.vals [0, n) by key bits [0, bits); the whole
// CTA calls, the arrays written and synchronised before.
__device__ __forceinline__ void one_cta_sort(OneSmem &S, uint32_t n, int bits) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t per = (n + kOneThreads - 1) / kOneThreads;  // keys per thread
    const uint32_t mine = warp * per * 32 + lane;
    const uint32_t lt = lanemask_lt();
    for (int shift = 0; shift < bits; shift += 8) {
        const uint32_t mask = bits - shift >= 8 ? 255u : (1u << (bits - shift)) - 1u;
        for (int k = lane; k < kRadix; k += 32) S.hist[warp][k] = 0;
        __syncwarp();
        uint32_t key[kOneItems], rank[kOneItems];
        uint16_t val[kOneItems];
#pragma unroll
        for (int j = 0; j < kOneItems; j++) {
            if ((uint32_t)j >= per) break;
            const uint32_t pos = mine + j * 32;
            const bool valid = pos < n;
            key[j] = valid ? S.keys[pos] : 0u;
            val[j] = valid ? S.vals[pos] : (uint16_t)0;
            const uint32_t d = (key[j] >> shift) & mask;
            uint32_t peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
            for (int bit = 0; bit < 8; bit++) {
                const bool on = (d >> bit) & 1u;
                const uint32_t b = __ballot_sync(0xffffffffu, on);
                peers &= on ? b : ~b;
            }
            uint32_t before = 0;
            if (valid) before = S.hist[warp][d];
            __syncwarp();
            if (valid && (peers & lt) == 0) S.hist[warp][d] = (uint16_t)(before + __popc(peers));
            __syncwarp();
            rank[j] = before + __popc(peers & lt);
        }
        __syncthreads();
        uint32_t cnt = 0;
        if (tid < kRadix) {
            uint32_t c[kOneWarps];
#pragma unroll
            for (int w = 0; w < kOneWarps; w++) c[w] = S.hist[w][tid];
#pragma unroll
            for (int w = 0; w < kOneWarps; w++) {
                S.hist[w][tid] = (uint16_t)cnt;
                cnt += c[w];
            }
        }
        uint32_t tot;
        const uint32_t ex = block_excl_scan(cnt, S.scan, &tot);
        if (tid < kRadix) S.start[tid] = ex;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kOneItems; j++) {
            if ((uint32_t)j >= per) break;
            if (mine + j * 32 >= n) continue;
            const uint32_t d = (key[j] >> shift) & mask;
            const uint32_t p = S.start[d] + S.hist[warp][d] + rank[j];
            S.keys[p] = key[j];
            S.vals[p] = val[j];
        }
        __syncthreads();
    }
}

// Compaction of the visible items and their depth sort.
__global__ void __launch_bounds__(kOneThreads) k_small_depth_sort(const uint32_t *__restrict__ cnt,
                                                                  const uint32_t *__restrict__ zkey, uint32_t n,
                                                                  uint32_t *__restrict__ szkey,
                                                                  uint32_t *__restrict__ sgid,
                                                                  uint32_t *__restrict__ inv, uint32_t *d_m) {
    pdl_enter();
    extern __shared__ uint4 s_one[];
    OneSmem &S = *reinterpret_cast<OneSmem *>(s_one);
    const int tid = threadIdx.x;
    const uint32_t per = (n + kOneThreads - 1) / kOneThreads, first = tid * per;
    bool vis[kOneItems];
    uint32_t z[kOneItems], mine = 0;
#pragma unroll
    for (int j = 0; j < kOneItems; j++) {
        const uint32_t i = first + j;
        const bool have = (uint32_t)j < per && i < n;
        vis[j] = have && cnt[i] > 0u;
        z[j] = have ? zkey[i] : 0u;  // (not written for invisible items, and not used then)
        if (have && !vis[j]) inv[i] = 0xffffffffu;
        mine += vis[j] ? 1u : 0u;
    }
    uint32_t M;
    uint32_t off = block_excl_scan(mine, S.scan, &M);
#pragma unroll
    for (int j = 0; j < kOneItems; j++)
        if (vis[j]) {
            S.keys[off] = z[j];
            S.vals[off++] = (uint16_t)(first + j);
        }
    __syncthreads();
    one_cta_sort(S, M, 31);
    for (uint32_t p = tid; p < M; p += kOneThreads) {
        const uint32_t g = S.vals[p];
        szkey[p] = S.keys[p];
        sgid[p] = g;
        inv[g] = p;
    }
    if (tid == 0) *d_m = M;
}

// Scan of the visible items' tile counts: first pair position per item, the
// pair count K and the overflow flag, the first item of every expansion
// chunk (of kEmitChunkSmall), and the tile ranges zeroed.
__global__ void __launch_bounds__(kOneThreads) k_small_count(const uint32_t *__restrict__ vis_cnt, const uint32_t *d_m,
                                                             uint32_t *__restrict__ vis_off,
                                                             uint32_t *__restrict__ chunk_start, uint32_t capacity,
                                                             uint32_t *d_k, uint32_t *overflow,
                                                             uint32_t *__restrict__ ranges, uint32_t n_ranges) {
    pdl_enter();
    __shared__ uint32_t smem[33];
    const int tid = threadIdx.x;
    for (uint32_t i = tid; i < n_ranges; i += kOneThreads) ranges[i] = 0u;
    const uint32_t M = *d_m, per = (M + kOneThreads - 1) / kOneThreads, first = tid * per;
    uint32_t v[kOneItems], sum = 0;
#pragma unroll
    for (int j = 0; j < kOneItems; j++) {
        v[j] = (uint32_t)j < per && first + j < M ? vis_cnt[first + j] : 0u;
        sum += v[j];
    }
    uint32_t K;
    uint32_t off = block_excl_scan(sum, smem, &K);
#pragma unroll
    for (int j = 0; j < kOneItems; j++) {
        if ((uint32_t)j >= per || first + j >= M) break;
        vis_off[first + j] = off;
        const uint32_t end = min(off + v[j], capacity);
        for (uint32_t c = (off + kEmitChunkSmall - 1) / kEmitChunkSmall; v[j] > 0u && c * kEmitChunkSmall < end; c++)
            chunk_start[c] = first + j;
        off += v[j];
    }
    if (tid == 0) {
        *d_k = K;
        if (K > capacity) *overflow = 1u;
    }
}

// Tile sort of the K pairs, the tiles' ranges (zeroed before) and, with
// `order`, the compositor's launch order (walk zeroed too).
__global__ void __launch_bounds__(kOneThreads) k_small_tile_sort(const uint32_t *__restrict__ keys,
                                                                 const uint32_t *__restrict__ vals,
                                                                 uint32_t *__restrict__ vals_out, const uint32_t *d_k,
                                                                 uint32_t capacity, int bits,
                                                                 uint2 *__restrict__ ranges, uint32_t n_tiles,
                                                                 uint32_t *__restrict__ order,
                                                                 uint32_t *__restrict__ walk) {
    pdl_enter();
    extern __shared__ uint4 s_one[];
    OneSmem &S = *reinterpret_cast<OneSmem *>(s_one);
    const int tid = threadIdx.x;
    const uint32_t K = min(*d_k, capacity);
    if (order && walk)
        for (uint32_t t = tid; t < n_tiles; t += kOneThreads) walk[t] = 0u;
    for (uint32_t p = tid; p < K; p += kOneThreads) {
        S.keys[p] = keys[p];
        S.vals[p] = (uint16_t)vals[p];
    }
    __syncthreads();
    one_cta_sort(S, K, bits);
    for (uint32_t p = tid; p < K; p += kOneThreads) {
        const uint32_t t = S.keys[p];
        vals_out[p] = S.vals[p];
        if (p == 0 || S.keys[p - 1] != t) ranges[t].x = p;
        if (p + 1 == K || S.keys[p + 1] != t) ranges[t].y = p + 1;
    }
    if (order) {
        __syncthreads();  // the ranges, read by this CTA
        tile_order<1>(0, ranges, nullptr, n_tiles, order);
    }
}

}  // namespace

cudaError_t set_small_frame_smem() {
    cudaError_t e = cudaFuncSetAttribute(k_small_depth_sort, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(OneSmem));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_small_tile_sort, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(OneSmem));
    return e;
}

void small_depth_sort(const Params &p, cudaStream_t s) {
    note_launch();
    pdl_launch(k_small_depth_sort, 1, kOneThreads, sizeof(OneSmem), s, p.item_cnt, p.item_zkey, p.n_items, p.szkey,
               p.sgid, p.inv, &p.counters[0]);
}

void small_count_pairs(const Params &p, cudaStream_t s) {
    note_launch();
    pdl_launch(k_small_count, 1, kOneThreads, 0, s, p.vis_cnt, (const uint32_t *)&p.counters[0], p.vis_off,
               p.chunk_start, p.pair_capacity, &p.counters[1], &p.counters[2], reinterpret_cast<uint32_t *>(p.ranges),
               2 * p.total_tiles);
}

void small_emit_pairs(const Params &p, void *temp, bool count_digits, cudaStream_t s) {
    TempLayout t = temp_layout(temp);
    // the general tile sort counts its first digits in the expansion
    const int sort_items = p.pair_capacity <= kSmallSort ? kSmallItems : kSortItems;
    const int sort_G = sort_blocks(p.pair_capacity, kSortThreads * sort_items);
    if (count_digits) cudaMemsetAsync(t.hist, 0, sizeof(uint32_t) * kRadix * sort_G, s);
    const uint32_t grid = std::min(std::max((p.pair_capacity + kEmitChunkSmall - 1) / kEmitChunkSmall, 1u),
                                   (uint32_t)(8 * device_sm_count()));
    note_launch();
    pdl_launch(k_expand_pairs<kEmitChunkSmall>, grid, kEmitThreads, 0, s, p.vis_off, p.vis_cnt, p.chunk_start, p.rect,
               p.rowtab, p.ell, p.tile_w, p.tile_h, p.vis_tile, p.vis_stride, p.views, p.n_views, &p.counters[0],
               &p.counters[1], p.pair_capacity, p.pair_keys, p.pair_vals, count_digits ? t.hist : nullptr, sort_G,
               (uint32_t)(kSortThreads * sort_items));
}

void small_tile_sort(const Params &p, uint32_t *vals_out, int bits, cudaStream_t s) {
    const bool order = p.total_tiles <= kSmallOrderTiles;
    note_launch();
    pdl_launch(k_small_tile_sort, 1, kOneThreads, sizeof(OneSmem), s, p.pair_keys, p.pair_vals, vals_out,
               (const uint32_t *)&p.counters[1], p.pair_capacity, bits, p.ranges, p.total_tiles,
               order ? p.tile_order : nullptr, p.tile_walk);
    if (!order) launch_tile_order(p, s);
}

void launch_tile_order(const Params &p, cudaStream_t s) {
    if (p.total_tiles == 0) return;
    note_launch();
    pdl_launch(k_tile_order, kOrderCtas, 1024, 0, s, p.ranges, p.total_tiles, p.tile_order, p.tile_walk);
}

void launch_bwd_prep(const Params &p, const uint32_t *walk, uint32_t *order, cudaStream_t s) {
    note_launch();
    const int zero_ctas = (device_sm_count() + kOrderCtas - 1) / kOrderCtas * kOrderCtas;  // whole clusters
    pdl_launch(k_bwd_prep, zero_ctas + kOrderCtas, 1024, 0, s, p.g2m, p.g2d, (const uint32_t *)&p.counters[0], walk,
               p.total_tiles, order, &p.counters[3]);
}

// ranges: zeroed by the pair count scan (scan_count_pairs)
void launch_ranges(const Params &p, cudaStream_t s) {
    note_launch();
    pdl_launch(k_ranges, 8 * device_sm_count(), 256, 0, s, p.pair_keys, &p.counters[1], p.pair_capacity, p.ranges);
}

}  // namespace pvg
