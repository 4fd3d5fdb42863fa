// ssim.cu -- the photometric loss of the objective (Sec. 3.4),
//   L = (1 - lambda_r) L1 + lambda_r (1 - SSIM),
// and dL/dpred in one fused pass, so a training step with the paper's RGB
// supervision needs no kernel outside this library.
//
// SSIM follows 3D Gaussian Splatting, whose losses the paper reuses: per
// channel, an 11 x 11 Gaussian window (sigma 1.5, normalised) applied with
// zero padding, C1 = 0.01^2, C2 = 0.03^2, averaged over channels and
// pixels; L1 is the mean absolute difference (sign(0) = 0).
//
// One CTA per 32 x 32 output tile and channel.  The window is separable
// and symmetric, so the gradient of SSIM is itself a windowed sum:
//   dSSIM/dx_p = sum_q G(q - p) [a_q + 2 x_p b_q + y_p c_q],
// a, b, c the derivatives of S_q with respect to the windowed moments
// G*x, G*x^2, G*xy.  The CTA stages x and y with a 10-pixel halo in
// shared memory, computes the five moments (row pass, then column pass) on
// the tile plus a 5-pixel halo, turns them into S, a, b, c (zero outside
// the image), filters a, b, c the same way and writes the gradient of its
// 32 x 32 pixels.  HBM traffic is one read of both images and one write of
// the gradient; the per-CTA sums of S and |x - y| go to a partial array
// that one small kernel adds in a fixed order (the loss is deterministic).
//
// The taps are 288 multiply-adds per pixel and channel with the halos (26
// bytes of HBM).  Every filter runs on packed pairs: a row pass filters two
// rows at once, a column pass two columns, and the values a row pass reads are
// stored as row pairs (3x1280x1920: 190 us by scalars, 175 us).  Each half
// rounds as the scalar filter did.  Nothing is full: 64 % of the shared-memory
// wavefronts, 54 % of the issue slots and 47 % of the FMA pipe at 17 warps per
// SM, which wait for one another's halos at the barriers between the passes.
#include <cooperative_groups.h>

#include <utility>

#include "pvg_internal.cuh"

namespace pvg {
namespace {

constexpr int kT = 32;               // output tile
constexpr int kR = 5;                // window radius
constexpr int kA = kT + 2 * kR;      // S / a / b / c region (42)
constexpr int kX = kT + 4 * kR;      // staged input region (52)
constexpr int kThreads = 192;  // one round of the largest pass (182 strips)
constexpr float kC1 = 0.01f * 0.01f, kC2 = 0.03f * 0.03f;

// shared layout, in floats: x and y as row pairs, [kX / 2][kXs] float2 each;
// the staged inputs are dead after the first row pass, so a, b, c (row pairs
// too, [3][kA / 2][kA] float2) take their place, and the gradient pass reads
// x and y of its own pixels from global memory again, where they are L2
// hits: 68 KB per CTA, three CTAs per SM.
constexpr int kXs = 58;  // row stride of the staged pairs: eight consecutive strips read distinct banks
constexpr int kH2 = 36;  // row stride of the row-filtered a, b, c
constexpr int kOffX = 0, kOffY = kX * kXs;
constexpr int kOffABC = 0;                         // [3][kA][kA] over the inputs
static_assert(3 * kA * kA <= 2 * kX * kXs, "a, b, c fit where the inputs were");
constexpr int kOffH = 2 * kX * kXs;                // 5 row-filtered moments [5][kX][kA]
constexpr int kOffH2 = kOffH;                      // row-filtered a, b, c [3][kA][kH2] (reuses the moments)
constexpr int kOffG = kOffH + 5 * kX * kA;         // 11 window taps
constexpr int kOffRed = kOffG + 12;                // 2 x 8 warp partials
constexpr int kSmemFloats = kOffRed + 16;

__global__ void __launch_bounds__(kThreads, 3) k_rgb_loss(const float *__restrict__ pred,
                                                       const float *__restrict__ tgt, int H, int W,
                                                       float lambda_r, float inv_n, float *__restrict__ dl,
                                                       float2 *__restrict__ partial) {
    pdl_enter();
    extern __shared__ float sm[];
    float *sx = sm + kOffX, *sy = sm + kOffY, *hm = sm + kOffH, *abc = sm + kOffABC, *h2 = sm + kOffH2;
    float *g = sm + kOffG, *red = sm + kOffRed;
    const int tid = threadIdx.x;
    const size_t plane = (size_t)H * W;
    const float *X = pred + blockIdx.z * plane, *Y = tgt + blockIdx.z * plane;
    const int tx0 = blockIdx.x * kT, ty0 = blockIdx.y * kT;
    if (tid < 11) {
        float s = 0.f;
        for (int j = 0; j < 11; j++) s += expf(-(float)((j - kR) * (j - kR)) / (2.0f * 1.5f * 1.5f));
        g[tid] = expf(-(float)((tid - kR) * (tid - kR)) / (2.0f * 1.5f * 1.5f)) / s;
    }
    // inputs with a 2R halo, zero outside the image, as row pairs
    float2 *sx2 = reinterpret_cast<float2 *>(sx), *sy2 = reinterpret_cast<float2 *>(sy);
    // (all loads of a thread in flight together: their latency, not their
    // bytes, is what the staging costs)
    constexpr int kLoads = (kX / 2 * kX + kThreads - 1) / kThreads;
    float2 vx[kLoads], vy[kLoads];
#pragma unroll
    for (int i = 0; i < kLoads; i++) {
        const int k = tid + i * kThreads;
        const int r = k / kX * 2, c = k % kX, gy = ty0 - 2 * kR + r, gx = tx0 - 2 * kR + c;
        const bool in = k < kX / 2 * kX && gx >= 0 && gx < W;
        const bool in0 = in && gy >= 0 && gy < H, in1 = in && gy + 1 >= 0 && gy + 1 < H;
        const size_t at = (size_t)gy * W + gx;
        vx[i] = make_float2(in0 ? X[at] : 0.f, in1 ? X[at + W] : 0.f);
        vy[i] = make_float2(in0 ? Y[at] : 0.f, in1 ? Y[at + W] : 0.f);
    }
#pragma unroll
    for (int i = 0; i < kLoads; i++) {
        const int k = tid + i * kThreads;
        if (k >= kX / 2 * kX) break;
        sx2[k / kX * kXs + k % kX] = vx[i];
        sy2[k / kX * kXs + k % kX] = vy[i];
    }
    __syncthreads();
    float gw[11];  // the taps, in registers
#pragma unroll
    for (int j = 0; j < 11; j++) gw[j] = g[j];
    auto tap = [&](int j) { return make_float2(gw[j], gw[j]); };
    // Each pass is register-blocked: a thread filters a strip of outputs
    // along the pass direction from one run of staged values, so a value is
    // read from shared memory once per strip instead of once per tap.
    //
    // row pass of the five moments: every pair of staged rows, strips of 6
    // columns of the 42-wide S region (7 per row)
    for (int k = tid; k < kX / 2 * 7; k += kThreads) {
        const int rp = k / 7, c0 = (k % 7) * 6;
        float2 xa[16], ya[16];
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
            const float4 u = reinterpret_cast<const float4 *>(&sx2[rp * kXs + c0 + j])[0];
            const float4 v = reinterpret_cast<const float4 *>(&sy2[rp * kXs + c0 + j])[0];
            xa[j] = make_float2(u.x, u.y); xa[j + 1] = make_float2(u.z, u.w);
            ya[j] = make_float2(v.x, v.y); ya[j + 1] = make_float2(v.z, v.w);
        }
        // one moment after another, its 16 values made in place
        auto moment = [&](int q, const float2 (&v)[16]) {
            float2 m[6];
#pragma unroll
            for (int o = 0; o < 6; o++) {
                float2 acc = make_float2(0.f, 0.f);
#pragma unroll
                for (int j = 0; j < 11; j++) acc = fma2(tap(j), v[o + j], acc);
                m[o] = acc;
            }
#pragma unroll
            for (int o = 0; o < 6; o += 2) {
                float *h = &hm[q * kX * kA + 2 * rp * kA + c0 + o];
                reinterpret_cast<float2 *>(h)[0] = make_float2(m[o].x, m[o + 1].x);
                reinterpret_cast<float2 *>(h + kA)[0] = make_float2(m[o].y, m[o + 1].y);
            }
        };
        moment(0, xa);
        moment(1, ya);
        float2 p[16];
#pragma unroll
        for (int j = 0; j < 16; j++) p[j] = mul2(xa[j], ya[j]);
        moment(4, p);
#pragma unroll
        for (int j = 0; j < 16; j++) p[j] = mul2(xa[j], xa[j]);
        moment(2, p);
#pragma unroll
        for (int j = 0; j < 16; j++) p[j] = mul2(ya[j], ya[j]);
        moment(3, p);
    }
    __syncthreads();
    // column pass -> S and its moment derivatives a, b, c on the tile + R
    // halo: every pair of columns, strips of 6 rows (7 per pair).  The row
    // pass was the inputs' last reader (barrier above), so a, b, c are
    // written over them.
    float ssum = 0.f, l1sum = 0.f;
    float2 *abc2 = reinterpret_cast<float2 *>(abc);  // [3][kA / 2][kA] row pairs
    for (int k = tid; k < kA / 2 * 7; k += kThreads) {
        const int c = (k % (kA / 2)) * 2, r0 = (k / (kA / 2)) * 6;
        float2 m[5][6];
#pragma unroll
        for (int q = 0; q < 5; q++) {
            float2 v[16];
#pragma unroll
            for (int i = 0; i < 16; i++) v[i] = reinterpret_cast<const float2 *>(&hm[q * kX * kA + (r0 + i) * kA + c])[0];
#pragma unroll
            for (int o = 0; o < 6; o++) {
                float2 acc = make_float2(0.f, 0.f);
#pragma unroll
                for (int i = 0; i < 11; i++) acc = fma2(tap(i), v[o + i], acc);
                m[q][o] = acc;
            }
        }
        float d[2][3];  // a, b, c of the even row's two columns, waiting for the odd row's
#pragma unroll
        for (int o = 0; o < 6; o++) {
            const int r = r0 + o, gy = ty0 - kR + r;
            float e[2][3];
#pragma unroll
            for (int t = 0; t < 2; t++) {
                const int gx = tx0 - kR + c + t;
                float a = 0.f, b = 0.f, cc = 0.f;
                if (gx >= 0 && gx < W && gy >= 0 && gy < H) {
                    auto at = [&](int q) { return t ? m[q][o].y : m[q][o].x; };
                    const float mx = at(0), my = at(1);
                    const float vx = fmaf(-mx, mx, at(2)), vy = fmaf(-my, my, at(3));
                    const float cxy = fmaf(-mx, my, at(4));
                    const float A1 = fmaf(2.f * mx, my, kC1), A2 = fmaf(2.f, cxy, kC2);
                    const float B1 = fmaf(mx, mx, fmaf(my, my, kC1)), B2 = vx + vy + kC2;
                    // SFU reciprocals (within 2 ulp)
                    const float iA1 = __fdividef(1.f, A1), iA2 = __fdividef(1.f, A2);
                    const float iB1 = __fdividef(1.f, B1), iB2 = __fdividef(1.f, B2);
                    const float S = A1 * A2 * iB1 * iB2;
                    const float dmu = 2.f * S * fmaf(my, iA1, -mx * iB1);
                    const float dvx = -S * iB2, dcxy = 2.f * S * iA2;
                    a = fmaf(-2.f * mx, dvx, fmaf(-my, dcxy, dmu));
                    b = dvx;
                    cc = dcxy;
                    if (r >= kR && r < kR + kT && c + t >= kR && c + t < kR + kT) ssum += S;
                }
                e[t][0] = a; e[t][1] = b; e[t][2] = cc;
            }
#pragma unroll
            for (int t = 0; t < 3; t++) {
                if (o & 1)
                    reinterpret_cast<float4 *>(&abc2[(t * (kA / 2) + r / 2) * kA + c])[0] =
                        make_float4(d[0][t], e[0][t], d[1][t], e[1][t]);
                d[0][t] = e[0][t];
                d[1][t] = e[1][t];
            }
        }
    }
    __syncthreads();
    // row pass of a, b, c (into the moments' space, no longer needed):
    // every pair of rows of the S region, strips of 4 of the 32 tile columns
    for (int k = tid; k < kA / 2 * 8; k += kThreads) {
        const int rp = k % (kA / 2), c0 = k / (kA / 2) * 4;  // consecutive rows read distinct banks
#pragma unroll
        for (int t = 0; t < 3; t++) {
            float2 v[14];
#pragma unroll
            for (int j = 0; j < 14; j += 2) {
                const float4 u = reinterpret_cast<const float4 *>(&abc2[(t * (kA / 2) + rp) * kA + c0 + j])[0];
                v[j] = make_float2(u.x, u.y);
                v[j + 1] = make_float2(u.z, u.w);
            }
            float2 m[4];
#pragma unroll
            for (int o = 0; o < 4; o++) {
                float2 acc = make_float2(0.f, 0.f);
#pragma unroll
                for (int j = 0; j < 11; j++) acc = fma2(tap(j), v[o + j], acc);
                m[o] = acc;
            }
            float *h = &h2[t * kA * kH2 + 2 * rp * kH2 + c0];
            reinterpret_cast<float4 *>(h)[0] = make_float4(m[0].x, m[1].x, m[2].x, m[3].x);
            reinterpret_cast<float4 *>(h + kH2)[0] = make_float4(m[0].y, m[1].y, m[2].y, m[3].y);
        }
    }
    __syncthreads();
    // column pass and the gradient of the tile's pixels (pairs of columns,
    // strips of 3 rows), and the L1 term of those pixels (x, y again from
    // global memory)
    {
        const float kl1 = (1.0f - lambda_r) * inv_n, kss = lambda_r * inv_n;
        float *D = dl ? dl + blockIdx.z * plane : nullptr;
        constexpr int kRows = 3, kStrips = (kT + kRows - 1) / kRows;  // 11 strips, the last of 2 rows
        for (int k = tid; k < kT / 2 * kStrips; k += kThreads) {
            const int c = (k % (kT / 2)) * 2, r0 = (k / (kT / 2)) * kRows;
            float px[kRows][2], py[kRows][2];  // loaded ahead of the filters
#pragma unroll
            for (int o = 0; o < kRows; o++)
#pragma unroll
                for (int t = 0; t < 2; t++) {
                    const bool in = r0 + o < kT && ty0 + r0 + o < H && tx0 + c + t < W;
                    const size_t at = (size_t)(ty0 + r0 + o) * W + tx0 + c + t;
                    px[o][t] = in ? X[at] : 0.f;
                    py[o][t] = in ? Y[at] : 0.f;
                }
            float2 q[3][kRows];
            if (D) {
#pragma unroll
                for (int t = 0; t < 3; t++) {
                    float2 v[kRows + 10];
#pragma unroll
                    for (int i = 0; i < kRows + 10; i++)  // (a row beyond the region belongs to no output)
                        v[i] = reinterpret_cast<const float2 *>(&h2[t * kA * kH2 + min(r0 + i, kA - 1) * kH2 + c])[0];
#pragma unroll
                    for (int o = 0; o < kRows; o++) {
                        float2 acc = make_float2(0.f, 0.f);
#pragma unroll
                        for (int i = 0; i < 11; i++) acc = fma2(tap(i), v[o + i], acc);
                        q[t][o] = acc;
                    }
                }
            }
#pragma unroll
            for (int o = 0; o < kRows; o++) {
                const int r = r0 + o, gy = ty0 + r;
                if (r >= kT || gy >= H) continue;
#pragma unroll
                for (int t = 0; t < 2; t++) {
                    const int gx = tx0 + c + t;
                    if (gx >= W) continue;
                    const float x = px[o][t], y = py[o][t], d = x - y;
                    l1sum += fabsf(d);
                    if (D) {
                        const float sgn = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f);
                        const float qa = t ? q[0][o].y : q[0][o].x, qb = t ? q[1][o].y : q[1][o].x;
                        const float dssim = qa + 2.f * x * qb + y * (t ? q[2][o].y : q[2][o].x);
                        D[(size_t)gy * W + gx] = kl1 * sgn - kss * dssim;
                    }
                }
            }
        }
    }
    // per-CTA sums
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ssum += __shfl_xor_sync(0xffffffffu, ssum, o);
        l1sum += __shfl_xor_sync(0xffffffffu, l1sum, o);
    }
    if ((tid & 31) == 0) {
        red[tid >> 5] = ssum;
        red[8 + (tid >> 5)] = l1sum;
    }
    __syncthreads();
    if (tid == 0) {
        float a = 0.f, b = 0.f;
        for (int w = 0; w < kThreads / 32; w++) {
            a += red[w];
            b += red[8 + w];
        }
        partial[(blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = make_float2(a, b);
    }
}

// loss[0..2] = (L, L1, SSIM) from the per-CTA partial sums, added in a
// fixed order in double precision by one cluster of kFinish CTAs (the 64-bit
// adders are few: one CTA takes 13 us for 7,200 partial sums).  Another CTA's
// shared memory may be written only once that CTA has started: every CTA
// arrives at a cluster barrier on entry and waits for it before its store.
constexpr int kFinish = 8, kFinishThreads = 256;

__global__ void __cluster_dims__(kFinish, 1, 1) __launch_bounds__(kFinishThreads)
    k_rgb_loss_finish(const float2 *__restrict__ partial, int n, double inv_n, float lambda_r, float *loss) {
    auto cluster = cooperative_groups::this_cluster();
    auto started = cluster.barrier_arrive();
    pdl_enter();
    __shared__ double s_warp[2][kFinishThreads / 32];
    __shared__ double s_cta[2][kFinish];  // CTA 0's: every CTA's sums
    double a = 0.0, b = 0.0;
    for (int i = blockIdx.x * kFinishThreads + threadIdx.x; i < n; i += kFinish * kFinishThreads) {
        const float2 p = partial[i];
        a += (double)p.x;
        b += (double)p.y;
    }
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if ((threadIdx.x & 31) == 0) {
        s_warp[0][threadIdx.x >> 5] = a;
        s_warp[1][threadIdx.x >> 5] = b;
    }
    __syncthreads();
    cluster.barrier_wait(std::move(started));
    if (threadIdx.x < 2) {
        double t = 0.0;
        for (int w = 0; w < kFinishThreads / 32; w++) t += s_warp[threadIdx.x][w];
        cluster.map_shared_rank(&s_cta[0][0], 0)[threadIdx.x * kFinish + blockIdx.x] = t;
    }
    cluster.sync();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        double s[2] = {0.0, 0.0};
        for (int k = 0; k < 2; k++)
            for (int w = 0; w < kFinish; w++) s[k] += s_cta[k][w];
        const double ssim = s[0] * inv_n, l1 = s[1] * inv_n;
        loss[0] = (float)((1.0 - lambda_r) * l1 + lambda_r * (1.0 - ssim));
        loss[1] = (float)l1;
        loss[2] = (float)ssim;
    }
}

}  // namespace

size_t rgb_loss_partials(int channels, int height, int width) {
    return (size_t)channels * ((height + kT - 1) / kT) * ((width + kT - 1) / kT);
}

cudaError_t launch_rgb_loss(const float *pred, const float *target, int channels, int height, int width,
                            float lambda_r, float *dl, float *loss, void *partials, cudaStream_t s) {
    const size_t smem = sizeof(float) * kSmemFloats;
    static_assert(sizeof(float) * kSmemFloats <= 227 * 1024, "shared memory of the loss kernel");
    cudaError_t e = cudaFuncSetAttribute(k_rgb_loss, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((width + kT - 1) / kT, (height + kT - 1) / kT, channels);
    const double n = (double)channels * height * width;
    note_launch();
    pdl_launch(k_rgb_loss, grid, kThreads, smem, s, pred, target, height, width, lambda_r, (float)(1.0 / n), dl,
                                            reinterpret_cast<float2 *>(partials));
    note_launch();
    pdl_launch(k_rgb_loss_finish, kFinish, kFinishThreads, 0, s, reinterpret_cast<const float2 *>(partials),
                                         (int)rgb_loss_partials(channels, height, width), 1.0 / n, lambda_r, loss);
    return cudaGetLastError();
}

}  // namespace pvg
