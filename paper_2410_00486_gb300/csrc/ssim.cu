// Photometric loss of Eq. 9 (Sec. III-C.3, CaRtGS) with its SSIM term:
//   L_v = w_v [ (1 - l) mean |img - tgt| + l (1 - mean SSIM(img, tgt)) + lambda_d mean_valid |D - D*| ]
// and its pixel gradients, for the raster backward's pixel-gradient input.
//
// SSIM per pixel and channel from window means (11x11 Gaussian, sigma 1.5, zero padding):
//   S = (2 mx my + C1)(2 sxy + C2) / ((mx^2 + my^2 + C1)(sx + sy + C2)),
//   sx = E[x^2] - mx^2, sy = E[y^2] - my^2, sxy = E[xy] - mx my.
// dS/dx at pixel q gathers, through the window, dS/dmx, dS/dE[x^2] and dS/dE[xy] of every
// pixel p whose window covers q:  dL/dx(q) = -(l / M) [ G*a + 2 x G*b + y G*c ](q),
// M = 3 H W, with a, b, c the per-pixel partials (k_ssim_fwd writes them; k_ssim_bwd blurs
// them).  Both kernels walk strips of 32x32 output tiles with a 5-pixel apron
// staged in shared memory, one separable pass per direction.
#include <math.h>
#include <stdio.h>

#include "cgs_internal.cuh"

namespace cgs {

constexpr int kSsimR = 5;                    // window radius
constexpr int kSsimN = 2 * kSsimR + 1;       // window taps
constexpr int kSsimT = 32;                   // edge of the output tile of a step
constexpr int kSsimIn = kSsimT + 2 * kSsimR;  // staged edge
constexpr float kC1 = 0.0001f, kC2 = 0.0009f;
constexpr int kRB = 4;                       // outputs per thread along a blur pass
constexpr int kSsimThreads = kSsimT * kSsimT / kRB;
constexpr int kSsimMaxSteps = 8;       // steps of a strip at most
// Blocks a window should keep when its strips get longer: about five for each place on the GPU
// (four blocks fit an SM).  Measured on four 1200x680 views only: strips of three steps, 3648
// blocks, 193 us; of one step 229.
constexpr int kSsimMinBlocks = 3000;
static_assert(kSsimT * (kSsimT / kRB) == kSsimThreads, "a pass over a tile is one round of the block");

struct SsimTaps {
    float2 g[kSsimR + 1];   // taps 0..5 (the window is symmetric), each twice for packed multiply-adds
};

// per-view accumulators: sum S, sum |x - y|, sum |D - D*| (valid)
constexpr int kSsimAcc = 3;

// A block walks down a strip of kSsimT columns in steps of kSsimT rows.  Each step stages its
// rows with the apron of columns (the first also the apron of rows), blurs them along the
// row into shared memory below the last ten blurred rows of the step before, then down the
// columns.  So no row is blurred along twice inside a strip, and the next step's rows are on
// their way while the columns are blurred.  In both passes a thread forms kRB adjacent
// outputs, streaming their kRB + 10 inputs through kRB accumulators; lanes lie along the
// rows in the row pass and along the columns in the column pass, and the odd row strides
// keep both free of bank conflicts.
//
// Bound by issue in the forward (two thirds of the slots) and by the latency of the staged
// maps in the backward, not by HBM.  Four 1200x680 views, both kernels and the launches
// around them: 193 us, where a tile a block, its staging loop of loads and stores one latency
// after another and each mean in a multiply-add of its own took 254; 198 with eight outputs a
// thread, 204 with the multiply-adds not packed, 214 with blocks that go on to other strips,
// 229 with one step a strip.
__device__ __forceinline__ void async_copy4(float *dst, const float *src, bool in)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(in ? 4 : 0) : "memory");
}
__device__ __forceinline__ void async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// f(staged row, staged column, offset in the plane, inside the image) for this thread's
// elements of `rows` staged rows from image row y0: a thread keeps one column, and every
// element is an asynchronous copy (zero outside the image), all of them in flight at once.
template <class F>
__device__ __forceinline__ void for_staged(int rows, int y0, int W, int H, F f)
{
    constexpr int kAtOnce = kSsimThreads / kSsimIn;
    const int c = threadIdx.x % kSsimIn, r0 = threadIdx.x / kSsimIn, gx = blockIdx.x * kSsimT - kSsimR + c;
    if (r0 >= kAtOnce) return;
    const bool inx = gx >= 0 && gx < W;
    // rows of this column from `lo` on, `n` of them, are inside the image
    const int lo = -y0, n = inx ? H : 0;
    int64_t q = (int64_t)(y0 + r0) * W + gx;
#pragma unroll 4
    for (int r = r0; r < rows; r += kAtOnce, q += kAtOnce * W) {
        const bool in = (unsigned)(r - lo) < (unsigned)n;
        f(r, c, in ? q : (int64_t)0, in);
    }
}

// Row pass of one step: f(staged row, blurred row, first column) for this thread's items.
template <class F>
__device__ __forceinline__ void for_row_items(bool first, F f)
{
    const int r = threadIdx.x % kSsimT, c0 = threadIdx.x / kSsimT * kRB;
    if (!first) {
        f(r, r + 2 * kSsimR, c0);
    } else {
        f(r, r, c0);
        if (threadIdx.x < 2 * kSsimR * (kSsimT / kRB))
            f(kSsimT + threadIdx.x % (2 * kSsimR), kSsimT + threadIdx.x % (2 * kSsimR),
              threadIdx.x / (2 * kSsimR) * kRB);
    }
}

// Sum over the block in double, in thread 0.
__device__ __forceinline__ double block_total(PairSum x, PairSum *red)
{
    for (int o = 16; o > 0; o >>= 1) {
        PairSum y;
        y.h = __shfl_xor_sync(kFull, x.h, o);
        y.l = __shfl_xor_sync(kFull, x.l, o);
        x.add(y);
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < kSsimThreads / 32; i++) t += red[i].value();
    return t;
}

// Five window means per pixel (of x, y, x^2, y^2 and xy), two pairs of them in packed
// multiply-adds.
__global__ void __launch_bounds__(kSsimThreads, 4)
k_ssim_fwd(const float *__restrict__ img, const float *__restrict__ tgt, int W, int H, int steps,
           const __grid_constant__ SsimTaps t, float *__restrict__ amap, float *__restrict__ bmap,
           float *__restrict__ cmap, double *__restrict__ acc)
{
    __shared__ float2 sxy[kSsimIn][kSsimIn + 1];
    __shared__ float4 hm[kSsimIn][kSsimT + 1];   // blurred along the row: x, y, x^2, y^2
    __shared__ float hp[kSsimIn][kSsimT + 1];    // and xy
    __shared__ PairSum red[2][kSsimThreads / 32];
    const int vc = blockIdx.z;                     // view * 3 + channel
    const size_t plane = (size_t)vc * W * H;
    const int x0 = blockIdx.x * kSsimT, y0 = blockIdx.y * kSsimT * steps;
    const int yend = min(H, y0 + kSsimT * steps);
    float2 g[kSsimR + 1];
#pragma unroll
    for (int k = 0; k <= kSsimR; k++) g[k] = t.g[k];
    auto tap = [&](int k) { return g[k <= kSsimR ? k : kSsimN - 1 - k]; };
    auto stage = [&](int rows, int y) {
        for_staged(rows, y, W, H, [&](int r, int c, int64_t q, bool in) {
            async_copy4(&sxy[r][c].x, img + plane + q, in);
            async_copy4(&sxy[r][c].y, tgt + plane + q, in);
        });
    };
    stage(kSsimIn, y0 - kSsimR);
    PairSum sS, sR;
    for (int y = y0; y < yend; y += kSsimT) {
        const bool first = y == y0;
        const int yst = first ? y - kSsimR : y + kSsimR;   // image row of the first staged row
        async_wait();
        __syncthreads();
        if (!first) {
            for (int i = threadIdx.x; i < 2 * kSsimR * kSsimT; i += kSsimThreads) {
                hm[i / kSsimT][i % kSsimT] = hm[kSsimT + i / kSsimT][i % kSsimT];
                hp[i / kSsimT][i % kSsimT] = hp[kSsimT + i / kSsimT][i % kSsimT];
            }
            __syncthreads();
        }
        float absd = 0.f;
        for_row_items(first, [&](int r, int hr, int c0) {
            float2 m[kRB], q[kRB];
            float p[kRB];
#pragma unroll
            for (int o = 0; o < kRB; o++) {
                m[o] = q[o] = make_float2(0.f, 0.f);
                p[o] = 0.f;
            }
            // the row's pixels are outputs of this strip up to column cend
            const int cend = yst + r >= y0 && yst + r < yend ? W - x0 - c0 : 0;
#pragma unroll
            for (int k = 0; k < kRB + 2 * kSsimR; k++) {
                const float2 v = sxy[r][c0 + k];
                const float2 vv = __fmul2_rn(v, v);
                const float xy = v.x * v.y;
                if (k >= kSsimR && k < kSsimR + kRB) absd += k - kSsimR < cend ? fabsf(v.x - v.y) : 0.f;
#pragma unroll
                for (int o = 0; o < kRB; o++)
                    if (k - o >= 0 && k - o < kSsimN) {
                        m[o] = __ffma2_rn(tap(k - o), v, m[o]);
                        q[o] = __ffma2_rn(tap(k - o), vv, q[o]);
                        p[o] = fmaf(tap(k - o).x, xy, p[o]);
                    }
            }
#pragma unroll
            for (int o = 0; o < kRB; o++) {
                hm[hr][c0 + o] = make_float4(m[o].x, m[o].y, q[o].x, q[o].y);
                hp[hr][c0 + o] = p[o];
            }
        });
        sR.add(absd);
        __syncthreads();
        if (y + kSsimT < yend) stage(kSsimT, y + kSsimT + kSsimR);
        const int c = threadIdx.x % kSsimT, r0 = threadIdx.x / kSsimT * kRB, gx = x0 + c;
        float2 m[kRB], q[kRB];
        float p[kRB];
#pragma unroll
        for (int o = 0; o < kRB; o++) {
            m[o] = q[o] = make_float2(0.f, 0.f);
            p[o] = 0.f;
        }
#pragma unroll
        for (int k = 0; k < kRB + 2 * kSsimR; k++) {
            const float4 v = hm[r0 + k][c];
            const float w = hp[r0 + k][c];
#pragma unroll
            for (int o = 0; o < kRB; o++)
                if (k - o >= 0 && k - o < kSsimN) {
                    m[o] = __ffma2_rn(tap(k - o), make_float2(v.x, v.y), m[o]);
                    q[o] = __ffma2_rn(tap(k - o), make_float2(v.z, v.w), q[o]);
                    p[o] = fmaf(tap(k - o).x, w, p[o]);
                }
        }
        float sum = 0.f;
#pragma unroll
        for (int o = 0; o < kRB; o++) {
            const int gy = y + r0 + o;
            if (gx >= W || gy >= H) continue;
            const float mx = m[o].x, my = m[o].y;
            const float sxx = q[o].x - mx * mx, syy = q[o].y - my * my, cov = p[o] - mx * my;
            const float A1 = 2.f * mx * my + kC1, A2 = 2.f * cov + kC2;
            const float B1 = mx * mx + my * my + kC1, B2 = sxx + syy + kC2;
            const float inv = __fdividef(1.f, B1 * B2);
            const float S = A1 * A2 * inv;
            const float dA1 = A2 * inv, dA2 = A1 * inv, dB1 = -S * (B2 * inv), dB2 = -S * (B1 * inv);
            const size_t i = plane + (size_t)gy * W + gx;
            amap[i] = 2.f * my * (dA1 - dA2) + 2.f * mx * (dB1 - dB2);
            bmap[i] = dB2;
            cmap[i] = 2.f * dA2;
            sum += S;
        }
        sS.add(sum);
    }
    const double a = block_total(sS, red[0]), b = block_total(sR, red[1]);
    if (threadIdx.x == 0) {
        atomicAdd(acc + kSsimAcc * (vc / 3) + 0, a);
        atomicAdd(acc + kSsimAcc * (vc / 3) + 1, b);
    }
}

// Blurs the three partials back (a and b as a packed pair) and writes the pixel gradients;
// the block that finishes last writes the views' losses.
__global__ void __launch_bounds__(kSsimThreads, 4)
k_ssim_bwd(const float *__restrict__ img, const float *__restrict__ tgt, const float *__restrict__ depth,
           const float *__restrict__ tgt_depth, const int32_t *__restrict__ depth_count,
           const float *__restrict__ weight, int W, int H, int steps, const __grid_constant__ SsimTaps t, float lam,
           float lambda_d, const float *__restrict__ amap, const float *__restrict__ bmap,
           const float *__restrict__ cmap, float *__restrict__ dl_dimg, float *__restrict__ dl_ddepth,
           double *__restrict__ acc, uint32_t *__restrict__ done, float *__restrict__ loss_view,
           int32_t *__restrict__ status)
{
    __shared__ float2 sab[kSsimIn][kSsimIn + 1];
    __shared__ float sc[kSsimIn][kSsimIn + 1];
    __shared__ float2 hab[kSsimIn][kSsimT + 1];
    __shared__ float hc[kSsimIn][kSsimT + 1];
    __shared__ PairSum red[kSsimThreads / 32];
    __shared__ bool s_last;
    const int vc = blockIdx.z, v = vc / 3, ch = vc % 3;
    const size_t plane = (size_t)vc * W * H;
    const int x0 = blockIdx.x * kSsimT, y0 = blockIdx.y * kSsimT * steps;
    const int yend = min(H, y0 + kSsimT * steps);
    float2 g[kSsimR + 1];
#pragma unroll
    for (int k = 0; k <= kSsimR; k++) g[k] = t.g[k];
    auto tap = [&](int k) { return g[k <= kSsimR ? k : kSsimN - 1 - k]; };
    auto stage = [&](int rows, int y) {
        for_staged(rows, y, W, H, [&](int r, int c, int64_t q, bool in) {
            async_copy4(&sab[r][c].x, amap + plane + q, in);
            async_copy4(&sab[r][c].y, bmap + plane + q, in);
            async_copy4(&sc[r][c], cmap + plane + q, in);
        });
    };
    stage(kSsimIn, y0 - kSsimR);
    const float M = 3.f * (float)W * (float)H;
    const float wv = weight ? weight[v] : 1.f;
    const int cnt = depth_count ? depth_count[v] : 0;
    PairSum sD;
    for (int y = y0; y < yend; y += kSsimT) {
        const bool first = y == y0;
        async_wait();
        __syncthreads();
        if (!first) {
            for (int i = threadIdx.x; i < 2 * kSsimR * kSsimT; i += kSsimThreads) {
                hab[i / kSsimT][i % kSsimT] = hab[kSsimT + i / kSsimT][i % kSsimT];
                hc[i / kSsimT][i % kSsimT] = hc[kSsimT + i / kSsimT][i % kSsimT];
            }
            __syncthreads();
        }
        const int c = threadIdx.x % kSsimT, r0 = threadIdx.x / kSsimT * kRB, gx = x0 + c;
        // image and target of the thread's pixels, on their way during both passes
        float xs[kRB], ys[kRB];
#pragma unroll
        for (int o = 0; o < kRB; o++) {
            const bool in = gx < W && y + r0 + o < H;
            const size_t q = plane + (in ? (size_t)(y + r0 + o) * W + gx : (size_t)0);
            xs[o] = in ? __ldg(img + q) : 0.f;
            ys[o] = in ? __ldg(tgt + q) : 0.f;
        }
        for_row_items(first, [&](int r, int hr, int c0) {
            float2 ab[kRB];
            float cc[kRB];
#pragma unroll
            for (int o = 0; o < kRB; o++) {
                ab[o] = make_float2(0.f, 0.f);
                cc[o] = 0.f;
            }
#pragma unroll
            for (int k = 0; k < kRB + 2 * kSsimR; k++) {
                const float2 p = sab[r][c0 + k];
                const float q = sc[r][c0 + k];
#pragma unroll
                for (int o = 0; o < kRB; o++)
                    if (k - o >= 0 && k - o < kSsimN) {
                        ab[o] = __ffma2_rn(tap(k - o), p, ab[o]);
                        cc[o] = fmaf(tap(k - o).x, q, cc[o]);
                    }
            }
#pragma unroll
            for (int o = 0; o < kRB; o++) {
                hab[hr][c0 + o] = ab[o];
                hc[hr][c0 + o] = cc[o];
            }
        });
        __syncthreads();
        if (y + kSsimT < yend) stage(kSsimT, y + kSsimT + kSsimR);
        float2 ab[kRB];
        float cc[kRB];
#pragma unroll
        for (int o = 0; o < kRB; o++) {
            ab[o] = make_float2(0.f, 0.f);
            cc[o] = 0.f;
        }
#pragma unroll
        for (int k = 0; k < kRB + 2 * kSsimR; k++) {
            const float2 p = hab[r0 + k][c];
            const float q = hc[r0 + k][c];
#pragma unroll
            for (int o = 0; o < kRB; o++)
                if (k - o >= 0 && k - o < kSsimN) {
                    ab[o] = __ffma2_rn(tap(k - o), p, ab[o]);
                    cc[o] = fmaf(tap(k - o).x, q, cc[o]);
                }
        }
        float absd = 0.f;
#pragma unroll
        for (int o = 0; o < kRB; o++) {
            const int gy = y + r0 + o;
            if (gx >= W || gy >= H) continue;
            const size_t q = plane + (size_t)gy * W + gx;
            const float xv = xs[o], yv = ys[o];
            const float sgn = xv > yv ? 1.f : (xv < yv ? -1.f : 0.f);
            dl_dimg[q] = wv * ((1.f - lam) * sgn / M - lam / M * (ab[o].x + 2.f * xv * ab[o].y + yv * cc[o]));
            if (ch == 0 && dl_ddepth) {
                const size_t pix = (size_t)v * W * H + (size_t)gy * W + gx;
                float gd = 0.f;
                if (tgt_depth && cnt > 0) {
                    const float td = tgt_depth[pix];
                    if (td > 0.f) {
                        const float dd = depth[pix] - td;
                        gd = wv * lambda_d * (dd > 0.f ? 1.f : (dd < 0.f ? -1.f : 0.f)) / (float)cnt;
                        absd += fabsf(dd);
                    }
                }
                dl_ddepth[pix] = gd;
            }
        }
        // (scaled so that a warp's sum over a strip leaves float's range no sooner than one over a tile)
        sD.add(absd * (1.f / kSsimMaxSteps));
    }
    if (ch == 0) {
        const double s = kSsimMaxSteps * block_total(sD, red);
        if (threadIdx.x == 0) atomicAdd(acc + kSsimAcc * v + 2, s);
    }
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(done, 1u) == gridDim.x * gridDim.y * gridDim.z - 1u;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const int views = (int)gridDim.z / 3;
    const double Md = 3.0 * (double)W * (double)H;
    for (int i = threadIdx.x; i < views; i += kSsimThreads) {
        const double w = weight ? (double)weight[i] : 1.0;
        const int n = depth_count ? depth_count[i] : 0;
        const double *a = acc + kSsimAcc * i;
        const double L = w * ((1.0 - lam) * __ldcg(a + 1) / Md + lam * (1.0 - __ldcg(a) / Md) +
                              (n > 0 ? (double)lambda_d * __ldcg(a + 2) / n : 0.0));
        loss_view[i] = (float)L;
        if (!isfinite(L)) set_status(status, CGS_ERR_NONFINITE);
    }
}

// Steps a block walks: the strip's apron of rows costs 10 rows in 32 steps, but short strips
// fill the GPU.
static int ssim_steps(int W, int H, int V)
{
    const int64_t cols = (W + kSsimT - 1) / kSsimT, rows = (H + kSsimT - 1) / kSsimT;
    int steps = 1;
    while (steps < kSsimMaxSteps && cols * ((rows + steps) / (steps + 1)) * 3 * V >= kSsimMinBlocks) steps++;
    return steps;
}

}  // namespace cgs

using namespace cgs;

extern "C" {

size_t cgs_ssim_workspace(int32_t V, const cgs_config *cfg)
{
    if (!cfg || V < 1 || cfg->width < 1 || cfg->height < 1) return 0;
    const size_t maps = 3 * (size_t)V * 3 * (size_t)cfg->width * cfg->height * sizeof(float);
    return ((maps + 255) & ~(size_t)255) + (size_t)V * kSsimAcc * sizeof(double) + sizeof(uint32_t);
}

int cgs_ssim_loss(const float *img, const float *tgt_rgb, const float *depth, const float *tgt_depth,
                  const int32_t *depth_count, int32_t V, const cgs_config *cfg, const float *view_weight,
                  float lambda_ssim, float *loss_view, float *dl_dimg, float *dl_ddepth, void *workspace,
                  size_t workspace_bytes, int32_t *status_dev, void *stream)
{
    if (!img || !tgt_rgb || !loss_view || !dl_dimg || !workspace || !cfg || V < 1) return CGS_ERR_ARG;
    if (cfg->width < 1 || cfg->height < 1 || cfg->width > (1 << 16) || cfg->height > (1 << 16)) return CGS_ERR_ARG;
    if (tgt_depth && (!depth || !depth_count || !dl_ddepth)) return CGS_ERR_ARG;
    if (!(lambda_ssim >= 0.f && lambda_ssim <= 1.f)) return CGS_ERR_ARG;
    if (workspace_bytes < cgs_ssim_workspace(V, cfg) || ((uintptr_t)workspace & 255) != 0) return CGS_ERR_WORKSPACE;
    const int W = cfg->width, H = cfg->height;
    const size_t plane_all = (size_t)V * 3 * W * H;
    float *amap = static_cast<float *>(workspace);
    float *bmap = amap + plane_all, *cmap = bmap + plane_all;
    const size_t maps = 3 * plane_all * sizeof(float);
    double *acc = reinterpret_cast<double *>(static_cast<char *>(workspace) + ((maps + 255) & ~(size_t)255));
    uint32_t *done = reinterpret_cast<uint32_t *>(acc + (size_t)kSsimAcc * V);
    SsimTaps t;
    double sum = 0.0, gd[2 * kSsimR + 1];
    for (int k = 0; k < 2 * kSsimR + 1; k++) {
        const double x = k - kSsimR;
        gd[k] = exp(-(x * x) / (2.0 * 1.5 * 1.5));
        sum += gd[k];
    }
    for (int k = 0; k <= kSsimR; k++) t.g[k].x = t.g[k].y = (float)(gd[k] / sum);
    const int steps = ssim_steps(W, H, V);
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaMemsetAsync(acc, 0, sizeof(double) * kSsimAcc * V + sizeof(uint32_t), s);
    const dim3 grid((W + kSsimT - 1) / kSsimT, (H + kSsimT * steps - 1) / (kSsimT * steps), 3 * V);
    if (e == cudaSuccess) {
        k_ssim_fwd<<<grid, kSsimThreads, 0, s>>>(img, tgt_rgb, W, H, steps, t, amap, bmap, cmap, acc);
        k_ssim_bwd<<<grid, kSsimThreads, 0, s>>>(img, tgt_rgb, depth, tgt_depth, tgt_depth ? depth_count : nullptr,
                                                 view_weight, W, H, steps, t, lambda_ssim, cfg->lambda_depth, amap,
                                                 bmap, cmap, dl_dimg, tgt_depth ? dl_ddepth : nullptr, acc, done, loss_view,
                                                 status_dev);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        fprintf(stderr, "libcgs: CUDA error: %s\n", cudaGetErrorString(e));
        return CGS_ERR_CUDA;
    }
    return CGS_OK;
}

}  // extern "C"
