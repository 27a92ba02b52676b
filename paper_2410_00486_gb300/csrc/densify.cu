// Adaptive density control (Sec. III-A.3 "splitting and cloning ... guided by gradients
// and the size", Sec. IV-A: densify with the positional-gradient threshold tau_p and
// remove Gaussians with opacity below eps_alpha), on the device.
//
// k_densify_plan classifies every Gaussian in float32 (0 prune, 1 keep, 2 keep + clone,
// 3 split into two) from its average view-space gradient accum/denom, its largest
// log-scale and its opacity logit, against thresholds rounded once from double on the
// host, and sums the outputs of its span of Gaussians; k_span_scan turns the codes into
// output positions and the new Gaussian count; k_densify_apply writes the new parameter
// vector and Adam state (clones and split children start with zero moments), each Gaussian's
// outputs consecutive.  Split children are mean + R(q) (s * z) with caller-supplied standard
// normal z, scale s / 1.6, other attributes copied.
#include <math.h>
#include <stdio.h>

#include "cgs_internal.cuh"

namespace cgs {

constexpr float kLogSplitDiv = 0.47000362924573558f;   // ln(1.6)

// Exclusive scan of count[0..n) into off[0..n], off[n] = total, in two launches over at most
// kScanBlocks spans of scan_span(n) entries: the totals of the spans (formed by whichever
// kernel has the counts at hand), then every block adds the totals before its own and scans
// its span, 4 entries a thread.  One block walking all entries, 32 lanes of each warp at a
// time, left the chip idle for the latency of thousands of dependent steps (200k entries 79
// us, two launches now 3.6 us with the totals formed by the plan; 357k cells 135 -> 7 us).
constexpr int kScanThreads = 256, kScanChunk = 4 * kScanThreads, kScanBlocks = 1024;

inline int64_t scan_span(int64_t n)
{
    const int64_t per = (n + kScanBlocks - 1) / kScanBlocks;
    return (per + kScanChunk - 1) / kScanChunk * kScanChunk;
}
inline int scan_blocks(int64_t n) { return (int)((n + scan_span(n) - 1) / scan_span(n)); }

// Sum of x over the block, returned to every thread.
__device__ __forceinline__ unsigned long long block_sum(unsigned long long x)
{
    __shared__ unsigned long long ws[32];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    __syncthreads();   // the previous sum has been read
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = x;
    __syncthreads();
    unsigned long long t = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); i++) t += ws[i];
    return t;
}

__global__ void __launch_bounds__(kScanThreads)
k_span_totals(const uint32_t *__restrict__ count, int64_t n, int64_t span, unsigned long long *__restrict__ part)
{
    const int64_t lo = blockIdx.x * span, hi = min(n, lo + span);
    unsigned long long s = 0;
#pragma unroll 4
    for (int64_t t = lo + threadIdx.x; t < hi; t += kScanThreads) s += count[t];
    s = block_sum(s);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// Entries of a scan: a count array, or densification codes (a pruned Gaussian leaves no
// output, a kept one one, a cloned or split one two).
struct CountEntry {
    const uint32_t *count;
    __device__ __forceinline__ uint32_t operator()(int64_t i) const { return count[i]; }
};
struct CodeEntry {
    const uint32_t *code;
    __device__ __forceinline__ uint32_t operator()(int64_t i) const { return min(code[i], 2u); }
};

template <class Entry>
__global__ void __launch_bounds__(kScanThreads)
k_span_scan(Entry entry, int64_t n, int64_t span, const unsigned long long *__restrict__ part,
            uint32_t *__restrict__ off, int64_t *__restrict__ total_out)
{
    __shared__ uint32_t wtot[kScanThreads / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned long long before = 0;
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += kScanThreads) before += part[b];
    unsigned long long run = block_sum(before);
    const int64_t lo = blockIdx.x * span, hi = min(n, lo + span);
    for (int64_t base = lo; base < hi; base += kScanChunk) {
        const int64_t t0 = base + 4 * (int64_t)threadIdx.x;
        uint32_t c[4], tot = 0;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            c[k] = t0 + k < hi ? entry(t0 + k) : 0u;
            tot += c[k];
        }
        uint32_t incl = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) wtot[w] = incl;
        __syncthreads();
        uint32_t pre = 0, all = 0;
#pragma unroll
        for (int i = 0; i < kScanThreads / 32; i++) {
            pre += i < w ? wtot[i] : 0u;
            all += wtot[i];
        }
        unsigned long long o = run + pre + incl - tot;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            if (t0 + k < hi) off[t0 + k] = (uint32_t)o;
            o += c[k];
        }
        run += all;
        __syncthreads();   // wtot is rewritten by the next chunk
    }
    if (hi == n && threadIdx.x == 0) {   // the last span
        off[n] = (uint32_t)run;
        if (total_out) *total_out = (int64_t)run;
    }
}

// One span of Gaussians a block: their codes and the span's output count.
__global__ void __launch_bounds__(kScanThreads)
k_densify_plan(const float *__restrict__ P, int64_t n, int64_t span, const float *__restrict__ accum,
               const float *__restrict__ denom, float t_grad, float t_logs, float t_logit,
               uint32_t *__restrict__ code, unsigned long long *__restrict__ part)
{
    const int64_t lo = blockIdx.x * span, hi = min(n, lo + span);
    unsigned long long outs = 0;
#pragma unroll 4
    for (int64_t g = lo + threadIdx.x; g < hi; g += kScanThreads) {
        const float den = denom[g];
        const float grad = den > 0.f ? __fdiv_rn(accum[g], den) : 0.f;
        const bool high = grad >= t_grad;
        const float *ls = P + 3 * n + 3 * g;
        const bool small = fmaxf(fmaxf(ls[0], ls[1]), ls[2]) <= t_logs;
        const bool prune = P[10 * n + g] < t_logit;
        const uint32_t c = prune ? 0u : (high ? (small ? 2u : 3u) : 1u);
        code[g] = c;
        outs += min(c, 2u);
    }
    outs = block_sum(outs);
    if (threadIdx.x == 0) part[blockIdx.x] = outs;
}

// A block of kDenG consecutive Gaussians, whose outputs are consecutive too: a map in
// shared memory says which Gaussian each output copies, and every group is then written
// as one contiguous run of floats, lanes along it, so stores are whole lines and loads
// nearly so (the copies of a Gaussian repeat its floats, a pruned one leaves a gap).  Bound
// by HBM and its latency: 200k Gaussians of SH degree 3 in 61 us, 4.7 TB/s; one thread per
// Gaussian, copying it float by float with the rows of a warp 180 bytes apart, took 266 us,
// the groups one after another and a load and a store at a time 78.  Eight floats ahead, or
// blocks of 64 Gaussians, measure the same.
constexpr int kDenG = 128, kDenThreads = 256, kDenAhead = 4;
constexpr uint16_t kDenFresh = 0x4000, kDenSplit = 0x8000;   // zero moments; mean and scale drawn anew

template <int DEG>
__global__ void __launch_bounds__(kDenThreads)
k_densify_apply(const float *__restrict__ P, const float *__restrict__ Mi, const float *__restrict__ Vi, int64_t n,
                const uint32_t *__restrict__ code, const uint32_t *__restrict__ off,
                const float *__restrict__ normals, int64_t m, float *__restrict__ Po, float *__restrict__ Mo,
                float *__restrict__ Vo)
{
    constexpr int R3 = 3 * ((DEG + 1) * (DEG + 1) - 1);
    __shared__ uint16_t src[2 * kDenG];
    __shared__ int s_outs;
    const int64_t g0 = (int64_t)blockIdx.x * kDenG;
    const int cnt = (int)min((int64_t)kDenG, n - g0);
    const int64_t j0 = off[g0];
    if (threadIdx.x == 0) s_outs = 0;
    for (int i = threadIdx.x; i < 2 * kDenG; i += kDenThreads) src[i] = kDenFresh;   // whatever the workspace holds
    __syncthreads();
    for (int gl = threadIdx.x; gl < cnt; gl += kDenThreads) {
        const int64_t g = g0 + gl, j = off[g];
        const uint32_t c = code[g];
        if (c == 0u) continue;
        const int outs = c == 1u ? 1 : 2;
        const int64_t jl = j - j0;
        // never write past the caller's n_out, nor past the map
        if (j + outs > m || jl < 0 || jl + outs > 2 * kDenG) continue;
        atomicMax(&s_outs, (int)jl + outs);
        src[jl] = (uint16_t)(gl | (c == 3u ? kDenFresh | kDenSplit : 0));
        if (outs == 2) src[jl + 1] = (uint16_t)(gl | kDenFresh | (c == 3u ? kDenSplit : 0));
        if (c == 3u) {
            const float *q = P + 6 * n + 4 * g;
            const float inv = 1.0f / sqrtf(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
            const float w = q[0] * inv, x = q[1] * inv, y = q[2] * inv, z = q[3] * inv;
            const float R[9] = {1.f - 2.f * (y * y + z * z), 2.f * (x * y - w * z), 2.f * (x * z + w * y),
                                2.f * (x * y + w * z), 1.f - 2.f * (x * x + z * z), 2.f * (y * z - w * x),
                                2.f * (x * z - w * y), 2.f * (y * z + w * x), 1.f - 2.f * (x * x + y * y)};
            const float *ls = P + 3 * n + 3 * g;
            const float s[3] = {expf(ls[0]), expf(ls[1]), expf(ls[2])};
            for (int k = 0; k < 2; k++) {
                const int64_t jj = j + k;
                const float *zz = normals + 6 * g + 3 * k;
                const float d0 = s[0] * zz[0], d1 = s[1] * zz[1], d2 = s[2] * zz[2];
                for (int r = 0; r < 3; r++)
                    Po[3 * jj + r] = P[3 * g + r] + (R[3 * r] * d0 + R[3 * r + 1] * d1 + R[3 * r + 2] * d2);
                for (int r = 0; r < 3; r++) Po[3 * m + 3 * jj + r] = ls[r] - kLogSplitDiv;
            }
        }
    }
    __syncthreads();
    // the groups side by side: a warp for means and scales, one for rotations, opacities and
    // DC colours, the others for the higher bands, so no group waits for another's loads,
    // and a thread's kDenAhead floats of each array on their way together
    const int outs = s_outs;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int widths[6] = {3, 3, 4, 1, 3, R3};
    int64_t oi = 0, oo = 0;
#pragma unroll
    for (int gi = 0; gi < 6; gi++) {
        const int w = widths[gi];
        if (w == 0) continue;
        const bool mine = gi < 2 ? wp == 0 : (gi < 5 ? wp == 1 : wp >= 2);   // warp-uniform
        if (mine) {
            const float *pi = P + oi + w * g0, *mi = Mi + oi + w * g0, *vi = Vi + oi + w * g0;
            float *po = Po + oo + w * j0, *mo = Mo + oo + w * j0, *vo = Vo + oo + w * j0;
            const int first = gi < 5 ? lane : lane + 32 * (wp - 2), step = gi < 5 ? 32 : kDenThreads - 64;
            for (int i0 = first; i0 < w * outs; i0 += kDenAhead * step) {
                float x[kDenAhead], y[kDenAhead], z[kDenAhead];   // every load before the first store
                uint32_t e[kDenAhead];
#pragma unroll
                for (int q = 0; q < kDenAhead; q++) {
                    const int i = i0 + q * step, jl = i / w;
                    const bool in = i < w * outs;
                    e[q] = in ? src[jl] : kDenFresh;
                    const int from = w * (int)(e[q] & (kDenFresh - 1)) + i - w * jl;
                    x[q] = in ? __ldg(pi + from) : 0.f;
                    y[q] = e[q] & kDenFresh ? 0.f : __ldg(mi + from);
                    z[q] = e[q] & kDenFresh ? 0.f : __ldg(vi + from);
                }
#pragma unroll
                for (int q = 0; q < kDenAhead; q++) {
                    const int i = i0 + q * step;
                    if (i >= w * outs) break;
                    if (gi >= 2 || !(e[q] & kDenSplit)) po[i] = x[q];
                    mo[i] = y[q];
                    vo[i] = z[q];
                }
            }
        }
        oi += (int64_t)w * n;
        oo += (int64_t)w * m;
    }
}

// ------------------------------------------------------------ geometric densification
// A keyframe's coloured point cloud becomes Gaussians (Sec. III-A.3, III-B; the 3DGS
// initialisation): mean = point, isotropic log-scale log sqrt(max(d2, 1e-7)) with d2 the
// mean squared distance to the 3 nearest other points (exact), identity rotation,
// opacity logit(init), SH DC (rgb - 1/2) / Y_0^0, higher bands 0.
//
// Exact k-NN on a uniform grid: bounding box and moments, then the grid (k_bbox); the grid
// spans the box cut to mean +- 3 standard deviations per axis, points outside fall into the
// border cells (so a few far outliers do not stretch the cells); cell size about one point
// per cell of the box's volume, face area or length, whichever is largest, and at most
// kGridCap cells per axis; counting sort of the points by cell (k_cell_count, the scan,
// k_cell_scatter), which copies their coordinates into cell order, so a row of cells along x
// is one contiguous run of points.  Per point a search over growing rings of cells stops
// once the distance to the unsearched region, less a rounding margin, is at least the
// third-best distance (k_knn); points not settled within kNearRings rings are listed and
// searched by a block each (knn_far).

constexpr int kGridCap = 128;
constexpr int kKnn = 3;
constexpr float kKnnFloor = 1e-7f;
constexpr float kShC0 = 0.28209479177387814f;
// Rings a single thread searches.  A stray point far outside the room has to look at
// every cell of the grid: one thread walking them alone took 122 ms on a 307k-point frame
// with two such points, where k_knn takes 160 us and a block for each of the two 17 us.  Four
// rings were not compared with other counts.  Clouds of a dense part and some widely spread
// points, whole call, each thread walking on to the end and now (ms): 307k with 3% spread, 6887
// of them left to the blocks, 3.86 and 1.04; 100k with 10%, 927 left, 2.45 and 0.92; 20k with
// 10% far wider, 12.8 and 7.1 (its dense part in few cells).
constexpr int kNearRings = 4;
constexpr int kFarThreads = 512, kFarBlocks = 304, kFarSample = 4096;

struct GridInfo {
    float lo[3];
    float h;
    int G[3];
    float margin;
    uint32_t box[6];   // sortable encodings, all maxima: complements of min x, y, z, then max x, y, z
    uint32_t done;     // blocks of k_bbox that have added their part
    uint32_t nfar;     // points listed for knn_far
    uint32_t nbad;     // points with a coordinate that is not finite
    double sum[3], sumsq[3];
};

__host__ __device__ inline int64_t grid_cell_budget(int64_t m)
{
    return m + 3 * (int64_t)kGridCap * kGridCap + 3 * kGridCap + 1;
}

__device__ __forceinline__ uint32_t f2sortable(float f)
{
    const uint32_t b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float sortable2f(uint32_t u)
{
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// Grid of the points from their box and moments (one thread).
__device__ void grid_setup(GridInfo *gi, int64_t m, int64_t budget)
{
    float lo[3], ext[3];
    float emax = 0.f, amax = 0.f;
    const double mm = (double)(m > 0 ? m : 1);
    for (int a = 0; a < 3; a++) {
        const uint32_t bmin = __ldcg(&gi->box[a]), bmax = __ldcg(&gi->box[3 + a]);
        const bool any = bmax != 0u;
        const float blo = any ? sortable2f(~bmin) : 0.f;
        const float bhi = any ? sortable2f(bmax) : 0.f;
        const double mu = __ldcg(&gi->sum[a]) / mm;
        const double sd = sqrt(fmax(__ldcg(&gi->sumsq[a]) / mm - mu * mu, 0.0));
        lo[a] = fmaxf(blo, (float)(mu - 3.0 * sd));
        const float hi = fmaxf(fminf(bhi, (float)(mu + 3.0 * sd)), lo[a]);
        ext[a] = fmaxf(hi - lo[a], 0.f);
        emax = fmaxf(emax, ext[a]);
        amax = fmaxf(amax, fmaxf(fabsf(blo), fabsf(bhi)));
    }
    // extents in ascending order: e0 <= e1 <= e2
    float e0 = fminf(ext[0], fminf(ext[1], ext[2])), e2 = emax;
    float e1 = ext[0] + ext[1] + ext[2] - e0 - e2;
    const double vol = (double)ext[0] * ext[1] * ext[2];
    double h = cbrt(vol / mm);
    h = fmax(h, sqrt((double)e1 * e2 / mm));
    h = fmax(h, (double)e2 / mm);
    h = fmax(h, (double)emax / kGridCap);
    if (!(h > 0.0)) h = 1.0;
    float hf = (float)h;
    int G[3];
    for (int it = 0; it < 64; it++) {          // the cell count stays within the caller's budget
        for (int a = 0; a < 3; a++) {
            const int c = (int)ceil((double)ext[a] / hf);
            G[a] = c < 1 ? 1 : (c > kGridCap ? kGridCap : c);
        }
        if ((int64_t)G[0] * G[1] * G[2] <= budget) break;
        hf *= 1.0625f;
    }
    for (int a = 0; a < 3; a++) {
        gi->G[a] = G[a];
        gi->lo[a] = lo[a];
    }
    gi->h = hf;
    // the float cell index of a point can be off by one near a cell face: a point counted in
    // an unsearched cell may lie this much closer than the face
    gi->margin = 8.f * 1.2e-7f * (amax + 2.f * hf);
}

// gi starts all zero; the block that finishes last sets up the grid.  Each block adds its
// part with twelve atomics: a set from every warp queued tens of thousands on the same
// words (307k points 95 us and 8 us for the set-up's own launch, now 20 us together).
constexpr int kBoxThreads = 256;
__global__ void __launch_bounds__(kBoxThreads)
k_bbox(const float *__restrict__ xyz, int64_t m, int64_t budget, GridInfo *__restrict__ gi, int32_t *status)
{
    __shared__ uint32_t sbox[8][6];
    __shared__ double smom[6][kBoxThreads];
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    double s1[3] = {0.0, 0.0, 0.0}, s2[3] = {0.0, 0.0, 0.0};
    int bad = 0;
#pragma unroll 4
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        bool finite = true;
        for (int a = 0; a < 3; a++) {
            const float x = xyz[3 * i + a];
            if (!isfinite(x)) {
                finite = false;
                continue;
            }
            lo[a] = fminf(lo[a], x);
            hi[a] = fmaxf(hi[a], x);
            s1[a] += x;
            s2[a] += (double)x * x;
        }
        bad += finite ? 0 : 1;
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int a = 0; a < 3; a++) {
        for (int o = 16; o > 0; o >>= 1) {
            lo[a] = fminf(lo[a], __shfl_xor_sync(kFull, lo[a], o));
            hi[a] = fmaxf(hi[a], __shfl_xor_sync(kFull, hi[a], o));
        }
        smom[a][threadIdx.x] = s1[a];
        smom[3 + a][threadIdx.x] = s2[a];
        if (lane == 0) {
            const bool any = lo[a] <= hi[a];
            sbox[w][a] = any ? ~f2sortable(lo[a]) : 0u;
            sbox[w][3 + a] = any ? f2sortable(hi[a]) : 0u;
        }
    }
    bad = __reduce_add_sync(kFull, bad);
    if (bad > 0 && lane == 0) {
        atomicAdd(&gi->nbad, (uint32_t)bad);
        set_status(status, CGS_ERR_NONFINITE);
    }
    __syncthreads();
    // one warp per sum: FP64 is slow on this part, a shuffle tree in every warp took most of
    // the kernel
    if (w < 6) {
        double y = 0.0;
        for (int i = lane; i < kBoxThreads; i += 32) y += smom[w][i];
        for (int o = 16; o > 0; o >>= 1) y += __shfl_xor_sync(kFull, y, o);
        if (lane == 0) {
            uint32_t x = 0;
            for (int i = 0; i < kBoxThreads / 32; i++) x = max(x, sbox[i][w]);
            atomicMax(&gi->box[w], x);
            atomicAdd(w < 3 ? &gi->sum[w] : &gi->sumsq[w - 3], y);
            __threadfence();
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(&gi->done, 1u) == gridDim.x - 1) {
        __threadfence();
        grid_setup(gi, m, budget);
    }
}

__device__ __forceinline__ int cell_axis(float x, float lo, float h, int G)
{
    int c = (int)floorf((x - lo) / h);
    return c < 0 ? 0 : (c >= G ? G - 1 : c);
}

// Cell of every point, and its rank among the cell's points (whatever order the atomics took).
__global__ void k_cell_count(const float *__restrict__ xyz, int64_t m, const GridInfo *__restrict__ gi,
                             uint32_t *__restrict__ cell_of, uint32_t *__restrict__ rank,
                             uint32_t *__restrict__ count)
{
    const GridInfo g = *gi;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const int cx = cell_axis(xyz[3 * i], g.lo[0], g.h, g.G[0]);
        const int cy = cell_axis(xyz[3 * i + 1], g.lo[1], g.h, g.G[1]);
        const int cz = cell_axis(xyz[3 * i + 2], g.lo[2], g.h, g.G[2]);
        const uint32_t c = (uint32_t)cx + (uint32_t)g.G[0] * ((uint32_t)cy + (uint32_t)g.G[1] * (uint32_t)cz);
        cell_of[i] = c;
        rank[i] = atomicAdd(count + c, 1u);
    }
}

__global__ void k_cell_scatter(const float *__restrict__ xyz, int64_t m, const uint32_t *__restrict__ cell_of,
                               const uint32_t *__restrict__ rank, const uint32_t *__restrict__ off,
                               float4 *__restrict__ pts)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
        pts[off[cell_of[i]] + rank[i]] =
            make_float4(xyz[3 * i], xyz[3 * i + 1], xyz[3 * i + 2], __uint_as_float((uint32_t)i));
}

// The three smallest distances, ascending (infinite until found).
struct Best {
    float b0 = INFINITY, b1 = INFINITY, b2 = INFINITY;
    __device__ __forceinline__ void insert(float d)
    {
        if (!(d < b2)) return;
        const float t = fmaxf(b0, d);
        b0 = fminf(b0, d);
        b2 = fmaxf(b1, t);
        b1 = fminf(b1, t);
    }
    __device__ __forceinline__ float nth(int want) const { return want <= 1 ? b0 : (want == 2 ? b1 : b2); }
};

// A point, its cell, and the bounds that let the search leave cells out.
struct Query {
    GridInfo g;
    uint32_t self;     // position in cell order
    float p[3];
    int c[3];
    // neighbours to find: min(3, points - 1); none if fewer of the others are finite, when the
    // scale takes its floor (a missing neighbour's distance would be infinite)
    int want;

    __device__ __forceinline__ Query(const GridInfo &gi, const float4 &q, uint32_t at, int64_t m)
        : g(gi), self(at), p{q.x, q.y, q.z}, want(m - 1 < kKnn ? (int)(m - 1) : kKnn)
    {
        if (m - 1 - (int64_t)g.nbad < want) want = 0;
        for (int a = 0; a < 3; a++) c[a] = cell_axis(p[a], g.lo[a], g.h, g.G[a]);
    }
    __device__ __forceinline__ float dist2(const float4 &q) const
    {
        const float ex = q.x - p[0], ey = q.y - p[1], ez = q.z - p[2];
        return ex * ex + ey * ey + ez * ez;
    }
    // Squared distance from the point to every point of cells i0..i1 along axis a is at least
    // this (border cells reach outwards without end).
    __device__ __forceinline__ float gap2(int a, int i0, int i1) const
    {
        float d = 0.f;
        if (i0 > 0) d = fmaxf(d, (g.lo[a] + (float)i0 * g.h) - p[a]);
        if (i1 < g.G[a] - 1) d = fmaxf(d, p[a] - (g.lo[a] + (float)(i1 + 1) * g.h));
        d = fmaxf(d - g.margin, 0.f);
        return d * d;
    }
    __device__ __forceinline__ bool beyond(float low2, const Best &b) const
    {
        return low2 >= b.nth(want) * (1.f + 1e-6f);
    }
    // Cells up to Chebyshev distance r have been searched: is every other point too far?
    __device__ __forceinline__ bool settled(int r, const Best &b) const
    {
        float bound = INFINITY;
        for (int a = 0; a < 3; a++) {
            if (c[a] - r > 0) bound = fminf(bound, p[a] - (g.lo[a] + (float)(c[a] - r) * g.h));
            if (c[a] + r < g.G[a] - 1) bound = fminf(bound, (g.lo[a] + (float)(c[a] + r + 1) * g.h) - p[a]);
        }
        if (bound == INFINITY) return true;   // every cell searched
        const float d = bound - g.margin;
        return d > 0.f && beyond(d * d, b);
    }
    __device__ __forceinline__ float log_scale(const Best &b) const
    {
        float d2 = 0.f;
        if (p[0] != p[0] || p[1] != p[1] || p[2] != p[2]) return 0.5f * logf(kKnnFloor);   // no distances at all
        if (want > 0) d2 += b.b0;
        if (want > 1) d2 += b.b1;
        if (want > 2) d2 += b.b2;
        if (want > 0) d2 = d2 / (float)want;
        return 0.5f * logf(fmaxf(d2, kKnnFloor));
    }
};

// One thread per point, in cell order: log-scale of Gaussian n + id into ls (3 per Gaussian).
// Bound by the latency of its loads: a row of cells costs two offsets and one run of
// coordinates, and rows and cells that lie beyond the third-best distance are not read.
__global__ void __launch_bounds__(128)
k_knn(const float4 *__restrict__ pts, int64_t m, GridInfo *__restrict__ gi, const uint32_t *__restrict__ off,
      uint32_t *__restrict__ far, float *__restrict__ ls)
{
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < m; t += (int64_t)gridDim.x * blockDim.x) {
        const float4 me = pts[t];
        const Query Q(*gi, me, (uint32_t)t, m);
        const GridInfo &g = Q.g;
        Best best;
        bool found = Q.want == 0;
        for (int r = 0; r <= kNearRings && !found; r++) {
            const int z0 = max(-r, -Q.c[2]), z1 = min(r, g.G[2] - 1 - Q.c[2]);
            const int y0 = max(-r, -Q.c[1]), y1 = min(r, g.G[1] - 1 - Q.c[1]);
            const int x0 = max(Q.c[0] - r, 0), x1 = min(Q.c[0] + r, g.G[0] - 1);
            for (int dz = z0; dz <= z1; dz++) {
                const float gz = Q.gap2(2, Q.c[2] + dz, Q.c[2] + dz);
                if (Q.beyond(gz, best)) continue;
                for (int dy = y0; dy <= y1; dy++) {
                    const float gyz = gz + Q.gap2(1, Q.c[1] + dy, Q.c[1] + dy);
                    if (Q.beyond(gyz, best)) continue;
                    // cells at Chebyshev distance exactly r: whole rows on the faces dz = +-r or
                    // dy = +-r, else only dx = -r and dx = +r
                    const bool face = dz == -r || dz == r || dy == -r || dy == r;
                    const uint32_t row =
                        (uint32_t)g.G[0] * ((uint32_t)(Q.c[1] + dy) + (uint32_t)g.G[1] * (uint32_t)(Q.c[2] + dz));
                    for (int side = 0; side < (face ? 1 : 2); side++) {
                        const int a0 = face ? x0 : (side ? Q.c[0] + r : Q.c[0] - r), a1 = face ? x1 : a0;
                        if (a0 < 0 || a1 >= g.G[0] || Q.beyond(gyz + Q.gap2(0, a0, a1), best)) continue;
                        const uint32_t q1 = off[row + (uint32_t)a1 + 1];
                        for (uint32_t q = off[row + (uint32_t)a0]; q < q1; q++)
                            if (q != Q.self) best.insert(Q.dist2(pts[q]));
                    }
                }
            }
            found = Q.settled(r, best);
        }
        if (!found) {
            far[atomicAdd(&gi->nfar, 1u)] = (uint32_t)t;
            continue;
        }
        const float l = Q.log_scale(best);
        float *o = ls + 3 * (int64_t)__float_as_uint(me.w);
        o[0] = l;
        o[1] = l;
        o[2] = l;
    }
}

// The listed points, one block each (of `blocks`).  An evenly spaced sample of the cloud
// bounds the third-best distance first; then the lanes of a warp take 32 rows of cells at a
// time, cut to the cells within that distance, and those rows' points together.
__device__ __forceinline__ void knn_far(uint32_t block, uint32_t blocks, const float4 *__restrict__ pts, int64_t m,
                                        const GridInfo *__restrict__ gi, const uint32_t *__restrict__ off,
                                        const uint32_t *__restrict__ far, float *__restrict__ ls)
{
    constexpr int NW = kFarThreads / 32;
    __shared__ Best sbest[NW];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    auto merge = [](Best &a, const Best &b) {
        a.insert(b.b0);
        a.insert(b.b1);
        a.insert(b.b2);
    };
    auto block_best = [&](Best best) {   // the block's three smallest, in every thread
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            Best other;
            other.b0 = __shfl_down_sync(kFull, best.b0, o);
            other.b1 = __shfl_down_sync(kFull, best.b1, o);
            other.b2 = __shfl_down_sync(kFull, best.b2, o);
            if (lane < o) merge(best, other);
        }
        __syncthreads();   // the previous result has been read
        if (lane == 0) sbest[w] = best;
        __syncthreads();
        best = sbest[0];
        for (int i = 1; i < NW; i++) merge(best, sbest[i]);
        return best;
    };
    const uint32_t nfar = gi->nfar;
    for (uint32_t f = block; f < nfar; f += blocks) {
        const uint32_t t = far[f];
        const float4 me = pts[t];
        const Query Q(*gi, me, t, m);
        const GridInfo &g = Q.g;
        Best best;
        const int64_t step = (m + kFarSample - 1) / kFarSample;
#pragma unroll 4
        for (int64_t q = threadIdx.x * step; q < m; q += kFarThreads * step)
            if (q != t) best.insert(Q.dist2(pts[q]));
        const Best bound = block_best(best);
        const float reach2 = bound.nth(Q.want) * (1.f + 1e-6f);
        best = Best();
        const int rows = g.G[1] * g.G[2];
        for (int r0 = 32 * w; r0 < rows; r0 += kFarThreads) {   // warp-uniform
            const int rr = r0 + lane, y = rr % g.G[1], z = rr / g.G[1];
            uint32_t q0 = 0u, len = 0u;
            if (rr < rows) {
                const float low2 = Q.gap2(1, y, y) + Q.gap2(2, z, z);
                if (low2 <= reach2) {
                    // the cells along x within reach, one more on each side for the rounding
                    // (distances past an int's range end at the border cells)
                    const float d = sqrtf(fmaxf(reach2 - low2, 0.f)) + g.margin;
                    const int x0 = max(cell_axis(Q.p[0] - d, g.lo[0], g.h, g.G[0]) - 1, 0);
                    const int x1 = min(cell_axis(Q.p[0] + d, g.lo[0], g.h, g.G[0]) + 1, g.G[0] - 1);
                    const uint32_t row = (uint32_t)rr * (uint32_t)g.G[0];
                    q0 = off[row + (uint32_t)x0];
                    len = off[row + (uint32_t)x1 + 1] - q0;
                }
            }
            uint32_t incl = len;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y2 = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += y2;
            }
            const uint32_t total = __shfl_sync(kFull, incl, 31), first = q0 - (incl - len);
            for (uint32_t j0 = 0; j0 < total; j0 += 32) {   // warp-uniform
                const uint32_t j = j0 + lane;
                int L = 0;   // owner: the number of lanes whose inclusive prefix is <= j
#pragma unroll
                for (int b = 16; b > 0; b >>= 1)
                    if (__shfl_sync(kFull, incl, L + b - 1) <= j) L += b;
                const uint32_t q = __shfl_sync(kFull, first, L) + j;
                if (j < total && q != t) best.insert(Q.dist2(pts[q]));
            }
        }
        best = block_best(best);
        if (threadIdx.x < 3) ls[3 * (int64_t)__float_as_uint(me.w) + threadIdx.x] = Q.log_scale(best);
    }
}

// The rest of the output as runs of floats: the old Gaussians' groups copied, and the new
// ones' appended, a run per (array, group, old or new).  Every block fills one chunk of a
// run, so the kind of run is uniform and both sides are contiguous.  Bound by HBM: 100k old
// and 307k new Gaussians of SH degree 3 in 60 us, 6.0 TB/s; a thread per Gaussian took 141 us
// for the old, 212 us for the new ones' moments and part of the neighbour search for the rest.
enum RunKind { kRunCopy, kRunFill, kRunQuat, kRunColor };
struct Run {
    float *dst;
    const float *src;
    int64_t len, block0;   // floats; first block
    float value;
    int kind;
};
constexpr int kMaxRuns = 36, kRunThreads = kFarThreads, kRunChunk = 16 * kRunThreads;
struct Runs {
    Run run[kMaxRuns];
    int n;
    int64_t blocks;
};

__device__ __forceinline__ void fill_run(const Runs &R, int64_t block)
{
    int k = 0;
    while (k + 1 < R.n && block >= R.run[k + 1].block0) k++;
    const Run &r = R.run[k];
    const int64_t e0 = (block - r.block0) * kRunChunk;
    const int cnt = (int)min((int64_t)kRunChunk, r.len - e0);
    float *d = r.dst + e0;
    const float *s = r.src ? r.src + e0 : nullptr;
    switch (r.kind) {
    case kRunCopy: {
        // all of the chunk's loads in flight before the first store
        float x[kRunChunk / kRunThreads];
#pragma unroll
        for (int q = 0; q < kRunChunk / kRunThreads; q++) {
            const int i = q * kRunThreads + (int)threadIdx.x;
            x[q] = i < cnt ? __ldg(s + i) : 0.f;
        }
#pragma unroll
        for (int q = 0; q < kRunChunk / kRunThreads; q++) {
            const int i = q * kRunThreads + (int)threadIdx.x;
            if (i < cnt) d[i] = x[q];
        }
        break;
    }
    case kRunFill: {
        // whole 16-byte words from the first aligned one
        const int head = min(cnt, (int)(((16u - ((uint32_t)(uintptr_t)d & 15u)) & 15u) >> 2)), words = (cnt - head) / 4;
        const float4 v4 = make_float4(r.value, r.value, r.value, r.value);
        for (int i = threadIdx.x; i < words; i += kRunThreads) reinterpret_cast<float4 *>(d + head)[i] = v4;
        for (int i = threadIdx.x; i < cnt; i += kRunThreads)
            if (i < head || i >= head + 4 * words) d[i] = r.value;
        break;
    }
    case kRunQuat:   // identity rotations
        for (int i = threadIdx.x; i < cnt; i += kRunThreads) d[i] = (i & 3) == 0 ? 1.f : 0.f;
        break;
    default:   // colours as SH DC coefficients
        for (int i = threadIdx.x; i < cnt; i += kRunThreads) d[i] = (__ldg(s + i) - 0.5f) / kShC0;
    }
}
static_assert(kRunChunk % 4 == 0, "a chunk of quaternions starts at a whole one");

__global__ void __launch_bounds__(kRunThreads) k_runs(const __grid_constant__ Runs R) { fill_run(R, blockIdx.x); }

// The far points' search beside the runs: a few blocks waiting on memory, hidden by the copies
// (17 us of a 307k-point frame with two strays).
__global__ void __launch_bounds__(kFarThreads)
k_far_runs(const __grid_constant__ Runs R, const float4 *__restrict__ pts, int64_t m,
           const GridInfo *__restrict__ gi, const uint32_t *__restrict__ off, const uint32_t *__restrict__ far,
           float *__restrict__ ls)
{
    if (blockIdx.x < kFarBlocks)
        knn_far(blockIdx.x, kFarBlocks, pts, m, gi, off, far, ls);
    else
        fill_run(R, (int64_t)blockIdx.x - kFarBlocks);
}

static void add_run(Runs &R, float *dst, const float *src, int64_t len, int kind, float value = 0.f)
{
    if (len <= 0) return;
    R.run[R.n++] = Run{dst, src, len, R.blocks, value, kind};
    R.blocks += (len + kRunChunk - 1) / kRunChunk;
}

}  // namespace cgs

using namespace cgs;

namespace {
size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }
int st_of(cudaError_t e)
{
    if (e == cudaSuccess) return CGS_OK;
    fprintf(stderr, "libcgs: CUDA error: %s\n", cudaGetErrorString(e));
    return CGS_ERR_CUDA;
}
}  // namespace

extern "C" {

size_t cgs_densify_workspace(int64_t n)
{
    if (n < 0) return 0;
    return al256(sizeof(uint32_t) * (size_t)n) * 2 + al256(sizeof(uint32_t) * ((size_t)n + 1));
}

int cgs_densify_plan(const float *params, int64_t n, int32_t sh_degree, const float *accum, const float *denom,
                     double tau_p, double scale_thr, double eps_alpha, void *workspace, size_t workspace_bytes,
                     int64_t *n_out_dev, void *stream)
{
    if (!params || !accum || !denom || !workspace || !n_out_dev || n < 1 || sh_degree < 0 || sh_degree > 3)
        return CGS_ERR_ARG;
    if (!(scale_thr > 0.0) || !(eps_alpha > 0.0 && eps_alpha < 1.0) || !(tau_p >= 0.0)) return CGS_ERR_ARG;
    if (2 * n + 1 >= ((int64_t)1 << 32)) return CGS_ERR_ARG;
    if (((uintptr_t)workspace & 255) != 0) return CGS_ERR_ARG;
    if (workspace_bytes < cgs_densify_workspace(n)) return CGS_ERR_WORKSPACE;
    uint32_t *code = static_cast<uint32_t *>(workspace);
    // span totals: at most one per kScanChunk Gaussians
    unsigned long long *part =
        reinterpret_cast<unsigned long long *>(static_cast<char *>(workspace) + al256(sizeof(uint32_t) * n));
    uint32_t *off = reinterpret_cast<uint32_t *>(static_cast<char *>(workspace) + 2 * al256(sizeof(uint32_t) * n));
    const float t_grad = (float)tau_p;
    const float t_logs = (float)log(scale_thr);
    const float t_logit = (float)log(eps_alpha / (1.0 - eps_alpha));
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t span = scan_span(n);
    const int blocks = scan_blocks(n);
    k_densify_plan<<<blocks, kScanThreads, 0, s>>>(params, n, span, accum, denom, t_grad, t_logs, t_logit, code, part);
    k_span_scan<<<blocks, kScanThreads, 0, s>>>(CodeEntry{code}, n, span, part, off, n_out_dev);
    return st_of(cudaGetLastError());
}

int cgs_densify_apply(const float *params, const float *m, const float *v, int64_t n, int32_t sh_degree,
                      const void *workspace, size_t workspace_bytes, const float *normals, int64_t n_out,
                      float *params_out, float *m_out, float *v_out, void *stream)
{
    if (!params || !m || !v || !workspace || !normals || n < 1 || n_out < 0 || sh_degree < 0 || sh_degree > 3)
        return CGS_ERR_ARG;
    if (n_out > 0 && (!params_out || !m_out || !v_out)) return CGS_ERR_ARG;
    if (workspace_bytes < cgs_densify_workspace(n)) return CGS_ERR_WORKSPACE;
    if (n_out > 2 * n) return CGS_ERR_ARG;
    const uint32_t *code = static_cast<const uint32_t *>(workspace);
    const uint32_t *off =
        reinterpret_cast<const uint32_t *>(static_cast<const char *>(workspace) + 2 * al256(sizeof(uint32_t) * n));
    cudaStream_t s = (cudaStream_t)stream;
    auto k = sh_degree == 0   ? k_densify_apply<0>
             : sh_degree == 1 ? k_densify_apply<1>
             : sh_degree == 2 ? k_densify_apply<2>
                              : k_densify_apply<3>;
    k<<<(unsigned)((n + kDenG - 1) / kDenG), kDenThreads, 0, s>>>(params, m, v, n, code, off, normals, n_out,
                                                                  params_out, m_out, v_out);
    return st_of(cudaGetLastError());
}

size_t cgs_points_workspace(int64_t n_points)
{
    if (n_points < 1) return 0;
    const int64_t B = grid_cell_budget(n_points);
    return al256(sizeof(GridInfo)) + 2 * al256(sizeof(uint32_t) * ((size_t)B + 1)) +
           2 * al256(sizeof(uint32_t) * (size_t)n_points) + al256(sizeof(float4) * (size_t)n_points) +
           al256(sizeof(unsigned long long) * kScanBlocks);
}

int cgs_points_to_gaussians(const float *params, const float *m, const float *v, int64_t n, int32_t sh_degree,
                            const float *xyz, const float *rgb, int64_t n_points, float init_opacity,
                            void *workspace, size_t workspace_bytes, float *params_out, float *m_out,
                            float *v_out, int32_t *status_dev, void *stream)
{
    if (n < 0 || n_points < 0 || n + n_points < 1 || sh_degree < 0 || sh_degree > 3) return CGS_ERR_ARG;
    if (n > 0 && (!params || !m || !v)) return CGS_ERR_ARG;
    if (!params_out || !m_out || !v_out) return CGS_ERR_ARG;
    if (n_points > 0 && (!xyz || !rgb || !workspace)) return CGS_ERR_ARG;
    if (!(init_opacity > 0.f && init_opacity < 1.f)) return CGS_ERR_ARG;
    if (grid_cell_budget(n_points) + 1 >= ((int64_t)1 << 32)) return CGS_ERR_ARG;
    const int64_t n_out = n + n_points;
    const int widths[6] = {3, 3, 4, 1, 3, 3 * ((sh_degree + 1) * (sh_degree + 1) - 1)};
    const float logit = logf(init_opacity / (1.f - init_opacity));
    cudaStream_t s = (cudaStream_t)stream;
    Runs R{};
    float *out[3] = {params_out, m_out, v_out};
    const float *in[3] = {params, m, v};
    for (int k = 0; k < 3; k++) {
        int64_t oi = 0, oo = 0;
        for (int gi = 0; gi < 6; gi++) {
            const int64_t w = widths[gi];
            if (n > 0) add_run(R, out[k] + oo, in[k] + oi, w * n, kRunCopy);
            float *tail = out[k] + oo + w * n;
            const int64_t len = w * n_points;
            if (k > 0 || gi == 5)
                add_run(R, tail, nullptr, len, kRunFill);   // moments and higher bands start at zero
            else if (gi == 0)
                add_run(R, tail, xyz, len, kRunCopy);
            else if (gi == 2)
                add_run(R, tail, nullptr, len, kRunQuat);
            else if (gi == 3)
                add_run(R, tail, nullptr, len, kRunFill, logit);
            else if (gi == 4)
                add_run(R, tail, rgb, len, kRunColor);
            oi += w * n;
            oo += w * n_out;
        }
    }
    if (n_points > 0 && ((uintptr_t)workspace & 255) != 0) return CGS_ERR_ARG;
    if (n_points > 0 && workspace_bytes < cgs_points_workspace(n_points)) return CGS_ERR_WORKSPACE;
    if (R.blocks + kFarBlocks >= (int64_t)1 << 31) return CGS_ERR_ARG;
    if (n_points == 0) {
        k_runs<<<(unsigned)R.blocks, kRunThreads, 0, s>>>(R);
        return st_of(cudaGetLastError());
    }
    const int64_t B = grid_cell_budget(n_points);
    char *w = static_cast<char *>(workspace);
    GridInfo *gi = reinterpret_cast<GridInfo *>(w);
    w += al256(sizeof(GridInfo));
    uint32_t *count = reinterpret_cast<uint32_t *>(w);   // next to gi: one memset clears both
    w += al256(sizeof(uint32_t) * (B + 1));
    uint32_t *off = reinterpret_cast<uint32_t *>(w);
    w += al256(sizeof(uint32_t) * (B + 1));
    uint32_t *cell_of = reinterpret_cast<uint32_t *>(w);   // later the list of far points
    w += al256(sizeof(uint32_t) * n_points);
    uint32_t *rank = reinterpret_cast<uint32_t *>(w);
    w += al256(sizeof(uint32_t) * n_points);
    float4 *pts = reinterpret_cast<float4 *>(w);
    w += al256(sizeof(float4) * n_points);
    unsigned long long *part = reinterpret_cast<unsigned long long *>(w);
    const cudaError_t e = cudaMemsetAsync(gi, 0, al256(sizeof(GridInfo)) + sizeof(uint32_t) * (B + 1), s);
    if (e != cudaSuccess) return st_of(e);
    const int pb = (int)((n_points + 255) / 256 < 1024 ? (n_points + 255) / 256 : 1024);
    k_bbox<<<pb < 304 ? pb : 304, 256, 0, s>>>(xyz, n_points, B, gi, status_dev);
    k_cell_count<<<pb, 256, 0, s>>>(xyz, n_points, gi, cell_of, rank, count);
    const int64_t span = scan_span(B);
    const int sb = scan_blocks(B);
    k_span_totals<<<sb, kScanThreads, 0, s>>>(count, B, span, part);
    k_span_scan<<<sb, kScanThreads, 0, s>>>(CountEntry{count}, B, span, part, off, nullptr);
    k_cell_scatter<<<pb, 256, 0, s>>>(xyz, n_points, cell_of, rank, off, pts);
    const int kb = (int)((n_points + 127) / 128 < 8192 ? (n_points + 127) / 128 : 8192);
    float *ls = params_out + 3 * n_out + 3 * n;   // log-scales of the new Gaussians
    k_knn<<<kb, 128, 0, s>>>(pts, n_points, gi, off, cell_of, ls);
    k_far_runs<<<(unsigned)(kFarBlocks + R.blocks), kFarThreads, 0, s>>>(R, pts, n_points, gi, off, cell_of, ls);
    return st_of(cudaGetLastError());
}

}  // extern "C"
