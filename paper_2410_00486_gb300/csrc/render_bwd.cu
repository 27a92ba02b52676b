// Backward of the blend (Eqs. 2-4, Sec. III-C.1, CaRtGS), pixel-parallel.
//
// One block per (view, tile), eight pixels of one column per thread (one warp per 16x16
// tile; two pixels on 8x8 tiles), walking the tile's list back to front from the block's
// largest `last`.
// A tile's list holds only splats that can reach alpha >= 1/255 in it (the binning's
// test), the same list the forward walked.  Each pixel recomputes alpha exactly as the
// forward did (same rounding, same decisions) and its transmittance from the stored final T,
// T_j = T_{j+1} / (1 - alpha_j), so no per-pixel splat list is kept.  A thread blends its
// pixels in pairs: when either pixel of a pair blends splat j, both run through the blend
// (the other with alpha = 0, which leaves its state as it is), so the two dependency chains
// interleave.
//
// With R_j the colour behind splat j normalised by the transmittance just after it,
// R_last = bg and R_{j-1} = a_j c_j + (1 - a_j) R_j (depth alike, starting at 0),
//   dL/dalpha_j = T_j [ gI . (c_j - R_j) + gD (z_j - Rz_j) ],
// so a pixel only carries the scalar S_j = gI . R_j + gD Rz_j, updated by the same
// recursion with c_j . gI + z_j gD in place of the colour.
//
// The per-(splat, pixel) gradients of a thread's pixels are added in registers (the
// pixels share dx, so the dx moments are formed once per thread), then a warp's rows of
// ten sums are added through shared memory (each lane stores its row, thirty lanes add
// one field over a third of the rows each, two shuffles join the thirds), after which
// ten lanes each issue one atomic add into the slot's gradient record; when only a few
// lanes contributed they add their own sums directly instead.  Warps where no pixel
// blended the splat skip it (vote).
//
// The per-pixel loss gradients (three channels and depth) are constant during the walk and
// live in shared memory, read once per blended pixel; that leaves 72 registers a thread,
// so 28 warps stay resident.  With a work counter the grid is persistent: as many blocks
// as are resident on the GPU take (view, tile) items in the sort's longest-first order
// from the counter until none is left.
//
// Windows of few tiles split each 16x16 tile into two or four parts, a warp and four or two
// pixels a thread each, and the smallest its list into two segments (bwd_split): one 640x480
// view of 40k Gaussians 190 -> 100 us, three of 637x479 343 -> 280 us.
#include "raster.cuh"

namespace cgs {

// Splats to which at most this many lanes of a warp contribute are added with per-lane
// atomics (L2 reductions); more contributors go through the warp sum.  Measured on the
// 16-view window with the persistent 28-warp kernel (raster backward ms): 4 lanes 3.366,
// 8 lanes 3.347, 10 lanes 3.340, 12 lanes 3.344, 16 lanes 3.419, 20 lanes 3.580, 24 lanes
// 3.877; folding a half-warp onto the other and adding from 16 lanes was twice as slow
// (same-address atomics serialise).
constexpr int kDirectLanes = 10;

// Row stride (floats) of the per-warp reduction buffer: ten fields padded to 12.
constexpr int kRedStride = 12;
constexpr int kRedRows = 33;   // 32 lanes and a zero row

__device__ __forceinline__ float sgnf(float x) { return x > 0.f ? 1.f : (x < 0.f ? -1.f : 0.f); }

// Shared memory of one work item: the staged batch, the loss gradients of its pixels (pixel p
// of thread t at [p NT + t]: three channels, depth) and a reduction buffer per warp.
template <int BD, int PIX, int NW>
struct BwdSmem {
    float4 s0[BD], s1[BD], s2[BD];
    uint32_t slot[BD];
    uint32_t smax[NW];
    __align__(16) float red[NW * kRedRows * kRedStride];
    float4 gi[PIX];
};

// One work item: the tile at a place of the work order by NT threads of PPT pixels each, or
// (S > 1) one of S parts of it by a warp on its own in a block of several: a half of eight
// rows, or one of the four 8x8 blocks, whose short outline the fewest splats cross.  With SEG
// > 1 an item is also one of SEG segments of the list: the splats behind its segment only
// take the pixels' transmittance and colour behind to the segment's end, by the same steps
// (the same bits) as the item that owns them.
template <int B, int BD, int NT, int PPT, int S, int SEG, class Smem>
__device__ __forceinline__ void bwd_item(const RasterBwdArgs &a, uint32_t place, int part, int seg, int tid, Smem &sm)
{
    constexpr int NW = NT / 32;
    constexpr bool kWarp = S > 1, kBlocks = S == 4;
    float4 *s0 = sm.s0, *s1 = sm.s1, *s2 = sm.s2, *sgi = sm.gi;
    uint32_t *sslot = sm.slot;
    auto item_sync = [] {
        if (kWarp) __syncwarp();
        else __syncthreads();
    };
    const int lane = threadIdx.x & 31;
    int64_t tile;
    int view, tx, ty;
    item_tile(a.order, a.g, tile, view, tx, ty, place);
    // row of pixel p: py0 + G p
    constexpr int G = kBlocks ? 4 : row_step<B>();
    const int px = tx * B + (kBlocks ? 8 * (part & 1) + (lane & 7) : tid % B);
    const int py0 = ty * B + (kBlocks ? 8 * (part >> 1) + (lane >> 3) : part * (B / S) + thread_row0<B, PPT>(tid));
    const float fx = (float)px;
    const uint32_t start = a.ranges[2 * tile];
    const uint32_t len = a.ranges[2 * tile + 1] - start;
    const size_t HW = (size_t)a.g.W * a.g.H;

    // per-pixel state: transmittance, pixel gradients, and S = (colour behind) . gI +
    // (depth behind) gD, where "behind" starts as the background (no depth) and follows
    // R <- alpha c + (1 - alpha) R towards the front
    float T[PPT], Sb[PPT];
    const float fy0 = (float)py0;   // row of pixel p: fy0 + G p (exact)
    uint32_t lst[PPT];
    uint32_t m = 0;
#pragma unroll
    for (int p = 0; p < PPT; p++) {
        const int py = py0 + G * p;
        lst[p] = 0;
        T[p] = 1.f;
        Sb[p] = 0.f;
        float gI0 = 0.f, gI1 = 0.f, gI2 = 0.f, gD = 0.f;
        if (!(px < a.g.W && py < a.g.H)) {
            sgi[p * NT + tid] = make_float4(0.f, 0.f, 0.f, 0.f);
            continue;
        }
        const size_t q = (size_t)py * a.g.W + px;
        const size_t pix = (size_t)view * HW + q;
        // never walk past the tile's list, whatever `last` holds
        lst[p] = min(a.last[pix], len);
        T[p] = a.tfin[pix];
        if (a.dl_dimg) {
            const float *gi = a.dl_dimg + (size_t)view * 3 * HW + q;
            gI0 = gi[0];
            gI1 = gi[HW];
            gI2 = gi[2 * HW];
            gD = a.dl_ddepth ? a.dl_ddepth[pix] : 0.f;
        } else {
            const float w = a.weight ? a.weight[view] : 1.f;
            const float sc = w / (3.f * (float)HW);
            const float *im = a.img + (size_t)view * 3 * HW + q;
            const float *tr = a.tgt_rgb + (size_t)view * 3 * HW + q;
            gI0 = sc * sgnf(im[0] - tr[0]);
            gI1 = sc * sgnf(im[HW] - tr[HW]);
            gI2 = sc * sgnf(im[2 * HW] - tr[2 * HW]);
            if (a.tgt_depth) {
                const float td = a.tgt_depth[pix];
                const int cnt = a.depth_count[view];
                if (td > 0.f && cnt > 0) gD = w * a.lambda_d * sgnf(a.depth[pix] - td) / (float)cnt;
            }
        }
        sgi[p * NT + tid] = make_float4(gI0, gI1, gI2, gD);
        Sb[p] = a.bg0 * gI0 + a.bg1 * gI1 + a.bg2 * gI2;
        m = max(m, lst[p]);
    }
    // block-wide largest `last`: the walk starts there
    for (int off = 16; off > 0; off >>= 1) m = max(m, __shfl_xor_sync(kFull, m, off));
    uint32_t maxlast = kWarp ? m : 0u;
    if (!kWarp) {
        if (lane == 0) sm.smax[threadIdx.x / 32] = m;
        __syncthreads();
        for (int i = 0; i < NW; i++) maxlast = max(maxlast, sm.smax[i]);
    }

    // A part stages one splat a lane per batch, and the next batch's records are on their way
    // while this one is walked (few warps: nothing else hides their latency)
    constexpr bool kAhead = kWarp;
    static_assert(!kAhead || BD == 32, "a splat a lane");
    float4 n0, n1, n2;
    uint32_t nslot = 0;
    auto fetch = [&](int at) {   // the lane's splat of the batch ending at `at`
        const int i = at - BD + lane;
        if (i >= 0) {
            nslot = a.vals[start + i];
            const float4 *r = a.rec + kRec4 * (size_t)nslot;
            n0 = r[0];
            n1 = r[1];
            n2 = r[2];
        }
    };
    const int seg0 = SEG > 1 ? (int)((uint64_t)maxlast * seg / SEG) : 0;
    const int seg1 = SEG > 1 ? (int)((uint64_t)maxlast * (seg + 1) / SEG) : (int)maxlast;
    if (SEG > 1 && seg0 == seg1) return;   // item-uniform
    if (kAhead) fetch((int)maxlast);
    for (int bend = (int)maxlast; bend > seg0; bend -= BD) {
        const int bstart = kAhead ? bend - BD : max(0, bend - BD);   // below 0: the batch's first lanes are empty
        const int nraw = bend - bstart;
        item_sync();
        // stage positions [bstart, bend) (every entry can reach the tile: the binning's test)
        if (kAhead) {
            if (bstart + lane >= 0) {
                stage_splat(n0, n1, n2.w, s0[lane], s1[lane]);
                s2[lane] = n2;
                sslot[lane] = nslot;
            }
            fetch(bstart);
        } else {
            for (int c0 = 0; c0 < BD; c0 += NT) {
                const int i = c0 + tid;
                if (i >= nraw) break;
                const uint32_t slot = a.vals[start + bstart + i];
                const float4 *r = a.rec + kRec4 * (size_t)slot;
                const float4 r2 = r[2];
                stage_splat(r[0], r[1], r2.w, s0[i], s1[i]);
                s2[i] = r2;
                sslot[i] = slot;
            }
        }
        item_sync();
        const int j0 = kAhead ? max(0, seg0 - bstart) : 0;
        int jtop = nraw - 1;
        if (SEG > 1) {
            // behind the segment: transmittance and colour behind only
#pragma unroll 4
            for (; jtop >= max(j0, seg1 - bstart); jtop--) {
                const uint32_t pos = (uint32_t)(bstart + jtop);
                const float4 q0 = s0[jtop], q1 = s1[jtop], q2 = s2[jtop];
                const PowerX pxs = power_x(q0, __fsub_rn(q0.x, fx));
#pragma unroll
                for (int p = 0; p < PPT; p++) {
                    const float pw = power_at(pxs, q1.x, __fsub_rn(q0.y, fy0 + (float)(G * p)));
                    if (!(pos < lst[p] && fabsf(pw) <= q1.w)) continue;
                    const float4 gi = sgi[p * NT + tid];
                    const float alpha = fminf(kAlphaMax, __fmul_rn(q1.y, exp2_fast(pw)));
                    T[p] = T[p] * rcp_fast(__fsub_rn(1.f, alpha));
                    const float cg = fmaf(q1.z, gi.w, fmaf(q2.z, gi.z, fmaf(q2.y, gi.y, q2.x * gi.x)));
                    Sb[p] = fmaf(alpha, cg - Sb[p], Sb[p]);
                }
            }
        }
        // two splats per loop trip, so one splat's loads and tests overlap the other's blend and
        // sums (3.470 -> 3.426 ms on the 16-view window; four per trip spill: 3.87 ms)
#pragma unroll 2
        for (int j = jtop; j >= j0; j--) {
            const uint32_t pos = (uint32_t)(bstart + j);   // list position of splat j
            const float4 q0 = s0[j];
            const float4 q1 = s1[j];
            const float4 q2 = s2[j];
            const float dx = __fsub_rn(q0.x, fx);
            const PowerX pxs = power_x(q0, dx);
            // per-thread sums over its pixels: colour / depth / opacity gradients, and the
            // moments sum dp, sum dp dy, sum dp dy^2 of dp = dL/dpower (dx is shared)
            float gr = 0.f, gg = 0.f, gb = 0.f, gz = 0.f, go = 0.f, sdp = 0.f, sdpy = 0.f, sdpyy = 0.f;
            bool contrib = false;
            unsigned who = 0u;   // lanes with a pixel that blends
            // pixels in pairs: a pair where either pixel blends runs both through the blend
            // (the other with G = 0, so alpha = 0 and its state is kept), so the two chains
            // interleave
#pragma unroll
            for (int p2 = 0; p2 < PPT; p2 += 2) {
                float dyv[2], pw[2];
                bool k[2];
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const int p = p2 + h;
                    dyv[h] = __fsub_rn(q0.y, fy0 + (float)(G * p));
                    pw[h] = power_at(pxs, q1.x, dyv[h]);
                    k[h] = pos < lst[p] && fabsf(pw[h]) <= q1.w;
                }
                // a warp-uniform branch (vote) rather than a divergent one: a lane whose pair
                // blends nothing runs the pair with alpha = 0, which changes nothing (3.337 ->
                // 3.297 ms on the 16-view window)
                const bool pair = k[0] || k[1];
                contrib = contrib || pair;
                if (PPT > 2 && !__any_sync(kFull, pair)) continue;
                if (PPT == 2) {
                    who = __ballot_sync(kFull, pair);
                    if (who == 0u) break;
                }
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const int p = p2 + h;
                    const float dy = dyv[h];
                    const float4 gi = sgi[p * NT + tid];   // dL/dimg, dL/ddepth of pixel p
                    const float G = k[h] ? exp2_fast(pw[h]) : 0.f;
                    const float araw = __fmul_rn(q1.y, G);
                    const float alpha = fminf(kAlphaMax, araw);
                    const float inv_om = rcp_fast(__fsub_rn(1.f, alpha));
                    T[p] = k[h] ? T[p] * inv_om : T[p];               // transmittance before splat j
                    const float wT = alpha * T[p];
                    gr = fmaf(wT, gi.x, gr);
                    gg = fmaf(wT, gi.y, gg);
                    gb = fmaf(wT, gi.z, gb);
                    gz = fmaf(wT, gi.w, gz);
                    const float cg = fmaf(q1.z, gi.w, fmaf(q2.z, gi.z, fmaf(q2.y, gi.y, q2.x * gi.x)));
                    const float diff = cg - Sb[p];
                    Sb[p] = fmaf(alpha, diff, Sb[p]);
                    // dalpha/dpower = alpha, dalpha/dopacity = G, both 0 where alpha is clamped
                    const float dLda = araw > kAlphaMax ? 0.f : diff * T[p];
                    go = fmaf(dLda, G, go);
                    const float dp = dLda * alpha;
                    const float dpy = dp * dy;
                    sdp += dp;
                    sdpy += dpy;
                    sdpyy = fmaf(dpy, dy, sdpyy);
                }
            }
            if (PPT > 2) who = __ballot_sync(kFull, contrib);
            if (who == 0u) continue;
            // raw moments of dp over this thread's pixels: sum dp dx, dp dy, dp dx^2, dp dx dy, dp dy^2
            const float m0 = sdp * dx, m3 = sdpy * dx;
            if (__popc(who) <= kDirectLanes) {
                // few contributing lanes: each adds its sums directly
                if (contrib) {
                    float *g = a.sgrad + (size_t)sslot[j] * 12;
                    const float hA = q0.z, nB = q0.w, hC = q1.x;
                    atomicAdd(g + 0, kLn2 * (2.f * hA * m0 + nB * sdpy));   // staged terms carry log2 e
                    atomicAdd(g + 1, kLn2 * (2.f * hC * sdpy + nB * m0));
                    atomicAdd(g + 2, -0.5f * (m0 * dx));
                    atomicAdd(g + 3, -m3);
                    atomicAdd(g + 4, -0.5f * sdpyy);
                    atomicAdd(g + 5, go);
                    atomicAdd(g + 6, gz);
                    atomicAdd(g + 8, gr);
                    atomicAdd(g + 9, gg);
                    atomicAdd(g + 10, gb);
                }
                continue;
            }
            {
                // warp sum of the ten fields through shared memory: every lane stores its
                // row, then lanes 10g + f (g < 3, f < 10) add field f over rows g, g + 3,
                // g + 6, ... and three shuffles combine the groups (row stride 12 floats:
                // the 16-byte stores are conflict-free, the column reads nearly so)
                float *buf = sm.red + (kWarp ? 0 : (size_t)(threadIdx.x >> 5) * (kRedRows * kRedStride));
                __syncwarp();   // the previous sum's column reads are done before the rows are rewritten
                float4 *row = reinterpret_cast<float4 *>(buf + lane * kRedStride);
                row[0] = make_float4(m0, sdpy, m0 * dx, m3);
                row[1] = make_float4(sdpyy, go, gz, gr);
                row[2] = make_float4(gg, gb, 0.f, 0.f);
                __syncwarp();
                const int g = lane / 10, f = lane - 10 * g;
                float sum = 0.f;
                if (lane < 30) {
                    // rows g, g + 3, ..., g + 30; row 32 (group 2's last) is a zero row
                    const float *col = buf + g * kRedStride + f;
#pragma unroll
                    for (int k = 0; k < 11; k++) sum += col[3 * k * kRedStride];
                }
                {
                    const float p1 = __shfl_down_sync(kFull, sum, 10), p2 = __shfl_down_sync(kFull, sum, 20);
                    sum += p1 + p2;   // lanes 0..9: field sums (groups 0, 1, 2)
                }
                // fields 0 and 1 (first moments) sit in lanes 0 and 1: exchange them
                const float other = __shfl_xor_sync(kFull, sum, 1);
                // power = -(A dx^2 + C dy^2)/2 - B dx dy with dx = u - x:
                //   dL/du = -(A S_dx + B S_dy), dL/dv = -(C S_dy + B S_dx),
                //   dL/dA = -S_xx / 2, dL/dB = -S_xy, dL/dC = -S_yy / 2
                // (staged q0.z = -A/2, q0.w = -B, q1.x = -C/2)
                const float hC = q1.x;
                if (f == 0) sum = kLn2 * (2.f * q0.z * sum + q0.w * other);   // staged terms carry log2 e
                else if (f == 1) sum = kLn2 * (2.f * hC * sum + q0.w * other);
                else if (f == 2 || f == 4) sum = -0.5f * sum;
                else if (f == 3) sum = -sum;
                // record fields 0..6 (u, v, A, B, C, o, z), 8..10 (r, g, b)
                if (lane < 10) atomicAdd(a.sgrad + (size_t)sslot[j] * 12 + (f < 7 ? f : f + 1), sum);
            }
        }
    }
}

// The zero rows of a block's reduction buffers.
template <int N>
__device__ __forceinline__ void zero_rows(float (&red)[N], int t, int threads)
{
    for (int i = t; i < N / kRedRows; i += threads)
        red[(i / kRedStride) * (kRedRows * kRedStride) + 32 * kRedStride + i % kRedStride] = 0.f;
}

// A block takes a tile at a time, the next one in the work order from the work counter (a
// persistent launch), or its own.
template <int B, int BD>
__global__ void __launch_bounds__(B *B / ppt_for<B, kPPTBwd>(), (min_blocks_for<B, kPPTBwd, kBwdMinWarps>())) k_render_bwd(RasterBwdArgs a)
{
    pdl_begin();   // plain loads below: none moves ahead of the wait
    constexpr int PPT = ppt_for<B, kPPTBwd>();
    constexpr int NT = B * B / PPT;
    __shared__ BwdSmem<BD, NT * PPT, NT / 32> sm;
    __shared__ uint32_t s_item;
    zero_rows(sm.red, threadIdx.x, NT);
    const uint32_t n_items = (uint32_t)(a.g.Tv * a.V);
    for (uint32_t it = 0;; it++) {
        uint32_t item = blockIdx.x;
        if (a.work) {
            __syncthreads();   // the previous item's reads of s_item and of the shared state are done
            if (threadIdx.x == 0) s_item = atomicAdd(a.work, 1u);
            __syncthreads();
            item = s_item;
            if (item >= n_items) break;
        } else if (it > 0) {
            break;
        }
        bwd_item<B, BD, NT, PPT, 1, 1>(a, item, 0, 0, threadIdx.x, sm);
    }
}

// Windows of few 16x16 tiles (bwd_split): the warps of a block of four take parts of tiles,
// each on its own.
constexpr int kPartWarps = 4, kPartMinBlocks = 5, kPartBatch = 32;   // a splat of a batch per lane
template <int S, int SEG>
__global__ void __launch_bounds__(32 * kPartWarps, kPartMinBlocks) k_render_bwd_parts(RasterBwdArgs a)
{
    pdl_begin();   // plain loads below: none moves ahead of the wait
    __shared__ BwdSmem<kPartBatch, 256 / S, 1> smem[kPartWarps];
    auto &sm = smem[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    zero_rows(sm.red, lane, 32);
    const uint32_t n_items = (uint32_t)(a.g.Tv * a.V) * (S * SEG);
    for (uint32_t it = 0;; it++) {
        uint32_t item = blockIdx.x * kPartWarps + (threadIdx.x >> 5);
        __syncwarp();   // the zero rows are written; the previous item's reads of the shared state are done
        if (a.work) {
            if (lane == 0) item = atomicAdd(a.work, 1u);
            item = __shfl_sync(kFull, item, 0);
        } else if (it > 0) {
            break;
        }
        if (item >= n_items) break;
        bwd_item<16, kPartBatch, 32, 8 / S, S, SEG>(a, item / (S * SEG), (int)(item / SEG % S), (int)(item % SEG), lane,
                                                    sm);
    }
}

// Parts of a tile and segments of its list.  With one of each the warp sums cover most pixels,
// which is best when the window has work for the whole GPU; a window of few tiles is bound by
// the walk of its longest list, one warp's chain of dependent steps, each shorter the fewer
// pixels the warp blends, and fewer with the list in segments.
// Measured together with the projection's backward (us; one, two and four parts,
// four parts in two and in four segments): 80 tiles 49, 34, 27, 23, 23; 300 tiles 67, 45, 37,
// 34, 36; 475 tiles 97, 68, 57, 49, 44; 1200 tiles 193, 146, 128, 105, 132; with longer lists
// 312, 233, 200, 194, 238; 1900 tiles 237, 194, 164, 193, 247; 2394 tiles 135, 111, 109, 131,
// 173; 3225 tiles 307, 276, 333; 3600 tiles 365, 275, 325; 5700 tiles 464, 521, 632; 9600 tiles
// 767, 833, 966.  Two parts in two segments: 158 at 1900 tiles, 106 at 2394, else slower.
// Splitting only the longest lists' tiles: 3225 tiles 314 to 395, 5700 tiles 493 to 602.
// The lines lie between measured sizes: 1200 and 1900 tiles, 2394 and 3225, 3600 and 5700.
struct BwdSplit {
    int parts, segments;
};
static BwdSplit bwd_split(int64_t tiles, int sms)
{
    if (tiles <= 8 * (int64_t)sms) return BwdSplit{4, 2};
    if (tiles <= 16 * (int64_t)sms) return BwdSplit{4, 1};
    return BwdSplit{tiles <= 32 * (int64_t)sms ? 2 : 1, 1};
}

int raster_bwd_batch(int64_t tiles, int B, int BD, int sms)
{
    return B == 16 && bwd_split(tiles, sms).parts > 1 ? kPartBatch : BD;
}

// Blocks of a persistent launch: as many as are resident on the GPU (queried once per device
// and kernel), at most `items` of them; clears the work counter.
template <class K>
static cudaError_t persistent_blocks(const RasterBwdArgs &a, K kernel, int threads, int (&resident)[64], int sms,
                                     int64_t &blocks, cudaStream_t s)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!resident[dev]) {
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0);
        if (e != cudaSuccess) return e;
        resident[dev] = max(1, per_sm) * max(1, sms);
    }
    blocks = min(blocks, (int64_t)resident[dev]);
    return clear_words(a.work, 1, s);
}

template <int B, int BD>
static cudaError_t launch_bwd(const RasterBwdArgs &a, int sms, cudaStream_t s)
{
    const int nt = B * B / ppt_for<B, kPPTBwd>();
    int64_t blocks = a.g.Tv * a.V;
    if (a.work) {
        static int resident[64] = {0};
        const cudaError_t e = persistent_blocks(a, k_render_bwd<B, BD>, nt, resident, sms, blocks, s);
        if (e != cudaSuccess) return e;
    }
    // Not a dependent launch: placed beside its predecessor's last blocks, a grid of few large
    // blocks lies unevenly on the SMs and the longest lists share one.  Forward to parameter
    // gradients, placed early and not (us): one 640x480 view of 46k in 32x32 tiles 488, 448
    // (184k: 773, 709); 800x600 of 72k 589, 562; eight of 46k in 16x16 tiles 679, 656; one in
    // 8x8 tiles 248, 222; four 1200x680 views of 122k 1244 both.
    if (blocks > 0) launch<false>(k_render_bwd<B, BD>, (unsigned)blocks, nt, 0, s, a);
    return cudaGetLastError();
}

template <int S, int SEG>
static cudaError_t launch_bwd_parts(const RasterBwdArgs &a, int sms, cudaStream_t s)
{
    int64_t blocks = (a.g.Tv * a.V * (S * SEG) + kPartWarps - 1) / kPartWarps;
    if (a.work) {
        static int resident[64] = {0};
        const cudaError_t e = persistent_blocks(a, k_render_bwd_parts<S, SEG>, 32 * kPartWarps, resident, sms, blocks, s);
        if (e != cudaSuccess) return e;
    }
    launch(k_render_bwd_parts<S, SEG>, (unsigned)blocks, 32 * kPartWarps, 0, s, a);
    return cudaGetLastError();
}

template <int B>
static cudaError_t launch_bwd_bd(const RasterBwdArgs &a, int BD, int sms, cudaStream_t s)
{
    if (B == 16) {
        const BwdSplit split = bwd_split(a.g.Tv * a.V, sms);
        if (split.parts == 4 && split.segments == 2) return launch_bwd_parts<4, 2>(a, sms, s);
        if (split.parts == 4) return launch_bwd_parts<4, 1>(a, sms, s);
        if (split.parts == 2) return launch_bwd_parts<2, 1>(a, sms, s);
    }
    switch (BD) {
    case 32: return launch_bwd<B, 32>(a, sms, s);
    case 64: return launch_bwd<B, 64>(a, sms, s);
    case 128: return launch_bwd<B, 128>(a, sms, s);
    default: return launch_bwd<B, 256>(a, sms, s);
    }
}

cudaError_t raster_bwd(const RasterBwdArgs &a, int B, int BD, int sms, cudaStream_t s)
{
    switch (B) {
    case 8: return launch_bwd_bd<8>(a, BD, sms, s);
    case 16: return launch_bwd_bd<16>(a, BD, sms, s);
    default: return launch_bwd_bd<32>(a, BD, sms, s);
    }
}

}  // namespace cgs
