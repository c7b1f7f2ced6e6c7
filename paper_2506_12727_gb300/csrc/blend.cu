// Tile-based alpha blending (Eq. 1) and its backward.
//
// In the supplement's rasterizer every (tile, view) pair gets its own thread
// block, and Alg. 2 has a tile's threads fetch its depth-sorted Gaussians
// into shared memory batch by batch and blend them.  Here the unit of work is a strip of
// a (tile, view) pair -- 8 columns (blend_strip_width) by (32 / 8) * PPT rows,
// strips side by side across wider tiles -- owned by one warp: each lane owns
// PPT pixels of one column, the warp stages batches
// of the tile's list in its own slice of shared memory, and leaves the strip
// as soon as all its pixels have stopped.  Warps of a persistent launch take
// strips from a queue that lists the tiles with the longest lists first, so
// the whole batch of views (any mix of resolutions) is one launch without a
// tail of heavy tiles, and no block-wide barrier couples unrelated strips.
//
// Each staged batch keeps only the Gaussians whose support and alpha >= 1/255
// region reach a pixel centre of the strip (an exact test of the quadratic
// form over the strip's rectangle), compacted with a ballot; the list
// positions are kept for the per-pixel bookkeeping.
//
// Forward per pixel (front to back): alpha = min(0.99, o G), skip alpha <
// 1/255, stop before T (1 - alpha) < 1e-4, C += c alpha T, T *= 1 - alpha;
// output C + T bg.  G is evaluated in base 2 from the staged coefficients
// and the column terms of the lane's pixel column (pair_eval).
//
// Backward per pixel (back to front from the last contributor), with T
// recovered by an (approximate) reciprocal:  dC/dc_i = alpha_i T_i,
// dC/dalpha_i = c_i T_i - S_i / (1 - alpha_i), S_i the colour blended behind
// i plus T_final bg.  The gradients of one Gaussian are summed over the
// lane's pixels (in a strip, as sums of dL/dpower times 1, dy, dy^2 for the
// lane's one column), then over the warp: the lanes' values of three Gaussians
// go through shared memory, where one lane per value adds up the 32 of them
// and adds the sum to the record with one atomic.
#include <map>
#include <mutex>
#include <type_traits>

#include "kernels.h"

namespace mvgs {
namespace {

constexpr unsigned kFull = 0xffffffffu;

constexpr int WARPS_PER_BLOCK = 4;

// One warp's work item: PPT pixels per lane of one (view, tile) pair -- a
// strip of the tile, or (sampled mode) a run of 32 * PPT of the tile's pixel
// samples.
template <int PPT>
struct Work {
    long long gt;               // global (view, tile) id, -1 when the queue is empty
    const DevCam* cam;
    float fx[PPT], fy[PPT];     // pixel centres (strips: one column, fx[k] all equal)
    int pix[PPT];               // pixel index in the view (y W + x); -1 for an idle slot
    float sx0, sx1, sy0, sy1;   // bounds of the warp's pixel centres
};

__device__ __forceinline__ int take_item(int* counter, int lane) {
    int item = 0;
    if (lane == 0) item = atomicAdd(counter, 1);
    return __shfl_sync(kFull, item, 0);
}

__device__ __forceinline__ const DevCam* view_of(const BlendArgs& a, long long gt, int lane) {
    int v = 0;
    if (lane == 0) v = find_view(a.cams, a.V, gt);
    v = __shfl_sync(kFull, v, 0);
    return &a.cams[v];
}

// Next strip for the warp.  With a pixel mask (the naive partial rendering
// of Fig. 3b) masked pixels are idle slots of their lanes.
template <int PPT>
__device__ __forceinline__ bool next_strip(const BlendArgs& a, int* counter, int lane, Work<PPT>& w) {
    const int item = take_item(counter, lane);
    if ((long long)item >= a.tiles * a.strips) return false;
    w.gt = (long long)a.order[item / a.strips];
    const int strip = item % a.strips;
    w.cam = view_of(a, w.gt, lane);
    const DevCam& cam = *w.cam;
    const long long local = w.gt - cam.tile_base;
    const int tx = (int)(local % cam.tiles_x), ty = (int)(local / cam.tiles_x);
    const int across = a.tw / a.sw;  // strips side by side in a tile
    const int step = 32 / a.sw;      // thread rows of the warp
    const int x0 = tx * a.tw + (strip % across) * a.sw, y0 = ty * a.th + (strip / across) * a.strip_h;
    const int px = x0 + lane % a.sw;
    const int py0 = y0 + lane / a.sw;
#pragma unroll
    for (int k = 0; k < PPT; k++) {
        const int py = py0 + k * step;
        w.fx[k] = px + 0.5f;
        w.fy[k] = py + 0.5f;
        int p = -1;
        if (px < cam.W && py < cam.H) {
            p = py * cam.W + px;
            if (a.pixel_mask && !a.pixel_mask[cam.pix_base + p]) p = -1;
        }
        w.pix[k] = p;
    }
    w.sx0 = x0 + 0.5f;
    w.sx1 = (float)min(x0 + a.sw, cam.W) - 0.5f;
    w.sy0 = y0 + 0.5f;
    w.sy1 = (float)min(y0 + a.strip_h, cam.H) - 0.5f;
    return true;
}

// Next run of pixel samples (Alg. 3): lanes take consecutive samples of the
// tile's list, so every lane of the warp has a pixel to blend except in the
// tile's last run.  Runs whose samples are all invalid are skipped.
template <int PPT>
__device__ __forceinline__ bool next_samples(const BlendArgs& a, int* counter, int lane, long long total,
                                             Work<PPT>& w) {
    for (;;) {
        const int item = take_item(counter, lane);
        if ((long long)item >= total) return false;
        const int i = a.chunk_map[item];
        w.gt = (long long)a.order[i];
        const long long chunk = (long long)item - a.chunk_off[i];
        w.cam = view_of(a, w.gt, lane);
        const DevCam& cam = *w.cam;
        const long long local = w.gt - cam.tile_base;
        const int tx = (int)(local % cam.tiles_x), ty = (int)(local / cam.tiles_x);
        const long long s0 = a.s_off[w.gt] + chunk * 32 * PPT, s1 = a.s_off[w.gt + 1];
        int xmin = 0x7fffffff, ymin = 0x7fffffff, xmax = -1, ymax = -1;
#pragma unroll
        for (int k = 0; k < PPT; k++) {
            const long long si = s0 + k * 32 + lane;
            int p = -1, px = 0, py = 0;
            if (si < s1) {
                const int li = a.s_pix[si];
                const int lx = li % a.tw, ly = li / a.tw;
                px = tx * a.tw + lx;
                py = ty * a.th + ly;
                if (ly < a.th && px < cam.W && py < cam.H) {
                    p = py * cam.W + px;
                    xmin = min(xmin, px);
                    xmax = max(xmax, px);
                    ymin = min(ymin, py);
                    ymax = max(ymax, py);
                }
            }
            w.fx[k] = px + 0.5f;
            w.fy[k] = py + 0.5f;
            w.pix[k] = p;
        }
        xmax = __reduce_max_sync(kFull, xmax);
        if (xmax < 0) continue;  // no valid sample in this run
        xmin = __reduce_min_sync(kFull, xmin);
        ymin = __reduce_min_sync(kFull, ymin);
        ymax = __reduce_max_sync(kFull, ymax);
        w.sx0 = xmin + 0.5f;
        w.sx1 = xmax + 0.5f;
        w.sy0 = ymin + 0.5f;
        w.sy1 = ymax + 0.5f;
        return true;
    }
}

template <int PPT, bool SAMPLED>
__device__ __forceinline__ bool next_work(const BlendArgs& a, int* counter, int lane, long long total,
                                          Work<PPT>& w) {
    if constexpr (SAMPLED) return next_samples<PPT>(a, counter, lane, total, w);
    else return next_strip<PPT>(a, counter, lane, w);
}

// A Gaussian staged by the forward: the values of the per-pixel arithmetic
// twice each, as operands of the packed instructions.
struct alignas(16) FwdEntry {
    float4 m;     // -mx, -mx, -my, -my
    float4 qab;   // qa, qa, qb, qb
    float4 qco;   // qc, qc, -o, -o
    float4 rg;    // -r, -r, -g, -g
    float4 brp;   // -b, -b, radius, list position (bit 31: pixel by pixel)
};
static_assert(sizeof(FwdEntry) == 80, "five 16-byte reads");
constexpr uint32_t kByPixel = 0x80000000u;  // a list has fewer than 2^31 entries, one per record at most

// The forward looks at FWD_SCAN list entries at a time until more than FWD_FLUSH
// of them reach the work item (or the list ends), then blends those: where few
// do, the scan goes on at the pace of its own loads.  The staging takes 30 KB
// per block; with 40 KB the L1 cache that is left thrashes under the fetches.
constexpr int FWD_SCAN = 64, FWD_FLUSH = 32, FWD_STAGE = FWD_SCAN + FWD_FLUSH;

// Resident blocks per SM the forward is compiled for: four (at most 128
// registers) for 4 pixels per lane without the depth and statistics outputs.
// More warps fetch more records at once than the L1 cache holds (five blocks:
// 3M Gaussians x 8 views 3.13 -> 3.44 ms, 500k x 4 0.62 -> 0.73), fewer leave
// latency open (three: 3.6 ms).  No bound elsewhere: more state there.
constexpr int fwd_min_blocks(int ppt, bool extra) { return ppt == 4 && !extra ? 4 : 1; }

// DEPTH: also the expected depth per pixel; STATS: also the per-pixel
// statistics (list position where the pixel stopped, Gaussians blended).
//
// Bound by instruction issue where most staged Gaussians are blended, by the L2
// sectors of the scanned list entries where few are.  So a lane's pixels are
// taken two at a time with packed float32 arithmetic and without branches: a
// pixel that the Gaussian does not reach blends it with alpha 0, which leaves T
// and C as they are, bit for bit; a stopped pixel's threshold is raised out of
// reach; the rare stop is found with one vote per Gaussian.  Gaussians for which
// that could differ (not ordinary_gaussian) take the pixels one by one.  Batches
// with a Gaussian that the clamp at 0.99 or a rounded exponent above 0 may touch
// (not plain, make_geom) take a variant of the step with those two tests, two
// instructions more per pixel: 500k x 4 views with 0, 10, 40, 100% of the
// opacities above 0.993 618, 708, 652, 607 us, where taking those Gaussians pixel
// by pixel cost 618, 740, 777, 879.  Warp instructions per staged Gaussian (128 pixels) 109 -> 75, per 32
// list entries scanned 193 -> 110, L2 sectors per entry 3.1 -> 1.4 (Geom).
// 3M Gaussians x 8 views at 32 x 64 tiles (2.1e9 blended pairs) 5.46 -> 3.13 ms,
// 1M x 16 views at 16 x 64 3.59 -> 2.60, 500k x 4 views 0.94 -> 0.62, 2M x 5
// views 2.34 -> 1.28, 500k x 1 view at 16 x 16 0.33 -> 0.21.
template <int PPT, bool SAMPLED, bool DEPTH, bool STATS>
__global__ void __launch_bounds__(32 * WARPS_PER_BLOCK, fwd_min_blocks(PPT, DEPTH || STATS))
    blend_forward_kernel(BlendArgs a, int* __restrict__ counter, float* __restrict__ img,
                         float* __restrict__ final_T, uint32_t* __restrict__ n_contrib,
                         uint2* __restrict__ pixel_stats) {
    __shared__ FwdEntry s_ent[WARPS_PER_BLOCK][FWD_STAGE];
    __shared__ uint32_t s_rid[WARPS_PER_BLOCK][FWD_STAGE];
    __shared__ float s_dep[WARPS_PER_BLOCK][DEPTH ? FWD_STAGE : 1];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    FwdEntry* ent = s_ent[w];
    uint32_t* wrid = s_rid[w];
    float* wdep = s_dep[w];
    constexpr float kStopped = 2.f;  // no alpha reaches it
    constexpr int NP = (PPT + 1) / 2, NK = 2 * NP;  // pairs, pixel slots (one idle slot with 1 pixel per lane)
    float one1, one2;  // kept in registers (a constant would be moved there at every use)
    asm volatile("mov.f32 %0, %1;" : "=f"(one1) : "f"(1.f));
    asm volatile("mov.f32 %0, %1;" : "=f"(one2) : "f"(1.f));
    const f32x2 one = pack2(one1, one2);
    const long long total = SAMPLED ? min(a.chunk_off[a.tiles], a.chunk_cap) : 0;
    Work<PPT> st;
    while (next_work<PPT, SAMPLED>(a, counter, lane, total, st)) {
        const DevCam& cam = *st.cam;
        const long long start = a.ranges[2 * st.gt], end = a.ranges[2 * st.gt + 1];
        f32x2 T[NP], C0[NP], C1[NP], C2[NP], D[NP], FX[SAMPLED ? NP : 1], FY[NP];
        float nmin[NK];  // minus the least alpha that blends; -kStopped once the pixel has stopped
        uint32_t last[NK], stop[NK], nblend[NK];
#pragma unroll
        for (int p = 0; p < NP; p++) {
            const int k = 2 * p, l = k + 1 < PPT ? k + 1 : k;
            T[p] = pack2(1.f, 1.f);
            C0[p] = C1[p] = C2[p] = D[p] = pack2(0.f, 0.f);
            if (SAMPLED || p == 0) FX[SAMPLED ? p : 0] = pack2(st.fx[k], st.fx[l]);
            FY[p] = pack2(st.fy[k], st.fy[l]);
        }
#pragma unroll
        for (int k = 0; k < NK; k++) {
            last[k] = 0;
            stop[k] = (uint32_t)(end - start);  // list position where the pixel stopped
            nblend[k] = 0;
            nmin[k] = k >= PPT || st.pix[k < PPT ? k : 0] < 0 ? -kStopped : -kAlphaMin;
        }
        auto all_stopped = [&]() {
            bool d = true;
#pragma unroll
            for (int k = 0; k < NK; k++) d = d && nmin[k] == -kStopped;
            return d;
        };
        const uint32_t len = (uint32_t)(end - start);  // one entry per record at most: below 2^31
        const uint32_t* list = a.sorted + start;
        // one ordinary Gaussian on all pixels, with the tests of pair_eval that a
        // plain one does without (TESTS); true when the warp's last pixel has
        // stopped (votes keep the warp together)
        auto packed_step = [&](auto tests, const FwdEntry& e, float dep) {
            constexpr bool TESTS = decltype(tests)::value;
            const float4 em = e.m, eq = e.qab, eo = e.qco, ec = e.rg, eb = e.brp;
            const uint32_t pos1 = __float_as_uint(eb.w) + 1;
            const float radius = eb.z;
            const f32x2 nmx = pack2(em.x, em.y), nmy = pack2(em.z, em.w), qa = pack2(eq.x, eq.y),
                        qb = pack2(eq.z, eq.w), qc = pack2(eo.x, eo.y), no = pack2(eo.z, eo.w);
            f32x2 xx{}, x{}, na[NP], om[NP];  // na: minus alpha, om: 1 - alpha
            bool in0 = true, in1 = true, ok[NK];
            float tmin;
#pragma unroll
            for (int p = 0; p < NP; p++) {
                const int k = 2 * p, l = 2 * p + 1;
                if (SAMPLED || p == 0) {
                    const f32x2 dx = add2(FX[SAMPLED ? p : 0], nmx);
                    xx = mul2(mul2(qa, dx), dx);
                    x = mul2(qb, dx);
                    float dx0, dx1;
                    unpack2(dx, dx0, dx1);
                    in0 = fabsf(dx0) <= radius;
                    in1 = SAMPLED ? fabsf(dx1) <= radius : in0;
                }
                const f32x2 dy = add2(FY[p], nmy);
                float dy0, dy1, e0, e1, v0, v1, t0, t1;
                unpack2(dy, dy0, dy1);
                unpack2(fma2(dy, fma2(qc, dy, x), xx), e0, e1);
                unpack2(mul2(no, pack2(ex2_approx(e0), ex2_approx(e1))), v0, v1);
                if (TESTS) {
                    v0 = fmaxf(v0, -kAlphaMax);
                    v1 = fmaxf(v1, -kAlphaMax);
                }
                ok[k] = in0 & (fabsf(dy0) <= radius) & (v0 <= nmin[k]) & (!TESTS || e0 <= 0.f);
                ok[l] = in1 & (fabsf(dy1) <= radius) & (v1 <= nmin[l]) & (!TESTS || e1 <= 0.f);
                na[p] = pack2(ok[k] ? v0 : 0.f, ok[l] ? v1 : 0.f);
                om[p] = add2(na[p], one);
                unpack2(mul2(T[p], om[p]), t0, t1);
                tmin = p == 0 ? fminf(t0, t1) : fminf(tmin, fminf(t0, t1));
            }
            const f32x2 r2 = pack2(ec.x, ec.y), g2 = pack2(ec.z, ec.w), b2 = pack2(eb.x, eb.y);
            auto add_colour = [&](int p, f32x2 nal) {
                const f32x2 nw = mul2(nal, T[p]);  // minus the weight, times minus the colour
                C0[p] = fma2(r2, nw, C0[p]);
                C1[p] = fma2(g2, nw, C1[p]);
                C2[p] = fma2(b2, nw, C2[p]);
                if (DEPTH) D[p] = fma2(pack2(-dep, -dep), nw, D[p]);
            };
            if (!__any_sync(kFull, tmin < kTMin)) {
#pragma unroll
                for (int p = 0; p < NP; p++) {
                    add_colour(p, na[p]);
                    T[p] = mul2_fresh(T[p], om[p]);
                }
#pragma unroll
                for (int k = 0; k < NK; k++) {
                    last[k] = ok[k] ? pos1 : last[k];
                    if (STATS) nblend[k] += ok[k];
                }
                return false;
            }
            // some pixel of the warp stops here: its alpha becomes 0
#pragma unroll
            for (int p = 0; p < NP; p++) {
                float t[2], al[2];
                unpack2(mul2(T[p], om[p]), t[0], t[1]);
                unpack2(na[p], al[0], al[1]);
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const int k = 2 * p + h;
                    if (t[h] < kTMin) {
                        al[h] = 0.f;
                        nmin[k] = -kStopped;
                        if (STATS) stop[k] = pos1;
                    }
                    if (al[h] < 0.f) {
                        last[k] = pos1;
                        if (STATS) nblend[k]++;
                    }
                }
                const f32x2 nal = pack2(al[0], al[1]);
                add_colour(p, nal);
                T[p] = mul2(T[p], add2(nal, one));
            }
            return (bool)__all_sync(kFull, all_stopped());
        };
        // any Gaussian, pixel by pixel
        auto general_step = [&](const FwdEntry& e, float dep) {
            const float4 em = e.m, eq = e.qab, eo = e.qco, ec = e.rg, eb = e.brp;
            const float radius = eb.z;
            const float4 q = make_float4(eq.x, eq.z, eo.x, -eo.z);
            const uint32_t pos1 = (__float_as_uint(eb.w) & ~kByPixel) + 1;
            auto blend_one = [&](int k, float fx, float fy, float& Tk, float& c0, float& c1, float& c2, float& d) {
                if (nmin[k] == -kStopped) return;
                const float dx = fx + em.x;
                float alpha, G;
                if (!pair_eval(dx, fy + em.z, col_terms(dx, q), q, radius, alpha, G)) return;
                const float Tn = __fmul_rn(Tk, __fsub_rn(1.f, alpha));
                if (Tn < kTMin) {
                    nmin[k] = -kStopped;
                    if (STATS) stop[k] = pos1;
                    return;
                }
                const float wgt = __fmul_rn(alpha, Tk);
                c0 = __fmaf_rn(-ec.x, wgt, c0);
                c1 = __fmaf_rn(-ec.z, wgt, c1);
                c2 = __fmaf_rn(-eb.x, wgt, c2);
                if (DEPTH) d = __fmaf_rn(dep, wgt, d);
                Tk = Tn;
                last[k] = pos1;
                if (STATS) nblend[k]++;
            };
#pragma unroll
            for (int p = 0; p < NP; p++) {
                float u[5][2], f0, f1, y0, y1;
                unpack2(T[p], u[0][0], u[0][1]);
                unpack2(C0[p], u[1][0], u[1][1]);
                unpack2(C1[p], u[2][0], u[2][1]);
                unpack2(C2[p], u[3][0], u[3][1]);
                unpack2(D[p], u[4][0], u[4][1]);
                unpack2(FX[SAMPLED ? p : 0], f0, f1);
                unpack2(FY[p], y0, y1);
                blend_one(2 * p, f0, y0, u[0][0], u[1][0], u[2][0], u[3][0], u[4][0]);
                blend_one(2 * p + 1, f1, y1, u[0][1], u[1][1], u[2][1], u[3][1], u[4][1]);
                T[p] = pack2(u[0][0], u[0][1]);
                C0[p] = pack2(u[1][0], u[1][1]);
                C1[p] = pack2(u[2][0], u[2][1]);
                C2[p] = pack2(u[3][0], u[3][1]);
                if (DEPTH) D[p] = pack2(u[4][0], u[4][1]);
            }
            return (bool)__all_sync(kFull, all_stopped());
        };
        // the next batch's geometry (and the ids of the one after it) is fetched
        // while the present one is blended
        uint32_t rec[2], nid[2];
        Geom g[2];
        auto fetch_ids = [&](uint32_t b) {
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const uint32_t i = b + 32 * h + lane;
                nid[h] = i < len ? list[i] : 0u;
            }
        };
        auto fetch_geometry = [&](uint32_t b) {
#pragma unroll
            for (int h = 0; h < 2; h++) {
                rec[h] = nid[h];
                if (b + 32 * h + lane < len) g[h] = load_geom(a.geom + rec[h]);
            }
        };
        fetch_ids(0);
        fetch_geometry(0);
        fetch_ids(FWD_SCAN);
        for (uint32_t b = 0; b < len;) {
            if (__all_sync(kFull, all_stopped())) break;
            // stage the Gaussians that can reach a pixel of the work item
            __syncwarp();
            int n = 0;
            bool odd = false, tests = false;
            do {
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const bool hit = b + 32 * h + lane < len && rect_reaches(st.sx0, st.sx1, st.sy0, st.sy1, g[h]);
                    const uint32_t bal = __ballot_sync(kFull, hit);
                    if (hit) {
                        const int slot = n + __popc(bal & lt);
                        const bool ordinary = g[h].radius >= 0.f;
                        odd |= !ordinary;
                        tests |= g[h].o < 0.f;
                        const float no = -fabsf(g[h].o);
                        ent[slot].m = make_float4(-g[h].mx, -g[h].mx, -g[h].my, -g[h].my);
                        ent[slot].qab = make_float4(g[h].qa, g[h].qa, g[h].qb, g[h].qb);
                        ent[slot].qco = make_float4(g[h].qc, g[h].qc, no, no);
                        ent[slot].brp.w = __uint_as_float((b + 32 * h + lane) | (ordinary ? 0u : kByPixel));
                        wrid[slot] = rec[h];
                    }
                    n += __popc(bal);
                }
                b += FWD_SCAN;
                if (b < len) {
                    fetch_geometry(b);
                    fetch_ids(b + FWD_SCAN);
                }
            } while (n <= FWD_FLUSH && b < len);
            __syncwarp();
            // their colours, each lane's entries (at most three) in flight together
            float4 cr[(FWD_STAGE + 31) / 32];
#pragma unroll
            for (int i = 0; i < (FWD_STAGE + 31) / 32; i++)
                if (32 * i + lane < n) cr[i] = a.rgb_r[wrid[32 * i + lane]];
#pragma unroll
            for (int i = 0; i < (FWD_STAGE + 31) / 32; i++) {
                const int e = 32 * i + lane;
                if (e < n) {
                    ent[e].rg = make_float4(-cr[i].x, -cr[i].x, -cr[i].y, -cr[i].y);
                    *reinterpret_cast<float2*>(&ent[e].brp) = make_float2(-cr[i].z, -cr[i].z);
                    ent[e].brp.z = cr[i].w;
                    if (DEPTH) wdep[e] = a.rec_depth[wrid[e]];
                }
            }
            __syncwarp();
            odd = __any_sync(kFull, odd);
            if (!odd && !__any_sync(kFull, tests)) {
                for (int j = 0; j < n; j++)
                    if (packed_step(std::false_type(), ent[j], DEPTH ? wdep[j] : 0.f)) break;
            } else {
                for (int j = 0; j < n; j++) {
                    const float dep = DEPTH ? wdep[j] : 0.f;
                    if (odd && __any_sync(kFull, __float_as_uint(ent[j].brp.w) >= kByPixel)
                            ? general_step(ent[j], dep)
                            : packed_step(std::true_type(), ent[j], dep))
                        break;
                }
            }
        }
        const long long HW = (long long)cam.W * cam.H;
        float* out = img + 3 * cam.pix_base;
#pragma unroll
        for (int k = 0; k < PPT; k++) {
            const long long p = st.pix[k];
            if (p >= 0) {
                auto half = [k](f32x2 v) {
                    float lo, hi;
                    unpack2(v, lo, hi);
                    return k & 1 ? hi : lo;
                };
                const float t = half(T[k / 2]);
                out[p] = __fmaf_rn(t, a.bg[0], half(C0[k / 2]));
                out[HW + p] = __fmaf_rn(t, a.bg[1], half(C1[k / 2]));
                out[2 * HW + p] = __fmaf_rn(t, a.bg[2], half(C2[k / 2]));
                final_T[cam.pix_base + p] = t;
                n_contrib[cam.pix_base + p] = last[k];
                if (STATS) pixel_stats[cam.pix_base + p] = make_uint2(stop[k], nblend[k]);
                if (DEPTH) a.depth_out[cam.pix_base + p] = half(D[k / 2]);
            }
        }
    }
}

// The backward's staging: list entries looked at together, staged entries that
// end a scan, and Gaussians whose lane sums are added up together (three: ten
// values each take 30 lanes).
constexpr int BWD_GROUP = 3;
constexpr int BWD_SCAN = 64, BWD_FLUSH = 16, BWD_STAGE = (BWD_SCAN + BWD_FLUSH + BWD_GROUP - 1) / BWD_GROUP * BWD_GROUP;

// A Gaussian staged by the backward (operands of the packed instructions twice).
struct alignas(16) BwdEntry {
    float4 m;     // -mx, -mx, -my, -my
    float4 qab;   // qa, qa, qb, qb
    float4 qco;   // qc, qc, -o, -o
    float4 rg;    // r, r, g, g
    float4 brp;   // b, b, radius, list position (bit 31: pixel by pixel)
};

// The lane sums of a group of Gaussians: ten rows of 32 lanes each, added up by
// one lane per row.  Rows are 136 bytes apart, so that the 16 lanes of an
// 8-byte read hit different banks.
struct BwdSums {
    static constexpr int ROW = 34;  // floats
    float v[32 * ROW];
};

// Resident blocks per SM the backward is compiled for: four (at most 128
// registers; three: 3M Gaussians x 8 views 6.39 -> 6.88 ms, five spill: 6.86).
constexpr int bwd_min_blocks(int ppt) { return ppt == 4 ? 4 : 1; }

// Bound by instruction issue and the FMA pipe (two thirds of the issue slots,
// half of the pipe's cycles, 16 warps per SM).  As in the forward, pixels are
// taken two at a time with packed arithmetic and without branches: a pixel that
// the Gaussian does not reach takes part with alpha 0, which leaves T and the
// sums as they are.  That needs finite factors: strips with an image gradient
// that is not of ordinary size, and Gaussians that are not ordinary, take the
// pixels one by one.  Batches with one that is not plain take the variant with
// the two tests, four instructions more per pixel: 500k x 4 views with 0, 10, 40,
// 100% of the opacities above 0.993 1308, 1376, 1267, 1160 us, where pixel by
// pixel they cost 1341, 1397, 1440, 1383.
// The steps of a group of three Gaussians follow each
// other without a branch, so one's latency hides behind the next.  A warp's
// sums go through shared memory (ten stores a lane, 16 reads by one lane
// per value: half the instructions of a shuffle reduction with its selects).  Every sum is
// taken in a fixed order -- a lane's pixels one after the other, then lanes 16,
// 8, 4, 2, 1 apart: the conic gradients of long thin Gaussians cancel to a small
// rest, and their error is the order's.
// With LOOK a group's alphas come first, and a group that no pixel blends is
// passed over (launch_blend_backward says where that pays).
// Warp instructions per staged Gaussian (128 pixels) 240 -> 180.  3M Gaussians x
// 8 views at 32 x 64 tiles 8.44 -> 6.35 ms, 1M x 16 views at 16 x 64 7.70 ->
// 5.36, 500k x 4 views 1.74 -> 1.31, the sampled pixels of 500k x 4 at 16 x 16
// 1.21 -> 1.02, 10k at 128 x 128 0.224 -> 0.123.
template <int PPT, bool SAMPLED, bool LOOK>
__global__ void __launch_bounds__(32 * WARPS_PER_BLOCK, bwd_min_blocks(PPT))
    blend_backward_kernel(BlendArgs a, int* __restrict__ counter, const float* __restrict__ dimg,
                          const float* __restrict__ final_T, const uint32_t* __restrict__ n_contrib,
                          float* __restrict__ rec_grad, double* __restrict__ rec_conic) {
    __shared__ BwdEntry s_ent[WARPS_PER_BLOCK][BWD_STAGE];
    __shared__ uint32_t s_rid[WARPS_PER_BLOCK][BWD_STAGE];
    __shared__ __align__(16) BwdSums s_sum[WARPS_PER_BLOCK];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    BwdEntry* ent = s_ent[w];
    uint32_t* wrid = s_rid[w];
    BwdSums& sums = s_sum[w];
    constexpr int NP = (PPT + 1) / 2, NK = 2 * NP;  // pairs, pixel slots (one idle slot with 1 pixel per lane)
    constexpr float LN2 = 0.6931471805599453f;
    float one1, one2;  // kept in registers (a constant would be moved there at every use)
    asm volatile("mov.f32 %0, %1;" : "=f"(one1) : "f"(1.f));
    asm volatile("mov.f32 %0, %1;" : "=f"(one2) : "f"(1.f));
    const f32x2 one = pack2(one1, one2);
    // the row this lane adds up: Gaussian of the group, value, and what the sum
    // is multiplied with
    const int my_group = lane / 10, my_val = lane % 10;
    const float my_factor = my_val < 6 ? -1.f : my_val == 6 ? LN2 : my_val == 8 ? 1.f : 0.5f;

    // adds the sums of the k Gaussians from entry j on to their records (lanes
    // l and l + 16 first, then 8, 4, 2 and 1 apart)
    auto add_sums = [&](int j, int k) {
        __syncwarp();
        const float2* row = reinterpret_cast<const float2*>(sums.v + lane * BwdSums::ROW);
        f32x2 t[8];
#pragma unroll
        for (int i = 0; i < 8; i++) t[i] = add2(row[i], row[i + 8]);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1)
#pragma unroll
            for (int i = 0; i < o; i++) t[i] = add2(t[i], t[i + o]);
        const float sum = t[0].x + t[0].y;
        const float other = __shfl_xor_sync(kFull, sum, 1);
        float out = my_factor * sum;
        // a Gaussian that no pixel of the strip blends has sums of 0: not added (the
        // atomics of 20k Gaussians in three small views 546 -> 534 us, with all
        // opaque 618 -> 576; the position takes both its sums, so it always is)
        if (my_group < k && (my_val < 2 || sum != 0.f)) {
            const BwdEntry& e = ent[j + my_group];
            const uint32_t r = wrid[j + my_group];
            // dL/d mean = sum dL/dpower (A dx + B dy, B dx + C dy), in base-2 coefficients
            if (my_val < 2)
                out = LN2 * fmaf(2.f * (my_val == 0 ? e.qab.x : e.qco.x), sum, e.qab.z * other);
            // the conic gradients sum terms weighted by dx^2 ~ 1e4 px^2 of both
            // signs: they are added across warps in double precision
            if (my_val < 7) atomicAdd(rec_grad + (size_t)kGradStride * r + my_val, out);
            else atomicAdd(rec_conic + (size_t)3 * r + (my_val - 7), (double)out);
        }
        __syncwarp();
    };

    const long long total = SAMPLED ? min(a.chunk_off[a.tiles], a.chunk_cap) : 0;
    Work<PPT> st;
    while (next_work<PPT, SAMPLED>(a, counter, lane, total, st)) {
        const DevCam& cam = *st.cam;
        const long long HW = (long long)cam.W * cam.H;
        const float* din = dimg + 3 * cam.pix_base;
        // per pixel: T in front of the current Gaussian, dL/dC, and V = minus
        // dL/dC . (colour blended behind the current Gaussian + T_final bg)
        f32x2 T[NP], d0[NP], d1[NP], d2[NP], V[NP], FX[SAMPLED ? NP : 1], FY[NP];
        uint32_t last[NK];
        uint32_t mylast = 0;
        bool odd_pixels = false;
        {
            float t[NK], e0[NK], e1[NK], e2[NK], u[NK];
#pragma unroll
            for (int k = 0; k < NK; k++) {
                t[k] = 1.f;
                e0[k] = e1[k] = e2[k] = 0.f;
                last[k] = 0;
                const long long p = k < PPT ? st.pix[k < PPT ? k : 0] : -1;
                if (p >= 0) {
                    e0[k] = din[p];
                    e1[k] = din[HW + p];
                    e2[k] = din[2 * HW + p];
                    t[k] = final_T[cam.pix_base + p];
                    last[k] = n_contrib[cam.pix_base + p];
                }
                u[k] = -t[k] * (e0[k] * a.bg[0] + e1[k] * a.bg[1] + e2[k] * a.bg[2]);
                mylast = last[k] > mylast ? last[k] : mylast;
                // gradients a Gaussian of weight 0 may be multiplied with
                odd_pixels |= !(fabsf(e0[k]) + fabsf(e1[k]) + fabsf(e2[k]) <= 1e25f && fabsf(u[k]) <= 1e35f);
            }
#pragma unroll
            for (int p = 0; p < NP; p++) {
                const int k = 2 * p, l = 2 * p + 1;
                T[p] = pack2(t[k], t[l]);
                d0[p] = pack2(e0[k], e0[l]);
                d1[p] = pack2(e1[k], e1[l]);
                d2[p] = pack2(e2[k], e2[l]);
                V[p] = pack2(u[k], u[l]);
                if (SAMPLED || p == 0) FX[SAMPLED ? p : 0] = pack2(st.fx[k], st.fx[l < PPT ? l : k]);
                FY[p] = pack2(st.fy[k], st.fy[l < PPT ? l : k]);
            }
        }
        odd_pixels = __any_sync(kFull, odd_pixels);
        const uint32_t len = __reduce_max_sync(kFull, mylast);
        const uint32_t* list = a.sorted + a.ranges[2 * st.gt];
        // back to front: entry i of the walk is list position len - 1 - i
        uint32_t rec[2], nid[2];
        Geom g[2];
        auto fetch_ids = [&](uint32_t b) {
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const uint32_t i = b + 32 * h + lane;
                nid[h] = i < len ? list[len - 1 - i] : 0u;
            }
        };
        auto fetch_geometry = [&](uint32_t b) {
#pragma unroll
            for (int h = 0; h < 2; h++) {
                rec[h] = nid[h];
                if (b + 32 * h + lane < len) g[h] = load_geom(a.geom + rec[h]);
            }
        };
        auto hand_over = [&](int u, float v0, float v1, float v2, float v3, float v4, float v5, float v6, float v7,
                             float v8, float v9) {
            const float v[10] = {v0, v1, v2, v3, v4, v5, v6, v7, v8, v9};
#pragma unroll
            for (int i = 0; i < 10; i++) sums.v[(10 * u + i) * BwdSums::ROW + lane] = v[i];
        };
        // Minus one Gaussian's alpha at all pixels, 0 where it takes no part; with the
        // tests of pair_eval that a plain one does without (TESTS).
        auto packed_alpha = [&](auto tests, const BwdEntry& e, f32x2* na) {
            constexpr bool TESTS = decltype(tests)::value;
            const float4 em = e.m, eq = e.qab, eo = e.qco, eb = e.brp;
            const uint32_t tag = __float_as_uint(eb.w);
            const float radius = eb.z;
            const f32x2 nmx = pack2(em.x, em.y), nmy = pack2(em.z, em.w), qa = pack2(eq.x, eq.y),
                        qb = pack2(eq.z, eq.w), qc = pack2(eo.x, eo.y), no = pack2(eo.z, eo.w);
            f32x2 xx{}, x{};
            bool in0 = true, in1 = true;
#pragma unroll
            for (int p = 0; p < NP; p++) {
                const int k = 2 * p, l = 2 * p + 1;
                if (SAMPLED || p == 0) {
                    const f32x2 dx = add2(FX[SAMPLED ? p : 0], nmx);
                    xx = mul2(mul2(qa, dx), dx);
                    x = mul2(qb, dx);
                    float dx0, dx1;
                    unpack2(dx, dx0, dx1);
                    in0 = fabsf(dx0) <= radius;
                    in1 = SAMPLED ? fabsf(dx1) <= radius : in0;
                }
                const f32x2 dy = add2(FY[p], nmy);
                float dy0, dy1, e0, e1, v0, v1;
                unpack2(dy, dy0, dy1);
                unpack2(fma2(dy, fma2(qc, dy, x), xx), e0, e1);
                unpack2(mul2(no, pack2(ex2_approx(e0), ex2_approx(e1))), v0, v1);
                if (TESTS) {
                    v0 = fmaxf(v0, -kAlphaMax);
                    v1 = fmaxf(v1, -kAlphaMax);
                }
                const bool ok0 = in0 & (fabsf(dy0) <= radius) & (v0 <= -kAlphaMin) & (tag < last[k]) & (!TESTS || e0 <= 0.f);
                const bool ok1 = in1 & (fabsf(dy1) <= radius) & (v1 <= -kAlphaMin) & (tag < last[l]) & (!TESTS || e1 <= 0.f);
                na[p] = pack2(ok0 ? v0 : 0.f, ok1 ? v1 : 0.f);
            }
        };
        // One Gaussian with these on all pixels: the lane's sums over its pixels -- minus
        // dL/dpower times 1, dy, dy^2, dx, dx^2 and dx dy, minus the colour
        // gradients, the E_1 term -- into place u of the group.
        auto packed_step = [&](auto tests, const BwdEntry& e, int u, const f32x2* na) {
            constexpr bool TESTS = decltype(tests)::value;
            const float4 em = e.m, eq = e.qab, eo = e.qco, ec = e.rg, eb = e.brp;
            const f32x2 nmx = pack2(em.x, em.y), nmy = pack2(em.z, em.w), qa = pack2(eq.x, eq.y),
                        qb = pack2(eq.z, eq.w), qc = pack2(eo.x, eo.y), r2 = pack2(ec.x, ec.y),
                        g2 = pack2(ec.z, ec.w), b2 = pack2(eb.x, eb.y);
            const f32x2 qc2 = add2(qc, qc);
            f32x2 dx{}, t2{}, x{}, sr{}, sg{}, sb{};
            float P0 = 0.f, P1 = 0.f, P2 = 0.f, Sx = 0.f, Sxx = 0.f, Sxy = 0.f;
            float E = 0.f;
#pragma unroll
            for (int p = 0; p < NP; p++) {
                if (SAMPLED || p == 0) {
                    dx = add2(FX[SAMPLED ? p : 0], nmx);
                    const f32x2 t = mul2(qa, dx);
                    t2 = add2(t, t);
                    x = mul2(qb, dx);
                }
                const f32x2 dy = add2(FY[p], nmy);
                float dy0, dy1, o0, o1;
                unpack2(dy, dy0, dy1);
                unpack2(add2(na[p], one), o0, o1);
                const f32x2 inv = pack2(rcp_approx(o0), rcp_approx(o1));
                T[p] = mul2(T[p], inv);  // transmittance in front of this Gaussian
                const f32x2 nw = mul2(na[p], T[p]);
                const f32x2 dc = fma2(d2[p], b2, fma2(d0[p], r2, mul2(d1[p], g2)));
                const f32x2 da = fma2(T[p], dc, mul2(V[p], inv));  // dL/dalpha
                V[p] = fma2(dc, nw, V[p]);
                f32x2 nd = mul2(da, na[p]);  // minus dL/dpower
                if (TESTS) {  // none at the clamp
                    nd.x = na[p].x > -kAlphaMax ? nd.x : 0.f;
                    nd.y = na[p].y > -kAlphaMax ? nd.y : 0.f;
                }
                const f32x2 ed = mul2(nd, dy);
                const f32x2 ax = fma2(qb, dy, t2), ay = fma2(qc2, dy, x);
                float n0, n1, h0, h1, w0, w1;
                unpack2(fma2(ay, ay, mul2(ax, ax)), n0, n1);
                unpack2(nd, h0, h1);
                unpack2(ed, w0, w1);
                E = fmaf(fabsf(h0), sqrt_approx(n0), E);
                E = fmaf(fabsf(h1), sqrt_approx(n1), E);
                // pixel by pixel: where these cancel, a result is as good as their order
                P0 = p == 0 ? h0 + h1 : P0 + h0 + h1;
                P1 = p == 0 ? w0 + w1 : P1 + w0 + w1;
                P2 = fmaf(w1, dy1, p == 0 ? w0 * dy0 : fmaf(w0, dy0, P2));
                if (SAMPLED) {
                    float dx0, dx1;
                    unpack2(dx, dx0, dx1);
                    const float x0 = h0 * dx0, x1 = h1 * dx1;
                    Sx += x0 + x1;
                    Sxx = fmaf(x1, dx1, fmaf(x0, dx0, Sxx));
                    Sxy = fmaf(x1, dy1, fmaf(x0, dy0, Sxy));
                }
                sr = p == 0 ? mul2(d0[p], nw) : fma2(d0[p], nw, sr);
                sg = p == 0 ? mul2(d1[p], nw) : fma2(d1[p], nw, sg);
                sb = p == 0 ? mul2(d2[p], nw) : fma2(d2[p], nw, sb);
            }
            auto sum = [](f32x2 v) {
                float lo, hi;
                unpack2(v, lo, hi);
                return lo + hi;
            };
            if (!SAMPLED) {
                float dx0, dx1;
                unpack2(dx, dx0, dx1);
                Sx = dx0 * P0;
                Sxx = dx0 * dx0 * P0;
                Sxy = dx0 * P1;
            }
            hand_over(u, Sx, P1, P0, sum(sr), sum(sg), sum(sb), E, Sxx, Sxy, P2);
        };
        // the same for any Gaussian and gradient, pixel by pixel
        auto general_step = [&](const BwdEntry& e, int u) {
            const float4 em = e.m, eq = e.qab, eo = e.qco, ec = e.rg, eb = e.brp;
            const uint32_t tag = __float_as_uint(eb.w);
            const float radius = eb.z;
            const float4 q = make_float4(eq.x, eq.z, eo.x, -eo.z);
            const uint32_t pos = tag & ~kByPixel;
            float P0 = 0.f, P1 = 0.f, P2 = 0.f, Sx = 0.f, Sxx = 0.f, Sxy = 0.f, R = 0.f, Gn = 0.f, B = 0.f, E = 0.f;
            auto one_pixel = [&](int k, float fx, float fy, float e0, float e1, float e2, float& Tk, float& Vk) {
                if (pos >= last[k]) return;
                const float dx = fx + em.x, dy = fy + em.z;
                float alpha, G;
                if (!pair_eval(dx, dy, col_terms(dx, q), q, radius, alpha, G)) return;
                const float inv = rcp_approx(1.f - alpha);
                Tk *= inv;
                const float nw = -alpha * Tk;
                R += e0 * nw;
                Gn += e1 * nw;
                B += e2 * nw;
                const float dc = e0 * ec.x + e1 * ec.z + e2 * eb.x;
                const float da = fmaf(Tk, dc, Vk * inv);
                Vk += dc * nw;
                if (alpha < kAlphaMax) {  // below the clamp alpha = o G
                    const float nd = -da * alpha, nx = nd * dx, ny = nd * dy;
                    const float ax = fmaf(q.y, dy, 2.f * q.x * dx), ay = fmaf(2.f * q.z, dy, q.y * dx);
                    P0 += nd;
                    P1 += ny;
                    P2 = fmaf(ny, dy, P2);
                    if (SAMPLED) {
                        Sx += nx;
                        Sxx = fmaf(nx, dx, Sxx);
                        Sxy = fmaf(nx, dy, Sxy);
                    }
                    E = fmaf(fabsf(nd), sqrt_approx(ax * ax + ay * ay), E);
                }
            };
#pragma unroll
            for (int p = 0; p < NP; p++) {
                float t[2], u[2], f[2], y[2], a0[2], a1[2], a2[2];
                unpack2(T[p], t[0], t[1]);
                unpack2(V[p], u[0], u[1]);
                unpack2(FX[SAMPLED ? p : 0], f[0], f[1]);
                unpack2(FY[p], y[0], y[1]);
                unpack2(d0[p], a0[0], a0[1]);
                unpack2(d1[p], a1[0], a1[1]);
                unpack2(d2[p], a2[0], a2[1]);
#pragma unroll
                for (int h = 0; h < 2; h++) one_pixel(2 * p + h, f[h], y[h], a0[h], a1[h], a2[h], t[h], u[h]);
                T[p] = pack2(t[0], t[1]);
                V[p] = pack2(u[0], u[1]);
            }
            if (!SAMPLED) {  // one column per lane: the products of the sums, as in packed_step
                float f0, f1;
                unpack2(FX[0], f0, f1);
                const float dx0 = f0 + em.x;
                if (fabsf(dx0) <= radius) {
                    Sx = dx0 * P0;
                    Sxx = dx0 * dx0 * P0;
                    Sxy = dx0 * P1;
                }
            }
            hand_over(u, Sx, P1, P0, R, Gn, B, E, Sxx, Sxy, P2);
        };
        fetch_ids(0);
        fetch_geometry(0);
        fetch_ids(BWD_SCAN);
        for (uint32_t b = 0; b < len;) {
            // stage the Gaussians that can reach a pixel of the work item
            __syncwarp();
            int n = 0;
            bool tests = false;
            do {
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const uint32_t i = b + 32 * h + lane;
                    const bool hit = i < len && rect_reaches(st.sx0, st.sx1, st.sy0, st.sy1, g[h]);
                    const uint32_t bal = __ballot_sync(kFull, hit);
                    if (hit) {
                        const int slot = n + __popc(bal & lt);
                        tests |= g[h].o < 0.f;
                        const float no = -fabsf(g[h].o);
                        ent[slot].m = make_float4(-g[h].mx, -g[h].mx, -g[h].my, -g[h].my);
                        ent[slot].qab = make_float4(g[h].qa, g[h].qa, g[h].qb, g[h].qb);
                        ent[slot].qco = make_float4(g[h].qc, g[h].qc, no, no);
                        ent[slot].brp.w = __uint_as_float((len - 1 - i) | (g[h].radius >= 0.f && !odd_pixels ? 0u : kByPixel));
                        wrid[slot] = rec[h];
                    }
                    n += __popc(bal);
                }
                b += BWD_SCAN;
                if (b < len) {
                    fetch_geometry(b);
                    fetch_ids(b + BWD_SCAN);
                }
            } while (n <= BWD_FLUSH && b < len);
            __syncwarp();
            float4 cr[(BWD_STAGE + 31) / 32];
#pragma unroll
            for (int i = 0; i < (BWD_STAGE + 31) / 32; i++)
                if (32 * i + lane < n) cr[i] = a.rgb_r[wrid[32 * i + lane]];
#pragma unroll
            for (int i = 0; i < (BWD_STAGE + 31) / 32; i++) {
                const int e = 32 * i + lane;
                if (e < n) {
                    ent[e].rg = make_float4(cr[i].x, cr[i].x, cr[i].y, cr[i].y);
                    *reinterpret_cast<float2*>(&ent[e].brp) = make_float2(cr[i].z, cr[i].z);
                    ent[e].brp.z = cr[i].w;
                }
            }
            // fill the last group with Gaussians that reach no pixel
            if (lane < BWD_GROUP - 1 && (n + lane) % BWD_GROUP != 0 && (n + lane) / BWD_GROUP == (n - 1) / BWD_GROUP) {
                const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
                ent[n + lane].m = ent[n + lane].qab = ent[n + lane].qco = ent[n + lane].rg = ent[n + lane].brp = zero;
            }
            __syncwarp();
            tests = __any_sync(kFull, tests);
            // in groups, straight through: the steps of a group overlap
            for (int j = 0; j < n; j += BWD_GROUP) {
                uint32_t tags = 0;
#pragma unroll
                for (int u = 0; u < BWD_GROUP; u++) tags |= __float_as_uint(ent[j + u].brp.w);
                if (!__any_sync(kFull, tags >= kByPixel)) {
                    f32x2 na[BWD_GROUP][NP];
                    if (LOOK) {  // groups that no pixel blends are passed over
                        if (!tests) {
#pragma unroll
                            for (int u = 0; u < BWD_GROUP; u++) packed_alpha(std::false_type(), ent[j + u], na[u]);
                        } else {
#pragma unroll
                            for (int u = 0; u < BWD_GROUP; u++) packed_alpha(std::true_type(), ent[j + u], na[u]);
                        }
                        float least = 0.f;
#pragma unroll
                        for (int u = 0; u < BWD_GROUP; u++)
#pragma unroll
                            for (int p = 0; p < NP; p++) least = fminf(least, fminf(na[u][p].x, na[u][p].y));
                        if (!__any_sync(kFull, least < 0.f)) continue;
                    }
                    if (!tests) {
#pragma unroll
                        for (int u = 0; u < BWD_GROUP; u++) {
                            if (!LOOK) packed_alpha(std::false_type(), ent[j + u], na[u]);
                            packed_step(std::false_type(), ent[j + u], u, na[u]);
                        }
                    } else {
#pragma unroll
                        for (int u = 0; u < BWD_GROUP; u++) {
                            if (!LOOK) packed_alpha(std::true_type(), ent[j + u], na[u]);
                            packed_step(std::true_type(), ent[j + u], u, na[u]);
                        }
                    }
                } else {
#pragma unroll 1
                    for (int u = 0; u < BWD_GROUP; u++) general_step(ent[j + u], u);
                }
                add_sums(j, min(n - j, BWD_GROUP));
            }
        }
    }
}

// Resident blocks over the whole GPU for a kernel (cached per kernel and device).
int persistent_blocks(const void* kernel) {
    static std::mutex mu;
    static std::map<std::pair<const void*, int>, int> cache;
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    const auto key = std::make_pair(kernel, dev);
    auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 32 * WARPS_PER_BLOCK, 0);
    const int n = (per_sm > 0 ? per_sm : 1) * (sms > 0 ? sms : 1);
    cache[key] = n;
    return n;
}

template <class K>
unsigned grid_for(K kernel, long long items) {
    const long long blocks = (items + WARPS_PER_BLOCK - 1) / WARPS_PER_BLOCK;
    const long long n = persistent_blocks(reinterpret_cast<const void*>(kernel));
    return (unsigned)(blocks < n ? blocks : n);
}

}  // namespace

// Strips are 8 columns wide whatever the tile width: with 4 pixels per lane
// an 8 x 16 strip, whose perimeter (and so the Gaussians that cross into it)
// is smaller than that of a full-width 32 x 4 strip of the same 128 pixels
// (3M Gaussians x 8 views at 32 x 64 tiles: blend forward + backward 16.7 ->
// 13.6 ms; 16-column strips 13.9 ms, 4-column 15.4 ms).
int blend_strip_width(int tw) { return tw > 8 ? 8 : tw; }

int blend_pixels_per_thread(int tw, int th, int req) {
    if (req > 0) return req;
    for (int p = 4; p >= 1; p >>= 1)
        if (th % ((32 / blend_strip_width(tw)) * p) == 0) return p;
    return 1;
}

// The forward's images do not depend on the pixels per lane (each pixel's
// arithmetic is its own), so a small render may use fewer and fill the chip with
// more, shorter strips; the backward sums a lane's pixels together and keeps its
// count.  2432 warps are resident.  Up to 2048 strips of 4 pixels per lane all
// warps have at most one strip and 1 pixel is fastest: 10k Gaussians at 128 x 128
// (128 strips) 69 -> 38 us, 20k in three small views (1077) 256 -> 144, 300k at
// 480 x 400 (1500) 179 -> 110, with 2 pixels 45, 179, 122.  Above, a strip's
// staging is repeated too often, and 2 are fastest while the queue is short:
// 100k at 800 x 600 (3750 strips) 83 us with 4, 73 with 2, 101 with 1; two views
// of unlike sizes (7394) 267, 170, 202; from about three strips of 4 per warp on
// it is even (7734 strips: 157 and 148, 55 and 59; 8216: 101 and 107).
int blend_forward_pixels_per_thread(int tw, int th, int req, long long tiles) {
    const int most = blend_pixels_per_thread(tw, th, req);
    if (req > 0) return most;
    const long long strips = tiles * tw * th / 128;
    const int want = strips <= 2048 ? 1 : strips <= 7500 ? 2 : 4;
    return want < most ? want : most;
}

void launch_blend_forward(const BlendArgs& a, int* counter, float* img, float* final_T, uint32_t* n_contrib,
                          uint2* pixel_stats, cudaStream_t s) {
    if (a.tiles == 0) return;
    const bool sampled = a.s_off != nullptr;
    // sampled mode: the number of runs is only known on the device; launch a
    // full persistent grid
    const bool depth = a.depth_out != nullptr, stats = pixel_stats != nullptr;
    const long long items = sampled ? (1LL << 40) : a.tiles * a.strips;
#define MVGS_BF1(P, S, D, ST)                                                                             \
    blend_forward_kernel<P, S, D, ST><<<grid_for(blend_forward_kernel<P, S, D, ST>, items),               \
                                        32 * WARPS_PER_BLOCK, 0, s>>>(a, counter, img, final_T, n_contrib, \
                                                                      pixel_stats)
#define MVGS_BF(P, S)                        \
    do {                                     \
        if (depth && stats)                  \
            MVGS_BF1(P, S, true, true);      \
        else if (depth)                      \
            MVGS_BF1(P, S, true, false);     \
        else if (stats)                      \
            MVGS_BF1(P, S, false, true);     \
        else                                 \
            MVGS_BF1(P, S, false, false);    \
    } while (0)
#define MVGS_BF2(P)              \
    do {                         \
        if (sampled)             \
            MVGS_BF(P, true);    \
        else                     \
            MVGS_BF(P, false);   \
    } while (0)
    switch (a.ppt) {
        case 1: MVGS_BF2(1); break;
        case 2: MVGS_BF2(2); break;
        case 8: MVGS_BF2(8); break;
        default: MVGS_BF2(4); break;
    }
#undef MVGS_BF2
#undef MVGS_BF
#undef MVGS_BF1
    note_launches(1);
}

// Strips up to which the backward looks at a group's alphas before it takes the
// group.  A strip's list is walked by one warp, and the longest walks are what is
// waited for when there are few strips, or when they are small (up to 2 pixels per
// lane: tiles 8 high): most of a list's Gaussians then reach the strip but no pixel
// of it.  375k Gaussians on 64 views of some 200 x 200 65 -> 32 ms, 921k x 9 views
// at 8 x 8 tiles 38 -> 18, 25k x 8 small views at 16 x 8 1.10 -> 0.68, 20k x 3 534
// -> 493 us; where every group is blended it costs 3 to 10% (500k at 1000 x 800
// 458 -> 500 us), so not for the large renders of tall tiles (sampled pixels of 500k
// x 4 views 1028 -> 1107, masked ones of 3M x 8 6.1 -> 6.6 ms).  Over 400 random
// calls it gives 1.08 to 1.21x (geometric mean per range of strips, 0.82 to 2.04x)
// up to this line and 1.00x beyond it.  Sampled or masked pixels fill a part of the
// strips (a quarter of them with four views to a group), so their line lies four
// times as far: 1.23 and 1.34x beyond 7500 and 15000 strips (61k Gaussians on 64
// small views 4.98 -> 2.93 ms).
constexpr long long kFewStrips = 7500;

void launch_blend_backward(const BlendArgs& a, int* counter, const float* dimg, const float* final_T,
                           const uint32_t* n_contrib, float* rec_grad, double* rec_conic, cudaStream_t s) {
    if (a.tiles == 0) return;
    cudaMemsetAsync(counter, 0, sizeof(int), s);
    const bool sampled = a.s_off != nullptr;
    const long long items = sampled ? (1LL << 40) : a.tiles * a.strips;
#define MVGS_BB(P, S, L)                                                                                         \
    blend_backward_kernel<P, S, L><<<grid_for(blend_backward_kernel<P, S, L>, items), 32 * WARPS_PER_BLOCK, 0, s>>>( \
        a, counter, dimg, final_T, n_contrib, rec_grad, rec_conic)
#define MVGS_BB2(P, L) if (sampled) MVGS_BB(P, true, L); else MVGS_BB(P, false, L)
    switch (a.ppt) {
        case 1: MVGS_BB2(1, true); break;
        case 2: MVGS_BB2(2, true); break;
        case 8: MVGS_BB2(8, true); break;
        default:
            if (a.tiles * a.strips <= (sampled || a.pixel_mask ? 4 : 1) * kFewStrips) MVGS_BB2(4, true);
            else MVGS_BB2(4, false);
            break;
    }
#undef MVGS_BB2
#undef MVGS_BB
    note_launches(1);
}

}  // namespace mvgs
