// Shared definitions of the sm_103a kernels (device side of libmvgs).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace mvgs {

// Rasterizer constants the paper inherits from 3DGS without printing them
// (Sec. 3 cites the 3DGS rasterizer and EWA splatting): low-pass dilation of
// the projected covariance, alpha clamp, alpha skip threshold, transmittance
// cutoff, guard band of the projection Jacobian, 3-sigma radius and the
// eigenvalue floor used for it.
constexpr float kDilation = 0.3f;
constexpr float kAlphaMax = 0.99f;
constexpr float kAlphaMin = 1.0f / 255.0f;
constexpr float kTMin = 1e-4f;
constexpr float kGuard = 1.3f;
constexpr float kSigmas = 3.0f;
constexpr float kEigFloor = 0.1f;

// What the projection reads of a view.
struct ProjCam {
    float R[9];      // world -> camera rotation, row-major
    float t[3];
    float fx, fy, cx, cy;
    float campos[3];
    float near_z;
    float limx, limy;  // guard band on x/z and y/z
    int W, H, tiles_x, tiles_y;
};

// Per-view camera table entry, built on the host from mvgs_camera and
// uploaded once per call; every kernel reads it from global memory.
struct __align__(16) DevCam : ProjCam {
    long long tile_base;  // first global tile id of the view
    long long pix_base;   // first pixel of the view in the packed layout
    long long bin_base;   // first bin of the view (8 x 8 tiles each, row-major)
};
static_assert(sizeof(DevCam) == 128, "camera table entry is 128 bytes");

// An element count: known on the host (max), or -- in the capturable mode,
// where no count is read back -- held in device memory and bounded by the
// capacity the buffers were sized for: min(max, *dev).
struct Count {
    unsigned long long max;
    const unsigned long long* dev;
    __host__ __device__ Count(unsigned long long m = 0, const unsigned long long* d = nullptr) : max(m), dev(d) {}
    __device__ __forceinline__ unsigned long long get() const {
        if (!dev) return max;
        const unsigned long long v = *dev;
        return v < max ? v : max;
    }
    __device__ __forceinline__ bool over() const { return dev && *dev > max; }
};

// Kernels launched with launch_chained begin while the kernel before them on the
// stream ends: chained() comes first in every thread, before any return, lets the
// next kernel's blocks take their places and then waits until the kernel before is
// complete and its writes are visible.  The predecessor has waited for its own in
// the same way, so this holds for every kernel before on the stream, whatever it
// wrote: the chain's arrays, and the scene a caller's kernel has just updated.
// The wait orders ordinary loads only.  A const __restrict__ pointer (or __ldg)
// would promise that nobody writes the data while the kernel runs, which is not so
// -- it may be resident while all of those still write -- and would allow loads
// through the non-coherent cache or ahead of the wait.  So no pointer of a chained
// kernel is __restrict__; where that costs something (a load behind a store that
// might alias it), the kernel loads first.  The 30
// launches from the participation to the blend wait about 1 us less each: a
// 500k-Gaussian frame 531 -> 483 us, 20k in three small views 877 -> 839, 500k x 4
// views 2900 -> 2845.  Not for the persistent blends: their waiting blocks cost
// more than the launch (five views of 2M Gaussians 3061 -> 3139 us).
__device__ __forceinline__ void chained() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Blocks up to which a launch is chained: a longer kernel gains nothing (3M
// Gaussians x 8 views with all of them: 14.42 against 14.39 ms).
constexpr unsigned kChainedBlocks = 4096;

template <class... P, class... A>
void launch_chained(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t s, A... args) {
    // not into a graph: a captured step runs 2% slower with these edges (15.08
    // against 14.79 ms at 3M Gaussians x 8 views)
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    cudaStreamIsCapturing(s, &capture);
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = capture == cudaStreamCaptureStatusNone && grid <= kChainedBlocks ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Asynchronous copies from global to shared memory: no register holds the data,
// so a warp goes on until it waits for them.  N: 4, 8 or 16 bytes, both sides
// aligned to it.
template <int N>
__device__ __forceinline__ void cp_async(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "n"(N)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
}

constexpr int kCamChunk = 32;
struct CamChunk {
    DevCam c[kCamChunk];
};

// Per-record float gradient slots written by the blend backward and read by
// the preprocessing backward: mean2d x, y, opacity (times the opacity), r, g, b,
// E_1 term, padding (the conic's three go to a separate double array).
constexpr int kGradStride = 8;

// Single-instruction approximations (PTX rcp.approx / sqrt.approx, about
// 1 ulp; flush-to-zero) for per-pair arithmetic, where the correctly rounded
// forms (__frcp_rn, IEEE sqrtf and division) are instruction sequences with a
// slow path.  The blend backward recovers T by a reciprocal and sums
// |dL/dmean2d| with a square root on every blended pair: the exact forms cost
// a fifth of that kernel, and the approximations are far inside the gradient
// tolerance of 1e-3 relative.
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float sqrt_approx(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ int find_view(const DevCam* cams, int V, long long gt) {
    int lo = 0, hi = V - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (cams[mid].tile_base <= gt) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// SplitMix64 (Steele, Lea & Flood, OOPSLA 2014): output number k of the
// stream seeded with s is mix(s + k * 0x9e3779b97f4a7c15).  The partial-render
// sample slot of cell (x, y) in a group of `group` views is
// floor(group * (h >> 32) / 2^32) with h output number 2^32 y + x + 1; a
// pixel's cell is (px / cell_w, py / cell_h).
__device__ __forceinline__ unsigned long long splitmix64_mix(unsigned long long z) {
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
    return z ^ (z >> 31);
}

__device__ __forceinline__ int sample_slot(unsigned long long seed, int x, int y, int group) {
    const unsigned long long c = ((unsigned long long)y << 32) | (unsigned)x;
    const unsigned long long h = splitmix64_mix(seed + (c + 1ULL) * 0x9e3779b97f4a7c15ULL);
    return (int)(((h >> 32) * (unsigned long long)group) >> 32);
}

// 2^x for the blend exponent (PTX ex2.approx, relative error near 2^-22;
// results below 2^-126 flush to zero, far under the 1/255 skip threshold).
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// The blend exponent in base 2.  With conic (A, B, C), d = pixel centre
// minus projected mean and L = log2 e,
//   power L = -(A dx^2 + 2 B dx dy + C dy^2) L / 2 = qa dx^2 + qb dx dy + qc dy^2,
// q = (qa, qb, qc) = (-A L / 2, -B L, -C L / 2), so G = exp(power) is one
// ex2 of a two-FMA polynomial in dy once the column terms (qa dx^2, qb dx)
// of the pixel's column are known.  A lane of a strip owns one column: it
// computes the column terms once per Gaussian and reuses them for its PPT
// pixels.
__device__ __forceinline__ float4 exp2_coeffs(float4 co) {
    constexpr float L = 1.4426950408889634f;
    return make_float4(__fmul_rn(-0.5f * L, co.x), __fmul_rn(-L, co.y), __fmul_rn(-0.5f * L, co.z), co.w);
}

// A record's tile rectangle and view for the duplication, in 8 bytes: the
// corners x0, y0, x1, y1 (tile coordinates, end exclusive, each below 2^12)
// in bits 0-47 and the view in bits 48-63.
__device__ __forceinline__ unsigned long long pack_tile_desc(short4 rc, int view) {
    return (unsigned long long)(uint16_t)rc.x | (unsigned long long)(uint16_t)rc.y << 12 |
           (unsigned long long)(uint16_t)rc.z << 24 | (unsigned long long)(uint16_t)rc.w << 36 |
           (unsigned long long)view << 48;
}
__device__ __forceinline__ short4 tile_desc_rect(unsigned long long d) {
    return make_short4((short)(d & 0xfffu), (short)(d >> 12 & 0xfffu), (short)(d >> 24 & 0xfffu),
                       (short)(d >> 36 & 0xfffu));
}
__device__ __forceinline__ int tile_desc_view(unsigned long long d) { return (int)(d >> 48); }

// Bins of 8 x 8 tiles (sort.cu): bins along an axis of `tiles` tiles, and the
// bins a tile rectangle reaches.
__host__ __device__ __forceinline__ int bins_across(int tiles) { return (tiles + 7) >> 3; }
__device__ __forceinline__ uint32_t bins_touched(short4 rc) {
    if (rc.z <= rc.x || rc.w <= rc.y) return 0u;
    return (uint32_t)((((rc.z - 1) >> 3) - (rc.x >> 3) + 1) * (((rc.w - 1) >> 3) - (rc.y >> 3) + 1));
}

// Packed float32 arithmetic of sm_100 and later on a pair of registers: one
// instruction, two IEEE round-to-nearest results (the bits of the scalar
// operations).  It takes the FMA pipe as long as two scalar instructions but
// one issue slot.
typedef float2 f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) { a = v.x; b = v.y; }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) { return __ffma2_rn(a, b, c); }

// A product the compiler may not merge with an equal one before it: where the
// first is only looked at and the second replaces its factor, merging them
// would cost a register copy per value.
__device__ __forceinline__ f32x2 mul2_fresh(f32x2 a, f32x2 b) {
    f32x2 r;
    asm volatile("{.reg .b64 a, b, r; mov.b64 a, {%2, %3}; mov.b64 b, {%4, %5}; mul.rn.f32x2 r, a, b; mov.b64 {%0, %1}, r;}"
                 : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}

struct ColTerms {
    float xx, x;  // qa dx^2 and qb dx
};

__device__ __forceinline__ ColTerms col_terms(float dx, float4 q) {
    return ColTerms{__fmul_rn(__fmul_rn(q.x, dx), dx), __fmul_rn(q.y, dx)};
}

// The blend decision and opacity of one (pixel, Gaussian) pair (Eq. 1 with
// the 3DGS clamp and skip rules and the per-pixel support rule); q holds the
// base-2 coefficients and the opacity (q.w), ct the column terms of dx.
// Everything is evaluated unconditionally; the return value says whether the
// Gaussian takes part at this pixel, and alpha and G = exp(power) are valid
// when it does.  The forward and the backward call this same function with
// the same inputs, so both take the same decision for every pair.  The
// products and fused multiply-adds are spelled out (no contraction left to
// the compiler), and the column terms are the same products whether a lane
// reuses them (strips) or computes them per pixel (sample runs), so every
// kernel rounds a pair the same way.
__device__ __forceinline__ bool pair_eval(float dx, float dy, ColTerms ct, float4 q, float radius, float& alpha,
                                          float& G) {
    const float e = __fmaf_rn(dy, __fmaf_rn(q.z, dy, ct.x), ct.xx);
    G = ex2_approx(e);
    alpha = fminf(kAlphaMax, __fmul_rn(q.w, G));
    return fabsf(dx) <= radius && fabsf(dy) <= radius && e <= 0.f && alpha >= kAlphaMin;
}

// What the blend kernels read of a record to decide whether it reaches a
// strip, in one 32-byte sector (a list entry is looked at by every strip of its
// tile; the separate arrays of the state took three sectors).  The colour is
// fetched for the entries that do.
struct alignas(32) Geom {
    float mx, my;        // projected mean
    float qa, qb, qc;    // base-2 exponent coefficients (exp2_coeffs)
    float o;             // opacity; negative: blended with the tests that a plain one does without
    float radius;        // in pixels; negative: blended pixel by pixel (ordinary_gaussian)
    float reach;         // alpha >= 1/255 needs an exponent of at least -reach (base 2), with a margin
};
static_assert(sizeof(Geom) == 32, "one sector");

__device__ __forceinline__ Geom load_geom(const Geom* g) {
    const float4 a = reinterpret_cast<const float4*>(g)[0], b = reinterpret_cast<const float4*>(g)[1];
    return Geom{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
}

// Whether the quadratic form of the conic (A, B, C) of a covariance (a, b, c) stays
// clear of its rounding: with det = ac - b^2 >= 0.01 ac, so B^2 <= 0.99 AC, it is
// at least 1/400 of the sum of its terms' magnitudes.  With the dilation's 0.3 in a
// and c, A and C are at most 334; the bound on a and c keeps the terms of a pixel
// distance (0, or at least 2^-25) clear of underflow.  NaN fails.
__device__ __forceinline__ bool well_conditioned(float a, float c, float det) {
    return (det >= 0.01f * (a * c)) & (a + c <= 1e15f);
}

// Whether blending a Gaussian with alpha 0 changes nothing, so that the packed
// blend steps may take it without branches: everything they multiply with that 0
// is finite -- the exponent's terms and the squares of its derivatives over the
// support (and a work item's 64 pixels past it), the colour (not negative, and small
// enough for its product with any image gradient the backward takes this way, see
// there) and the depth.  NaN fails every comparison.
__device__ __forceinline__ bool ordinary_gaussian(float4 co, float radius, float3 rgb, float depth, bool well) {
    return (well || (fabsf(co.x) + fabsf(co.y) + fabsf(co.z)) * (radius + 64.f) <= 1e15f) &&
           (co.w <= 1.f) & (rgb.x + rgb.y + rgb.z <= 1e10f) & (fabsf(depth) <= 3e38f);
}

// A record's Geom; well: well_conditioned.
__device__ __forceinline__ Geom make_geom(float2 m, float4 co, float radius, float3 rgb, float depth, bool well) {
    const float4 q = exp2_coeffs(co);
    const float l2 = __log2f(255.f * co.w);  // o G >= 1/255 where the exponent is -l2 or more
    float reach = -1.f;
    if (l2 > 0.f) {
        reach = l2 * 1.001f + 1e-3f;
        // What rounding may add to a pixel's exponent and take from rect_reaches'
        // maximum: 3 2^-24 each of the terms' magnitudes, together below 2^-21 of
        // their sum at the support's corner (rect_reaches may look up to a work
        // item's 64 pixels past it).  At most 400 l2 2^-21 for a well-conditioned
        // form, inside the margin above; of the order of 1 for needles of 500
        // pixels, whose terms are a million times the exponent.
        if (!well) {
            const float far = radius + 64.f;
            reach += 0x1p-21f * (fabsf(q.x) + fabsf(q.y) + fabsf(q.z)) * far * far;
        }
    }
    // plain: two tests of pair_eval cannot matter, and the packed steps leave them out
    //   - e <= 0: rounding (a few 2^-24 of the sum of the terms' magnitudes) cannot
    //     turn a well-conditioned form negative.
    //   - the clamp at 0.99: o G stays below it when o does (G <= 1 up to the
    //     error of ex2.approx).
    const bool plain = well & (co.w <= 0.989f);
    return Geom{m.x, m.y, q.x, q.y, q.z, plain ? co.w : -co.w,
                ordinary_gaussian(co, radius, rgb, depth, well) ? radius : -radius, reach};
}

// Whether a Gaussian can pass the support rule and alpha >= 1/255 at any
// pixel centre of the rectangle [x0, x1] x [y0, y1].  From the point of the
// rectangle (relative to the mean) where the exponent is largest, the way to
// the mean, along which it grows, must leave the rectangle, so that point lies
// on an edge facing the mean: at most one in x and one in y, and on an edge the
// exponent is a 1D quadratic with its maximum in closed form.  (On an axis on
// which the rectangle holds the mean there is no such edge; its candidate below
// is then some point of the rectangle, and the mean itself when that is
// inside.)  The margin in `reach` (make_geom) keeps the test a superset of what
// any pixel's float32 evaluation lets through, so what a pixel blends does not
// depend on the work item it is in, and the forward and the backward, whose strips
// may differ, blend the same pairs; a maximiser off by a relative 1e-7 (the
// approximate reciprocals) lowers the exponent by a second-order amount, far
// inside it.  NaN fails the first comparisons or the last.
__device__ __forceinline__ bool rect_reaches(float sx0, float sx1, float sy0, float sy1, const Geom& g) {
    const float x0 = sx0 - g.mx, x1 = sx1 - g.mx, y0 = sy0 - g.my, y1 = sy1 - g.my, r = fabsf(g.radius);
    const float xe = fminf(fmaxf(0.f, x0), x1), ye = fminf(fmaxf(0.f, y0), y1);
    const float hb = -0.5f * g.qb;
    const float ys = fminf(fmaxf(hb * xe * rcp_approx(g.qc), y0), y1);
    const float xs = fminf(fmaxf(hb * ye * rcp_approx(g.qa), x0), x1);
    const float e1 = fmaf(xe, fmaf(g.qb, ys, g.qa * xe), g.qc * ys * ys);
    const float e2 = fmaf(xs, fmaf(g.qb, ye, g.qa * xs), g.qc * ye * ye);
    return (x0 <= r) & (x1 >= -r) & (y0 <= r) & (y1 >= -r) & (fmaxf(e1, e2) >= -g.reach) & (g.reach > 0.f);
}

}  // namespace mvgs
