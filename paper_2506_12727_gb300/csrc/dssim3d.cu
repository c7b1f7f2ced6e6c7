// 3D distance-aware D-SSIM (Sec. 5.1.2) on the merged images of a partially
// rendered batch (Fig. 3c), and the two copies around it.
//
// merge:  for every pixel of merged image m (views m*group .. m*group+group-1,
//         one resolution), the owner view v = m*group + slot(x, y) -- the view
//         that rendered the pixel in the partial render -- gives the merged
//         colour and target, and the pixel's surface point: the expected depth
//         z = D / (1 - T_final) (D = sum alpha T z_i from the forward) lifted
//         through the pixel centre of v's camera, X = R^T (z K^-1 (x+.5, y+.5,
//         1) - t), with the kernel width s = sigma_px z / f_x (the window's
//         sigma in pixels carried to the surface).  1 - T_final < 1e-3: no
//         surface point (s = 0).
// loss:   K*(p, q) = exp(-|X_q - X_p|^2 / (2 s_p^2)) over the 11x11 window of
//         the centre p, normalised to sum 1 over the neighbours inside the
//         image that have a surface point (a centre without one keeps only
//         itself); SSIM with K* in place of the 2D window, C1 = 0.01^2,
//         C2 = 0.03^2; L_m = (1 - lambda) mean|I - I*| + lambda (1 - mean SSIM),
//         the weights held constant.
//         Kernel 1 (per 32x8 pixels, halo 42x18 in shared memory) forms the
//         weights, the moments, SSIM and, per centre p and channel, the
//         coefficients A_p, B_p, C_p / Z_p of dSSIM_p/dI1(q) = w_pq (A + 2 B
//         I1(q) + C I2(q)) / Z_p; kernel 2 gathers them back per pixel q over
//         the centres whose window holds q; kernel 3 reduces the block sums per
//         image in a fixed order.
// split:  dL/d(merged pixel) goes to the owner view's pixel, 0 to the group's
//         other views there.
#include <cfloat>
#include <cmath>

#include "kernels.h"

namespace mvgs {
namespace {

// 32 x 8 pixels per block: a lane holds two pixels one above the other, so that
// a neighbour read from shared memory serves both, and a warp two rows of 32,
// so that its reads of a neighbour offset fall in different banks.
constexpr int TSX = 32, TSY = 8;
constexpr int THREADS = TSX * TSY / 2;
constexpr int RAD = 5;
constexpr int HSX = TSX + 2 * RAD, HSY = TSY + 2 * RAD;  // 42 x 18 staged
constexpr float kC1 = 0.01f * 0.01f;
constexpr float kC2 = 0.03f * 0.03f;
constexpr int kMaxImages = 64;
constexpr float kMinOpacity = 1e-3f;

struct Images {
    int count;
    int H[kMaxImages], W[kMaxImages], tiles_x[kMaxImages];
    long long pix[kMaxImages];      // first pixel of the image in the packed layout
    long long blk[kMaxImages + 1];  // first block of the image
    int first;                      // global index of image 0
};

__device__ __forceinline__ int image_of(const Images& im, long long b) {
    int i = 0;
    while (i + 1 < im.count && im.blk[i + 1] <= b) i++;
    return i;
}

struct Blk {
    int i, H, W, x0, y0;
    long long pix;
};

__device__ __forceinline__ Blk block_of(const Images& im) {
    Blk b;
    b.i = image_of(im, blockIdx.x);
    const long long t = blockIdx.x - im.blk[b.i];
    b.H = im.H[b.i];
    b.W = im.W[b.i];
    b.x0 = (int)(t % im.tiles_x[b.i]) * TSX;
    b.y0 = (int)(t / im.tiles_x[b.i]) * TSY;
    b.pix = im.pix[b.i];
    return b;
}

// The window sums of one centre.
struct Sums {
    float Z;
    f32x2 m1, m2, m3;     // sums of w I1, w I2 (channels 0, 1; m3: channel 2 of both)
    f32x2 e11, e22, e33;  // of w I1^2, w I2^2
    f32x2 e12;            // of w I1 I2
    float e12c;           // channel 2
};

// One tap's terms, each product and sum rounded as in w * a * q accumulated
// term by term.
__device__ __forceinline__ void add_tap(Sums& s, float w, f32x2 a, f32x2 q, f32x2 c) {
    const f32x2 ww = pack2(w, w);
    const f32x2 wa = mul2(ww, a), wq = mul2(ww, q), wc = mul2(ww, c);
    s.Z += w;
    s.m1 = add2(s.m1, wa);
    s.m2 = add2(s.m2, wq);
    s.m3 = add2(s.m3, wc);
    s.e11 = fma2(wa, a, s.e11);
    s.e22 = fma2(wq, q, s.e22);
    s.e33 = fma2(wc, c, s.e33);
    s.e12 = fma2(wa, q, s.e12);
    s.e12c = __fmaf_rn(wc.x, c.y, s.e12c);
}

// Whether the fast loops below may take these values: images finite (a zero
// weight then adds nothing), and where there is a surface point, coordinates and
// widths far from the ends of the float range.
constexpr float kMaxCoord = 0x1p30f, kMinWidth = 0x1p-30f, kMaxWidth = 0x1p20f;
__device__ __forceinline__ bool finite(float v) { return fabsf(v) <= FLT_MAX; }
__device__ __forceinline__ bool in_domain(float x, float y, float z, float s) {
    if (!(s > 0.f)) return true;
    return fabsf(x) <= kMaxCoord && fabsf(y) <= kMaxCoord && fabsf(z) <= kMaxCoord && s >= kMinWidth && s <= kMaxWidth;
}
// A pixel without a surface point sits this far off as a neighbour, and as far on
// the other side as a centre: its distance to any other gives a weight of zero
// (at least 2^63 over 2^41), and d2 y stays below 2^126.
constexpr float kFar = 0x1p32f;

// The weights of one neighbour for two centres (or of two neighbours for one
// centre) whose squared distances are d2: exp(-d2 / c), c = 2 s^2, nc = -c, y
// the correctly rounded 1 / c.  The quotient d2 y is corrected once by its exact
// remainder (Markstein 1990, whose theorem gives the correctly rounded quotient
// when d2 y is faithful; of 1.7e10 drawn pairs, near the worst cases too, none
// differed from the division, nor of the millions a host test draws): 3 instructions for both against about 10 each.
__device__ __forceinline__ f32x2 weights(f32x2 d2, f32x2 nc, f32x2 y) {
    f32x2 q = mul2(d2, y);
    q = fma2(fma2(q, nc, d2), y, q);
    return pack2(__expf(-q.x), __expf(-q.y));
}

__device__ __forceinline__ f32x2 dist2(f32x2 dx, f32x2 dy, f32x2 dz) {
    return fma2(dz, dz, fma2(dx, dx, mul2(dy, dy)));
}

// Blocks with values out of the fast loops' domain: a pixel without a surface
// point is marked in the staged x coordinate by a NaN of its own (one that comes in
// as a coordinate is made another), and the loops below test for it.
__device__ __forceinline__ float no_point() { return __uint_as_float(0x7fffdeadu); }
__device__ __forceinline__ bool is_point(float x) { return __float_as_uint(x) != 0x7fffdeadu; }

// Called by every thread of the block.
__device__ __forceinline__ void mark_points(const Blk& b, long long HW, const float* __restrict__ pts,
                                            const float* __restrict__ sig, float (&sX)[HSY][HSX + 1]) {
    for (int k = threadIdx.x; k < HSX * HSY; k += THREADS) {
        const int r = k / HSX, c = k % HSX;
        const int y = b.y0 + r - RAD, x = b.x0 + c - RAD;
        const bool in = x >= 0 && y >= 0 && x < b.W && y < b.H;
        const long long o = (long long)y * b.W + x;
        float v = no_point();
        if (in && sig[b.pix + o] > 0.f) {
            v = pts[3 * b.pix + o];
            if (!is_point(v)) v = __uint_as_float(0x7fffffffu);
        }
        sX[r][c] = v;
    }
    __syncthreads();
}

// The weights for any values: as above where nothing of that can leave the float
// range, else by division.
__device__ __forceinline__ float any_weight(float w, float d2, float c, float y) {
    if (d2 * y > 200.f) w = 0.f;  // the correction may have been infinite
    return c >= 0x1p-90f && c <= 0x1p120f ? w : __expf(-d2 / c);
}
__device__ __forceinline__ f32x2 any_weights(f32x2 d2, f32x2 nc, f32x2 y) {
    const f32x2 w = weights(d2, nc, y);
    return pack2(any_weight(w.x, d2.x, -nc.x, y.x), any_weight(w.y, d2.y, -nc.y, y.y));
}
// What has no weight may be anything.
__device__ __forceinline__ f32x2 if_some(float w, f32x2 v) { return pack2(w != 0.f ? v.x : 0.f, w != 0.f ? v.y : 0.f); }

// Bound by the FMA pipe (two thirds busy): for two pixels a neighbour takes 9
// passes of the shared-memory unit, 9 packed instructions for both weights, two
// exponentials and 11 each for the 16 sums, where one pixel per lane took 10
// reads, two slow divisions' worth of instructions and 21 for the sums.  One
// 1264 x 832 image: 303 -> 180 us, of which the arithmetic is 120.
__global__ void __launch_bounds__(THREADS) dssim3d_forward_kernel(Images im, long long P, const float* __restrict__ img,
                                                                 const float* __restrict__ tgt,
                                                                 const float* __restrict__ pts,
                                                                 const float* __restrict__ sig,
                                                                 float* __restrict__ coef, float2* __restrict__ bsum,
                                                                 long long blk_offset) {
    __shared__ float sX[HSY][HSX + 1], sY[HSY][HSX + 1], sZ[HSY][HSX + 1];
    __shared__ f32x2 sA[HSY][HSX + 1], sQ[HSY][HSX + 1], sC[HSY][HSX + 1];  // I1, I2 of channels 0, 1; both of 2
    __shared__ float red[2][THREADS / 32];
    const Blk b = block_of(im);
    const long long HW = (long long)b.H * b.W;
    bool odd = false;
    for (int k = threadIdx.x; k < HSX * HSY; k += THREADS) {
        const int r = k / HSX, c = k % HSX;
        const int y = b.y0 + r - RAD, x = b.x0 + c - RAD;
        const bool in = x >= 0 && y >= 0 && x < b.W && y < b.H;
        const long long o = (long long)y * b.W + x;
        const float s = in ? sig[b.pix + o] : -1.f;
        float X[3], u[3], v[3];
#pragma unroll
        for (int ch = 0; ch < 3; ch++) {
            X[ch] = in ? pts[3 * b.pix + ch * HW + o] : 0.f;
            u[ch] = in ? img[3 * b.pix + ch * HW + o] : 0.f;
            v[ch] = in ? tgt[3 * b.pix + ch * HW + o] : 0.f;
            odd |= !finite(u[ch]) || !finite(v[ch]);
        }
        odd |= !in_domain(X[0], X[1], X[2], s);
        const bool point = s > 0.f;
        sX[r][c] = point ? X[0] : kFar;
        sY[r][c] = point ? X[1] : 0.f;
        sZ[r][c] = point ? X[2] : 0.f;
        sA[r][c] = pack2(u[0], u[1]);
        sQ[r][c] = pack2(v[0], v[1]);
        sC[r][c] = pack2(u[2], v[2]);
    }
    odd = __syncthreads_or(odd);
    const int lane = threadIdx.x & 31, c0 = lane + RAD, r0 = 2 * (threadIdx.x >> 5) + RAD;
    const int x = b.x0 + lane, y = b.y0 + r0 - RAD;
    Sums s[2]{};
    if (odd) {
        mark_points(b, HW, pts, sig, sX);
        // the loops below with every test (a NaN in every block of a 1264 x 832 image:
        // 540 us with the backward, without one 333)
        float c2[2], npx[2];
        bool point[2];
#pragma unroll
        for (int k = 0; k < 2; k++) {
            const float sp = x < b.W && y + k < b.H ? sig[b.pix + (long long)(y + k) * b.W + x] : -1.f;
            point[k] = sp > 0.f;
            c2[k] = point[k] ? 2.f * sp * sp : 1.f;
            npx[k] = -sX[r0 + k][c0];
        }
        const f32x2 nx = pack2(npx[0], npx[1]), ny = pack2(-sY[r0][c0], -sY[r0 + 1][c0]),
                    nz = pack2(-sZ[r0][c0], -sZ[r0 + 1][c0]);
        const f32x2 nc = pack2(-c2[0], -c2[1]), yc = pack2(1.f / c2[0], 1.f / c2[1]);
        for (int rr = r0 - RAD; rr <= r0 + RAD + 1; rr++) {
            const bool upper = point[0] && rr <= r0 + RAD, lower = point[1] && rr > r0 - RAD;
#pragma unroll
            for (int du = -RAD; du <= RAD; du++) {
                const int cc = c0 + du;
                const float qx = sX[rr][cc], qy = sY[rr][cc], qz = sZ[rr][cc];
                f32x2 w = any_weights(
                    dist2(add2(pack2(qx, qx), nx), add2(pack2(qy, qy), ny), add2(pack2(qz, qz), nz)), nc, yc);
                const bool neighbour = is_point(qx);
                w.x = upper && neighbour ? w.x : 0.f;
                w.y = lower && neighbour ? w.y : 0.f;
                if (du == 0 && rr == r0) w.x = 1.f;
                if (du == 0 && rr == r0 + 1) w.y = 1.f;
                const f32x2 a = sA[rr][cc], q = sQ[rr][cc], ch2 = sC[rr][cc];
                add_tap(s[0], w.x, if_some(w.x, a), if_some(w.x, q), if_some(w.x, ch2));
                add_tap(s[1], w.y, if_some(w.y, a), if_some(w.y, q), if_some(w.y, ch2));
            }
        }
    } else {
        float sp[2], npx[2];
#pragma unroll
        for (int k = 0; k < 2; k++) {
            sp[k] = x < b.W && y + k < b.H ? sig[b.pix + (long long)(y + k) * b.W + x] : -1.f;
            npx[k] = sp[k] > 0.f ? -sX[r0 + k][c0] : kFar;
        }
        const f32x2 nx = pack2(npx[0], npx[1]), ny = pack2(-sY[r0][c0], -sY[r0 + 1][c0]),
                    nz = pack2(-sZ[r0][c0], -sZ[r0 + 1][c0]);
        const float ca = sp[0] > 0.f ? 2.f * sp[0] * sp[0] : 1.f, cb = sp[1] > 0.f ? 2.f * sp[1] * sp[1] : 1.f;
        const f32x2 nc = pack2(-ca, -cb), yc = pack2(1.f / ca, 1.f / cb);
        // neighbours in rows; the first row is in the upper pixel's window only, the
        // last in the lower one's
        auto row = [&](int rr, bool upper, bool lower) {
#pragma unroll
            for (int du = -RAD; du <= RAD; du++) {
                const int cc = c0 + du;
                const float qx = sX[rr][cc], qy = sY[rr][cc], qz = sZ[rr][cc];
                const f32x2 w = weights(dist2(add2(pack2(qx, qx), nx), add2(pack2(qy, qy), ny), add2(pack2(qz, qz), nz)),
                                        nc, yc);
                const f32x2 a = sA[rr][cc], q = sQ[rr][cc], ch2 = sC[rr][cc];
                if (upper) add_tap(s[0], w.x, a, q, ch2);
                if (lower) add_tap(s[1], w.y, a, q, ch2);
            }
        };
        // a warp of background, without a surface point, has nothing to add up (an
        // image of it 335 -> 117 us with the backward)
        if (__any_sync(0xffffffffu, sp[0] > 0.f || sp[1] > 0.f)) {
            row(r0 - RAD, true, false);
            for (int rr = r0 - RAD + 1; rr <= r0 + RAD; rr++) row(rr, true, true);
            row(r0 + RAD + 1, false, true);
        }
#pragma unroll
        for (int k = 0; k < 2; k++) {
            if (sp[k] > 0.f) continue;
            s[k] = Sums{};  // no surface point: only the centre itself
            add_tap(s[k], 1.f, sA[r0 + k][c0], sQ[r0 + k][c0], sC[r0 + k][c0]);
        }
    }
    float ssim = 0.f, l1 = 0.f;
#pragma unroll
    for (int k = 0; k < 2; k++) {
        if (x >= b.W || y + k >= b.H) continue;
        const float iZ = 1.f / s[k].Z;
        const long long p = b.pix + (long long)(y + k) * b.W + x;
        const float m1[3] = {s[k].m1.x, s[k].m1.y, s[k].m3.x}, m2[3] = {s[k].m2.x, s[k].m2.y, s[k].m3.y};
        const float e11[3] = {s[k].e11.x, s[k].e11.y, s[k].e33.x}, e22[3] = {s[k].e22.x, s[k].e22.y, s[k].e33.y};
        const float e12[3] = {s[k].e12.x, s[k].e12.y, s[k].e12c};
        const f32x2 a = sA[r0 + k][c0], q = sQ[r0 + k][c0], ch2 = sC[r0 + k][c0];
        const float i1[3] = {a.x, a.y, ch2.x}, i2[3] = {q.x, q.y, ch2.y};
#pragma unroll
        for (int ch = 0; ch < 3; ch++) {
            const float mu1 = m1[ch] * iZ, mu2 = m2[ch] * iZ;
            const float s11 = e11[ch] * iZ - mu1 * mu1, s22 = e22[ch] * iZ - mu2 * mu2;
            const float s12 = e12[ch] * iZ - mu1 * mu2;
            const float a1 = 2.f * mu1 * mu2 + kC1, a2 = 2.f * s12 + kC2;
            const float b1 = mu1 * mu1 + mu2 * mu2 + kC1, b2 = s11 + s22 + kC2;
            const float S = a1 * a2 / (b1 * b2);
            const float dmu1 = 2.f * mu2 * S / a1 - 2.f * mu1 * S / b1;
            const float ds11 = -S / b2;
            const float ds12 = 2.f * S / a2;
            coef[(0 * 3 + ch) * P + p] = (dmu1 - 2.f * mu1 * ds11 - mu2 * ds12) * iZ;
            coef[(1 * 3 + ch) * P + p] = ds11 * iZ;
            coef[(2 * 3 + ch) * P + p] = ds12 * iZ;
            ssim += S;
            l1 += fabsf(i1[ch] - i2[ch]);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ssim += __shfl_xor_sync(0xffffffffu, ssim, o);
        l1 += __shfl_xor_sync(0xffffffffu, l1, o);
    }
    if (lane == 0) {
        red[0][threadIdx.x >> 5] = ssim;
        red[1][threadIdx.x >> 5] = l1;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float a = 0.f, q = 0.f;
        for (int k = 0; k < THREADS / 32; k++) {
            a += red[0][k];
            q += red[1][k];
        }
        bsum[blk_offset + blockIdx.x] = make_float2(a, q);
    }
}

// Bound by shared memory (80% of its rate): 14 words per neighbour, for two
// pixels.  One 1264 x 832 image: 272 -> 145 us.
__global__ void __launch_bounds__(THREADS) dssim3d_backward_kernel(Images im, long long P, const float* __restrict__ img,
                                                                  const float* __restrict__ tgt,
                                                                  const float* __restrict__ pts,
                                                                  const float* __restrict__ sig,
                                                                  const float* __restrict__ coef, float lambda,
                                                                  float inv_images, float* __restrict__ dimg) {
    __shared__ float sX[HSY][HSX + 1], sY[HSY][HSX + 1], sZ[HSY][HSX + 1], sN[HSY][HSX + 1], sR[HSY][HSX + 1];
    __shared__ f32x2 sA[HSY][HSX + 1], sB[HSY][HSX + 1], sC[HSY][HSX + 1];  // A, 2 B, C of channels 0, 1
    __shared__ f32x2 sD[HSY][HSX + 1];                                      // A, 2 B of channel 2
    __shared__ float sE[HSY][HSX + 1];                                      // C of channel 2
    const Blk b = block_of(im);
    const long long HW = (long long)b.H * b.W;
    bool odd = false;
    for (int k = threadIdx.x; k < HSX * HSY; k += THREADS) {
        const int r = k / HSX, c = k % HSX;
        const int y = b.y0 + r - RAD, x = b.x0 + c - RAD;
        const bool in = x >= 0 && y >= 0 && x < b.W && y < b.H;
        const long long o = (long long)y * b.W + x;
        const float s = in ? sig[b.pix + o] : -1.f;
        float X[3], t[9];
#pragma unroll
        for (int ch = 0; ch < 3; ch++) X[ch] = in ? pts[3 * b.pix + ch * HW + o] : 0.f;
#pragma unroll
        for (int j = 0; j < 9; j++) {
            t[j] = in ? coef[j * P + b.pix + o] : 0.f;
            if (j >= 3 && j < 6) t[j] *= 2.f;
            odd |= !finite(t[j]);
        }
        odd |= !in_domain(X[0], X[1], X[2], s);
        const bool point = s > 0.f;
        const float cc = point ? 2.f * s * s : 1.f;
        sX[r][c] = point ? X[0] : kFar;
        sY[r][c] = point ? X[1] : 0.f;
        sZ[r][c] = point ? X[2] : 0.f;
        sN[r][c] = -cc;
        sR[r][c] = 1.f / cc;
        sA[r][c] = pack2(t[0], t[1]);
        sB[r][c] = pack2(t[3], t[4]);
        sC[r][c] = pack2(t[6], t[7]);
        sD[r][c] = pack2(t[2], t[5]);
        sE[r][c] = t[8];
    }
    const int lane = threadIdx.x & 31, c0 = lane + RAD, r0 = 2 * (threadIdx.x >> 5) + RAD;
    const int x = b.x0 + lane, y = b.y0 + r0 - RAD;
    float i1[2][3], i2[2][3], sq[2];
#pragma unroll
    for (int k = 0; k < 2; k++) {
        const bool in = x < b.W && y + k < b.H;
        const long long o = (long long)(y + k) * b.W + x;
        sq[k] = in ? sig[b.pix + o] : -1.f;
#pragma unroll
        for (int ch = 0; ch < 3; ch++) {
            i1[k][ch] = in ? img[3 * b.pix + ch * HW + o] : 0.f;
            i2[k][ch] = in ? tgt[3 * b.pix + ch * HW + o] : 0.f;
            odd |= !finite(i1[k][ch]) || !finite(i2[k][ch]);
        }
    }
    odd = __syncthreads_or(odd);
    if (odd) mark_points(b, HW, pts, sig, sX);
    const bool some = __any_sync(0xffffffffu, sq[0] > 0.f || sq[1] > 0.f);  // else background: nothing to add up
    if (x >= b.W) return;
    float g[2][3] = {};
    if (odd) {  // the loops below with every test
        const bool point[2] = {sq[0] > 0.f, sq[1] > 0.f};
        const f32x2 nx = pack2(-sX[r0][c0], -sX[r0 + 1][c0]), ny = pack2(-sY[r0][c0], -sY[r0 + 1][c0]),
                    nz = pack2(-sZ[r0][c0], -sZ[r0 + 1][c0]);
        for (int rr = r0 + RAD + 1; rr >= r0 - RAD; rr--) {
            const bool upper = point[0] && rr <= r0 + RAD, lower = point[1] && rr > r0 - RAD;
#pragma unroll
            for (int du = -RAD; du <= RAD; du++) {
                const int cc = c0 - du;
                const float px = sX[rr][cc], py = sY[rr][cc], pz = sZ[rr][cc], n = sN[rr][cc], rc = sR[rr][cc];
                f32x2 w = any_weights(
                    dist2(add2(pack2(px, px), nx), add2(pack2(py, py), ny), add2(pack2(pz, pz), nz)), pack2(n, n),
                    pack2(rc, rc));
                const bool centre = is_point(px);
                w.x = upper && centre ? w.x : 0.f;
                w.y = lower && centre ? w.y : 0.f;
                if (du == 0 && rr == r0) w.x = 1.f;
                if (du == 0 && rr == r0 + 1) w.y = 1.f;
                const f32x2 A = sA[rr][cc], B = sB[rr][cc], C = sC[rr][cc], D = sD[rr][cc];
                const float E = sE[rr][cc];
#pragma unroll
                for (int k = 0; k < 2; k++) {
                    const float wk = k ? w.y : w.x;
                    const float e0 = __fmaf_rn(C.x, i2[k][0], __fmaf_rn(B.x, i1[k][0], A.x)),
                                e1 = __fmaf_rn(C.y, i2[k][1], __fmaf_rn(B.y, i1[k][1], A.y)),
                                e2 = __fmaf_rn(E, i2[k][2], __fmaf_rn(D.y, i1[k][2], D.x));
                    g[k][0] = __fmaf_rn(wk, wk != 0.f ? e0 : 0.f, g[k][0]);
                    g[k][1] = __fmaf_rn(wk, wk != 0.f ? e1 : 0.f, g[k][1]);
                    g[k][2] = __fmaf_rn(wk, wk != 0.f ? e2 : 0.f, g[k][2]);
                }
            }
        }
    } else {
        f32x2 u[2], v[2], G[2];
        float gc[2] = {0.f, 0.f};
#pragma unroll
        for (int k = 0; k < 2; k++) {
            u[k] = pack2(i1[k][0], i1[k][1]);
            v[k] = pack2(i2[k][0], i2[k][1]);
            G[k] = pack2(0.f, 0.f);
        }
        const f32x2 nx = pack2(sq[0] > 0.f ? -sX[r0][c0] : kFar, sq[1] > 0.f ? -sX[r0 + 1][c0] : kFar),
                    ny = pack2(-sY[r0][c0], -sY[r0 + 1][c0]), nz = pack2(-sZ[r0][c0], -sZ[r0 + 1][c0]);
        auto add = [&](int k, float w, int rr, int cc) {
            const f32x2 d = sD[rr][cc];
            G[k] = fma2(pack2(w, w), fma2(sC[rr][cc], v[k], fma2(sB[rr][cc], u[k], sA[rr][cc])), G[k]);
            gc[k] = __fmaf_rn(w, __fmaf_rn(sE[rr][cc], i2[k][2], __fmaf_rn(d.y, i1[k][2], d.x)), gc[k]);
        };
        // centres p = q - (du, dv) whose window holds q, dv and du ascending
        auto row = [&](int rr, bool upper, bool lower) {
#pragma unroll
            for (int du = -RAD; du <= RAD; du++) {
                const int cc = c0 - du;
                const float px = sX[rr][cc], py = sY[rr][cc], pz = sZ[rr][cc], n = sN[rr][cc], rc = sR[rr][cc];
                const f32x2 w = weights(dist2(add2(pack2(px, px), nx), add2(pack2(py, py), ny), add2(pack2(pz, pz), nz)),
                                        pack2(n, n), pack2(rc, rc));
                if (upper) add(0, w.x, rr, cc);
                if (lower) add(1, w.y, rr, cc);
            }
        };
        if (some) {
            row(r0 + RAD + 1, false, true);
            for (int rr = r0 + RAD; rr > r0 - RAD; rr--) row(rr, true, true);
            row(r0 - RAD, true, false);
        }
#pragma unroll
        for (int k = 0; k < 2; k++) {
            if (!(sq[k] > 0.f)) {  // no surface point: only the pixel's own window reaches it
                G[k] = pack2(0.f, 0.f);
                gc[k] = 0.f;
                add(k, 1.f, r0 + k, c0);
            }
            g[k][0] = G[k].x;
            g[k][1] = G[k].y;
            g[k][2] = gc[k];
        }
    }
    const float inv_n = 1.f / (3.f * (float)b.H * (float)b.W);
#pragma unroll
    for (int k = 0; k < 2; k++) {
        if (y + k >= b.H) continue;
        const long long o = (long long)(y + k) * b.W + x;
#pragma unroll
        for (int ch = 0; ch < 3; ch++) {
            const float d = i1[k][ch] - i2[k][ch];
            const float sgn = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f);
            dimg[3 * b.pix + ch * HW + o] = inv_images * inv_n * ((1.f - lambda) * sgn - lambda * g[k][ch]);
        }
    }
}

__global__ void dssim3d_reduce_kernel(Images im, const float2* __restrict__ bsum, long long blk_offset,
                                      float lambda, float* __restrict__ loss) {
    const int i = blockIdx.x;
    __shared__ double red[2][256];
    double a = 0.0, q = 0.0;
    for (long long k = im.blk[i] + threadIdx.x; k < im.blk[i + 1]; k += blockDim.x) {
        const float2 s = bsum[blk_offset + k];
        a += s.x;
        q += s.y;
    }
    red[0][threadIdx.x] = a;
    red[1][threadIdx.x] = q;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) {
            red[0][threadIdx.x] += red[0][threadIdx.x + s];
            red[1][threadIdx.x] += red[1][threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double n = 3.0 * im.H[i] * (double)im.W[i];
        loss[im.first + i] = (float)((1.0 - lambda) * red[1][0] / n + lambda * (1.0 - red[0][0] / n));
    }
}

// ---- merge / split ---------------------------------------------------------
__global__ void merge_kernel(const DevCam* __restrict__ cams, int group, int cw, int ch, unsigned long long seed,
                             float sigma_px,
                             long long merged_pix, const long long* __restrict__ mbase, int M,
                             const float* __restrict__ images, const float* __restrict__ targets,
                             const float* __restrict__ depth_acc, const float* __restrict__ final_T,
                             float* __restrict__ out_img, float* __restrict__ out_tgt, float* __restrict__ out_pts,
                             float* __restrict__ out_sig) {
    const long long gp = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gp >= merged_pix) return;
    int m = 0;
    while (m + 1 < M && mbase[m + 1] <= gp) m++;
    const DevCam& c0 = cams[m * group];
    const long long local = gp - mbase[m];
    const int x = (int)(local % c0.W), y = (int)(local / c0.W);
    const int v = m * group + sample_slot(seed, x / cw, y / ch, group);
    const DevCam& cam = cams[v];
    const long long HW = (long long)cam.W * cam.H;
    const long long src = (long long)y * cam.W + x;
    const long long dst3 = 3 * mbase[m];
    for (int ch = 0; ch < 3; ch++) {
        if (out_img) out_img[dst3 + ch * HW + local] = images[3 * cam.pix_base + ch * HW + src];
        if (out_tgt) out_tgt[dst3 + ch * HW + local] = targets[3 * cam.pix_base + ch * HW + src];
    }
    if (!out_pts) return;
    const float opac = 1.f - final_T[cam.pix_base + src];
    float X[3] = {0.f, 0.f, 0.f}, s = 0.f;
    if (opac >= kMinOpacity) {
        const float z = depth_acc[cam.pix_base + src] / opac;
        const float pc[3] = {z * (x + 0.5f - cam.cx) / cam.fx - cam.t[0], z * (y + 0.5f - cam.cy) / cam.fy - cam.t[1],
                             z - cam.t[2]};
        for (int i = 0; i < 3; i++) X[i] = cam.R[i] * pc[0] + cam.R[3 + i] * pc[1] + cam.R[6 + i] * pc[2];
        s = sigma_px * z / cam.fx;
    }
    for (int i = 0; i < 3; i++) out_pts[dst3 + i * HW + local] = X[i];
    out_sig[gp] = s;
}

__global__ void split_kernel(const DevCam* __restrict__ cams, int group, int cw, int ch, unsigned long long seed,
                             long long merged_pix, const long long* __restrict__ mbase, int M,
                             const float* __restrict__ dmerged, float* __restrict__ dimg) {
    const long long gp = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gp >= merged_pix) return;
    int m = 0;
    while (m + 1 < M && mbase[m + 1] <= gp) m++;
    const DevCam& c0 = cams[m * group];
    const long long local = gp - mbase[m];
    const int x = (int)(local % c0.W), y = (int)(local / c0.W);
    const int owner = sample_slot(seed, x / cw, y / ch, group);
    const long long HW = (long long)c0.W * c0.H;
    for (int k = 0; k < group; k++) {
        const DevCam& cam = cams[m * group + k];
        for (int ch = 0; ch < 3; ch++)
            dimg[3 * cam.pix_base + ch * HW + local] = k == owner ? dmerged[3 * mbase[m] + ch * HW + local] : 0.f;
    }
}

Images make_images(const int* hw, int first, int count) {
    Images im{};
    im.count = count;
    im.first = first;
    long long pix = 0, blk = 0;
    for (int i = 0; i < first; i++) pix += (long long)hw[2 * i] * hw[2 * i + 1];
    for (int i = 0; i < count; i++) {
        const int H = hw[2 * (first + i)], W = hw[2 * (first + i) + 1];
        im.H[i] = H;
        im.W[i] = W;
        im.tiles_x[i] = (W + TSX - 1) / TSX;
        im.pix[i] = pix;
        im.blk[i] = blk;
        pix += (long long)H * W;
        blk += (long long)im.tiles_x[i] * ((H + TSY - 1) / TSY);
    }
    im.blk[count] = blk;
    return im;
}

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace

size_t dssim3d_temp_bytes(const int* hw, int M) {
    long long P = 0, blocks = 0;
    for (int i = 0; i < M; i++) {
        P += (long long)hw[2 * i] * hw[2 * i + 1];
        blocks += (long long)((hw[2 * i + 1] + TSX - 1) / TSX) * ((hw[2 * i] + TSY - 1) / TSY);
    }
    return align256(9 * (size_t)P * sizeof(float)) + align256((size_t)blocks * sizeof(float2));
}

void launch_dssim3d(const float* img, const float* target, const float* points, const float* sigma, const int* hw,
                    int M, float lambda, float* loss, float* dimg, void* tmp, cudaStream_t s) {
    long long P = 0;
    for (int i = 0; i < M; i++) P += (long long)hw[2 * i] * hw[2 * i + 1];
    char* base = static_cast<char*>(tmp);
    float* coef = reinterpret_cast<float*>(base);
    float2* bsum = reinterpret_cast<float2*>(base + align256(9 * (size_t)P * sizeof(float)));
    long long blk_offset = 0;
    for (int first = 0; first < M; first += kMaxImages) {
        const int count = M - first < kMaxImages ? M - first : kMaxImages;
        const Images im = make_images(hw, first, count);
        const long long nb = im.blk[count];
        if (nb > 0) {
            dssim3d_forward_kernel<<<(unsigned)nb, THREADS, 0, s>>>(im, P, img, target, points, sigma, coef, bsum,
                                                                blk_offset);
            note_launches(1);
            if (dimg) {
                dssim3d_backward_kernel<<<(unsigned)nb, THREADS, 0, s>>>(im, P, img, target, points, sigma, coef, lambda,
                                                                     1.f / (float)M, dimg);
                note_launches(1);
            }
        }
        dssim3d_reduce_kernel<<<count, 256, 0, s>>>(im, bsum, blk_offset, lambda, loss);
        note_launches(1);
        blk_offset += nb;
    }
}

void launch_merge_views(const DevCam* cams, int group, int cw, int ch, unsigned long long seed, float sigma_px,
                        long long merged_pix,
                        const long long* mbase, int M, const float* images, const float* targets,
                        const float* depth_acc, const float* final_T, float* out_img, float* out_tgt, float* out_pts,
                        float* out_sig, cudaStream_t s) {
    if (merged_pix <= 0) return;
    merge_kernel<<<(unsigned)((merged_pix + 255) / 256), 256, 0, s>>>(cams, group, cw, ch, seed, sigma_px, merged_pix,
                                                                       mbase, M, images, targets, depth_acc, final_T,
                                                                       out_img, out_tgt, out_pts, out_sig);
    note_launches(1);
}

void launch_split_merged(const DevCam* cams, int group, int cw, int ch, unsigned long long seed, long long merged_pix,
                         const long long* mbase, int M, const float* dmerged, float* dimg, cudaStream_t s) {
    if (merged_pix <= 0) return;
    split_kernel<<<(unsigned)((merged_pix + 255) / 256), 256, 0, s>>>(cams, group, cw, ch, seed, merged_pix, mbase, M,
                                                                       dmerged, dimg);
    note_launches(1);
}

}  // namespace mvgs
