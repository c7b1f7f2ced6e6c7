// Training-loop pieces around the rasterizer: the multi-view densification
// step (Sec. 5.2.2; supplement "Experiment details") and a fused Adam update.
//
// Densification decides every Gaussian on its own, in double precision from
// the float32 inputs (so the decision is exact and reproducible):
//   mean E_k = accum_E_k / denom (0 where denom = 0);
//   large    = max_i log_scale_i > log_dense_extent;
//   pruned   = logit < prune_logit (the opacity threshold, multiplied by the
//              views per iteration, in logit space);
//   split    = !pruned && large && mean E_1 >= split_threshold;
//   cloned   = !pruned && !large && mean E_2 >= clone_threshold;
// outputs, ordered by source Gaussian: none if pruned; two children if split
// (mean mu + R(q)(s * z_k) with the caller's standard normal samples z,
// log-scale - ln 1.6, the rest copied); the Gaussian and a copy if cloned;
// else the Gaussian.  Kind per output: 0 the Gaussian itself, 1 a copy, 2 a
// split child; carried per-Gaussian arrays (optimiser moments) are copied for
// kind 0 and zeroed for kinds 1 and 2.
//
// Adam (Kingma & Ba, ICLR 2015) with bias correction, one read and one write
// of parameter, gradient and both moments per element.
#include "kernels.h"

namespace mvgs {
namespace {

// Whether e / den >= threshold in double precision (0 / 0 and anything over a
// denominator that is not positive count as 0).  The quotient is taken in
// double only where float32 cannot tell: a double division is some twenty
// instructions of a pipe with a 64th of the float32 rate (the count pass over
// 1M Gaussians 52 -> 24 us).
__device__ __forceinline__ bool mean_reaches(float e, float den, double threshold) {
    if (!(den > 0.f)) return 0.0 >= threshold;
    const float q = e / den, t = (float)threshold, band = 1e-5f * fabsf(t);
    if (fabsf(q) > 1e-30f && fabsf(q) < 1e30f && fabsf(t) > 1e-30f && fabsf(t) < 1e30f) {
        if (q > t + band) return true;
        if (q < t - band) return false;
    }
    return (double)e / (double)den >= threshold;
}

__global__ void densify_count_kernel(DensifyArgs a, int* __restrict__ counts) {
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= a.n) return;
    const float den = a.denom[g];
    const float* ls = a.log_scales + 3 * g;
    const double mx = (double)fmaxf(ls[0], fmaxf(ls[1], ls[2]));
    const bool large = mx > a.log_dense_extent;
    const bool pruned = (double)a.logits[g] < a.prune_logit;
    const bool split = !pruned && large && mean_reaches(a.e1[g], den, a.split_threshold);
    const bool cloned = !pruned && !large && mean_reaches(a.e2[g], den, a.clone_threshold);
    counts[g] = pruned ? 0 : ((split || cloned) ? 2 : 1) | (split ? 4 : 0);
}

// counts carry the split bit (4) next to the output count (bits 0-1); the
// scan reads the count through the mask 3.  The SH rows are copied by
// copy_rows_kernel: a thread that writes its own 48-float row leaves every store
// of a warp spread over 32 rows (1M Gaussians at degree 3: 521 -> 111 us with it).
__global__ void densify_write_kernel(DensifyArgs a, const int* __restrict__ counts,
                                     const long long* __restrict__ off, DensifyOut o, uint32_t* __restrict__ map) {
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= a.n) return;
    const int c = counts[g];
    const int cnt = c & 3;
    if (cnt == 0) return;
    const bool split = (c & 4) != 0;
    const long long d0 = off[g];
    float q[4];
    float nq = 0.f;
    for (int i = 0; i < 4; i++) {
        q[i] = a.quats[4 * g + i];
        nq += q[i] * q[i];
    }
    const float inv = rsqrtf(nq);
    const float w = q[0] * inv, x = q[1] * inv, y = q[2] * inv, z = q[3] * inv;
    const float R[9] = {1.f - 2.f * (y * y + z * z), 2.f * (x * y - w * z), 2.f * (x * z + w * y),
                        2.f * (x * y + w * z), 1.f - 2.f * (x * x + z * z), 2.f * (y * z - w * x),
                        2.f * (x * z - w * y), 2.f * (y * z + w * x), 1.f - 2.f * (x * x + y * y)};
    for (int k = 0; k < cnt; k++) {
        const long long d = d0 + k;
        const int kind = split ? 2 : k;  // cloned: the Gaussian (0), then its copy (1)
        map[d] = (uint32_t)g;
        if (o.src) o.src[d] = g;
        if (o.kind) o.kind[d] = kind;
        for (int i = 0; i < 3; i++) {
            float m = a.means[3 * g + i];
            float l = a.log_scales[3 * g + i];
            if (split) {
                float off_i = 0.f;
                for (int j = 0; j < 3; j++)
                    off_i += R[3 * i + j] * (expf(a.log_scales[3 * g + j]) * a.normals[6 * g + 3 * k + j]);
                m += off_i;
                l -= kLogSplitDiv;
            }
            o.means[3 * d + i] = m;
            o.log_scales[3 * d + i] = l;
        }
        for (int i = 0; i < 4; i++) o.quats[4 * d + i] = a.quats[4 * g + i];
        o.logits[d] = a.logits[g];
    }
}

// Rows of `width` elements: out[d] = in[src[d]], or zeros where kind (when
// given) is not 0.  A block takes `rows` consecutive output rows and walks their
// elements together, so reads and writes are coalesced; the row of an element is
// a multiplication (inv = ceil(2^32 / width), exact while rows * width * width <
// 2^32) instead of a 64-bit division per element (ten moment arrays of 1M SH-3
// Gaussians: 817 -> 217 us).
constexpr int ROW_ELEMS = 4096;  // elements per block, about
template <class T, class I>
__global__ void __launch_bounds__(256) copy_rows_kernel(long long n_out, const I* __restrict__ src,
                                                        const int* __restrict__ kind, uint32_t width, uint32_t rows,
                                                        uint32_t inv, const T* __restrict__ in, T* __restrict__ out) {
    const long long d0 = (long long)blockIdx.x * rows;
    const uint32_t n = (uint32_t)(n_out - d0 < rows ? n_out - d0 : rows);
#pragma unroll 4
    for (uint32_t e = threadIdx.x; e < n * width; e += 256) {
        const uint32_t r = rows == 1 ? 0u : width == 1 ? e : __umulhi(e, inv);
        const long long d = d0 + r;
        T v{};
        if (!kind || kind[d] == 0) v = in[(size_t)src[d] * width + (e - r * width)];
        out[(size_t)d0 * width + e] = v;
    }
}

template <class I>
void copy_rows(long long n_out, const I* src, const int* kind, int width, const float* in, float* out, cudaStream_t s) {
    if (n_out <= 0) return;
    const bool vec = width % 4 == 0 && ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15) == 0;
    const uint32_t w = (uint32_t)(vec ? width / 4 : width);
    const uint32_t rows = w < ROW_ELEMS ? ROW_ELEMS / w : 1;
    const uint32_t inv = (uint32_t)(((1ull << 32) + w - 1) / w);
    const unsigned blocks = (unsigned)((n_out + rows - 1) / rows);
    if (vec)
        copy_rows_kernel<<<blocks, 256, 0, s>>>(n_out, src, kind, w, rows, inv, reinterpret_cast<const float4*>(in),
                                                reinterpret_cast<float4*>(out));
    else
        copy_rows_kernel<<<blocks, 256, 0, s>>>(n_out, src, kind, w, rows, inv, in, out);
    note_launches(1);
}

__global__ void adam_kernel(long long count, float* __restrict__ p, const float* __restrict__ g,
                            float* __restrict__ m, float* __restrict__ v, float lr, float b1, float b2, float eps,
                            float c1, float c2) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (long long)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        // p -= lr * (m / c1) / (sqrt(v / c2) + eps), c_k = 1 - beta_k^t
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

// The same update on float4 vectors (count4 = count / 4, all pointers 16-byte
// aligned); the caller handles a tail of count % 4 elements with adam_kernel.
__device__ __forceinline__ void adam1(float& p, float g, float& m, float& v, float lr, float b1, float b2, float eps,
                                      float c1, float c2) {
    m = b1 * m + (1.f - b1) * g;
    v = b2 * v + (1.f - b2) * g * g;
    p -= lr * (m / c1) / (sqrtf(v / c2) + eps);
}

__global__ void adam4_kernel(long long count4, float4* __restrict__ p, const float4* __restrict__ g,
                             float4* __restrict__ m, float4* __restrict__ v, float lr, float b1, float b2, float eps,
                             float c1, float c2) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count4;
         i += (long long)gridDim.x * blockDim.x) {
        float4 pp = p[i], mm = m[i], vv = v[i];
        const float4 gg = g[i];
        adam1(pp.x, gg.x, mm.x, vv.x, lr, b1, b2, eps, c1, c2);
        adam1(pp.y, gg.y, mm.y, vv.y, lr, b1, b2, eps, c1, c2);
        adam1(pp.z, gg.z, mm.z, vv.z, lr, b1, b2, eps, c1, c2);
        adam1(pp.w, gg.w, mm.w, vv.w, lr, b1, b2, eps, c1, c2);
        p[i] = pp;
        m[i] = mm;
        v[i] = vv;
    }
}

}  // namespace

namespace {
size_t align256(size_t x) { return (x + 255) / 256 * 256; }

// The scratch of one densification step: outputs per Gaussian, their offsets,
// the source of every output (at most two per Gaussian), the scan's.
struct DensifyTemp {
    size_t off, map, scan, bytes;
    explicit DensifyTemp(long long n) {
        const size_t m = (size_t)(n > 0 ? n : 1);
        off = align256(m * sizeof(int));
        map = off + align256((m + 1) * sizeof(long long));
        scan = map + align256(2 * m * sizeof(uint32_t));
        bytes = scan + scan_temp_bytes(m);
    }
};
}  // namespace

size_t densify_temp_bytes(long long n) { return DensifyTemp(n).bytes; }

// Pass 1: decisions and output offsets; returns the device pointer of the
// output count (off[n]).
const long long* launch_densify_plan(const DensifyArgs& a, void* tmp, cudaStream_t s) {
    const DensifyTemp T(a.n);
    char* base = static_cast<char*>(tmp);
    int* counts = reinterpret_cast<int*>(base);
    long long* off = reinterpret_cast<long long*>(base + T.off);
    if (a.n > 0) {
        densify_count_kernel<<<(unsigned)((a.n + 255) / 256), 256, 0, s>>>(a, counts);
        note_launches(1);
    }
    scan_masked_i32_to_i64(counts, 3, off, (uint64_t)a.n, base + T.scan, s);
    return off + a.n;
}

void launch_densify_write(const DensifyArgs& a, const DensifyOut& o, long long n_out, void* tmp, cudaStream_t s) {
    if (a.n <= 0) return;
    const DensifyTemp T(a.n);
    char* base = static_cast<char*>(tmp);
    uint32_t* map = reinterpret_cast<uint32_t*>(base + T.map);
    densify_write_kernel<<<(unsigned)((a.n + 255) / 256), 256, 0, s>>>(
        a, reinterpret_cast<const int*>(base), reinterpret_cast<const long long*>(base + T.off), o, map);
    note_launches(1);
    copy_rows(n_out, map, nullptr, a.nk, a.sh, o.sh, s);
}

void launch_carry(long long n_out, const long long* src, const int* kind, int width, const float* in, float* out,
                  cudaStream_t s) {
    copy_rows(n_out, src, kind, width, in, out, s);
}

void launch_adam(long long count, float* p, const float* g, float* m, float* v, float lr, float b1, float b2,
                 float eps, int step, cudaStream_t s) {
    if (count <= 0) return;
    const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    const bool aligned = ((reinterpret_cast<uintptr_t>(p) | reinterpret_cast<uintptr_t>(g) |
                           reinterpret_cast<uintptr_t>(m) | reinterpret_cast<uintptr_t>(v)) & 15) == 0;
    long long head = 0;
    if (aligned && count >= 4) {
        const long long c4 = count / 4;
        long long blocks = (c4 + 255) / 256;
        if (blocks > 152 * 8) blocks = 152 * 8;
        adam4_kernel<<<(unsigned)blocks, 256, 0, s>>>(c4, reinterpret_cast<float4*>(p),
                                                      reinterpret_cast<const float4*>(g),
                                                      reinterpret_cast<float4*>(m), reinterpret_cast<float4*>(v),
                                                      lr, b1, b2, eps, c1, c2);
        note_launches(1);
        head = 4 * c4;
    }
    if (head < count) {
        long long blocks = (count - head + 255) / 256;
        if (blocks > 152 * 16) blocks = 152 * 16;
        adam_kernel<<<(unsigned)blocks, 256, 0, s>>>(count - head, p + head, g + head, m + head, v + head, lr, b1,
                                                     b2, eps, c1, c2);
        note_launches(1);
    }
}

}  // namespace mvgs
