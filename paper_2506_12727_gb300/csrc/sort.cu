// Exclusive scans, stable LSD radix sort and the per-tile lists.
//
// The supplement ("Rasterization in multi-view training") sorts duplicated
// (tile, viewpoint, depth) keys so each (tile, view) list is depth ordered.
// Here the same lists are built without sorting the duplicated keys at all:
//   1. the visible records are sorted by depth (32-bit keys, one entry per
//      record);
//   2. in that order, one entry per (record, bin) is generated -- a bin is
//      8 x 8 tiles of one view, so a record has few of them -- and the entries
//      are sorted stably by bin (usually one 8-bit pass);
//   3. every chunk of a bin's entries is expanded to the bin's 64 tiles at
//      once: entry i covers tile t when bit t of its 64-bit coverage mask is
//      set, so transposing the masks of 32 entries gives each tile its part of
//      the list in depth order.  A first kernel counts per (chunk, tile), a
//      scan over the chunks gives every chunk its place in every tile's list,
//      and a second kernel writes the record ids there, in runs.
// Stability keeps depth order, and equal depths keep the record order, which
// is Gaussian-major, so ties inside a tile list are broken by Gaussian index.
#include <cstddef>

#include "../../include/mvgs.h"
#include "kernels.h"

namespace mvgs {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// Blocks of a launch that is sized by a capacity (capturable mode): they stride
// over what there is.  The tile lists' entries are a tenth of the key capacity
// that bounds them: at 3M Gaussians x 8 views the blocks without entries cost a
// captured step 0.64 ms (15.47 -> 14.83).  Kernels that the loop makes slower are
// variants of their own (STRIDE).
constexpr uint64_t GRID_CAP = 152 * 32;

// ---------------------------------------------------------------------------
// exclusive scan (reduce, spine, downsweep; fewer launches for fewer blocks)
// ---------------------------------------------------------------------------
constexpr int SC_THREADS = 256;
constexpr int SC_ITEMS = 16;
constexpr int SC_TILE = SC_THREADS * SC_ITEMS;
constexpr int SPINE_THREADS = 1024;

// Exclusive scan across the block of one value per thread.  `buf` holds
// at least 33 elements of shared memory.  Returns the thread's exclusive
// prefix and the block total.
template <class T>
__device__ __forceinline__ T block_exclusive_scan(T v, T* buf, T& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) buf[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        T w = lane < nw ? buf[lane] : T(0);
        T wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            T y = __shfl_up_sync(kFull, wi, o);
            if (lane >= o) wi += y;
        }
        buf[lane] = wi - w;
        if (lane == 31) buf[32] = wi;
    }
    __syncthreads();
    T res = inc - v + buf[warp];
    total = buf[32];
    __syncthreads();
    return res;
}

template <class Tin, class Tout>
struct LoadDirect {
    const Tin* in;
    __device__ __forceinline__ Tout operator()(uint64_t i) const { return (Tout)in[i]; }
};

struct LoadMasked {
    const int* in;
    int mask;
    __device__ __forceinline__ long long operator()(uint64_t i) const { return (long long)(in[i] & mask); }
};

template <class Load, class T>
__global__ void __launch_bounds__(SC_THREADS) scan_reduce_kernel(Load ld, Count cn, T* partials) {
    chained();
    __shared__ T buf[33];
    const uint64_t n = cn.get();
    const uint64_t base = (uint64_t)blockIdx.x * SC_TILE;
    T s = 0;
#pragma unroll 4
    for (int i = threadIdx.x; i < SC_TILE; i += SC_THREADS) {
        const uint64_t idx = base + i;
        if (idx < n) s += ld(idx);
    }
    T total;
    block_exclusive_scan<T>(s, buf, total);
    if (threadIdx.x == 0) partials[blockIdx.x] = total;
}

template <class T>
__global__ void __launch_bounds__(SPINE_THREADS) scan_spine_kernel(T* partials, uint64_t nb, T* end_out, Count cn) {
    chained();
    __shared__ T buf[33];
    T carry = 0;
    for (uint64_t start = 0; start < nb; start += SPINE_THREADS) {
        const uint64_t i = start + threadIdx.x;
        const T v = i < nb ? partials[i] : T(0);
        T tot;
        const T ex = block_exclusive_scan<T>(v, buf, tot);
        if (i < nb) partials[i] = ex + carry;
        carry += tot;
    }
    if (threadIdx.x == 0) end_out[cn.get()] = carry;
}

__device__ __forceinline__ int pad_index(int i) { return i + (i >> 5); }

// What the blocks before sum to: the scanned partials (SPINE), the sum of the
// raw ones (PARTIALS), or of their input read again (INPUT; not in place).
enum ScanBase { SPINE, PARTIALS, INPUT };

// (end_out is `out` again: as an argument of its own, 32 registers instead of 38,
// and 24M counts are scanned in 84 us instead of 99)
template <class Load, class T>
__global__ void __launch_bounds__(SC_THREADS) scan_down_kernel(Load ld, Count cn, ScanBase mode, const T* partials, T* out, T* end_out) {
    chained();
    __shared__ T tile[SC_TILE + SC_TILE / 32];
    __shared__ T buf[33];
    const uint64_t n = cn.get();
    const uint64_t base = (uint64_t)blockIdx.x * SC_TILE;
    for (int i = threadIdx.x; i < SC_TILE; i += SC_THREADS) {
        const uint64_t idx = base + i;
        tile[pad_index(i)] = idx < n ? ld(idx) : T(0);
    }
    __syncthreads();
    T local[SC_ITEMS];
    T sum = 0;
#pragma unroll
    for (int k = 0; k < SC_ITEMS; k++) {
        local[k] = tile[pad_index(threadIdx.x * SC_ITEMS + k)];
        sum += local[k];
    }
    T first = 0;
    if (mode == SPINE) {
        first = partials[blockIdx.x];
    } else {
        T before = 0;
        if (mode == PARTIALS) {
            for (unsigned i = threadIdx.x; i < blockIdx.x; i += SC_THREADS) before += partials[i];
        } else {
            const uint64_t end = base < n ? base : n;
#pragma unroll 8
            for (uint64_t i = threadIdx.x; i < end; i += SC_THREADS) before += ld(i);
        }
        block_exclusive_scan<T>(before, buf, first);
    }
    T total;
    T run = block_exclusive_scan<T>(sum, buf, total) + first;
    if (mode != SPINE && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) end_out[n] = first + total;
#pragma unroll
    for (int k = 0; k < SC_ITEMS; k++) {
        tile[pad_index(threadIdx.x * SC_ITEMS + k)] = run;
        run += local[k];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < SC_TILE; i += SC_THREADS) {
        const uint64_t idx = base + i;
        if (idx < n) out[idx] = tile[pad_index(i)];
    }
}

uint64_t ceil_div_u64(uint64_t a, uint64_t b) { return (a + b - 1) / b; }

// Exclusive scan of ld(0 .. n); the total goes to out[n].
template <class Load, class T>
void scan_impl(Load ld, T* out, Count n, void* tmp, cudaStream_t s) {
    if (n.max == 0) {
        cudaMemsetAsync(out, 0, sizeof(T), s);
        return;
    }
    const uint64_t nb = ceil_div_u64(n.max, SC_TILE);
    T* partials = static_cast<T*>(tmp);
    // A launch costs a dependent kernel some 3 us: up to 5 blocks sum what
    // lies before them from the input, up to 1024 from the blocks' sums.
    const ScanBase mode = nb <= 5 ? INPUT : nb <= 1024 ? PARTIALS : SPINE;
    if (mode != INPUT) {
        launch_chained(scan_reduce_kernel<Load, T>, (unsigned)nb, SC_THREADS, 0, s, ld, n, partials);
        note_launches(1);
    }
    if (mode == SPINE) {
        launch_chained(scan_spine_kernel<T>, 1, SPINE_THREADS, 0, s, partials, nb, out, n);
        note_launches(1);
    }
    launch_chained(scan_down_kernel<Load, T>, (unsigned)nb, SC_THREADS, 0, s, ld, n, mode, partials, out, out);
    note_launches(1);
}

// ---------------------------------------------------------------------------
// stable LSD radix sort of (uint32 key, uint32 value), 8-bit digits
// ---------------------------------------------------------------------------
// A pass is a histogram per block, a scan per digit over the blocks and the
// scatter: three launches instead of five (the scan over the digits is the
// scatter's own), two when there are few blocks.  Bound by the scatter: 16
// ballot rounds per key in the ranking, then runs of about 16 keys.  Sort of the
// depths: 22M (3M Gaussians x 8 views) 0.93 -> 0.61 ms, 500k 138 -> 57 us, 10k
// 118 -> 42 us, with three passes for four where their range allows it (below
// 2^24 apart: the farthest up to about four times as far as the nearest).
// Digits of 9 bits, three passes for 27 bits, took 0.77 ms at 22M keys against
// 0.74 with four passes, and as long at 2M.
constexpr int RS_THREADS = 256;  // == number of digit values
constexpr int RS_ITEMS = 16;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_SEG = RS_ITEMS * 32;  // contiguous keys per warp
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;
// Blocks up to which the scatter sums the histograms itself: at 64 blocks its
// loads take 1 us more than reading a scanned table, the scan 2 us and a launch.
constexpr uint64_t RS_DIRECT = 64;

// The histograms of a pass: per digit over the blocks (direct false: scanned
// in place, totals beside) or per block over the digits (direct true).
struct RadixTable {
    uint32_t* counts;
    uint32_t* totals;
    bool direct;
};

// Blocks of n keys.  A launch sized by a capacity has at most GRID_CAP blocks,
// which go on to further ones of the actual count.
__device__ __forceinline__ uint32_t rs_blocks(uint64_t n) { return (uint32_t)((n + RS_TILE - 1) / RS_TILE); }

struct RankSmem {
    uint32_t whist[RS_WARPS * 256];  // per-warp digit counts, then per-warp prefixes
    uint32_t boff[256];              // first output position of each digit of the block
    uint32_t dstart[256];            // first block-local position of each digit
    unsigned long long scan_buf[33];
    uint32_t skeys[RS_TILE];         // keys in block-local sorted order
    uint32_t svals[RS_TILE];         // values in block-local sorted order
};

// Keys of the thread's digit in all blocks and in the blocks before.
__device__ __forceinline__ void digit_counts(const RadixTable& tab, uint32_t nblocks, uint32_t block, uint32_t& tot,
                                             uint32_t& pre) {
    if (tab.direct) {
        tot = pre = 0;
#pragma unroll 8
        for (uint32_t b = 0; b < nblocks; b++) {
            const uint32_t c = tab.counts[b * 256 + threadIdx.x];
            if (b < block) pre += c;
            tot += c;
        }
    } else {
        pre = tab.counts[(uint64_t)threadIdx.x * nblocks + block];
        tot = tab.totals[threadIdx.x];
    }
}

// Per-block digit histogram.  sub (optional): subtracted from every key.
template <bool STRIDE>
__global__ void __launch_bounds__(RS_THREADS) rs_upsweep(const uint32_t* keys, Count cn, int shift,
                                                        const unsigned long long* sub, RadixTable tab) {
    chained();
    __shared__ uint32_t hist[RS_WARPS * 256];
    const uint64_t n = cn.get();
    const uint32_t nblocks = rs_blocks(n);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t k0 = sub ? (uint32_t)*sub : 0u;
    uint32_t block = blockIdx.x;
    if (block >= nblocks) return;
    do {
        const uint64_t base = (uint64_t)block * RS_TILE + warp * RS_SEG + lane;
        uint32_t k[RS_ITEMS];
#pragma unroll
        for (int j = 0; j < RS_ITEMS; j++) k[j] = base + (uint64_t)j * 32 < n ? keys[base + (uint64_t)j * 32] : 0u;
        for (int i = threadIdx.x; i < RS_WARPS * 256; i += RS_THREADS) hist[i] = 0;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < RS_ITEMS; j++)
            if (base + (uint64_t)j * 32 < n) atomicAdd(&hist[warp * 256 + (((k[j] - k0) >> shift) & 0xffu)], 1u);
        __syncthreads();
        uint32_t sum = 0;
#pragma unroll
        for (int w = 0; w < RS_WARPS; w++) sum += hist[w * 256 + threadIdx.x];
        if (tab.direct) tab.counts[(uint64_t)block * 256 + threadIdx.x] = sum;
        else tab.counts[(uint64_t)threadIdx.x * nblocks + block] = sum;
        if (STRIDE) __syncthreads();
    } while (STRIDE && (block += gridDim.x) < nblocks);
}

// The same table for a pass whose digits take at most 32 values (few bins, or
// the bin ids' high bits): each lane counts into its
// own column of a per-warp table (digit-major, lane-minor: a lane's updates
// hit its own bank, and are plain read-modify-writes, not atomics, since no
// other lane touches the column), then a skewed sweep sums the columns.
// Shared-memory atomics from 32 lanes on a handful of digits serialise.
__global__ void __launch_bounds__(RS_THREADS) rs_upsweep_narrow(const uint32_t* keys, Count cn, int shift,
                                                               uint32_t mask, RadixTable tab) {
    chained();
    __shared__ uint32_t cnt[RS_WARPS][32 * 32];
    __shared__ uint32_t wsum[RS_WARPS][32];
    const uint64_t n = cn.get();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t* c = cnt[warp];
    const uint32_t nblocks = rs_blocks(n);
    for (uint32_t block = blockIdx.x; block < nblocks; block += gridDim.x) {
        for (int i = lane; i < 32 * 32; i += 32) c[i] = 0;
        __syncwarp();
        const uint64_t base = (uint64_t)block * RS_TILE + warp * RS_SEG + lane;
#pragma unroll
        for (int j = 0; j < RS_ITEMS; j++) {
            const uint64_t idx = base + (uint64_t)j * 32;
            if (idx < n) c[((keys[idx] >> shift) & mask) * 32 + lane] += 1u;
        }
        __syncwarp();
        // lane d sums digit d's column, starting at a different lane per digit
        uint32_t sum = 0;
#pragma unroll 8
        for (int i = 0; i < 32; i++) sum += c[lane * 32 + ((i + lane) & 31)];
        wsum[warp][lane] = sum;
        __syncthreads();
        uint32_t total = 0;
        if (threadIdx.x < 32) {
#pragma unroll
            for (int w = 0; w < RS_WARPS; w++) total += wsum[w][threadIdx.x];
        }
        if (tab.direct) tab.counts[(uint64_t)block * 256 + threadIdx.x] = total;
        else tab.counts[(uint64_t)threadIdx.x * nblocks + block] = total;
        __syncthreads();
    }
}

// One block per digit: its counts become the number of its keys in the blocks
// before, and their sum its total.  A warp takes a stretch of the blocks.
__global__ void __launch_bounds__(RS_THREADS) rs_scan_kernel(RadixTable tab, Count cn) {
    chained();
    __shared__ uint32_t buf[33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t nblocks = rs_blocks(cn.get());
    uint32_t* row = tab.counts + (uint64_t)blockIdx.x * nblocks;
    const uint32_t per = (nblocks + RS_THREADS - 1) / RS_THREADS * 32;
    const uint32_t r0 = min(warp * per, nblocks), r1 = min(r0 + per, nblocks);
    uint32_t sum = 0;
#pragma unroll 4
    for (uint32_t r = r0 + lane; r < r1; r += 32) sum += row[r];
    uint32_t total;
    const uint32_t ex = block_exclusive_scan<uint32_t>(sum, buf, total);
    uint32_t run = __shfl_sync(kFull, ex, 0);
#pragma unroll 4
    for (uint32_t r = r0; r < r1; r += 32) {
        const uint32_t v = r + lane < r1 ? row[r + lane] : 0u;
        uint32_t inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, inc, o);
            if (lane >= o) inc += y;
        }
        if (r + lane < r1) row[r + lane] = run + inc - v;
        run += __shfl_sync(kFull, inc, 31);
    }
    if (threadIdx.x == 0) tab.totals[blockIdx.x] = total;
}

// Stable rank of the block's keys (held in registers, warp w owning the
// contiguous segment [w*SEG, (w+1)*SEG) in rounds of 32 lanes) and scatter:
// first into shared memory in block-local digit order, then to global memory
// in runs of consecutive positions per digit.  Equal digits inside a round are
// found with one ballot per digit bit.  Values are fetched after the ranking,
// so they do not occupy registers during it.
// NB: significant bits of this pass's digit.  vin == nullptr: the values are
// the keys' positions (an identity permutation, generated instead of read).
// sub: subtracted from every key (the keys written are the differences).
// gout != nullptr: also writes gout[pos] = gsrc[value] (a per-element array
// carried into sorted order).  STRIDE: a launch sized by a capacity; a variant of
// its own because the loop costs registers that spill.
template <bool WRITE_KEYS, int NB, bool STRIDE>
__global__ void __launch_bounds__(RS_THREADS, 3) rs_downsweep(const uint32_t* kin,
                                                             const uint32_t* vin,
                                                             uint32_t* kout, uint32_t* vout,
                                                             Count cn, int shift,
                                                             const unsigned long long* sub, RadixTable tab,
                                                             const uint32_t* gsrc = nullptr,
                                                             uint32_t* gout = nullptr) {
    chained();
    __shared__ RankSmem sm;
    const uint64_t n = cn.get();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t nblocks = rs_blocks(n);
    const uint32_t k0 = sub ? (uint32_t)*sub : 0u;
    uint32_t block = blockIdx.x;
    if (block >= nblocks) return;
    do {
        const uint64_t block0 = (uint64_t)block * RS_TILE;
        const int here = (int)(n - block0 < (uint64_t)RS_TILE ? n - block0 : (uint64_t)RS_TILE);
        const int local0 = warp * RS_SEG + lane;
        for (int i = threadIdx.x; i < RS_WARPS * 256; i += RS_THREADS) sm.whist[i] = 0;
        const uint32_t* in = kin + block0;
        uint32_t k[RS_ITEMS];
#pragma unroll
        for (int j = 0; j < RS_ITEMS; j++) k[j] = (local0 + j * 32 < here ? in[local0 + j * 32] : 0u) - k0;
        uint32_t tot, pre;
        digit_counts(tab, nblocks, block, tot, pre);
        __syncthreads();
        uint32_t* wh = sm.whist + warp * 256;
        uint32_t lr[RS_ITEMS];
#pragma unroll
        for (int j = 0; j < RS_ITEMS; j++) {
            const bool ok = local0 + j * 32 < here;
            const uint32_t d = (k[j] >> shift) & 0xffu;
            uint32_t peers = __ballot_sync(kFull, ok);
#pragma unroll
            for (int b = 0; b < NB; b++) {  // digit bits above NB are zero in this pass
                const uint32_t bit = (d >> b) & 1u;
                const uint32_t bb = __ballot_sync(kFull, bit);
                peers &= bit ? bb : ~bb;
            }
            const uint32_t rank = __popc(peers & lt);
            const uint32_t before = wh[d];
            __syncwarp();
            if (ok && rank == 0) wh[d] = before + __popc(peers);
            __syncwarp();
            lr[j] = before + rank;
        }
        uint32_t vv[RS_ITEMS];
#pragma unroll
        for (int j = 0; j < RS_ITEMS; j++)
            vv[j] = !vin ? (uint32_t)block0 + local0 + j * 32 : local0 + j * 32 < here ? vin[block0 + local0 + j * 32] : 0u;
        __syncthreads();
        uint32_t run = 0;
#pragma unroll
        for (int w = 0; w < RS_WARPS; w++) {
            const uint32_t c = sm.whist[w * 256 + threadIdx.x];
            sm.whist[w * 256 + threadIdx.x] = run;
            run += c;
        }
        // both prefixes over the digits in one scan: of the totals (high words) and
        // of the block's counts
        unsigned long long all;
        const unsigned long long at =
            block_exclusive_scan<unsigned long long>((unsigned long long)tot << 32 | run, sm.scan_buf, all);
        sm.dstart[threadIdx.x] = (uint32_t)at;
        sm.boff[threadIdx.x] = (uint32_t)(at >> 32) + pre;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < RS_ITEMS; j++) {
            if (local0 + j * 32 < here) {
                const uint32_t d = (k[j] >> shift) & 0xffu;
                const uint32_t lp = sm.dstart[d] + wh[d] + lr[j];
                sm.skeys[lp] = k[j];
                sm.svals[lp] = vv[j];
            }
        }
        __syncthreads();
        // four at a time: no carried value's fetch waits behind a store
        for (int i0 = threadIdx.x; i0 < here; i0 += 4 * RS_THREADS) {
            uint32_t carried[4] = {0u, 0u, 0u, 0u};
            if (gout) {
#pragma unroll
                for (int q = 0; q < 4; q++)
                    if (i0 + q * RS_THREADS < here) carried[q] = gsrc[sm.svals[i0 + q * RS_THREADS]];
            }
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int i = i0 + q * RS_THREADS;
                if (i >= here) break;
                const uint32_t key = sm.skeys[i];
                const uint32_t d = (key >> shift) & 0xffu;
                const uint32_t pos = sm.boff[d] + (uint32_t)i - sm.dstart[d];
                vout[pos] = sm.svals[i];
                if (WRITE_KEYS) kout[pos] = key;
                if (gout) gout[pos] = carried[q];
            }
        }
        if (STRIDE) __syncthreads();
    } while (STRIDE && (block += gridDim.x) < nblocks);
}

// ---------------------------------------------------------------------------
// per-tile lists through bins of 8 x 8 tiles
// ---------------------------------------------------------------------------
// Sorting one entry per (record, tile) moved 28 bytes per entry (generation,
// histogram, two radix passes).  Here only the (record, bin) entries are
// sorted -- about 1.7 per record at 32 x 64 tiles and 4 at 16 x 16, against 14
// and 58 tiles -- and the record id of a (record, tile) pair is written once,
// straight into its tile's list.  Bound by the random descriptor fetches of
// the entries and the 4 bytes written per (record, tile) pair.  Tile sort with
// ranges, radix sort of all pairs -> bins: 3M Gaussians x 8 views at 32 x 64
// tiles (340M pairs, 41M entries) 4.83 -> 1.64 ms; 1M x 16 views at 16 x 64
// (236M pairs) 3.83 -> 1.21 ms; 500k x 4 views at 16 x 16 (116M pairs, 8M
// entries) 1.81 -> 0.44 ms; 500k x 1 view at 16 x 16 0.49 -> 0.17 ms; 20k x 3
// small views 0.115 -> 0.097 ms.  Bins of 64 tiles because a coverage mask then
// is two words and a warp transposes 32 of them in ten shuffles.
//
// Sort key of an entry: the bin id above 12 bits holding the part of the
// record's rectangle inside the bin (x0, y0, x1, y1 inclusive, 3 bits each),
// so the expansion needs no record fetch.  With more than 2^20 bins (LOCAL
// false) the key is the bin id alone and the expansion clips the record's
// rectangle again.
constexpr int BIN_LOCAL_BITS = 12;
constexpr long long BIN_LOCAL_MAX = 1LL << (32 - BIN_LOCAL_BITS);
constexpr int BC_THREADS = 256;
constexpr int BC_WARPS = BC_THREADS / 32;
constexpr int BC_CHUNK = 1024;            // entries of one bin expanded together
constexpr int BC_GROUPS = BC_CHUNK / 32;  // groups of 32 entries, one lane per group when a list is placed
static_assert(BC_GROUPS == 32, "one lane per group");

// The part of rectangle rc inside bin (bx, by), packed as in the sort key.
__device__ __forceinline__ uint32_t clip_to_bin(short4 rc, int bx, int by) {
    const int x0 = max(rc.x - 8 * bx, 0), x1 = min(rc.z - 1 - 8 * bx, 7);
    const int y0 = max(rc.y - 8 * by, 0), y1 = min(rc.w - 1 - 8 * by, 7);
    return (uint32_t)(x0 | y0 << 3 | x1 << 6 | y1 << 9);
}

// Coverage mask over the bin's tiles (bit 8 y + x) of a packed local rectangle.
__device__ __forceinline__ uint2 bin_mask(uint32_t l) {
    const int x0 = l & 7, y0 = (l >> 3) & 7, x1 = (l >> 6) & 7, y1 = (l >> 9) & 7;
    const uint32_t rep = ((0xffu >> (7 - x1)) & (0xffu << x0)) * 0x01010101u;
    const unsigned long long rows = (~0ull >> (8 * (7 - y1))) & (~0ull << (8 * y0));
    return make_uint2(rep & (uint32_t)rows, rep & (uint32_t)(rows >> 32));
}

__device__ __forceinline__ int find_bin_view(const DevCam* cams, int V, long long bin) {
    int lo = 0, hi = V - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (cams[mid].bin_base <= bin) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// One entry per (record, bin), in depth order; off is the exclusive scan of
// the records' bin counts in that order.  A warp takes 32 records and walks
// their entries 32 at a time (each lane finds its entry's record by a search
// over the warp's offsets), so the stores are coalesced however uneven the
// records' counts are.  The bins' bounds are zeroed on the way.  32-bit offsets:
// 22M records (3M Gaussians x 8 views) are scanned in 80 us instead of 147 and
// read here in 376 us with the descriptors, 394 before; the descriptors' random
// 32-byte sectors are most of that.
template <bool LOCAL>
__global__ void __launch_bounds__(256) bin_entries_kernel(const uint32_t* order,
                                                          const uint32_t* off, Count Rc,
                                                          Count Sc, const unsigned long long* desc,
                                                          const DevCam* cams,
                                                          uint32_t* keys, uint32_t* vals,
                                                          uint32_t* zero, long long zero_count) {
    chained();
    const uint64_t R = Rc.get(), S = Sc.get();
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (long long k = (long long)i; k < zero_count; k += (long long)gridDim.x * blockDim.x) zero[k] = 0;
    const int lane = threadIdx.x & 31;
    const uint64_t w0 = i - lane;
    if (w0 >= R) return;  // the whole warp
    const uint64_t r = i < R ? i : R;
    const uint32_t o = off[r];
    const uint32_t first = __shfl_sync(kFull, o, 0);
    const uint32_t total = off[w0 + 32 < R ? w0 + 32 : R] - first;
    uint32_t rec = 0, b0 = 0;
    int bxs = 1;
    float inv = 1.f;  // 1 / (bins across the record)
    unsigned long long d = 0;
    if (i < R) {
        rec = order[i];
        d = desc[rec];
        const short4 rc = tile_desc_rect(d);
        const DevCam& c = cams[tile_desc_view(d)];
        bxs = bins_across(c.tiles_x);
        b0 = (uint32_t)(c.bin_base + (long long)(rc.y >> 3) * bxs + (rc.x >> 3));
        inv = 1.f / (float)max(((rc.z - 1) >> 3) - (rc.x >> 3) + 1, 1);
    }
    const uint32_t rel = o - first;
    for (uint32_t j0 = 0; j0 < total; j0 += 32) {
        const uint32_t j = j0 + lane;
        // the last record starting at or before entry j (records without
        // bins share the next one's offset)
        int src = 0;
#pragma unroll
        for (int step = 16; step > 0; step >>= 1) {
            const uint32_t v = __shfl_sync(kFull, rel, src + step);
            if (v <= j) src += step;
        }
        const uint32_t k = j - __shfl_sync(kFull, rel, src);
        const unsigned long long ds = __shfl_sync(kFull, d, src);
        const uint32_t recs = __shfl_sync(kFull, rec, src), b0s = __shfl_sync(kFull, b0, src);
        const int bxss = __shfl_sync(kFull, bxs, src);
        const short4 rc = tile_desc_rect(ds);
        const int bx0 = rc.x >> 3, by0 = rc.y >> 3;
        const int w = max(((rc.z - 1) >> 3) - bx0 + 1, 1);
        // k / w: k < 2^18 (512 x 512 bins per view), so (k + 1/2) / w is 1 / (2 w) or
        // more from an integer and the float32 product off by less than 1 / (16 w)
        const int ty = (int)(((float)k + 0.5f) * __shfl_sync(kFull, inv, src)), tx = (int)k - ty * w;
        const uint32_t bin = b0s + (uint32_t)ty * (uint32_t)bxss + (uint32_t)tx;
        if (j < total && (uint64_t)first + j < S) {
            keys[first + j] = LOCAL ? bin << BIN_LOCAL_BITS | clip_to_bin(rc, bx0 + tx, by0 + ty) : bin;
            vals[first + j] = recs;
        }
    }
}

// First and one past the last position of every bin's entries (zeroed before:
// a bin without entries keeps an empty range).
template <bool STRIDE>
__global__ void __launch_bounds__(256) bin_bounds_kernel(const uint32_t* keys, Count Sc, int shift,
                                                         uint32_t* begin, uint32_t* end) {
    chained();
    const uint64_t S = Sc.get();
    uint64_t i0 = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4;
    if (i0 >= S) return;
    do {
        uint32_t b[6];
        b[0] = i0 > 0 ? keys[i0 - 1] >> shift : 0xffffffffu;
#pragma unroll
        for (int q = 1; q < 6; q++) b[q] = i0 + q - 1 < S ? keys[i0 + q - 1] >> shift : 0xffffffffu;
#pragma unroll
        for (int q = 1; q < 5; q++) {
            const uint64_t i = i0 + q - 1;
            if (i >= S) break;
            if (i == 0 || b[q] != b[q - 1]) begin[b[q]] = (uint32_t)i;
            if (i + 1 == S || b[q] != b[q + 1]) end[b[q]] = (uint32_t)i + 1;
        }
    } while (STRIDE && (i0 += (uint64_t)gridDim.x * 1024) < S);
}

// First chunk of every bin (one block; bins that no entry touches have none).
// A single bin holds all S entries.
__global__ void __launch_bounds__(SPINE_THREADS) bin_chunks_kernel(uint32_t* begin,
                                                                   uint32_t* end, Count Sc, long long bins,
                                                                   uint32_t* chunk_off) {
    chained();
    __shared__ uint32_t buf[33];
    if (bins == 1) {
        if (threadIdx.x == 0) {
            const uint32_t S = (uint32_t)Sc.get();
            begin[0] = 0;
            end[0] = S;
            chunk_off[0] = 0;
            chunk_off[1] = S / BC_CHUNK + (S % BC_CHUNK != 0);
        }
        return;
    }
    uint32_t carry = 0;
    for (long long base = 0; base < bins; base += SPINE_THREADS) {
        const long long b = base + threadIdx.x;
        const uint32_t len = b < bins ? end[b] - begin[b] : 0u;
        uint32_t total;
        const uint32_t ex = block_exclusive_scan<uint32_t>(len / BC_CHUNK + (len % BC_CHUNK != 0), buf, total);
        if (b < bins) chunk_off[b] = carry + ex;
        carry += total;
    }
    if (threadIdx.x == 0) chunk_off[bins] = carry;
}

// The bin of chunk c: the last one whose first chunk is c or earlier (a warp
// narrows the range 32-fold per step).
__device__ __forceinline__ uint32_t bin_of_chunk(const uint32_t* chunk_off, uint32_t bins, uint32_t c, int lane) {
    uint32_t lo = 0, hi = bins;
    while (hi - lo > 1) {
        const uint32_t step = (hi - lo + 31) / 32, at = lo + (uint32_t)lane * step;
        const uint32_t n = __popc(__ballot_sync(kFull, at < hi && chunk_off[at] <= c));
        lo += (n - 1) * step;
        hi = lo + step < hi ? lo + step : hi;
    }
    return lo;
}

// 32 x 32 bit transpose over the warp: bit r of lane t's result is bit t of
// lane r's word.
__device__ __forceinline__ uint32_t warp_transpose(uint32_t x, int lane) {
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) {
        const uint32_t m = j == 16 ? 0x0000ffffu : j == 8 ? 0x00ff00ffu : j == 4 ? 0x0f0f0f0fu
                                               : j == 2 ? 0x33333333u : 0x55555555u;
        const uint32_t y = __shfl_xor_sync(kFull, x, j);
        x = lane & j ? (x & ~m) | ((y & ~m) >> j) : (x & m) | ((y & m) << j);
    }
    return x;
}

struct BinLists {
    const uint32_t* keys;              // entries sorted by bin
    const uint32_t* vals;              // their record ids
    const unsigned long long* desc;    // tile descriptors (LOCAL false only)
    const uint32_t* begin;             // [bins] the bin's entries: [begin, end)
    const uint32_t* end;
    const uint32_t* chunk_off;         // [bins + 1] first chunk of every bin
    uint32_t* chunk_bin;               // [chunks]
    uint32_t* counts;                  // [chunks, 64] entries per tile, then the entries of the chunks before
    uint32_t bins;
};

// Coverage mask of entry p (clipped to bin (bx, by) when the key does not hold it).
template <bool LOCAL>
__device__ __forceinline__ uint2 entry_mask(const BinLists& L, uint64_t p, int bx, int by) {
    if (LOCAL) return bin_mask(L.keys[p]);
    return bin_mask(clip_to_bin(tile_desc_rect(L.desc[L.vals[p]]), bx, by));
}

// Entries per tile of every chunk.
template <bool LOCAL>
__global__ void __launch_bounds__(BC_THREADS) bin_count_kernel(BinLists L, const DevCam* cams, int V) {
    chained();
    __shared__ uint32_t part[BC_WARPS][64];
    const uint32_t chunks = L.chunk_off[L.bins];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (uint32_t c = blockIdx.x; c < chunks; c += gridDim.x) {
        const uint32_t b = bin_of_chunk(L.chunk_off, L.bins, c, lane);
        const uint32_t p0 = L.begin[b] + (c - L.chunk_off[b]) * BC_CHUNK;
        const uint32_t cnt = min(L.end[b] - p0, (uint32_t)BC_CHUNK);
        int bx = 0, by = 0;
        if (!LOCAL) {
            const DevCam& cam = cams[find_bin_view(cams, V, b)];
            const long long lb = (long long)b - cam.bin_base;
            bx = (int)(lb % bins_across(cam.tiles_x));
            by = (int)(lb / bins_across(cam.tiles_x));
        }
        uint32_t lo = 0, hi = 0;
#pragma unroll
        for (int q = 0; q < BC_GROUPS / BC_WARPS; q++) {
            const uint32_t e = (warp * (BC_GROUPS / BC_WARPS) + q) * 32 + lane;
            const uint2 m = e < cnt ? entry_mask<LOCAL>(L, (uint64_t)p0 + e, bx, by) : make_uint2(0u, 0u);
            lo += __popc(warp_transpose(m.x, lane));
            hi += __popc(warp_transpose(m.y, lane));
        }
        part[warp][lane] = lo;
        part[warp][32 + lane] = hi;
        if (threadIdx.x == 0) L.chunk_bin[c] = b;
        __syncthreads();
        if (threadIdx.x < 64) {
            uint32_t sum = 0;
#pragma unroll
            for (int w = 0; w < BC_WARPS; w++) sum += part[w][threadIdx.x];
            L.counts[(uint64_t)c * 64 + threadIdx.x] = sum;
        }
        __syncthreads();
    }
}

// One block per bin: every chunk's counts become the number of entries in the
// chunks before it, tile by tile, and the totals the tiles' list lengths.
constexpr int BS_PARTS = 8;  // stretches of chunks scanned side by side
__global__ void __launch_bounds__(64 * BS_PARTS) bin_scan_kernel(BinLists L, const DevCam* cams, int V,
                                                                 uint32_t* tile_counts) {
    chained();
    __shared__ uint32_t sums[BS_PARTS][64];
    const uint32_t b = blockIdx.x;
    const int t = threadIdx.x & 63, part = threadIdx.x >> 6;
    const uint32_t c0 = L.chunk_off[b], n = L.chunk_off[b + 1] - c0;
    const uint32_t per = (n + BS_PARTS - 1) / BS_PARTS;
    const uint32_t r0 = min(part * per, n), r1 = min(r0 + per, n);
    uint32_t* row = L.counts + (uint64_t)c0 * 64 + t;
    uint32_t sum = 0;
#pragma unroll 8
    for (uint32_t r = r0; r < r1; r++) sum += row[(uint64_t)r * 64];
    sums[part][t] = sum;
    __syncthreads();
    uint32_t run = 0;
    for (int q = 0; q < part; q++) run += sums[q][t];
#pragma unroll 8
    for (uint32_t r = r0; r < r1; r++) {
        const uint32_t v = row[(uint64_t)r * 64];
        row[(uint64_t)r * 64] = run;
        run += v;
    }
    if (part == BS_PARTS - 1) {
        const DevCam& cam = cams[find_bin_view(cams, V, b)];
        const int lb = (int)((long long)b - cam.bin_base), across = bins_across(cam.tiles_x);
        const int tx = (lb % across) * 8 + (t & 7), ty = (lb / across) * 8 + (t >> 3);
        if (tx < cam.tiles_x && ty < cam.tiles_y)
            tile_counts[cam.tile_base + (long long)ty * cam.tiles_x + tx] = run;
    }
}

// Writes every chunk's record ids into the tiles' lists.  A warp takes one
// tile at a time: lane g holds the tile's coverage word of the chunk's group g
// (32 entries), a warp scan of the popcounts gives each lane its part of the
// run, the set bits are compacted in shared memory and the run is stored by
// consecutive lanes.
template <bool LOCAL, bool STRIDE>
__global__ void __launch_bounds__(BC_THREADS) bin_place_kernel(BinLists L, const DevCam* cams, int V,
                                                               const long long* ranges, Count Kc, uint32_t* sorted) {
    chained();
    __shared__ uint32_t words[64][BC_GROUPS + 1];
    __shared__ uint32_t recs[BC_CHUNK];
    __shared__ uint32_t first[64];
    __shared__ uint16_t stage[BC_WARPS][BC_CHUNK];
    // nothing is placed when the lists do not fit (capturable mode)
    const uint32_t chunks = Kc.over() ? 0u : L.chunk_off[L.bins];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t c = blockIdx.x;
    if (c >= chunks) return;
    do {
        const uint32_t b = L.chunk_bin[c];
        const uint32_t p0 = L.begin[b] + (c - L.chunk_off[b]) * BC_CHUNK;
        const uint32_t cnt = min(L.end[b] - p0, (uint32_t)BC_CHUNK);
        const DevCam& cam = cams[find_bin_view(cams, V, b)];
        const int lb = (int)((long long)b - cam.bin_base), across = bins_across(cam.tiles_x);
        const int bx = lb % across, by = lb / across;
        if (threadIdx.x < 64) {
            const int tx = bx * 8 + (threadIdx.x & 7), ty = by * 8 + (threadIdx.x >> 3);
            first[threadIdx.x] = tx < cam.tiles_x && ty < cam.tiles_y
                                     ? (uint32_t)ranges[2 * (cam.tile_base + (long long)ty * cam.tiles_x + tx)] +
                                           L.counts[(uint64_t)c * 64 + threadIdx.x]
                                     : 0u;
        }
#pragma unroll
        for (int q = 0; q < BC_GROUPS / BC_WARPS; q++) {
            const int g = warp * (BC_GROUPS / BC_WARPS) + q;
            const uint32_t e = g * 32 + lane;
            uint2 m = make_uint2(0u, 0u);
            if (e < cnt) {
                m = entry_mask<LOCAL>(L, (uint64_t)p0 + e, bx, by);
                recs[e] = L.vals[(uint64_t)p0 + e];
            }
            words[lane][g] = warp_transpose(m.x, lane);
            words[32 + lane][g] = warp_transpose(m.y, lane);
        }
        __syncthreads();
        uint16_t* st = stage[warp];
        for (int t = warp; t < 64; t += BC_WARPS) {
            uint32_t word = words[t][lane];
            const uint32_t n = __popc(word);
            uint32_t inc = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(kFull, inc, o);
                if (lane >= o) inc += y;
            }
            const uint32_t all = __shfl_sync(kFull, inc, 31);
            if (all == 0) continue;
            uint32_t at = inc - n;
            while (word) {
                st[at++] = (uint16_t)(lane * 32 + __ffs(word) - 1);
                word &= word - 1;
            }
            __syncwarp();
            uint32_t* out = sorted + first[t];
            for (uint32_t j = lane; j < all; j += 32) out[j] = recs[st[j]];
            __syncwarp();
        }
        if (STRIDE) __syncthreads();
    } while (STRIDE && (c += gridDim.x) < chunks);
}

// Blend processing order: tiles by decreasing list length, in 256 length
// classes (8 per octave: the exponent and three mantissa bits of length + 1),
// tile id order inside a class; the persistent blend kernels take the longest
// lists first so that no heavy tile is left for the end of the queue.  One
// block sorts all tiles by counting in shared memory (one launch instead of a
// radix sort's ten).
constexpr int TO_THREADS = 1024;
constexpr int TO_WARPS = TO_THREADS / 32;

__device__ __forceinline__ uint32_t length_class(long long len) {
    const unsigned long long v = (unsigned long long)(len > 0 ? len : 0) + 1ull;
    const int e = 63 - __clzll((long long)v);
    const uint32_t m = e >= 3 ? (uint32_t)(v >> (e - 3)) & 7u : (uint32_t)(v << (3 - e)) & 7u;
    const uint32_t b = 8u * (uint32_t)e + m;  // grows with the length
    return 255u - (b < 255u ? b : 255u);      // 0: the longest lists
}

__global__ void __launch_bounds__(TO_THREADS) tile_order_kernel(const long long* ranges, long long tiles,
                                                                uint32_t* order) {
    chained();
    __shared__ uint32_t off[256];                // per class: next output position
    __shared__ uint32_t wcnt[TO_WARPS][256];     // per warp and class, within a chunk
    __shared__ uint32_t buf[33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    auto cls = [&](long long t) { return length_class(ranges[2 * t + 1] - ranges[2 * t]); };
    if (threadIdx.x < 256) off[threadIdx.x] = 0;
    __syncthreads();
    for (long long t = threadIdx.x; t < tiles; t += TO_THREADS) atomicAdd(&off[cls(t)], 1u);
    __syncthreads();
    uint32_t total;
    const uint32_t c0 = threadIdx.x < 256 ? off[threadIdx.x] : 0u;
    const uint32_t ex = block_exclusive_scan<uint32_t>(c0, buf, total);
    if (threadIdx.x < 256) off[threadIdx.x] = ex;
    __syncthreads();
    // stable scatter, chunk by chunk in tile order: rank inside the warp by
    // matching classes, then add the counts of the warps before
    uint32_t next = threadIdx.x < tiles ? cls(threadIdx.x) : 256u;
    for (long long base = 0; base < tiles; base += TO_THREADS) {
        const long long t = base + threadIdx.x;
        const bool valid = t < tiles;
        const uint32_t c = next;
        next = t + TO_THREADS < tiles ? cls(t + TO_THREADS) : 256u;  // read ahead of this chunk's stores
        const uint32_t peers = __match_any_sync(kFull, c);
        for (int i = lane; i < 256; i += 32) wcnt[warp][i] = 0;
        __syncwarp();
        if (valid && (peers & lt) == 0) wcnt[warp][c] = (uint32_t)__popc(peers);
        __syncthreads();
        if (threadIdx.x < 256) {
            uint32_t run = off[threadIdx.x];
            for (int w = 0; w < TO_WARPS; w++) {
                const uint32_t n = wcnt[w][threadIdx.x];
                wcnt[w][threadIdx.x] = run;
                run += n;
            }
            off[threadIdx.x] = run;
        }
        __syncthreads();
        if (valid) {
            const uint32_t pos = wcnt[warp][c] + (uint32_t)__popc(peers & lt);
            if ((long long)pos < tiles) order[pos] = (uint32_t)t;
        }
        __syncthreads();
    }
}

// [start, end) of every tile's list.  All lists are empty when they need more
// entries than there is room for (a capturable call that ran out of key
// capacity: nothing is placed then, so no range may point at the array).  The
// needed count decides, not the starts: those are of the (record, bin) entries
// that were kept, which may fill the room exactly.
__global__ void ranges_kernel(const unsigned long long* starts, long long tiles, Count Kc,
                              long long* ranges) {
    chained();
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= tiles) return;
    const bool fits = !Kc.over();
    ranges[2 * t] = fits ? (long long)starts[t] : 0;
    ranges[2 * t + 1] = fits ? (long long)starts[t + 1] : 0;
}

}  // namespace

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
size_t scan_temp_bytes(uint64_t n) { return (ceil_div_u64(n, SC_TILE) + 1) * sizeof(unsigned long long); }

void scan_i32_to_i64(const int* in, long long* out, uint64_t n, void* tmp, cudaStream_t s) {
    scan_impl(LoadDirect<int, long long>{in}, out, n, tmp, s);
}

void scan_masked_i32_to_i64(const int* in, int mask, long long* out, uint64_t n, void* tmp, cudaStream_t s) {
    scan_impl(LoadMasked{in, mask}, out, n, tmp, s);
}

void scan_u32_to_u64(const uint32_t* in, unsigned long long* out, uint64_t n, void* tmp, cudaStream_t s) {
    scan_impl(LoadDirect<uint32_t, unsigned long long>{in}, out, n, tmp, s);
}

void scan_u32(const uint32_t* in, uint32_t* out, Count n, void* tmp, cudaStream_t s) {
    scan_impl(LoadDirect<uint32_t, uint32_t>{in}, out, n, tmp, s);
}

static uint64_t radix_blocks(uint64_t n) { return ceil_div_u64(n, RS_TILE); }

size_t radix_temp_bytes(uint64_t n) { return (radix_blocks(n > 0 ? n : 1) + 1) * 256 * sizeof(uint32_t); }

namespace {
// One radix pass over the 8 bits from `shift` up; the keys' bits from
// shift + bits up are zero.
void radix_pass(const uint32_t* kin, const uint32_t* vin, uint32_t* kout, uint32_t* vout, Count n, int shift, int bits,
                bool write_keys, const unsigned long long* sub, void* tmp, cudaStream_t s,
                const uint32_t* gsrc = nullptr, uint32_t* gout = nullptr) {
    const uint64_t nb64 = radix_blocks(n.max);
    const unsigned nb = (unsigned)(n.dev && nb64 > GRID_CAP ? GRID_CAP : nb64);
    uint32_t* totals = static_cast<uint32_t*>(tmp);
    const RadixTable tab{totals + 256, totals, nb64 <= RS_DIRECT};
    if (bits <= 5 && !sub) launch_chained(rs_upsweep_narrow, nb, RS_THREADS, 0, s, kin, n, shift, (1u << bits) - 1u, tab);
    else if (nb < nb64) launch_chained(rs_upsweep<true>, nb, RS_THREADS, 0, s, kin, n, shift, sub, tab);
    else launch_chained(rs_upsweep<false>, nb, RS_THREADS, 0, s, kin, n, shift, sub, tab);
    if (!tab.direct) {
        launch_chained(rs_scan_kernel, 256, RS_THREADS, 0, s, tab, n);
        note_launches(1);
    }
#define MVGS_DOWN2(W, B, T) \
    launch_chained(rs_downsweep<W, B, T>, nb, RS_THREADS, 0, s, kin, vin, kout, vout, n, shift, sub, tab, gsrc, gout)
#define MVGS_DOWN(W, B) (nb < nb64 ? (MVGS_DOWN2(W, B, true)) : (MVGS_DOWN2(W, B, false)))
    if (bits <= 5 && !sub && write_keys) MVGS_DOWN(true, 5);
    else if (write_keys) MVGS_DOWN(true, 8);
    else MVGS_DOWN(false, 8);
#undef MVGS_DOWN
#undef MVGS_DOWN2
    note_launches(2);
}
}  // namespace

void radix_sort_ids(const uint32_t* keys, const unsigned long long* sub, uint32_t* keys_a, uint32_t* vals_a,
                    uint32_t* keys_b, uint32_t* vals_b, uint32_t* vals_out, Count n, int bits, void* tmp,
                    cudaStream_t s, const uint32_t* gather_src, uint32_t* gather_out) {
    if (n.max == 0) return;
    const int passes = (bits + 7) / 8 > 0 ? (bits + 7) / 8 : 1;
    const uint32_t* kin = keys;
    const uint32_t* vin = nullptr;
    for (int p = 0; p < passes; p++) {
        const bool last = p == passes - 1;
        uint32_t* kout = (p & 1) ? keys_a : keys_b;
        uint32_t* vout = last ? vals_out : ((p & 1) ? vals_a : vals_b);
        radix_pass(kin, vin, kout, vout, n, 8 * p, bits - 8 * p, !last, p == 0 ? sub : nullptr, tmp, s,
                   last ? gather_src : nullptr, last ? gather_out : nullptr);
        kin = kout;
        vin = vout;
    }
}

namespace {
uint64_t bin_chunks(uint64_t S, long long bins) { return S / BC_CHUNK + (uint64_t)bins; }
size_t round256(size_t x) { return (x + 255) / 256 * 256; }

// The scratch of the tile lists inside one buffer.
struct BinTemp {
    size_t begin, end, chunk_off, chunk_bin, counts, tile_counts, starts, scan, bytes;
    BinTemp(uint64_t S, long long bins, long long tiles) {
        size_t o = 0;
        auto take = [&](size_t n) { const size_t at = o; o += round256(n); return at; };
        const uint64_t chunks = bin_chunks(S, bins);
        begin = take((size_t)bins * sizeof(uint32_t));
        end = take((size_t)bins * sizeof(uint32_t));
        chunk_off = take((size_t)(bins + 1) * sizeof(uint32_t));
        chunk_bin = take(chunks * sizeof(uint32_t));
        counts = take(chunks * 64 * sizeof(uint32_t));
        tile_counts = take((size_t)tiles * sizeof(uint32_t));
        starts = take((size_t)(tiles + 1) * sizeof(unsigned long long));
        scan = take(scan_temp_bytes((uint64_t)tiles));
        bytes = o;
    }
};

template <class T>
T* part(void* tmp, size_t off) { return reinterpret_cast<T*>(static_cast<char*>(tmp) + off); }
}  // namespace

size_t tile_lists_temp_bytes(uint64_t S, long long bins, long long tiles) { return BinTemp(S, bins, tiles).bytes; }

bool tile_lists_keep_desc(long long bins) { return bins > BIN_LOCAL_MAX; }

void tile_lists(const uint32_t* order, const uint32_t* bin_off, Count R, Count S, Count K,
                const unsigned long long* desc, const DevCam* cams, int V, long long bins, long long tiles,
                uint32_t* keys_a, uint32_t* vals_a, uint32_t* keys_b, uint32_t* vals_b, uint32_t* sorted,
                long long* ranges, uint64_t S_cap, void* tmp, void* radix_tmp, cudaStream_t s) {
    const BinTemp T(S_cap, bins, tiles);
    uint32_t* tile_counts = part<uint32_t>(tmp, T.tile_counts);
    unsigned long long* starts = part<unsigned long long>(tmp, T.starts);
    const bool any = S.max > 0 && R.max > 0;
    const bool local = !tile_lists_keep_desc(bins);
    BinLists L{};
    const auto grid = [&](uint64_t blocks) { return (unsigned)(S.dev && blocks > GRID_CAP ? GRID_CAP : blocks); };
    const unsigned chunks = grid(bin_chunks(S.max, bins));
    if (!any) {
        cudaMemsetAsync(tile_counts, 0, (size_t)tiles * sizeof(uint32_t), s);
    } else {
        StageTimer timer(MVGS_STAGE_TILE_SORT, s);
        uint32_t *kin = keys_a, *vin = vals_a, *kout = keys_b, *vout = vals_b;
        const unsigned rblocks = (unsigned)ceil_div_u64(R.max, 256);
        uint32_t* begin = part<uint32_t>(tmp, T.begin);
        uint32_t* end = part<uint32_t>(tmp, T.end);
        const long long zeroed = bins > 1 ? (long long)((T.chunk_off - T.begin) / sizeof(uint32_t)) : 0;  // begin and end
        if (local) launch_chained(bin_entries_kernel<true>, rblocks, 256, 0, s, order, bin_off, R, S, desc, cams, kin, vin,
                                  begin, zeroed);
        else launch_chained(bin_entries_kernel<false>, rblocks, 256, 0, s, order, bin_off, R, S, desc, cams, kin, vin,
                                  begin, zeroed);
        const int low = local ? BIN_LOCAL_BITS : 0;
        int bits = 0;
        while ((1LL << bits) < bins) bits++;
        for (int p = 0; 8 * p < bits; p++) {
            radix_pass(kin, vin, kout, vout, S, low + 8 * p, bits - 8 * p, true, nullptr, radix_tmp, s);
            uint32_t *nk = kin, *nv = vin;
            kin = kout;
            vin = vout;
            kout = nk;
            vout = nv;
        }
        uint32_t* chunk_off = part<uint32_t>(tmp, T.chunk_off);
        L = BinLists{kin, vin, desc, begin, end, chunk_off, part<uint32_t>(tmp, T.chunk_bin),
                     part<uint32_t>(tmp, T.counts), (uint32_t)bins};
        if (bins > 1) {
            const uint64_t blocks = ceil_div_u64(S.max, 1024);
            if (grid(blocks) < blocks) launch_chained(bin_bounds_kernel<true>, grid(blocks), 256, 0, s, kin, S, low, begin, end);
            else launch_chained(bin_bounds_kernel<false>, grid(blocks), 256, 0, s, kin, S, low, begin, end);
            note_launches(1);
        }
        launch_chained(bin_chunks_kernel, 1, SPINE_THREADS, 0, s, begin, end, S, bins, chunk_off);
        if (local) launch_chained(bin_count_kernel<true>, chunks, BC_THREADS, 0, s, L, cams, V);
        else launch_chained(bin_count_kernel<false>, chunks, BC_THREADS, 0, s, L, cams, V);
        launch_chained(bin_scan_kernel, (unsigned)bins, 64 * BS_PARTS, 0, s, L, cams, V, tile_counts);
        note_launches(4);
    }
    {
        StageTimer timer(MVGS_STAGE_RANGES, s);
        scan_u32_to_u64(tile_counts, starts, (uint64_t)tiles, part<void>(tmp, T.scan), s);
        launch_chained(ranges_kernel, (unsigned)ceil_div_u64((uint64_t)tiles, 256), 256, 0, s, starts, tiles, K, ranges);
        note_launches(1);
    }
    if (any) {
        StageTimer timer(MVGS_STAGE_TILE_SORT, s);
#define MVGS_PLACE(L_, T) \
    launch_chained(bin_place_kernel<L_, T>, chunks, BC_THREADS, 0, s, L, cams, V, ranges, K, sorted)
        const bool stride = chunks < bin_chunks(S.max, bins);
        if (local) stride ? (MVGS_PLACE(true, true)) : (MVGS_PLACE(true, false));
        else stride ? (MVGS_PLACE(false, true)) : (MVGS_PLACE(false, false));
#undef MVGS_PLACE
        note_launches(1);
    }
}

void tile_order(const long long* ranges, long long tiles, uint32_t* order, cudaStream_t s) {
    if (tiles <= 0) return;
    launch_chained(tile_order_kernel, 1, TO_THREADS, 0, s, ranges, tiles, order);
    note_launches(1);
}

}  // namespace mvgs
