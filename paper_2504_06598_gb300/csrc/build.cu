// build.cu -- hierarchy construction over the Gaussians' bounding boxes
// (Sec. 3.2 builds a BVH over the boxes of Eq. 2; the paper delegates it to
// Embree/OptiX, here it is a linear BVH built on the GPU):
//   k_preprocess  box of each Gaussian's bounding ellipsoid + scene bounds
//   k_morton      63-bit key: Morton code of each mean in the scene bounds
//                 with a size class of the Gaussian's box below the top
//                 two octree levels
//   k_radix_pass  stable LSD sort of (code, id), 8 digits of 8 bits, one
//                 pass over the keys each
//   k_karras      binary radix tree over the sorted codes (Karras 2012),
//                 equal codes split by position
//   k_leaves      per-Gaussian record in tree order, then bottom-up box
//                 refit with one arrival counter per node; cuts the wide
//                 hierarchies on the way
//   k_wide_*      records of the 8- and 32-wide hierarchies
#include <cuda_runtime.h>
#include <math.h>

#include "gsrt_internal.cuh"

namespace gsrt {
namespace {

constexpr int kSortThreads = 256;
constexpr int kSortItems = 8;
constexpr int kSortTile = kSortThreads * kSortItems;
constexpr int kSortPasses = 8;  // 8-bit digits of a 64-bit key

// Order-preserving map float -> uint32 (for atomicMax; a minimum is kept as
// the maximum of the complement, so that zero starts both).
__device__ __forceinline__ unsigned int f2ord(float f) {
    unsigned int u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord2f(unsigned int u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

struct Activated {
    float mu[3];
    float opacity;
    float R[9];  // R_q, local to world, row-major
    float inv_s[3];
    float s[3];
    bool finite;
};

// Eq. 1 activation in float32: normalised quaternion -> rotation,
// exp of log-scales, sigmoid of the opacity logit.
__device__ __forceinline__ Activated activate(const float *means, const float *log_scales,
                                              const float *quats, const float *logits,
                                              int64_t g) {
    Activated a;
    float qw = quats[4 * g + 0], qx = quats[4 * g + 1], qy = quats[4 * g + 2],
          qz = quats[4 * g + 3];
    float n2 = qw * qw + qx * qx + qy * qy + qz * qz;
    float inv = 1.0f / sqrtf(n2);
    qw *= inv; qx *= inv; qy *= inv; qz *= inv;
    a.R[0] = 1.0f - 2.0f * (qy * qy + qz * qz);
    a.R[1] = 2.0f * (qx * qy - qw * qz);
    a.R[2] = 2.0f * (qx * qz + qw * qy);
    a.R[3] = 2.0f * (qx * qy + qw * qz);
    a.R[4] = 1.0f - 2.0f * (qx * qx + qz * qz);
    a.R[5] = 2.0f * (qy * qz - qw * qx);
    a.R[6] = 2.0f * (qx * qz - qw * qy);
    a.R[7] = 2.0f * (qy * qz + qw * qx);
    a.R[8] = 1.0f - 2.0f * (qx * qx + qy * qy);
    bool fin = isfinite(n2) && n2 > 0.0f;
    for (int k = 0; k < 3; ++k) {
        float ls = log_scales[3 * g + k];
        a.mu[k] = means[3 * g + k];
        a.s[k] = expf(ls);
        a.inv_s[k] = expf(-ls);
        fin = fin && isfinite(ls) && isfinite(a.mu[k]) && a.s[k] > 0.0f && isfinite(a.s[k]) &&
              isfinite(a.inv_s[k]);
    }
    float lg = logits[g];
    fin = fin && isfinite(lg);
    a.opacity = 1.0f / (1.0f + expf(-lg));
    a.finite = fin;
    return a;
}

// Box of the ellipsoid |S^-1 R_q^T (x - mu)| <= s: half extent along world
// axis i is s * sqrt(sum_k R_ik^2 s_k^2). Padded outward (relative 2^-10 of
// the extent plus 2^-18 of the coordinate magnitude) so that float32
// rounding in the ellipsoid and slab tests never loses a valid hit.
__device__ __forceinline__ void ellipsoid_box(const Activated &a, float box[6]) {
    const float s_cut = 2.8284271247461903f;
    for (int i = 0; i < 3; ++i) {
        float v = 0.0f;
        for (int k = 0; k < 3; ++k) {
            float r = a.R[3 * i + k] * a.s[k];
            v = fmaf(r, r, v);
        }
        float h = s_cut * sqrtf(v);
        float pad = h * 0x1p-10f + (fabsf(a.mu[i]) + h) * 0x1p-18f;
        box[i] = a.mu[i] - (h + pad);
        box[3 + i] = a.mu[i] + (h + pad);
    }
}

// Box of Gaussian g into aabb; a finite mean widens lo and hi.
__device__ __forceinline__ void gaussian_box(int64_t g, const float *means, const float *log_scales,
                                             const float *quats, const float *logits,
                                             float *__restrict__ aabb, uint32_t *status,
                                             float lo[3], float hi[3]) {
    const Activated a = activate(means, log_scales, quats, logits, g);
    float box[6];
    if (a.finite) {
        ellipsoid_box(a, box);
        for (int k = 0; k < 3; ++k) {
            lo[k] = fminf(lo[k], a.mu[k]);
            hi[k] = fmaxf(hi[k], a.mu[k]);
        }
    } else {
        // A non-finite Gaussian gets an empty box: it is never hit.
        for (int k = 0; k < 3; ++k) {
            box[k] = NAN;
            box[3 + k] = NAN;
        }
        atomicOr(status, kErrNonfinite);
    }
    for (int k = 0; k < 6; ++k) aabb[6 * g + k] = box[k];
}

__global__ void __launch_bounds__(256) k_preprocess(int64_t M, const float *__restrict__ means,
                             const float *__restrict__ log_scales, const float *__restrict__ quats,
                             const float *__restrict__ logits, float *__restrict__ aabb,
                             unsigned int *__restrict__ bounds, uint32_t *__restrict__ status) {
    int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    if (g < M) gaussian_box(g, means, log_scales, quats, logits, aabb, status, lo, hi);
    // reduction of the finite means over the block, then six atomics: one per
    // warp made the kernel wait on its six addresses (1M: 131 us)
    __shared__ float s_lo[3][8], s_hi[3][8];
    for (int k = 0; k < 3; ++k) {
        for (int off = 16; off > 0; off >>= 1) {
            lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], off));
            hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], off));
        }
        if ((threadIdx.x & 31) == 0) {
            s_lo[k][threadIdx.x >> 5] = lo[k];
            s_hi[k][threadIdx.x >> 5] = hi[k];
        }
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        const int k = threadIdx.x;
        float l = INFINITY, h = -INFINITY;
        for (int w = 0; w < 8; ++w) {
            l = fminf(l, s_lo[k][w]);
            h = fmaxf(h, s_hi[k][w]);
        }
        if (l <= h) {
            atomicMax(&bounds[k], ~f2ord(l));
            atomicMax(&bounds[3 + k], f2ord(h));
        }
    }
}

// Spread the low 21 bits of v to every third bit of a 64-bit word.
__device__ __forceinline__ unsigned long long spread3(unsigned long long v) {
    v &= 0x1fffffull;
    v = (v | (v << 32)) & 0x1f00000000ffffull;
    v = (v | (v << 16)) & 0x1f0000ff0000ffull;
    v = (v | (v << 8)) & 0x100f00f00f00f00full;
    v = (v | (v << 4)) & 0x10c30c30c30c30c3ull;
    v = (v | (v << 2)) & 0x1249249249249249ull;
    return v;
}

// Sort key of one Gaussian: its 63-bit Morton code with a 4-bit size class
// inserted below the top two octree levels (6 bits). Gaussians of very
// different extent then fall into different subtrees below the coarse
// spatial split, so a few large Gaussians no longer inflate the boxes of
// the many small ones around them. Size class = floor(-2 log2(e / E)),
// clamped to 0..15, with e the largest box edge of the Gaussian and E the
// largest edge of the bounds of the means (large Gaussians sort first).
constexpr int kKeyTopBits = 6;
constexpr int kKeySizeBits = 4;

__device__ __forceinline__ unsigned long long sort_code(int64_t g, const float *means,
                                                        const unsigned int *bounds,
                                                        const float *aabb) {
    unsigned long long q[3];
    float scene = 0.0f, edge = 0.0f;
    for (int k = 0; k < 3; ++k) {
        float lo = ord2f(~bounds[k]), hi = ord2f(bounds[3 + k]);
        float ext = hi - lo;
        scene = fmaxf(scene, ext);
        edge = fmaxf(edge, aabb[6 * g + 3 + k] - aabb[6 * g + k]);
        float x = means[3 * g + k];
        float u = (ext > 0.0f) ? (x - lo) / ext : 0.0f;
        u = fminf(fmaxf(u, 0.0f), 1.0f);  // NaN -> 0
        q[k] = (unsigned long long)(u * 2097151.0f);
    }
    const unsigned long long morton = (spread3(q[0]) << 2) | (spread3(q[1]) << 1) | spread3(q[2]);
    int cls = 0;
    if (scene > 0.0f && edge > 0.0f) {
        const float c = floorf(-2.0f * log2f(edge / scene));
        cls = (int)fminf(fmaxf(c, 0.0f), (float)((1 << kKeySizeBits) - 1));
    }
    const int low = 63 - kKeyTopBits - kKeySizeBits;
    const unsigned long long top = morton >> (63 - kKeyTopBits);
    const unsigned long long rest = (morton & ((1ull << (63 - kKeyTopBits)) - 1ull)) >> kKeySizeBits;
    return (top << (63 - kKeyTopBits)) | ((unsigned long long)cls << low) | rest;
}

// Codes and ids, and the histograms of every sort digit (kSortTile codes a
// block).
__global__ void __launch_bounds__(kSortThreads)
    k_morton(int64_t M, const float *__restrict__ means, const unsigned int *__restrict__ bounds,
             const float *__restrict__ aabb, unsigned long long *__restrict__ codes,
             uint32_t *__restrict__ vals, uint32_t *__restrict__ hist) {
    __shared__ uint32_t h[kSortPasses][256];
    for (int p = 0; p < kSortPasses; ++p) h[p][threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kSortTile;
    for (int r = 0; r < kSortItems; ++r) {
        const int64_t g = base + r * kSortThreads + threadIdx.x;
        if (g >= M) break;
        const unsigned long long c = sort_code(g, means, bounds, aabb);
        codes[g] = c;
        vals[g] = (uint32_t)g;
        for (int p = 0; p < kSortPasses; ++p) atomicAdd(&h[p][(uint32_t)(c >> (8 * p)) & 255u], 1u);
    }
    __syncthreads();
    for (int p = 0; p < kSortPasses; ++p) {
        const uint32_t v = h[p][threadIdx.x];
        if (v) atomicAdd(&hist[256 * p + threadIdx.x], v);
    }
}

// ---------------------------------------------------------------- radix sort

// Histograms of the digits of bits [8 * first, 64) (n below 2^32).
__global__ void __launch_bounds__(kSortThreads)
    k_radix_hist(int64_t n, const unsigned long long *__restrict__ keys, int first,
                 uint32_t *__restrict__ hist) {
    __shared__ uint32_t h[kSortPasses][256];
    for (int p = 0; p < kSortPasses; ++p) h[p][threadIdx.x] = 0;
    __syncthreads();
    const int64_t step = (int64_t)gridDim.x * kSortThreads;
    for (int64_t i = (int64_t)blockIdx.x * kSortThreads + threadIdx.x; i < n; i += step) {
        const unsigned long long c = keys[i];
        for (int p = first; p < kSortPasses; ++p)
            atomicAdd(&h[p][(uint32_t)(c >> (8 * p)) & 255u], 1u);
    }
    __syncthreads();
    for (int p = first; p < kSortPasses; ++p) {
        const uint32_t v = h[p][threadIdx.x];
        if (v) atomicAdd(&hist[256 * p + threadIdx.x], v);
    }
}

// Exclusive scan in three launches: per-block sums, a scan of the block
// sums by one block, then each block scans its own items and adds its
// block's offset. kScanItems consecutive entries per block.
constexpr int kScanItems = 1024;

__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t *total) {
    __shared__ uint32_t warp_sums[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = v;
    for (int off = 1; off < 32; off <<= 1) {
        uint32_t u = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += u;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < (int)(blockDim.x >> 5) ? warp_sums[lane] : 0u;
        for (int off = 1; off < 32; off <<= 1) {
            uint32_t u = __shfl_up_sync(0xffffffffu, w, off);
            if (lane >= off) w += u;
        }
        warp_sums[lane] = w;
    }
    __syncthreads();
    const uint32_t excl = incl - v + (warp > 0 ? warp_sums[warp - 1] : 0u);
    if (total) *total = warp_sums[(blockDim.x >> 5) - 1];
    __syncthreads();
    return excl;
}

__global__ void __launch_bounds__(256) k_scan_reduce(const uint32_t *__restrict__ a, int64_t n,
                                                     uint32_t *__restrict__ sums) {
    const int64_t base = (int64_t)blockIdx.x * kScanItems;
    uint32_t v = 0;
    for (int k = 0; k < kScanItems / 256; ++k) {
        const int64_t i = base + k * 256 + threadIdx.x;
        if (i < n) v += a[i];
    }
    uint32_t total = 0;
    block_exclusive_scan(v, &total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(1024) k_scan_top(uint32_t *__restrict__ sums, int64_t nb) {
    const int64_t chunk = (nb + 1023) / 1024;
    const int64_t b0 = threadIdx.x * chunk, b1 = min(b0 + chunk, nb);
    uint32_t v = 0;
    for (int64_t i = b0; i < b1; ++i) v += sums[i];
    uint32_t run = block_exclusive_scan(v, nullptr);
    for (int64_t i = b0; i < b1; ++i) {
        const uint32_t t = sums[i];
        sums[i] = run;
        run += t;
    }
}

__global__ void __launch_bounds__(256) k_scan_apply(uint32_t *__restrict__ a, int64_t n,
                                                    const uint32_t *__restrict__ sums) {
    const int64_t base = (int64_t)blockIdx.x * kScanItems;
    constexpr int P = kScanItems / 256;  // items per thread, consecutive
    uint32_t v[P];
    uint32_t local = 0;
    for (int k = 0; k < P; ++k) {
        const int64_t i = base + threadIdx.x * P + k;
        v[k] = i < n ? a[i] : 0u;
        local += v[k];
    }
    uint32_t run = block_exclusive_scan(local, nullptr) + sums[blockIdx.x];
    for (int k = 0; k < P; ++k) {
        const int64_t i = base + threadIdx.x * P + k;
        if (i < n) a[i] = run;
        run += v[k];
    }
}

void scan_exclusive(uint32_t *a, int64_t n, uint32_t *sums, cudaStream_t s) {
    const int64_t nb = (n + kScanItems - 1) / kScanItems;
    k_scan_reduce<<<(unsigned)nb, 256, 0, s>>>(a, n, sums);
    k_scan_top<<<1, 1024, 0, s>>>(sums, nb);
    k_scan_apply<<<(unsigned)nb, 256, 0, s>>>(a, n, sums);
}

// One digit of the stable sort in one pass over the keys (decoupled
// look-back: Merrill and Garland 2016; as a radix sort, Adinets and Merrill
// 2022). A block takes the next tile, ranks its keys by digit in input order
// (each warp its own consecutive keys, with warp-level digit matching and
// counters of its own, so no block barrier per round), publishes its digit
// counts, and adds up the tiles before it from theirs: thread d reads back
// the counts of digit d until a tile whose running total is known. The keys
// go through shared memory so that each digit's run is stored together.
// A tile is taken only after the tiles before it, so each waits only on
// blocks that are already running; the wait is bounded all the same, and a
// thread whose wait runs out counts its digit in the tile's keys itself: the
// order of the keys, which the rest of the build indexes by, never depends on it.
// Against a histogram, a three-kernel scan and a scatter per digit (40
// launches for eight digits): the whole rebuild 806 -> 557 us at 1M, 272 -> 132
// at 1,000. Bound by the chain of a tile, about 20 us a digit at 1M.
constexpr unsigned long long kTileCounted = 1ull << 62, kTileTotal = 2ull << 62;
constexpr unsigned long long kTileValue = (1ull << 40) - 1ull;
#ifndef GSRT_LOOKBACK_LIMIT  // (a test builds with 0)
#define GSRT_LOOKBACK_LIMIT (1 << 24)
#endif
constexpr int kLookbackLimit = GSRT_LOOKBACK_LIMIT;

// Four blocks per SM, so that the tiles of 1M keys run at once (three, at 74
// registers, left a second wave: 21 us a pass).
template <bool VALS>
__global__ void __launch_bounds__(kSortThreads, 4)
    k_radix_pass(int64_t n, const unsigned long long *__restrict__ kin,
                 const uint32_t *__restrict__ vin, unsigned long long *__restrict__ kout,
                 uint32_t *__restrict__ vout, int pass, const uint32_t *__restrict__ hist,
                 uint32_t *__restrict__ tickets, unsigned long long *__restrict__ tile_state) {
    constexpr int W = kSortThreads / 32;
    __shared__ unsigned long long s_key[kSortTile];
    __shared__ uint32_t s_val[VALS ? kSortTile : 1];
    __shared__ uint32_t wcount[W][256];
    __shared__ long long s_shift[256];  // global position minus position in the tile
    __shared__ uint32_t s_tile;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, shift = 8 * pass;
    if (tid == 0) s_tile = atomicAdd(&tickets[pass], 1u);
    for (int w = 0; w < W; ++w) wcount[w][tid] = 0;
    const uint32_t digit_total = hist[256 * pass + tid];
    __syncthreads();
    const int64_t tile = s_tile;
    const int64_t tile0 = tile * kSortTile;
    const int64_t warp0 = tile0 + warp * (kSortItems * 32);
    unsigned long long key[kSortItems];
    uint32_t val[kSortItems], rank[kSortItems];
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        const int64_t i = warp0 + 32 * j + lane;
        key[j] = i < n ? kin[i] : 0ull;
        if constexpr (VALS) val[j] = i < n ? vin[i] : 0u;
    }
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        const bool in = warp0 + 32 * j + lane < n;
        const uint32_t digit = (uint32_t)(key[j] >> shift) & 255u;
        const uint32_t peers = __match_any_sync(0xffffffffu, in ? digit : 256u + lane);
        const uint32_t before = in ? wcount[warp][digit] : 0u;
        rank[j] = before + __popc(peers & ((1u << lane) - 1u));
        __syncwarp();
        if (in && rank[j] == before) wcount[warp][digit] = before + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // thread d: the tile's count of digit d, made exclusive over the warps
    uint32_t count = 0;
    for (int w = 0; w < W; ++w) {
        const uint32_t c = wcount[w][tid];
        wcount[w][tid] = count;
        count += c;
    }
    const unsigned long long tag = (unsigned long long)(pass + 1) << 56;  // states of other passes
    volatile unsigned long long *mine = tile_state + tile * 256 + tid;
    *mine = (tile == 0 ? kTileTotal : kTileCounted) | tag | count;
    const uint32_t local = block_exclusive_scan(count, nullptr);
    const uint32_t digit_base = block_exclusive_scan(digit_total, nullptr);
    // eight tiles' states at a time: one after the other, the reads of the
    // tiles that start together were the whole time of a 1M pass
    unsigned long long prior = 0;
    int spins = 0;
    for (int64_t t = tile - 1; t >= 0;) {
        constexpr int B = 8;
        unsigned long long v[B];
#pragma unroll
        for (int q = 0; q < B; ++q)
            v[q] = t - q >= 0
                       ? *(volatile unsigned long long *)(tile_state + (t - q) * 256 + tid)
                       : kTileTotal | tag;
        int used = 0;
        bool done = false;
#pragma unroll
        for (int q = 0; q < B; ++q)
            if (!done && used == q && (v[q] & (63ull << 56)) == tag) {
                prior += v[q] & kTileValue;
                done = (v[q] & kTileTotal) != 0;
                ++used;
            }
        if (done) break;
        t -= used;
        if (used == 0 && spins++ >= kLookbackLimit) {
            const int64_t end = min((t + 1) * kSortTile, n);
            for (int64_t i = t * kSortTile; i < end; ++i)
                prior += ((uint32_t)(kin[i] >> shift) & 255u) == (uint32_t)tid;
            --t;
        }
    }
    if (tile > 0) *mine = kTileTotal | tag | (prior + count);
    s_shift[tid] = (long long)digit_base + (long long)prior - (long long)local;
    // positions within the tile: the digits' starts, then the warps', then ranks
    for (int w = 0; w < W; ++w) wcount[w][tid] += local;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        if (warp0 + 32 * j + lane >= n) continue;
        const uint32_t pos = wcount[warp][(uint32_t)(key[j] >> shift) & 255u] + rank[j];
        s_key[pos] = key[j];
        if constexpr (VALS) s_val[pos] = val[j];
    }
    __syncthreads();
    const int m = (int)min((int64_t)kSortTile, n - tile0);
    for (int i = tid; i < m; i += kSortThreads) {
        const unsigned long long k = s_key[i];
        const int64_t pos = s_shift[(uint32_t)(k >> shift) & 255u] + i;
        kout[pos] = k;
        if constexpr (VALS) vout[pos] = s_val[i];
    }
}

// Scratch that starts a sort or a build at zero, in one allocation: scene
// bounds, digit histograms, tile tickets, arrival counters and wide record
// allocators (of a build over `arrivals` Gaussians), tile states.
struct ZeroScratch {
    size_t hist, tickets, arrive, states, bytes;
    ZeroScratch(int64_t n, int64_t arrivals) {
        hist = 64;
        tickets = hist + kSortPasses * 256 * sizeof(uint32_t);
        arrive = tickets + 64;
        states = (arrive + (size_t)arrivals * sizeof(uint32_t) + 255) / 256 * 256;
        bytes = states + (size_t)radix_tiles(n) * 256 * sizeof(unsigned long long);
    }
};

// ---------------------------------------------------------------- hierarchy

// Common-prefix length of sorted keys i and j, extended by the index bits
// when the codes are equal; -1 outside [0, n).
template <typename I>
__device__ __forceinline__ int delta(const unsigned long long *codes, I n, I i, I j) {
    if (j < 0 || j >= n) return -1;
    unsigned long long a = codes[i], b = codes[j];
    if (a == b) return 64 + __clz((uint32_t)(i ^ j));
    return __clzll(a ^ b);
}

// Internal node i of the binary radix tree over n sorted codes.
template <typename I>
__device__ __forceinline__ void karras_node(I i, I n, const unsigned long long *codes,
                                            Node *__restrict__ nodes,
                                            uint32_t *__restrict__ parent_int,
                                            uint32_t *__restrict__ parent_leaf) {
    int d = (delta(codes, n, i, i + 1) - delta(codes, n, i, i - 1)) >= 0 ? 1 : -1;
    int dmin = delta(codes, n, i, i - d);
    I lmax = 2;
    while (delta(codes, n, i, i + lmax * d) > dmin) lmax <<= 1;
    I l = 0;
    for (I t = lmax >> 1; t >= 1; t >>= 1)
        if (delta(codes, n, i, i + (l + t) * d) > dmin) l += t;
    const I j = i + l * d;
    int dnode = delta(codes, n, i, j);
    I s = 0;
    for (I div = 2;; div <<= 1) {
        const I t = (l + div - 1) / div;
        if (delta(codes, n, i, i + (s + t) * d) > dnode) s += t;
        if (t <= 1) break;
    }
    const I gamma = i + s * d + (d < 0 ? -1 : 0);
    const I lo = i < j ? i : j, hi = i < j ? j : i;
    uint32_t left = (lo == gamma) ? (kLeafBit | (uint32_t)gamma) : (uint32_t)gamma;
    uint32_t right = (hi == gamma + 1) ? (kLeafBit | (uint32_t)(gamma + 1)) : (uint32_t)(gamma + 1);
    Node &nd = nodes[i];
    nd.child[0] = left;
    nd.child[1] = right;
    nd.leaf_range[0] = (uint32_t)lo;
    nd.leaf_range[1] = (uint32_t)hi;
    if (left & kLeafBit) parent_leaf[gamma] = (uint32_t)i; else parent_int[gamma] = (uint32_t)i;
    if (right & kLeafBit) parent_leaf[gamma + 1] = (uint32_t)i; else parent_int[gamma + 1] = (uint32_t)i;
}

// I: int where no index can pass 2^31 (n below 2^30), else 64 bits.
template <typename I>
__global__ void __launch_bounds__(256)
    k_karras(I n, const unsigned long long *__restrict__ codes,
                         Node *__restrict__ nodes, uint32_t *__restrict__ parent_int,
                         uint32_t *__restrict__ parent_leaf) {
    const I i = (I)blockIdx.x * 256 + (I)threadIdx.x;
    if (i < n - 1) karras_node<I>(i, n, codes, nodes, parent_int, parent_leaf);
}

// Up to kSmallMax Gaussians: boxes, bounds, codes, the sort and the tree in
// one launch of one block, everything between them in its shared memory. The
// eleven launches it stands for cost more than their work: a rebuild of 1,000
// Gaussians 132 -> 72 us, of 5,000 156 either way but 17 us of host time
// instead of 36; above, one block is the slower. Each digit is ranked as in
// k_radix_pass, the keys moving within shared memory.
constexpr int kSmallThreads = 1024, kSmallItems = 8;
constexpr int kSmallMax = kSmallThreads * kSmallItems;
constexpr size_t kSmallBytes = (size_t)kSmallMax * 12 + (size_t)(kSmallThreads / 32) * 256 * 4;

__global__ void __launch_bounds__(kSmallThreads, 1)
    k_small(int n, const float *__restrict__ means, const float *__restrict__ log_scales,
            const float *__restrict__ quats, const float *__restrict__ logits,
            float *__restrict__ aabb, unsigned long long *__restrict__ codes,
            uint32_t *__restrict__ vals, Node *__restrict__ nodes,
            uint32_t *__restrict__ parent_int, uint32_t *__restrict__ parent_leaf,
            uint32_t *__restrict__ arrive, int n_arrive, uint32_t *__restrict__ status) {
    constexpr int W = kSmallThreads / 32;
    extern __shared__ unsigned long long small_smem[];
    unsigned long long *s_key = small_smem;
    uint32_t *s_val = reinterpret_cast<uint32_t *>(s_key + kSmallMax);
    uint32_t(*wcount)[256] = reinterpret_cast<uint32_t(*)[256]>(s_val + kSmallMax);
    __shared__ unsigned int s_bounds[6];
    __shared__ uint32_t s_base[256];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < 6) s_bounds[tid] = 0;
    for (int i = tid; i < n_arrive; i += kSmallThreads) arrive[i] = 0;
    __syncthreads();
    {
        float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
        for (int g = tid; g < n; g += kSmallThreads) gaussian_box(g, means, log_scales, quats, logits, aabb, status, lo, hi);
        for (int k = 0; k < 3; ++k) {
            for (int off = 16; off > 0; off >>= 1) {
                lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], off));
                hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], off));
            }
            if (lane == 0 && lo[k] <= hi[k]) {
                atomicMax(&s_bounds[k], ~f2ord(lo[k]));
                atomicMax(&s_bounds[3 + k], f2ord(hi[k]));
            }
        }
    }
    __syncthreads();
    for (int g = tid; g < n; g += kSmallThreads) {
        s_key[g] = sort_code(g, means, s_bounds, aabb);
        s_val[g] = (uint32_t)g;
    }
    const int J = (n + kSmallThreads - 1) / kSmallThreads;  // keys per thread
    const int first = warp * J * 32 + lane;
    for (int shift = 0; shift < 64; shift += 8) {
        for (int i = tid; i < W * 256; i += kSmallThreads) (&wcount[0][0])[i] = 0;
        __syncthreads();
        unsigned long long key[kSmallItems];
        uint32_t val[kSmallItems], rank[kSmallItems];
#pragma unroll
        for (int j = 0; j < kSmallItems; ++j) {
            if (j >= J) break;
            const int i = first + 32 * j;
            const bool in = i < n;
            key[j] = in ? s_key[i] : 0ull;
            val[j] = in ? s_val[i] : 0u;
            const uint32_t digit = (uint32_t)(key[j] >> shift) & 255u;
            const uint32_t peers = __match_any_sync(0xffffffffu, in ? digit : 256u + lane);
            const uint32_t before = in ? wcount[warp][digit] : 0u;
            rank[j] = before + __popc(peers & ((1u << lane) - 1u));
            __syncwarp();
            if (in && rank[j] == before) wcount[warp][digit] = before + __popc(peers);
            __syncwarp();
        }
        __syncthreads();
        uint32_t count = 0;
        if (tid < 256)
            for (int w = 0; w < W; ++w) {
                const uint32_t c = wcount[w][tid];
                wcount[w][tid] = count;
                count += c;
            }
        const uint32_t base = block_exclusive_scan(count, nullptr);
        if (tid < 256) s_base[tid] = base;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kSmallItems; ++j) {
            if (j >= J) break;
            if (first + 32 * j < n) {
                const uint32_t digit = (uint32_t)(key[j] >> shift) & 255u;
                const uint32_t pos = s_base[digit] + wcount[warp][digit] + rank[j];
                s_key[pos] = key[j];
                s_val[pos] = val[j];
            }
        }
        __syncthreads();
    }
    for (int i = tid; i < n; i += kSmallThreads) {
        codes[i] = s_key[i];
        vals[i] = s_val[i];
        if (i < n - 1) karras_node<int>(i, n, s_key, nodes, parent_int, parent_leaf);
    }
}

__device__ __forceinline__ void write_record(PrimRec *__restrict__ prims, int64_t i, uint32_t g,
                                             const Activated &a) {
    PrimRec r;
    for (int k = 0; k < 3; ++k) r.mu[k] = a.mu[k];
    r.opacity = a.opacity;
    // M = S^-1 R_q^T: row k is column k of R_q divided by s_k
    for (int k = 0; k < 3; ++k)
        for (int j = 0; j < 3; ++j) r.m[3 * k + j] = a.R[3 * j + k] * a.inv_s[k];
    if (!a.finite)
        for (int k = 0; k < 9; ++k) r.m[k] = NAN;
    r.gid = g;
    r.pad[0] = 0.0f;
    r.pad[1] = 0.0f;
    float4 *dst = reinterpret_cast<float4 *>(prims + i);
    const float4 *src = reinterpret_cast<const float4 *>(&r);
    for (int k = 0; k < 4; ++k) dst[k] = src[k];
}

// The W-wide hierarchies (W = 8, 32) are cut out of the binary tree
// bottom-up, in the box refit: k_W(p) is the number of children that the
// wide node holding binary node p has below p, k_W(leaf) = 1. At a node
// whose children together exceed W, the one with more is closed: it becomes
// a wide node of its own and counts as one (both, if that still exceeds W).
// So every wide node but the root holds more than W / 2 children, and the
// records are at most M + M / (W / 2). Against cutting at fixed binary
// levels (mean 32-wide fill 6.6 children) the grouped walks take a third of
// the steps: 1M shell at 1080p, rebuild + trace, spp 64 47.6 -> 28.0 ms,
// N=4 spp 16 46.7 -> 33.8, 3M with 8-bit records 100.6 -> 48.7; and the cut
// costs the refit little where listing, counting and scanning each width
// took kernels of their own (frame at spp 1 6.65 -> 6.14 ms). Four words per internal node p, one
// byte (bits 0-7, 8-15) per W:
//   x  parent
//   y  children of its wide node left of p's within the parent (0 when p is
//      the left child); bit 24 + w: p is closed in tree w
//   z  k_W(p)
//   w  children below p's left child; bit 24 + w: that child is closed,
//      bit 27 + w: the right one is
constexpr uint32_t kLeafCounts = 0x0101u;  // one child in each of the two
constexpr uint32_t kRootClosed = 3u << 24;

__device__ __forceinline__ uint32_t close_children(uint32_t &kl, uint32_t &kr) {
    uint32_t closed = 0, nl = 0, nr = 0;
#pragma unroll
    for (int w = 0; w < kGroupTrees; ++w) {
        const uint32_t W = group_width(w);
        uint32_t a = (kl >> (8 * w)) & 255u, b = (kr >> (8 * w)) & 255u;
        if (a + b > W) {
            const bool left = a >= b;
            if (left) a = 1; else b = 1;
            closed |= (left ? 1u : 8u) << w;
            if (a + b > W) {
                if (left) b = 1; else a = 1;
                closed |= (left ? 8u : 1u) << w;
            }
        }
        nl |= a << (8 * w);
        nr |= b << (8 * w);
    }
    kl = nl;
    kr = nr;
    return closed;  // bits 0-2: the left child, 3-5: the right one
}

// Wide tree links of node p once both children are known (kl, kr: their
// counts); returns p's own counts.
__device__ __forceinline__ uint32_t cut_node(uint32_t p, uint2 child, uint32_t kl, uint32_t kr,
                                             uint4 *__restrict__ link) {
    const uint32_t closed = close_children(kl, kr);
    if (!(child.x & kLeafBit))
        __stcg(reinterpret_cast<uint2 *>(link + child.x), make_uint2(p, (closed & 7u) << 24));
    if (!(child.y & kLeafBit))
        __stcg(reinterpret_cast<uint2 *>(link + child.y), make_uint2(p, kl | (closed >> 3) << 24));
    if (p == 0) __stcg(reinterpret_cast<uint2 *>(link), make_uint2(0u, kRootClosed));
    __stcg(reinterpret_cast<uint2 *>(link + p) + 1, make_uint2(kl + kr, kl | closed << 24));
    return kl + kr;
}

// Records in tree order, box refit and the cut of the wide trees (link !=
// null). A Karras node is numbered by one end of its leaf range, so the nodes
// over leaves of one block lie among that block's node numbers: those (more
// than 9 of 10) are refitted in shared memory, in rounds: a round's ready
// nodes are listed densely, one thread each, and a node is ready when its
// second child arrives. (A thread per leaf that climbs while it arrives second
// leaves one lane in ten working.) What leaves the block is listed for
// k_climb.
constexpr int kLeafThreads = 256;

__global__ void __launch_bounds__(kLeafThreads)
    k_leaves(int64_t n, const uint32_t *__restrict__ order, const float *__restrict__ means,
             const float *__restrict__ log_scales, const float *__restrict__ quats,
             const float *__restrict__ logits, const float *__restrict__ aabb,
             PrimRec *__restrict__ prims, Node *__restrict__ nodes,
             const uint32_t *__restrict__ parent_int, const uint32_t *__restrict__ parent_leaf,
             uint4 *__restrict__ link, uint32_t *__restrict__ exits,
             uint32_t *__restrict__ n_exits) {
    __shared__ uint2 s_child[kLeafThreads];
    __shared__ uint32_t s_parent[kLeafThreads];
    __shared__ uint32_t s_arrive[kLeafThreads];
    __shared__ uint32_t s_counts[kLeafThreads][2];
    __shared__ float s_box[kLeafThreads][2][6];
    __shared__ bool s_near[kLeafThreads];  // the node covers leaves of this block only
    __shared__ uint16_t s_ready[2][kLeafThreads];
    __shared__ uint32_t s_exit[kLeafThreads];
    __shared__ uint32_t s_n[2], s_n_exit;
    const int tid = threadIdx.x;
    const uint32_t b0 = blockIdx.x * kLeafThreads;
    const int64_t i = (int64_t)b0 + tid;
    {
        bool near = false;
        if (i < n - 1) {
            const uint4 c = *reinterpret_cast<const uint4 *>(nodes[i].child);  // children, range
            s_child[tid] = make_uint2(c.x, c.y);
            s_parent[tid] = parent_int[i];
            near = c.z >= b0 && c.w < b0 + kLeafThreads;
        }
        s_near[tid] = near;
        s_arrive[tid] = 0;
        if (tid < 2) s_n[tid] = 0;
        if (tid == 2) s_n_exit = 0;
    }
    __syncthreads();
    // hands a finished child (its box, counts) to its parent q
    auto arrive_at = [&](uint32_t ref, uint32_t q, const float box[6], uint32_t counts, int next) {
        const uint32_t j = q - b0;
        if (j < (uint32_t)kLeafThreads && s_near[j]) {
            const int side = s_child[j].x == ref ? 0 : 1;
            for (int k = 0; k < 6; ++k) s_box[j][side][k] = box[k];
            s_counts[j][side] = counts;
            __threadfence_block();
            if (atomicAdd(&s_arrive[j], 1u) == 1u) s_ready[next][atomicAdd(&s_n[next], 1u)] = (uint16_t)j;
        } else {
            s_exit[atomicAdd(&s_n_exit, 1u)] = ref;
        }
    };
    if (i < n) {
        const uint32_t g = order[i];
        const Activated a = activate(means, log_scales, quats, logits, g);
        write_record(prims, i, g, a);
        float box[6];
        for (int k = 0; k < 6; ++k) box[k] = aabb[6 * (int64_t)g + k];
        arrive_at(kLeafBit | (uint32_t)i, parent_leaf[i], box, kLeafCounts, 0);
    }
    __syncthreads();
    for (int now = 0;; now ^= 1) {
        const uint32_t n_ready = s_n[now];
        __syncthreads();
        if (n_ready == 0) break;
        if (tid == 0) s_n[now] = 0;
        if (tid < (int)n_ready) {
            const int j = s_ready[now][tid];
            const uint32_t p = b0 + (uint32_t)j;
            const volatile float *l = s_box[j][0], *r = s_box[j][1];
            float bl[6], br[6], box[6];
            for (int k = 0; k < 6; ++k) {
                bl[k] = l[k];
                br[k] = r[k];
            }
            for (int k = 0; k < 3; ++k) {
                box[k] = fminf(bl[k], br[k]);
                box[3 + k] = fmaxf(bl[3 + k], br[3 + k]);
            }
            float4 *out = reinterpret_cast<float4 *>(nodes[p].box);
            out[0] = make_float4(bl[0], bl[1], bl[2], bl[3]);
            out[1] = make_float4(bl[4], bl[5], br[0], br[1]);
            out[2] = make_float4(br[2], br[3], br[4], br[5]);
            uint32_t counts = kLeafCounts;
            if (link) counts = cut_node(p, s_child[j], s_counts[j][0], s_counts[j][1], link);
            if (p != 0) arrive_at(p, s_parent[j], box, counts, now ^ 1);
        }
        __syncthreads();
    }
    // a block lists at most one exit per leaf
    if (tid == 0) s_n[0] = s_n_exit ? atomicAdd(n_exits, s_n_exit) : 0u;
    __syncthreads();
    if (tid < (int)s_n_exit) exits[s_n[0] + tid] = s_exit[tid];
}

// The exits of k_leaves, one thread each, carried to the root: the second to
// reach a node merges both boxes and continues. A launch of its own: climbing
// at the end of k_leaves, a few threads held their block's place on the SM
// through a dozen meetings in memory each.
__device__ __forceinline__ uint32_t arrive_acq_rel(uint32_t *counter) {
    uint32_t old;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(old) : "l"(counter) : "memory");
    return old;
}

__global__ void __launch_bounds__(64)
    k_climb(const uint32_t *__restrict__ exits, const uint32_t *__restrict__ n_exits,
            const uint32_t *__restrict__ order, const float *__restrict__ aabb,
            Node *__restrict__ nodes, const uint32_t *__restrict__ parent_int,
            const uint32_t *__restrict__ parent_leaf, uint32_t *__restrict__ arrive,
            uint4 *__restrict__ link) {
    const uint32_t e = blockIdx.x * 64 + threadIdx.x;
    if (e >= *n_exits) return;
    uint32_t ref = exits[e], p, counts = kLeafCounts;
    float box[6];
    if (ref & kLeafBit) {
        const uint32_t leaf = ref & ~kLeafBit;
        const int64_t g = order[leaf];
        for (int k = 0; k < 6; ++k) box[k] = aabb[6 * g + k];
        p = parent_leaf[leaf];
    } else {
        const float *l = nodes[ref].box[0], *r = nodes[ref].box[1];
        for (int k = 0; k < 3; ++k) {
            box[k] = fminf(l[k], r[k]);
            box[3 + k] = fmaxf(l[3 + k], r[3 + k]);
        }
        if (link) counts = link[ref].z;
        p = parent_int[ref];
    }
    for (int guard = 0; guard < 4096; ++guard) {
        Node *nd = nodes + p;
        const uint2 child = __ldcg(reinterpret_cast<const uint2 *>(nd->child));
        const uint32_t next = parent_int[p];
        const int side = child.x == ref ? 0 : 1;
        // a child's box is 24 bytes at an 8-byte boundary
        float2 *mine = reinterpret_cast<float2 *>(nd->box[side]);
        for (int k = 0; k < 3; ++k) __stcg(mine + k, make_float2(box[2 * k], box[2 * k + 1]));
        if (arrive_acq_rel(&arrive[p]) == 0u) return;
        const float2 *other = reinterpret_cast<const float2 *>(nd->box[1 - side]);
        float ob[6];
        for (int k = 0; k < 3; ++k) {
            const float2 v = __ldcg(other + k);
            ob[2 * k] = v.x;
            ob[2 * k + 1] = v.y;
        }
        if (link) {
            const uint32_t sib = side ? child.x : child.y;
            const uint32_t oc = (sib & kLeafBit) ? kLeafCounts : __ldcg(&link[sib].z);
            counts = cut_node(p, child, side ? oc : counts, side ? counts : oc, link);
        }
        for (int k = 0; k < 3; ++k) {
            box[k] = fminf(box[k], ob[k]);
            box[3 + k] = fmaxf(box[3 + k], ob[3 + k]);
        }
        if (p == 0) return;
        ref = p;
        p = next;
    }
}

// M == 1: a root whose two children are the same leaf. Draws are keyed by
// (ray, Gaussian, sample), so testing the leaf twice gives the same answer.
__global__ void k_single(const uint32_t *__restrict__ order, const float *__restrict__ means,
                         const float *__restrict__ log_scales, const float *__restrict__ quats,
                         const float *__restrict__ logits, const float *__restrict__ aabb,
                         PrimRec *__restrict__ prims, Node *__restrict__ nodes,
                         uint4 *__restrict__ link) {
    uint32_t g = order[0];
    Activated a = activate(means, log_scales, quats, logits, g);
    write_record(prims, 0, g, a);
    Node nd;
    for (int s = 0; s < 2; ++s) {
        for (int k = 0; k < 6; ++k) nd.box[s][k] = aabb[6 * (int64_t)g + k];
        nd.child[s] = kLeafBit;
    }
    nd.leaf_range[0] = nd.leaf_range[1] = 0;
    nodes[0] = nd;
    // a wide root of one child (k_wide_records writes the left one only)
    if (link) link[0] = make_uint4(0u, kRootClosed, kLeafCounts, kLeafCounts);
}

// Depth of every internal binary node (walk to the root).
__global__ void k_depth(int64_t n_int, const uint32_t *__restrict__ parent_int,
                        uint32_t *__restrict__ depth, uint32_t *__restrict__ flag) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_int) return;
    uint32_t d = 0, p = (uint32_t)i;
    while (p != 0 && d < 4096) {
        p = parent_int[p];
        ++d;
    }
    depth[i] = d;
    flag[i] = (d & 1u) ? 0u : 1u;  // wide nodes sit at even binary depth
}

// Quantisation of one axis of a node: planes origin + q * 2^e, q in 0..255.
__device__ __forceinline__ int quant_exponent(float ext) {
    if (!(ext > 0.0f)) return -120;
    int e = (int)ceilf(log2f(ext / 254.0f));
    e = max(e, -120);
    while (254.0f * ldexpf(1.0f, e) < ext) ++e;  // one unit of slack
    return min(e, 120);
}

__device__ __forceinline__ unsigned char quant_lo(float v, float origin, float scale) {
    if (!(v == v)) return 0;  // NaN box: full range
    float q = floorf((v - origin) / scale);
    q = fminf(fmaxf(q, 0.0f), 255.0f);
    while (q > 0.0f && __fadd_rn(origin, q * scale) > v) q -= 1.0f;
    return (unsigned char)q;
}

__device__ __forceinline__ unsigned char quant_hi(float v, float origin, float scale) {
    if (!(v == v)) return 255;
    float q = ceilf((v - origin) / scale);
    q = fminf(fmaxf(q, 0.0f), 255.0f);
    while (q < 255.0f && __fadd_rn(origin, q * scale) < v) q += 1.0f;
    return (unsigned char)q;
}

// One wide node per even-depth binary node: its children, or grandchildren
// where a child is internal; written at its compact index.
template <int FMT>
__global__ void k_collapse(int64_t n_int, const Node *__restrict__ nodes,
                           const uint32_t *__restrict__ depth, const uint32_t *__restrict__ wmap,
                           void *__restrict__ wide) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_int || (depth[i] & 1u)) return;
    float lo[3][4], hi[3][4];
    uint32_t child[4];
    int k = 0;
    const Node nd = nodes[i];
    for (int side = 0; side < 2; ++side) {
        const uint32_t c = nd.child[side];
        if (c & kLeafBit) {
            for (int a = 0; a < 3; ++a) { lo[a][k] = nd.box[side][a]; hi[a][k] = nd.box[side][3 + a]; }
            child[k++] = c;
        } else {
            const Node cn = nodes[c];
            for (int s2 = 0; s2 < 2; ++s2) {
                for (int a = 0; a < 3; ++a) { lo[a][k] = cn.box[s2][a]; hi[a][k] = cn.box[s2][3 + a]; }
                const uint32_t gc = cn.child[s2];
                child[k++] = (gc & kLeafBit) ? gc : wmap[gc];
            }
        }
    }
    const int used = k;
    for (; k < 4; ++k) {
        for (int a = 0; a < 3; ++a) { lo[a][k] = INFINITY; hi[a][k] = INFINITY; }
        child[k] = kEmpty;
    }
    const uint32_t w = wmap[i];
    if (FMT == GS_NODES_WIDE4) {
        Node4 n;
        for (int a = 0; a < 3; ++a)
            for (int j = 0; j < 4; ++j) { n.lo[a][j] = lo[a][j]; n.hi[a][j] = hi[a][j]; }
        for (int j = 0; j < 4; ++j) { n.child[j] = child[j]; n.reserved[j] = 0; }
        reinterpret_cast<Node4 *>(wide)[w] = n;
    } else {
        NodeQ4 n;
        n.used = (unsigned char)((1u << used) - 1u);
        for (int a = 0; a < 3; ++a) {
            float nlo = INFINITY, nhi = -INFINITY;
            for (int j = 0; j < used; ++j) { nlo = fminf(nlo, lo[a][j]); nhi = fmaxf(nhi, hi[a][j]); }
            if (!(nlo <= nhi)) { nlo = 0.0f; nhi = 0.0f; }
            const int e = quant_exponent(nhi - nlo);
            const float scale = ldexpf(1.0f, e);
            n.origin[a] = nlo;
            n.exp[a] = (signed char)e;
            for (int j = 0; j < 4; ++j) {
                if (j < used) {
                    n.qlo[a][j] = quant_lo(lo[a][j], nlo, scale);
                    n.qhi[a][j] = quant_hi(hi[a][j], nlo, scale);
                } else {
                    n.qlo[a][j] = 255;
                    n.qhi[a][j] = 0;
                }
            }
        }
        for (int j = 0; j < 4; ++j) n.child[j] = child[j];
        n.reserved[0] = n.reserved[1] = 0;
        reinterpret_cast<NodeQ4 *>(wide)[w] = n;
    }
}

// Reference of the wide node at every closed binary node: a block adds up its
// nodes' record counts (plus `header` units each), takes its range of the
// trees' records with one atomic per tree, and hands it out in node
// order. The order of the blocks' ranges varies from run to run; a reference
// is never compared, so no result depends on it.
struct WideRefs {
    uint32_t *ref[kGroupTrees];
};

__global__ void __launch_bounds__(256)
    k_wide_offsets(int64_t n_int, const uint4 *__restrict__ link, uint32_t *__restrict__ alloc,
                   uint32_t header, const WideRefs out) {
    constexpr int P = 4;  // consecutive nodes per thread
    __shared__ uint32_t base[kGroupTrees];
    __shared__ unsigned long long warp_sum[8];
    const int64_t i0 = ((int64_t)blockIdx.x * 256 + threadIdx.x) * P;
    uint32_t flags[P], cnt[P];
    // 21 bits per tree: at most 1024 nodes x 34 units
    unsigned long long local = 0;
#pragma unroll
    for (int j = 0; j < P; ++j) {
        flags[j] = 0;
        cnt[j] = 0;
        if (i0 + j < n_int) {
            const uint4 l = link[i0 + j];
            flags[j] = l.y >> 24;
            cnt[j] = l.z;
        }
#pragma unroll
        for (int w = 0; w < kGroupTrees; ++w)
            if ((flags[j] >> w) & 1u)
                local += (unsigned long long)(((cnt[j] >> (8 * w)) & 255u) + header) << (21 * w);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long incl = local;
    for (int off = 1; off < 32; off <<= 1) {
        const unsigned long long u = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += u;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    unsigned long long before = 0, total = 0;
    for (int k = 0; k < 8; ++k) {
        if (k < warp) before += warp_sum[k];
        total += warp_sum[k];
    }
    if (threadIdx.x < kGroupTrees) {
        const uint32_t t = (uint32_t)(total >> (21 * threadIdx.x)) & 0x1fffffu;
        base[threadIdx.x] = t ? atomicAdd(&alloc[threadIdx.x], t) : 0u;
    }
    __syncthreads();
    const unsigned long long excl = before + incl - local;
#pragma unroll
    for (int w = 0; w < kGroupTrees; ++w) {
        uint32_t run = base[w] + ((uint32_t)(excl >> (21 * w)) & 0x1fffffu);
#pragma unroll
        for (int j = 0; j < P; ++j) {
            if (!((flags[j] >> w) & 1u)) continue;
            const uint32_t c = (cnt[j] >> (8 * w)) & 255u;
            out.ref[w][i0 + j] = (c - 1u) << kWideCountShift | run;
            run += c + header;
        }
    }
}

// 8-bit planes of one child box against its node's frame (origin, scale):
// lower planes rounded down and upper planes rounded up, each by one more
// quantum, so that the traversal's decoding (whose rounding stays under
// half a quantum) still covers the FP32 box. A non-finite box is flagged.
__device__ __forceinline__ void quant_child(const float b[6], const float origin[3],
                                            const float scale[3], uint32_t &q0, uint32_t &q1) {
    uint32_t lo[3], hi[3];
    bool finite = true;
    for (int a = 0; a < 3; ++a) finite = finite && isfinite(b[a]) && isfinite(b[3 + a]);
    for (int a = 0; a < 3; ++a) {
        float ql = floorf((b[a] - origin[a]) / scale[a]) - 1.0f;
        float qh = ceilf((b[3 + a] - origin[a]) / scale[a]) + 1.0f;
        // exact checks in the frame (q * scale is exact for a power-of-two
        // scale): one quantum of room below lo and above hi
        while (ql > 0.0f && !(__fadd_rn(origin[a], (ql + 1.0f) * scale[a]) <= b[a])) ql -= 1.0f;
        while (qh < 255.0f && !(__fadd_rn(origin[a], (qh - 1.0f) * scale[a]) >= b[3 + a])) qh += 1.0f;
        lo[a] = finite ? (uint32_t)fminf(fmaxf(ql, 0.0f), 255.0f) : 0u;
        hi[a] = finite ? (uint32_t)fminf(fmaxf(qh, 0.0f), 255.0f) : 0u;
    }
    q0 = lo[0] | lo[1] << 8 | lo[2] << 16 | hi[0] << 24;
    q1 = hi[1] | hi[2] << 8 | (finite ? 0u : kQ8Skip);
}

// Frame of an 8-bit wide node from the union of its children's boxes:
// per axis a power-of-two scale with the extent plus two spare quanta
// within 255 quanta, and the origin one quantum below the lower bound.
__device__ __forceinline__ void quant_frame(const float lo[3], const float hi[3], float origin[3],
                                            float scale[3]) {
    for (int a = 0; a < 3; ++a) {
        float l = lo[a], h = hi[a];
        if (!(l <= h)) { l = 0.0f; h = 0.0f; }
        const float ext = h - l;
        int e = ext > 0.0f ? (int)ceilf(log2f(ext / 251.0f)) : -120;
        e = max(e, -120);
        while (251.0f * ldexpf(1.0f, e) < ext) ++e;
        e = min(e, 120);
        scale[a] = ldexpf(1.0f, e);
        origin[a] = l - scale[a];
    }
}

struct WideOut {
    const uint32_t *ref[kGroupTrees];
    void *rec[kGroupTrees];
};

// Writes the child records of the wide trees, one thread per binary
// internal node, each record by itself: the thread whose child is a leaf or
// closed climbs to the wide node it belongs to (a few levels, one link each)
// and adds up the children to its left on the way. All reads of its own node
// are coalesced and nothing is kept in arrays. In the 8-bit form the planes
// are taken against the wide node's own box, and the first child's thread
// also writes the header.
template <bool Q8>
__global__ void __launch_bounds__(256)
    k_wide_records(int64_t n_int, const Node *__restrict__ nodes, const uint4 *__restrict__ link,
                   const WideOut out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_int) return;
    const float4 *np = reinterpret_cast<const float4 *>(nodes + i);
    const float4 b0 = __ldg(np), b1 = __ldg(np + 1), b2 = __ldg(np + 2);
    const uint4 cref = __ldg(reinterpret_cast<const uint4 *>(np + 3));
    const float box[2][6] = {{b0.x, b0.y, b0.z, b0.w, b1.x, b1.y},
                             {b1.z, b1.w, b2.x, b2.y, b2.z, b2.w}};
    uint4 l = __ldg(link + i);
    const uint32_t left = l.w;
    uint32_t need[2];  // trees in which the child is a record of its own
    need[0] = (cref.x & kLeafBit) ? 3u : (left >> 24) & 3u;
    need[1] = (cref.y & kLeafBit) ? 3u : (left >> 27) & 3u;
    if (cref.x == cref.y) need[1] = 0u;  // a single Gaussian
    uint32_t todo = need[0] | need[1];
    uint32_t cur = (uint32_t)i, pos = 0;  // children left of node i, one byte per tree
    for (int guard = 0; todo && guard < 4096; ++guard) {
        const uint32_t here = (l.y >> 24) & todo;
#pragma unroll
        for (int w = 0; w < kGroupTrees; ++w) {
            if (!((here >> w) & 1u)) continue;
            const uint32_t first = __ldg(out.ref[w] + cur) & kWideOffsetMask;
            float origin[3], scale[3];
            if constexpr (Q8) {
                const float *rb = &nodes[cur].box[0][0];
                float lo[3], hi[3];
                for (int q = 0; q < 3; ++q) {
                    lo[q] = fminf(__ldg(rb + q), __ldg(rb + 6 + q));
                    hi[q] = fmaxf(__ldg(rb + 3 + q), __ldg(rb + 9 + q));
                }
                quant_frame(lo, hi, origin, scale);
            }
#pragma unroll
            for (int side = 0; side < 2; ++side) {
                if (!((need[side] >> w) & 1u)) continue;
                const uint32_t c = side ? cref.y : cref.x;
                const uint32_t r = (c & kLeafBit) ? c : __ldg(out.ref[w] + c);
                const uint32_t j = ((pos >> (8 * w)) & 255u) +
                                   (side ? (left >> (8 * w)) & 255u : 0u);
                const float *b = box[side];
                if constexpr (Q8) {
                    uint4 *dst = static_cast<uint4 *>(out.rec[w]) + first;
                    uint32_t q0, q1;
                    quant_child(b, origin, scale, q0, q1);
                    dst[kGroupQHeaderUnits + j] = make_uint4(q0, q1, r, 0u);
                    if (j == 0) {
                        dst[0] = make_uint4(__float_as_uint(origin[0]), __float_as_uint(origin[1]),
                                            __float_as_uint(origin[2]), __float_as_uint(scale[0]));
                        dst[1] = make_uint4(__float_as_uint(scale[1]), __float_as_uint(scale[2]), 0u, 0u);
                    }
                } else {
                    float4 *dst = reinterpret_cast<float4 *>(static_cast<ChildRec *>(out.rec[w]) + first + j);
                    // planes within +-1e30, so that sums and differences of
                    // them are numbers (NaN boxes, never hit, stay NaN)
                    float v[6];
#pragma unroll
                    for (int q = 0; q < 6; ++q)
                        v[q] = b[q] < -1e30f ? -1e30f : (b[q] > 1e30f ? 1e30f : b[q]);
                    dst[0] = make_float4(v[0], v[1], v[2], v[3]);
                    dst[1] = make_float4(v[4], v[5], __uint_as_float(r), 0.0f);
                }
            }
        }
        todo &= ~here;
        if (!todo) break;
        pos += l.y & 0xffffffu;  // at most W children per tree: no carry
        cur = l.x;
        l = __ldg(link + cur);
    }
}

inline unsigned grid_for(int64_t n, int threads) {
    return (unsigned)((n + threads - 1) / threads);
}

}  // namespace

int64_t radix_tiles(int64_t n) { return (n + kSortTile - 1) / kSortTile; }

size_t sort_scratch_bytes(int64_t n) { return ZeroScratch(n, 0).bytes; }
// (arrival counters, the wide record allocators, the number of exits)
constexpr int kBuildCounters = kGroupTrees + 1;

size_t build_scratch_bytes(int64_t n) { return ZeroScratch(n, n + kBuildCounters).bytes; }

int sort_keys64(unsigned long long *keys[2], int64_t n, int lo_bit, void *scratch,
                cudaStream_t s) {
    const ZeroScratch z(n, 0);
    unsigned char *base = static_cast<unsigned char *>(scratch);
    uint32_t *hist = reinterpret_cast<uint32_t *>(base + z.hist);
    // a failed call leaves its error for the caller's cudaGetLastError
    cudaMemsetAsync(base, 0, z.bytes, s);
    const int64_t tiles = radix_tiles(n);
    k_radix_hist<<<(unsigned)(tiles < 1216 ? tiles : 1216), kSortThreads, 0, s>>>(n, keys[0],
                                                                                lo_bit / 8, hist);
    int cur = 0;
    for (int pass = lo_bit / 8; pass < kSortPasses; ++pass) {
        k_radix_pass<false><<<(unsigned)tiles, kSortThreads, 0, s>>>(
            n, keys[cur], nullptr, keys[1 - cur], nullptr, pass, hist,
            reinterpret_cast<uint32_t *>(base + z.tickets),
            reinterpret_cast<unsigned long long *>(base + z.states));
        cur = 1 - cur;
    }
    return cur;
}

int64_t scan_tmp_entries(int64_t n) { return (n + kScanItems - 1) / kScanItems + 1; }

gs_status build_into(gs_bvh *b, const gs_gaussians *g, cudaStream_t s) {
    const int64_t M = g->M;
    b->M = M;
    b->n_nodes = M == 0 ? 0 : (M == 1 ? 1 : M - 1);
    if (M == 0) return GS_OK;
    cudaError_t e;
    const ZeroScratch z(M, M + kBuildCounters);
    unsigned char *base = static_cast<unsigned char *>(b->zero);
    unsigned int *bounds = reinterpret_cast<unsigned int *>(base);
    uint32_t *hist = reinterpret_cast<uint32_t *>(base + z.hist);
    uint32_t *arrive = reinterpret_cast<uint32_t *>(base + z.arrive);
    uint32_t *parent_int = b->parent, *parent_leaf = b->parent + M;
    int cur = 0;
    const bool small = M > 1 && M <= kSmallMax;
    if (small) {
        if ((e = cudaFuncSetAttribute(k_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)kSmallBytes)) != cudaSuccess)
            return cuda_fail(e, "small build setup");
        k_small<<<1, kSmallThreads, kSmallBytes, s>>>(
            (int)M, g->means, g->log_scales, g->quats, g->opacity_logits, b->aabb, b->codes[0],
            b->vals[0], b->nodes, parent_int, parent_leaf, arrive, (int)M + kBuildCounters, b->status);
    } else {
        if ((e = cudaMemsetAsync(base, 0, z.bytes, s)) != cudaSuccess)
            return cuda_fail(e, "memset build scratch");
        k_preprocess<<<grid_for(M, 256), 256, 0, s>>>(M, g->means, g->log_scales, g->quats,
                                                       g->opacity_logits, b->aabb, bounds, b->status);
        const int64_t tiles = radix_tiles(M);
        k_morton<<<(unsigned)tiles, kSortThreads, 0, s>>>(M, g->means, bounds, b->aabb, b->codes[0],
                                                           b->vals[0], hist);
        for (int pass = 0; pass < kSortPasses; ++pass) {
            k_radix_pass<true><<<(unsigned)tiles, kSortThreads, 0, s>>>(
                M, b->codes[cur], b->vals[cur], b->codes[1 - cur], b->vals[1 - cur], pass, hist,
                reinterpret_cast<uint32_t *>(base + z.tickets),
                reinterpret_cast<unsigned long long *>(base + z.states));
            cur = 1 - cur;
        }
    }
    b->final_buf = cur;
    const uint32_t *order = b->vals[cur];
    if (M == 1) {
        k_single<<<1, 1, 0, s>>>(order, g->means, g->log_scales, g->quats, g->opacity_logits,
                                 b->aabb, b->prims, b->nodes, b->link);
    } else {
        if (!small && M < (int64_t)1 << 30)
            k_karras<int><<<grid_for(M - 1, 256), 256, 0, s>>>((int)M, b->codes[cur], b->nodes,
                                                                parent_int, parent_leaf);
        else if (!small)
            k_karras<int64_t><<<grid_for(M - 1, 256), 256, 0, s>>>(M, b->codes[cur], b->nodes,
                                                                    parent_int, parent_leaf);
        k_leaves<<<grid_for(M, kLeafThreads), kLeafThreads, 0, s>>>(M, order, g->means, g->log_scales, g->quats,
                                                   g->opacity_logits, b->aabb, b->prims, b->nodes,
                                                   parent_int, parent_leaf, b->link,
                                                   b->vals[1 - cur], arrive + M + kGroupTrees);
        if (M > kLeafThreads)
            k_climb<<<grid_for(M, 64), 64, 0, s>>>(b->vals[1 - cur], arrive + M + kGroupTrees, order,
                                                   b->aabb, b->nodes, parent_int, parent_leaf, arrive,
                                                   b->link);
    }
    if (b->node_format == GS_NODES_WIDE4 || b->node_format == GS_NODES_WIDE4_Q8) {
        const int64_t n_int = b->n_nodes;
        if (M == 1) {
            if ((e = cudaMemsetAsync(b->depth, 0, 4, s)) != cudaSuccess) return cuda_fail(e, "memset depth");
            if ((e = cudaMemsetAsync(b->wmap, 0, 4, s)) != cudaSuccess) return cuda_fail(e, "memset map");
        } else {
            k_depth<<<grid_for(n_int, 256), 256, 0, s>>>(n_int, b->parent, b->depth, b->wmap);
            scan_exclusive(b->wmap, n_int, b->scan_tmp, s);
        }
        if (b->node_format == GS_NODES_WIDE4)
            k_collapse<GS_NODES_WIDE4><<<grid_for(n_int, 256), 256, 0, s>>>(n_int, b->nodes, b->depth,
                                                                            b->wmap, b->wide);
        else
            k_collapse<GS_NODES_WIDE4_Q8><<<grid_for(n_int, 256), 256, 0, s>>>(
                n_int, b->nodes, b->depth, b->wmap, b->wide);
    }
    if (b->link) {
        const int64_t n_int = b->n_nodes;
        const bool q8 = b->node_format == GS_NODES_BINARY_Q8;
        WideRefs refs;
        WideOut out;
        for (int w = 0; w < kGroupTrees; ++w) {
            refs.ref[w] = b->group[w].ref;
            out.ref[w] = b->group[w].ref;
            out.rec[w] = b->group[w].rec;
        }
        k_wide_offsets<<<grid_for(n_int, 1024), 256, 0, s>>>(
            n_int, b->link, arrive + M, q8 ? (uint32_t)kGroupQHeaderUnits : 0u, refs);
        if (q8) k_wide_records<true><<<grid_for(n_int, 256), 256, 0, s>>>(n_int, b->nodes, b->link, out);
        else k_wide_records<false><<<grid_for(n_int, 256), 256, 0, s>>>(n_int, b->nodes, b->link, out);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "build launch");
    return GS_OK;
}

}  // namespace gsrt
