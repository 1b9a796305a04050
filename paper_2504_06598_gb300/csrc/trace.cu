// trace.cu -- stochastic ray tracing of transparent Gaussians on sm_103a.
//
// One warp per tile of pixels. A lane carries S consecutive samples of its
// pixel (the launch's passes have N * S slots, see launch_trace); the 32
// lanes are split into pixels x lanes: the L lanes of one pixel trace passes
// sub, sub + L, ... of the same camera ray (L the largest power of two not
// above the passes, at most 32), so they share their ray and differ only in
// the random draws and the clips they cause; with one pass per pixel the
// tile is 8x4 pixels. With 8 or more lanes on a pixel the group walks a wide
// copy together (traverse_group), otherwise the warp traverses as a tile
// (traverse_tile) or, for the options that are about the per-lane walk and for
// very small or dense scenes, as a packet (traverse_packet); in small images a
// warp takes one pixel, and from 33 to 127 samples a pixel one walk may serve
// four pixels (k_trace_shared); choose_walk has the lines. Each pass is one
// traversal of the hierarchy
// (Sec. 3.2) keeping its closest accepted intersections (Sec. 3.5). At every
// leaf the intersection routine of Alg. 1 runs:
//   t    mean of the 1D Gaussian along the ray (Sec. 3.1)
//   cull if t <= t_min or t is not before the slot's hit, or if the mean
//        lies outside the bounding ellipsoid (Eq. 2: q > s^2 = 8)
//   alpha = opacity * exp(-q/2), q the minimum of the Mahalanobis form
//   accept iff xi < alpha (Eq. 4, Fig. 2), replacing the slot (Eq. 6) and
//        clipping the traversal range to the farthest slot.
// After the traversal each slot is shaded once (SH colour, Sec. 3.2) or gets
// the background, and the pixel accumulates the mean of Eq. 7. On request
// every sample's slot {tc, tau, id} is also stored, [pixel][sample], for a
// gradient launch that reads it instead of tracing again.
//
// Float32 formulation of the 1D Gaussian. With o the ray origin, d the unit
// direction, mu the mean and M = S^-1 R_q^T:
//   o - mu = h + l exactly (h rounded, l its rounding error),
//   tc = -(h . d) puts the base point P = o + tc d near the mean,
//   w = P - mu = fma(tc, d, h) + l is accurate to the rounding of its own
//       (small) magnitude, whatever rounding tc carries, because q does not
//       depend on which point of the ray is used as base,
//   tau = -(Mw . Md) / |Md|^2 is the 1D mean relative to P,
//   w2 = w + tau d, q = |M w2|^2 - (M w2 . Md)^2 / |Md|^2.
// The depth is t = tc + tau; depths are compared through (tc, tau) pairs so
// that two nearby hits are ordered to the accuracy of tau, not of t.
#include <cuda_runtime.h>
#include <math.h>

#include "trace_common.cuh"

namespace gsrt {
namespace {

// Template values of FMT for the cooperative traversal of the wide records by
// groups of L = 8, 16, 32 lanes on one pixel: kFmtGroup + log2 L for the
// FP32 records, kFmtGroupQ8 + log2 W for the 8-bit ones; the others are
// GS_NODES_*.
constexpr int kFmtGroup = 8;
constexpr int kFmtGroupQ8 = 16;
// Tile traversal of the 32-wide records by a warp of camera rays, with and
// without the test of each leaf's box.
constexpr int kFmtTileLeaf = 4, kFmtTileLeafQ8 = 5, kFmtTile = 6, kFmtTileQ8 = 7;
__host__ __device__ constexpr bool is_tile_fmt(int f) { return f >= kFmtTileLeaf && f <= kFmtTileQ8; }
__host__ __device__ constexpr bool is_group_fmt(int f) { return f >= kFmtGroup + 3; }
__host__ __device__ constexpr bool is_group_q8(int f) { return f >= kFmtGroupQ8 + 3; }

// Persistent kernel: each warp repeatedly takes the next tile (one atomic
// per tile, so the tail of the launch stays balanced), then runs all passes
// of its pixels. The grouped form is latency-bound and is built for eight
// resident blocks per SM with one or two slots per lane (64 registers),
// seven with four (72: fewer spills of the four slots), five with eight;
// the packets for eight with up to four slots (as packets of the 1M shell at
// 1080p, against five: spp 1 4.77 -> 4.31 ms, spp 16 with four slots 16.9 -> 15.9
// ms) and six with eight (85 registers; against one, four, five and eight blocks:
// spp 16 with eight slots 14.8, 13.3, 12.4, 11.7 and 12.1 ms). The tiles have the
// packets' bounds; seven blocks with eight slots gained 3% at 1080p and cost 4%
// at 411x307.
constexpr int group_min_blocks(int n) { return n >= 8 ? 5 : (n >= 4 ? 7 : kGroupMinBlocks); }

template <int N, bool COUNT, int FMT>
__global__ void __launch_bounds__(kThreads, is_group_fmt(FMT) ? group_min_blocks(N)
                                                               : (N >= 8 ? 6 : 8))
    k_trace(const __grid_constant__ TraceArgs a) {
    const int lane = threadIdx.x & 31;
    const uint32_t kAll = 0xffffffffu;
    const int lg = a.lpp_log2, L = 1 << lg;
    const int tw_lg = tile_w_log2(lg), th_lg = 5 - lg - tw_lg;
    const int sub = lane & (L - 1), pl = lane >> lg;
    const uint32_t tiles_x = (uint32_t)((a.width + (1 << tw_lg) - 1) >> tw_lg);
    const uint32_t tiles_y = (uint32_t)((a.height + (1 << th_lg) - 1) >> th_lg);
    const uint32_t n_tiles = tiles_x * tiles_y;
    const int64_t npix = (int64_t)a.width * a.height;
    uint32_t stack[kMaxStack];
    float stack_t[kMaxStack];
    uint32_t err = 0;
    Counts cnt;
    unsigned long long n_shaded = 0, n_rays = 0;
    // group stacks: each warp's pool split evenly among its groups (a tile's
    // warp is one group)
    constexpr bool grouped = is_group_fmt(FMT), tiled = is_tile_fmt(FMT);
    constexpr int LG = grouped ? (FMT & 7) : 5;
    constexpr bool pooled = grouped || tiled;
    constexpr int pool = tiled ? kTilePool : grouped ? kGroupPool : 1;
    __shared__ uint32_t s_ref[pooled ? kThreads / 32 : 1][pool];
    __shared__ float s_t[pooled ? kThreads / 32 : 1][pool];
    __shared__ __align__(16) float s_pyr[tiled ? kThreads / 32 : 1][tiled ? kTileFloats : 4];
    const int grp_off = grouped ? (lane >> LG) * (kGroupPool >> (5 - LG)) : 0;
    uint32_t *grp_ref = s_ref[pooled ? threadIdx.x >> 5 : 0] + grp_off;
    float *grp_t = s_t[pooled ? threadIdx.x >> 5 : 0] + grp_off;
    float *pyr = s_pyr[tiled ? threadIdx.x >> 5 : 0];
    // a warp on one pixel with more passes than its layout has lanes: the colours
    // (at most 64) pass through the walk's stack. (Otherwise each pass is a lane's
    // own in the layout too.)
    const bool relay = grouped && LG == 5 && !COUNT && a.sum_log2 < 5 && a.spp > 1 << a.sum_log2;
    float(*colour)[64] = reinterpret_cast<float(*)[64]>(grp_ref);
    const int sum_lanes = relay ? 1 << a.sum_log2 : L;
    for (;;) {
        uint32_t tile = 0;
        const int more = next_tile(a, tiles_x, n_tiles, tile);
        if (more == 0) break;
        if (more < 0) continue;
        const int x = (int)(((tile % tiles_x) << tw_lg) + (pl & ((1 << tw_lg) - 1)));
        const int y = (int)(((tile / tiles_x) << th_lg) + (pl >> tw_lg));
        const bool valid = x < a.width && y < a.height;
        const int64_t pix = valid ? (int64_t)y * a.width + x : 0;
        Ray<N> r;
        {
            float d[3];
            camera_ray(a, valid ? x : 0, valid ? y : 0, d);
            set_ray(r, a.eye, d);
        }
        r.ray_id = a.ray_id_offset + (uint32_t)pix;
        r.stream_tag = a.stream_tag;
        r.t_min = a.t_min;
        r.t_max = a.t_max;
        r.any_hit = false;
        if constexpr (tiled) tile_pyramid(r.d, valid, pyr);
        float acc[3] = {0.0f, 0.0f, 0.0f};
        const int n_rounds = (a.spp + L - 1) >> lg;
        for (int j = 0; j < n_rounds; ++j) {
            const int pass = (j << lg) + sub;
            const bool live = valid && pass < a.spp;
            const int s0 = pass * N;
            // an unused slot (sample index beyond the pixel's count) sits
            // at -inf: no candidate is closer, and it never sets the clip
#pragma unroll
            for (int k = 0; k < N; ++k)
                r.slot[k] = s0 + k < a.n_samples ? Slot{INFINITY, 0.0f, 0xffffffffu}
                                                 : Slot{-INFINITY, 0.0f, 0xffffffffu};
            update_clip(r, a.t_max);
            if (!live) r.t_far = -INFINITY;  // lanes off the image never hit
            if (a.n_nodes > 0) {
                if constexpr (tiled) {
                    trace_tile<N, (FMT & 1) != 0, FMT <= kFmtTileLeafQ8>(a, r, pass, a.eye, pyr, grp_ref, grp_t, err);
                } else if constexpr (grouped) {
                    uint32_t e = 0;
                    traverse_group<N, COUNT, LG, true, is_group_q8(FMT)>(a, r, pass, grp_ref,
                                                                          grp_t, e, cnt);
                    if (!COUNT && __any_sync(kAll, e & kErrStack)) {
                        e &= ~kErrStack;
                        start_over<N>(a, r, pass, e);
                    }
                    err |= e;
                }
                else if constexpr (FMT == GS_NODES_BINARY)
                    traverse_packet<N, COUNT>(a, r, pass, stack, stack_t, err, cnt);
                else
                    traverse_packet_wide<N, COUNT, FMT>(a, r, pass, stack, stack_t, err, cnt);
            }
            if (relay) __syncwarp();  // the walk's reads of the stack are done
            if (live) {
                // shade each slot once (Eq. 6) and accumulate (Eq. 7)
                float Y[16];
                sh_basis(a.sh_degree, r.d, Y);
#pragma unroll
                for (int k = 0; k < N; ++k) {
                    if (s0 + k >= a.n_samples) continue;
                    float c[3];
                    if (r.slot[k].gid != 0xffffffffu) {
                        sh_colour(a, r.slot[k].gid, Y, c);
                        if (COUNT) ++n_shaded;
                    } else {
                        c[0] = a.bg[0]; c[1] = a.bg[1]; c[2] = a.bg[2];
                    }
                    if (relay) {
                        for (int i = 0; i < 3; ++i) colour[i][s0 + k] = c[i];
                    } else {
                        acc[0] += c[0];
                        acc[1] += c[1];
                        acc[2] += c[2];
                    }
                    if (a.hit_id) {
                        const int64_t o = ((int64_t)s0 + k) * npix + pix;
                        a.hit_id[o] = r.slot[k].gid == 0xffffffffu ? -1 : (int32_t)r.slot[k].gid;
                        a.hit_t[o] = r.slot[k].t();
                    }
                }
                if (a.keys) {
                    gs_sample_key *key = a.keys + pix * a.n_samples + s0;
#pragma unroll
                    for (int k = 0; k < N; ++k) {
                        if (s0 + k >= a.n_samples) continue;
                        key[k].tc = r.slot[k].tc;
                        key[k].tau = r.slot[k].tau;
                        key[k].gid = r.slot[k].gid;
                    }
                }
            }
            __syncwarp();
            if (relay) {
                add_in_layout(colour, 0, a.n_samples, log2_of(N), a.sum_log2, lane, acc);
                __syncwarp();
            }
        }
        // the pixel's lanes add their partial sums (Eq. 7)
        for (int o = sum_lanes >> 1; o >= 1; o >>= 1) {
            acc[0] += __shfl_xor_sync(kAll, acc[0], o);
            acc[1] += __shfl_xor_sync(kAll, acc[1], o);
            acc[2] += __shfl_xor_sync(kAll, acc[2], o);
        }
        if (valid && sub == 0) {
            const float inv_n = 1.0f / (float)a.n_samples;
            a.rgb[3 * pix + 0] = acc[0] * inv_n;
            a.rgb[3 * pix + 1] = acc[1] * inv_n;
            a.rgb[3 * pix + 2] = acc[2] * inv_n;
            if (COUNT) ++n_rays;
        }
    }
    if (err) atomicOr(a.status, err);
    if (COUNT) {
        atomicAdd(a.counters + 0, cnt.nodes);
        atomicAdd(a.counters + 1, cnt.prims);
        atomicAdd(a.counters + 2, cnt.draws);
        atomicAdd(a.counters + 3, n_rays);
        atomicAdd(a.counters + 4, n_shaded);
        atomicAdd(a.counters + 5, cnt.node_fetch);
        atomicAdd(a.counters + 6, cnt.prim_fetch);
    }
}

// ---------------------------------------------------------------- shared walks
// From 33 to 127 samples a pixel: a warp holds a 2x2 tile, walks the 32-wide copy
// once for its four pixels (the pyramid test of traverse_tile), evaluates the
// surviving Gaussians with a lane per (pixel, Gaussian) pair, eight Gaussians
// for the four pixels at a time, and then draws for one pixel after the
// other, all 32 lanes with two samples each. A pixel's 64 samples are kept in
// shared memory (three words each) between its turns. The grouped form (one
// pixel a warp) spent more on its walk than on its draws (1M shell at 1080p:
// 13.6 ms of 23.0 at spp 64; now 17.8, issue 77%); evaluating per lane as the
// tiles do repeats each evaluation on the pixel's lanes.
constexpr int kSharedPx = 4;
constexpr int kSharedPool = 192;  // stack entries per warp

struct __align__(16) SharedWarp {
    float pyr[kTileFloats];
    float2 tc[kSharedPx][32], tau[kSharedPx][32];
    uint2 gid[kSharedPx][32];
    float dir[kSharedPx][4];
    union {
        uint32_t ref[kSharedPool];  // during a walk
        float colour[3][64];        // after it: of one pixel's samples
    };
    float t[kSharedPool];
    uint32_t leaves[32];
    float acc[kSharedPx][3][32];  // partial sums
};

__device__ __forceinline__ void load_slots(const SharedWarp &m, int p, int lane, Ray<2> &r) {
    const float2 tc = m.tc[p][lane], tau = m.tau[p][lane];
    const uint2 gid = m.gid[p][lane];
    r.slot[0] = Slot{tc.x, tau.x, gid.x};
    r.slot[1] = Slot{tc.y, tau.y, gid.y};
}

__device__ __forceinline__ void store_slots(SharedWarp &m, int p, int lane, const Ray<2> &r) {
    m.tc[p][lane] = make_float2(r.slot[0].tc, r.slot[1].tc);
    m.tau[p][lane] = make_float2(r.slot[0].tau, r.slot[1].tau);
    m.gid[p][lane] = make_uint2(r.slot[0].gid, r.slot[1].gid);
}

// The largest clip of the warp's lanes (-inf where none is in range).
__device__ __forceinline__ float warp_clip(float t_far, float t_min) {
    const uint32_t b = t_far >= t_min ? __float_as_uint(fmaxf(t_far, 0.0f)) + 1u : 0u;
    const uint32_t m = __reduce_max_sync(0xffffffffu, b);
    return m ? __uint_as_float(m - 1u) : -INFINITY;
}

// Two candidates of pixel p at a time, nearest first, as in traverse_group:
// an even lane draws for the first, an odd lane for the second, and the two
// swap the halves. ok: this lane holds a candidate (of its own pixel).
__device__ __forceinline__ float shared_draws(const TraceArgs &a, SharedWarp &m, int p, int lane,
                                              uint32_t ray_id, uint32_t counter, bool ok, float ct,
                                              float ck1, float ck2, float cal, uint32_t cgid,
                                              float G) {
    const uint32_t kAll = 0xffffffffu;
    const bool odd = lane & 1;
    Ray<2> r;
    load_slots(m, p, lane, r);
    r.t_min = a.t_min;
    r.t_max = a.t_max;
    r.any_hit = false;
    update_clip(r, a.t_max);
    if (!(r.t_far > -INFINITY)) r.t_far = -INFINITY;  // no sample here
    const uint32_t depth = (__float_as_uint(fmaxf(ct, 0.0f)) & ~31u) | (uint32_t)lane;
    bool drawn = false;
    for (;;) {
        const uint32_t k0 = __reduce_min_sync(kAll, ok ? depth : 0xffffffffu);
        if (k0 == 0xffffffffu) break;
        const int j0 = (int)(k0 & 31u);
        if (lane == j0) ok = false;
        const uint32_t k1 = __reduce_min_sync(kAll, ok ? depth : 0xffffffffu);
        const bool two = k1 != 0xffffffffu;
        const int j1 = two ? (int)(k1 & 31u) : j0;
        if (lane == j1) ok = false;
        const uint32_t gid0 = __shfl_sync(kAll, cgid, j0), gid1 = __shfl_sync(kAll, cgid, j1);
        const uint4 u = philox10_rk(make_uint4(ray_id, odd ? gid1 : gid0, counter, a.stream_tag), a.rk);
        const uint32_t x0 = __shfl_xor_sync(kAll, odd ? u.x : u.z, 1);
        const uint32_t x1 = __shfl_xor_sync(kAll, odd ? u.y : u.w, 1);
        const float far0 = r.t_far;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            if (q == 1 && !two) break;
            const int src = q ? j1 : j0;
            const float t = __shfl_sync(kAll, ct, src);
            const float key_tc = __shfl_sync(kAll, ck1, src);
            const float key_tau = __shfl_sync(kAll, ck2, src);
            const float alpha = __shfl_sync(kAll, cal, src);
            bool closer[2];
            if (closer_slots<2>(r, t, key_tc, key_tau, q ? gid1 : gid0, closer)) {
                drawn = true;
                const bool own = odd == (q == 1);
                uint32_t bits[2];
                bits[0] = own ? (odd ? u.z : u.x) : x0;
                bits[1] = own ? (odd ? u.w : u.y) : x1;
                apply_draws<2>(a, r, closer, bits, key_tc, key_tau, alpha, q ? gid1 : gid0);
            }
        }
        if (__any_sync(kAll, r.t_far != far0)) {
            G = warp_clip(r.t_far, a.t_min);
            ok = ok && ct <= G;
        }
    }
    if (drawn) store_slots(m, p, lane, r);
    return G;
}

template <bool Q8>
__global__ void __launch_bounds__(kThreads, 8) k_trace_shared(const __grid_constant__ TraceArgs a) {
    __shared__ SharedWarp s_warp[kThreads / 32];
    const uint32_t kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    SharedWarp &m = s_warp[threadIdx.x >> 5];
    const int ep = lane >> 3;  // the pixel this lane evaluates for
    const uint32_t tiles_x = (uint32_t)((a.width + 1) >> 1);
    const uint32_t n_tiles = tiles_x * (uint32_t)((a.height + 1) >> 1);
    const int64_t npix = (int64_t)a.width * a.height;
    uint32_t err = 0;
    for (;;) {
        uint32_t tile = 0;
        const int more = next_tile(a, tiles_x, n_tiles, tile);
        if (more == 0) break;
        if (more < 0) continue;
        const int x0 = (int)(tile % tiles_x) * 2, y0 = (int)(tile / tiles_x) * 2;
        Ray<1> er;  // the ray this lane evaluates along
        const bool valid = x0 + (ep & 1) < a.width && y0 + (ep >> 1) < a.height;
        camera_ray(a, valid ? x0 + (ep & 1) : 0, valid ? y0 + (ep >> 1) : 0, er.d);
        for (int i = 0; i < 3; ++i) er.o[i] = a.eye[i];
        er.t_min = a.t_min;
        er.t_max = a.t_max;
        tile_pyramid(er.d, valid, m.pyr);
        if ((lane & 7) < 3) m.dir[ep][lane & 7] = (lane & 7) == 0 ? er.d[0] : (lane & 7) == 1 ? er.d[1] : er.d[2];
        for (int base = 0; base < a.n_samples; base += 64) {
            const int s0 = base + 2 * lane;
            float G;
            {
                Ray<1> all;
                all.slot[0] = Slot{INFINITY, 0.0f, 0xffffffffu};
                update_clip(all, a.t_max);
                G = valid ? all.t_far : -INFINITY;
            }
#pragma unroll
            for (int p = 0; p < kSharedPx; ++p) {
                m.tc[p][lane] = make_float2(s0 < a.n_samples ? INFINITY : -INFINITY,
                                            s0 + 1 < a.n_samples ? INFINITY : -INFINITY);
                m.tau[p][lane] = make_float2(0.0f, 0.0f);
                m.gid[p][lane] = make_uint2(0xffffffffu, 0xffffffffu);
            }
            __syncwarp();
            float g = warp_clip(G, a.t_min), g2 = g * g;
            bool full = false;
            int sp = 0;
            uint32_t node = a.n_nodes > 0 ? __ldg(a.troot) : 0u, steps = 0;
            bool walk = a.n_nodes > 0 && g >= a.t_min;
            while (walk) {
                if (++steps > a.step_limit) {
                    err |= kErrSteps;
                    break;
                }
                const int n_child = (int)((node >> kWideCountShift) & 31u) + 1;
                uint32_t ref = kEmpty;
                float d2 = INFINITY, lo[3], hi[3];
                bool hit = false;
                if (lane < n_child)
                    hit = tile_child<Q8>(a.trec, node, lane, a.eye, m.pyr, g2, ref, d2, lo, hi);
                const bool leaf = (ref & kLeafBit) != 0u;
                const uint32_t lm = __ballot_sync(kAll, hit && leaf);
                if (lm) {
                    if (hit && leaf) m.leaves[__popc(lm & ((1u << lane) - 1u))] = ref & ~kLeafBit;
                    __syncwarp();
                    const int n_leaf = __popc(lm);
                    for (int b = 0; b < n_leaf; b += 8) {
                        const int c = b + (lane & 7);
                        float ct = 0.0f, ck1 = 0.0f, ck2 = 0.0f, cal = 0.0f;
                        uint32_t cgid = 0;
                        bool ok = false;
                        if (c < n_leaf && G >= a.t_min) {
                            CandGeom cg;
                            ok = cand_depth<1, true>(a, er, m.leaves[c], cg) && cg.t <= G &&
                                 cand_alpha<1, true>(a, er, cg, cal);
                            ct = cg.t;
                            ck1 = cg.key_tc;
                            ck2 = cg.key_tau;
                            cgid = cg.gid;
                        }
                        uint32_t okm = __ballot_sync(kAll, ok);
                        while (okm) {
                            const int p = (__ffs(okm) - 1) >> 3;
                            okm &= ~(0xffu << (8 * p));
                            const uint32_t id = a.ray_id_offset +
                                                (uint32_t)((int64_t)(y0 + (p >> 1)) * a.width + x0 + (p & 1));
                            const float Gp = __shfl_sync(kAll, G, 8 * p);
                            const float Gn =
                                shared_draws(a, m, p, lane, id, (uint32_t)(base >> 2) + (lane >> 1),
                                             ok && ep == p, ct, ck1, ck2, cal, cgid, Gp);
                            if (ep == p) G = Gn;
                        }
                    }
                    g = warp_clip(G, a.t_min);
                    g2 = g * g;
                    if (!(g >= a.t_min)) break;
                    __syncwarp();
                }
                const bool inner = hit && !leaf && d2 <= g2;
                const uint32_t im = __ballot_sync(kAll, inner);
                if (im) {
                    const uint32_t key = (__float_as_uint(d2) & ~31u) | (uint32_t)lane;
                    const int nj = (int)(__reduce_min_sync(kAll, inner ? key : 0xffffffffu) & 31u);
                    const uint32_t next = __shfl_sync(kAll, ref, nj);
                    const uint32_t others = im & ~(1u << nj);
                    const int npush = __popc(others);
                    if (sp + npush > kSharedPool >> kPoolShift) {
                        full = true;
                        break;
                    }
                    __syncwarp();
                    if (inner && lane != nj) {
                        const int pos = sp + __popc(others & ((1u << lane) - 1u));
                        m.ref[pos] = ref;
                        m.t[pos] = d2;
                    }
                    sp += npush;
                    __syncwarp();
                    node = next;
                    continue;
                }
                walk = false;
                while (sp > 0) {
                    const int k = sp - 1 - lane;
                    const uint32_t okm = __ballot_sync(kAll, k >= 0 && m.t[k >= 0 ? k : 0] <= g2);
                    if (okm) {
                        sp -= __ffs(okm);  // the lowest lane holds the topmost
                        node = m.ref[sp];
                        walk = true;
                        break;
                    }
                    sp = sp > 32 ? sp - 32 : 0;
                }
            }
            // shade each slot once (Eq. 6) and accumulate (Eq. 7)
#pragma unroll 1
            for (int p = 0; p < kSharedPx; ++p) {
                const int x = x0 + (p & 1), y = y0 + (p >> 1);
                if (x >= a.width || y >= a.height) continue;
                const int64_t pix = (int64_t)y * a.width + x;
                Ray<2> r;
                load_slots(m, p, lane, r);
                for (int i = 0; i < 3; ++i) r.d[i] = m.dir[p][i];
                if (full) {
                    // (the stack did not do: this pixel's samples again)
                    for (int i = 0; i < 3; ++i) r.o[i] = a.eye[i];
                    r.ray_id = a.ray_id_offset + (uint32_t)pix;
                    r.stream_tag = a.stream_tag;
                    r.t_min = a.t_min;
                    r.t_max = a.t_max;
                    r.any_hit = false;
                    update_clip(r, a.t_max);
                    if (!(r.t_far > -INFINITY)) r.t_far = -INFINITY;
                    start_over<2>(a, r, s0 >> 1, err);
                }
                float Y[16];
                sh_basis(a.sh_degree, r.d, Y);
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    if (s0 + k >= a.n_samples) continue;
                    float c[3];
                    if (r.slot[k].gid != 0xffffffffu) {
                        sh_colour(a, r.slot[k].gid, Y, c);
                    } else {
                        c[0] = a.bg[0]; c[1] = a.bg[1]; c[2] = a.bg[2];
                    }
                    for (int i = 0; i < 3; ++i) m.colour[i][2 * lane + k] = c[i];
                    if (a.hit_id) {
                        const int64_t o = ((int64_t)s0 + k) * npix + pix;
                        a.hit_id[o] = r.slot[k].gid == 0xffffffffu ? -1 : (int32_t)r.slot[k].gid;
                        a.hit_t[o] = r.slot[k].t();
                    }
                    if (a.keys) {
                        gs_sample_key *key = a.keys + pix * a.n_samples + s0 + k;
                        key->tc = r.slot[k].tc;
                        key->tau = r.slot[k].tau;
                        key->gid = r.slot[k].gid;
                    }
                }
                __syncwarp();
                float acc[3];
                for (int i = 0; i < 3; ++i) acc[i] = base > 0 ? m.acc[p][i][lane] : 0.0f;
                add_in_layout(m.colour, base, min(base + 64, a.n_samples), a.k_log2, a.sum_log2,
                              lane, acc);
                for (int i = 0; i < 3; ++i) m.acc[p][i][lane] = acc[i];
                __syncwarp();
            }
            __syncwarp();
        }
#pragma unroll 1
        for (int p = 0; p < kSharedPx; ++p) {
            const int x = x0 + (p & 1), y = y0 + (p >> 1);
            if (x >= a.width || y >= a.height) continue;
            float acc[3];
            for (int i = 0; i < 3; ++i) acc[i] = m.acc[p][i][lane];
            for (int o = (1 << a.sum_log2) >> 1; o >= 1; o >>= 1) {
                acc[0] += __shfl_xor_sync(kAll, acc[0], o);
                acc[1] += __shfl_xor_sync(kAll, acc[1], o);
                acc[2] += __shfl_xor_sync(kAll, acc[2], o);
            }
            if (lane == 0) {
                const float inv_n = 1.0f / (float)a.n_samples;
                const int64_t pix = (int64_t)y * a.width + x;
                for (int i = 0; i < 3; ++i) a.rgb[3 * pix + i] = acc[i] * inv_n;
            }
        }
        __syncwarp();
    }
    if (err) atomicOr(a.status, err);
}

template <bool Q8>
gs_status launch_shared(const TraceArgs &a, cudaStream_t s) {
    int dev = 0, sms = 0, per = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_trace_shared<Q8>, kThreads, 0);
    if (e != cudaSuccess) return cuda_fail(e, "trace launch setup");
    const int64_t tiles = (int64_t)((a.width + 1) >> 1) * ((a.height + 1) >> 1);
    const int64_t need = (tiles + kThreads / 32 - 1) / (kThreads / 32);
    const int64_t fit = (int64_t)sms * (per > 0 ? per : 1);
    if (a.order == nullptr &&
        (e = cudaMemsetAsync(a.work, 0, sizeof(uint32_t), s)) != cudaSuccess)
        return cuda_fail(e, "reset work counter");
    k_trace_shared<Q8><<<(unsigned)(need < fit ? need : fit), kThreads, 0, s>>>(a);
    return GS_OK;
}

template <int N, int FMT>
gs_status launch_nf(const TraceArgs &a, bool count, cudaStream_t s) {
    int dev = 0, sms = 0, per = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = count ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_trace<N, !is_tile_fmt(FMT), FMT>, kThreads, 0)
                  : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_trace<N, false, FMT>, kThreads, 0);
    if (e != cudaSuccess) return cuda_fail(e, "trace launch setup");
    // one resident grid; warps take tiles until none is left
    const int tw_lg = tile_w_log2(a.lpp_log2), th_lg = 5 - a.lpp_log2 - tw_lg;
    const uint32_t tiles = (uint32_t)(((a.width + (1 << tw_lg) - 1) >> tw_lg) *
                                      ((a.height + (1 << th_lg) - 1) >> th_lg));
    const uint32_t warps_needed = tiles;
    uint32_t blocks = (uint32_t)sms * (uint32_t)(per > 0 ? per : 1);
    const uint32_t max_blocks = (warps_needed + kThreads / 32 - 1) / (kThreads / 32);
    if (blocks > max_blocks) blocks = max_blocks;
    if (a.order == nullptr &&
        (e = cudaMemsetAsync(a.work, 0, sizeof(uint32_t), s)) != cudaSuccess)
        return cuda_fail(e, "reset work counter");
    if (count) k_trace<N, !is_tile_fmt(FMT), FMT><<<blocks, kThreads, 0, s>>>(a);
    else k_trace<N, false, FMT><<<blocks, kThreads, 0, s>>>(a);
    return GS_OK;
}

template <int N>
gs_status launch_n(const TraceArgs &a, int format, bool count, cudaStream_t s) {
    if (a.trec != nullptr && a.leaf_test)
        return a.gq8 ? launch_nf<N, kFmtTileLeafQ8>(a, false, s)
                     : launch_nf<N, kFmtTileLeaf>(a, false, s);
    if (a.trec != nullptr)
        return a.gq8 ? launch_nf<N, kFmtTileQ8>(a, false, s) : launch_nf<N, kFmtTile>(a, false, s);
    // groups of 8 or more lanes on one pixel take the cooperative form
    if (format == GS_NODES_BINARY && a.grec != nullptr) {
        if (a.lpp_log2 == 5) return launch_nf<N, kFmtGroup + 5>(a, count, s);
        if (a.lpp_log2 == 4) return launch_nf<N, kFmtGroup + 4>(a, count, s);
        if (a.lpp_log2 == 3) return launch_nf<N, kFmtGroup + 3>(a, count, s);
    }
    if (format == GS_NODES_BINARY_Q8 && a.grec != nullptr) {
        if (a.lpp_log2 == 5) return launch_nf<N, kFmtGroupQ8 + 5>(a, count, s);
        if (a.lpp_log2 == 4) return launch_nf<N, kFmtGroupQ8 + 4>(a, count, s);
        if (a.lpp_log2 == 3) return launch_nf<N, kFmtGroupQ8 + 3>(a, count, s);
    }
    switch (format) {
        case GS_NODES_WIDE4: return launch_nf<N, GS_NODES_WIDE4>(a, count, s);
        case GS_NODES_WIDE4_Q8: return launch_nf<N, GS_NODES_WIDE4_Q8>(a, count, s);
        default: return launch_nf<N, GS_NODES_BINARY>(a, count, s);
    }
}

// Samples one lane carries when the caller leaves the choice to the
// library (samples_per_lane = 0). The time follows the number of walks a
// pixel needs and grows slowly with the slots a walk carries. Measured on
// the 1M-Gaussian shell at 1080p with packets and groups, which every layout can
// take (the tiles and shared walks that the library prefers keep the layout's
// sums but take less: T = 1 2.9 ms, 16 8.4, 64 15.5), trace ms for K = n_hits * S
// slots per lane and T = spp * n_hits samples per pixel (one sample per lane
// first):
//   T = 4:   K 1 14.1, 2 7.6, 4 5.4 (per-lane packets)
//   T = 8:   K 1 20.1, 4 8.8, 8 7.1
//   T = 16:  K 1 24.2, 4 15.9, 8 11.7
//   T = 32:  K 1 27.5, 2 27.0, 4 25.5 (8 lanes a pixel, grouped), 8 21.0
//   T = 64:  K 1 52.3, 2 30.4 (32 lanes, grouped), 4 30.5, 8 38.5
//   T = 128: K 2 59.8, 4 34.4, 8 46.4;  T = 256: K 4 67.5, 8 52.5
// K is never below n_hits.
int auto_samples_per_lane(int spp, int n_hits, int node_format) {
    (void)node_format;
    const int64_t T = (int64_t)spp * n_hits;
    int K;
    if (T <= 2) K = (int)T;
    else if (T < 8) K = 4;
    else if (T < 64) K = 8;
    else if (T < 128) K = 2;
    else if (T < 256) K = 4;
    else K = 8;
    if (K < n_hits) K = n_hits;
    return K / n_hits;
}

}  // namespace

// Warps the current device holds at once at 64 registers a thread.
static int64_t resident_warps() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    return (int64_t)sms * 32;
}

// The walks of a launch: the layout's own (packets of the binary nodes, or
// groups of 8 and more lanes), tiles, a warp per pixel, or one walk for four
// pixels.
enum class Walk { kLayout, kTile, kWarp, kShared };

// Lines from the times (us) of shells of 10 to 1M Gaussians in images of 64x64 to
// 1080p, one to 256 samples a pixel.
static Walk choose_walk(const gs_bvh *b, const gs_pinhole *cam, const gs_trace_params *p, int n_eff,
                        int passes, int lpp_log2) {
    // the forms other than the layout's take depths along the ray from the eye
    // and none of the options that are about the per-lane walk
    if (!b->link || !(p->t_min >= 0.0f) || p->depth_mode != 0 || p->rng_mode != 0 ||
        p->stack_depth != 0 || p->counters != nullptr)
        return Walk::kLayout;
    const int64_t pix = (int64_t)cam->width * cam->height, T = (int64_t)p->spp * p->n_hits;
    const double waves = (double)pix / (double)resident_warps();  // of a warp per pixel
    const double field = field_pixels(cam);
    const bool many = p->samples_per_lane == 0 && T > 32;
    // A warp per pixel (most lanes without a sample, helping in the walk) evaluates
    // 32 Gaussians at a time, a tile's warp one after the other, so that the time
    // of few tiles is the longest tile's; but its work is the pixels'. Its share
    // of waves before it loses to tiles grows with the scene's size, as the
    // depth of a tile does: at one slot a lane 4 waves at 1,000 Gaussians (45 against
    // 62), 15 at 20,000 (233 against 313), 41 at 300,000 (1336 against 1367), 63 at
    // 1M (3108 against 2919); at eight slots two thirds, against shared walks a
    // quarter of that.
    if (lpp_log2 < 3 || (many && T < 64)) {
        double share = many ? 0.14 : n_eff < 8 ? 0.6 : 0.40 - 0.04 * lpp_log2;
        // (three or five to seven passes are two rounds of the layout's lanes)
        if (!many && passes > 1 << lpp_log2) share *= 1.6;
        if (waves < warp_waves(share, b->M, field, (double)resident_warps())) return Walk::kWarp;
    }
    // Eight to 31 passes of the caller's samples per lane: a whole warp does in one
    // round what groups of 8 or 16 lanes do in two, and more than groups of 16 do on
    // the 8-wide copy (spp 24, one a lane: 20,000 at 640x480 2036 -> 977, 1M 14.6 ->
    // 4.7 ms; spp 16: 90k 2213 -> 1686).
    if (!many && lpp_log2 >= 3 && passes < 32 && passes * n_eff <= 64 &&
        (passes > 1 << lpp_log2 ? b->M >= 4096 : lpp_log2 == 4 && b->M >= 65536))
        return Walk::kWarp;
    // Shared walks for 64 samples and more: a second walk for samples 64 to 127, where
    // the groups of four slots from 128 on still walk once. Below six waves of 2x2
    // tiles the groups' many small warps win (1M, spp 64: 320x240 1622 against 2305,
    // 500x400 3841 against 3305).
    if (many && T >= 64) return T < 128 && waves > 24.0 ? Walk::kShared : Walk::kLayout;
    // A few hundred Gaussians: the packets' steps are the cheapest, and with them a
    // launch is little more than its fixed cost (100 at 1080p, spp 4 90 against 119).
    if (b->M < 512) return Walk::kLayout;
    if (many) {
        // 33 to 63 samples are five to eight passes of tiles: with few Gaussians that
        // costs less than the draws of 64 (1,000 at 1080p 1448 against 1861; 20,000
        // 4222 against 3947)
        return b->M < 4096 && waves > 32.0 ? Walk::kTile : Walk::kShared;
    }
    if (lpp_log2 >= 3) return Walk::kLayout;
    // More than three Gaussians a ray of the tile: its farthest clip takes in so many
    // that packets, which clip per ray, do better (1M at 500x400, spp 8 4502 against
    // 5533; at 640x480 4428 against 4846).
    return (double)b->M > 3.0 * field * (double)(1 << lpp_log2) ? Walk::kLayout : Walk::kTile;
}

void trace_layout(const gs_bvh *b, const gs_trace_params *p, int *S_out, int *spp_eff_out,
                  int *lpp_log2_out, bool *grouped_out) {
    // A lane carries S consecutive samples: the launch runs ceil(spp / S)
    // passes of n_hits * S slots; sample s = pass * n_hits * S + k either way.
    int S = p->samples_per_lane > 0 ? p->samples_per_lane
                                    : auto_samples_per_lane(p->spp, p->n_hits, b->node_format);
    while (S > 1 && S > p->spp) S >>= 1;
    *S_out = S;
    *spp_eff_out = (p->spp + S - 1) / S;
    *lpp_log2_out = lanes_per_pixel_log2(*spp_eff_out);
    *grouped_out = (b->node_format == GS_NODES_BINARY || b->node_format == GS_NODES_BINARY_Q8) &&
                   b->link && *lpp_log2_out >= 3;
}

gs_status launch_trace(const gs_bvh *b, const gs_gaussians *g, const gs_pinhole *cam,
                       const gs_trace_params *p, float *rgb, int32_t *hit_id, float *hit_t,
                       gs_sample_key *keys, cudaStream_t s) {
    int S = 1, spp_eff = 1, lpp_log2 = 0;
    bool grouped = false;
    trace_layout(b, p, &S, &spp_eff, &lpp_log2, &grouped);
    const int n_eff = p->n_hits * S;
    const int sum_log2 = lpp_log2;
    const Walk walk = choose_walk(b, cam, p, n_eff, spp_eff, lpp_log2);
    const bool shared = walk == Walk::kShared, tile = walk == Walk::kTile;
    if (walk == Walk::kWarp) lpp_log2 = 5;
    TraceArgs a;
    a.nodes = b->nodes;
    a.wide = b->wide;
    a.lpp_log2 = lpp_log2;
    a.sum_log2 = sum_log2;
    if (b->link && a.lpp_log2 >= 3) {
        a.grec = b->group[group_tree(a.lpp_log2)].rec;
        a.groot = b->group[group_tree(a.lpp_log2)].ref;
    } else {
        a.grec = nullptr;
        a.groot = nullptr;
    }
    a.gq8 = b->node_format == GS_NODES_BINARY_Q8;
    a.trec = tile || shared ? b->group[kWarpTree].rec : nullptr;
    a.troot = tile || shared ? b->group[kWarpTree].ref : nullptr;
    a.leaf_test = leaf_test_pays(b->M, field_pixels(cam));
    a.prims = b->prims;
    a.sh = g->sh;
    a.n_nodes = b->n_nodes;
    a.sh_degree = g->sh_degree;
    a.sh_dtype = g->sh_dtype;
    a.width = cam->width;
    a.height = cam->height;
    a.ray_id_offset = cam->ray_id_offset;
    for (int i = 0; i < 3; ++i) {
        a.eye[i] = cam->eye[i];
        a.look_at[i] = cam->look_at[i];
        a.up[i] = cam->up[i];
        a.bg[i] = p->bg[i];
    }
    a.tan_half = (float)tan((double)cam->fov_y_deg * 3.14159265358979323846 / 360.0);
    a.key0 = (uint32_t)(p->seed & 0xffffffffu);
    a.key1 = (uint32_t)(p->seed >> 32);
    philox_round_keys(a.key0, a.key1, a.rk);
    a.stream_tag = p->stream_tag;
    a.spp = spp_eff;
    a.k_log2 = 0;
    while ((1 << a.k_log2) < n_eff) ++a.k_log2;
    a.n_samples = p->spp * p->n_hits;
    a.t_min = p->t_min;
    a.t_max = p->t_max;
    a.stack_depth = p->stack_depth == 0 ? kMaxStack : p->stack_depth;
    // a valid traversal visits every internal node at most once per pass
    a.step_limit = (uint32_t)(b->n_nodes + 8 < (int64_t)kStepLimit ? b->n_nodes + 8 : kStepLimit);
    a.rgb = rgb;
    a.hit_id = hit_id;
    a.hit_t = hit_t;
    a.keys = keys;
    a.n_gauss = (uint32_t)b->M;
    a.counters = p->counters;
    a.status = b->status;
    a.work = b->status + 1;
    a.depth_mode = p->depth_mode;
    a.rng_mode = p->rng_mode;
    {
        // camera forward axis, float32 normalise as for the camera rays
        float f[3];
        for (int i = 0; i < 3; ++i) f[i] = cam->look_at[i] - cam->eye[i];
        float n2 = f[0] * f[0];
        n2 = n2 + f[1] * f[1];
        n2 = n2 + f[2] * f[2];
        const float n = sqrtf(n2);
        for (int i = 0; i < 3; ++i) a.fwd[i] = f[i] / n;
    }
    const bool count = p->counters != nullptr;
    gs_status st;
    a.order = nullptr;
    // below three waves the longest tile decides, whatever the order (90k at
    // 411x307, 1.6 waves: 1119 us by rows, 1147 ordered), and a launch of 200 us does
    // not gain the two launches' 20 (1,000 at 1080p, spp 1 119 by rows, 137 ordered,
    // spp 8 303 and 276)
    const bool worth = b->M >= 4096 || (b->M >= 512 && (int64_t)p->spp * p->n_hits >= 8);
    const int tw_lg = shared ? 1 : tile_w_log2(a.lpp_log2), th_lg = shared ? 1 : 5 - a.lpp_log2 - tw_lg;
    const int64_t tiles = (((int64_t)a.width + (1 << tw_lg) - 1) >> tw_lg) *
                          (((int64_t)a.height + (1 << th_lg) - 1) >> th_lg);
    if ((shared || tile) && worth && tiles > 3 * resident_warps())
        order_regions(b, a, tw_lg, th_lg, s);
    if (shared) {
        st = a.gq8 ? launch_shared<true>(a, s) : launch_shared<false>(a, s);
        if (st != GS_OK) return st;
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_fail(e, "trace launch");
        return GS_OK;
    }
    switch (n_eff) {
        case 1: st = launch_n<1>(a, b->node_format, count, s); break;
        case 2: st = launch_n<2>(a, b->node_format, count, s); break;
        case 4: st = launch_n<4>(a, b->node_format, count, s); break;
        case 8: st = launch_n<8>(a, b->node_format, count, s); break;
        default: return fail(GS_ERR_INVALID_ARG, "n_hits must be 1, 2, 4 or 8");
    }
    if (st != GS_OK) return st;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "trace launch");
    return GS_OK;
}

}  // namespace gsrt
