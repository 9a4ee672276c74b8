// Device parts shared by the counts of one tree level by 4x4x4 bricks (nodecount.cu: the pinhole modes,
// panocount.cu: the panoramic mode): the cast of an image's rays by tiles, bounds of step counts and
// depths under a pixel box, float pixels with their exact fallbacks, a node's ancestors.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "bricks.cuh"
#include "interval.cuh"
#include "kernels.h"
#include "mig.h"

namespace mig {

namespace {

using namespace dev;

constexpr int kWarpsN = 8;  // warps per CTA of the kernels below

__device__ __forceinline__ const uint64_t *grid_umask(const GridView &g) {
    return reinterpret_cast<const uint64_t *>(g.g + umask_offset(g.nx, g.ny, g.nz));
}
__device__ __forceinline__ const uint64_t *grid_omask(const GridView &g) {
    return reinterpret_cast<const uint64_t *>(g.g + omask_offset(g.nx, g.ny, g.nz));
}

__device__ __forceinline__ float q16f(int v) { return (float)v * (1.0f / 65536.0f); }

// ------------------------------------------------------------------------- cast and render kernels
// The rays of an image are cast 8x4 pixels at a time, one ray per lane. Before that, lanes follow one
// such part each as a beam (beam_free): the part's rays start where the beam stopped, and are not
// cast at all if it met nothing within the range (60 % of the parts on the large workload, 16 % at
// paper scale). Three layouts, by the number of tiles of the launch:
//   large - one warp per 32x32 pixel tile, its 32 parts' beams on its 32 lanes, from 3 tiles per resident
//           warp on (6 and 1.5 measured the same or slower, 1.5 by a fifth in the smallest launches);
//   mid   - one CTA per 32x32 tile, the beams on its first warp;
//   small - one CTA per 16x16 tile, one part per warp, no beams and no 32x32 bounds, for levels that do
//           not fill the GPU: their time is one warp's chain of dependent steps.
// The level's size is only known on the device (tree_eval_device), so the kernels choose.
constexpr int kCastCtas = 4;  // resident CTAs per SM (64 registers; 3 CTAs of 80 are 2 % slower)
enum CastLayout { kCastSmall, kCastMid, kCastLarge };
__device__ __forceinline__ CastLayout cast_layout(long long images, int W, int H, int num_sms) {
    const long long tiles = images * ((W + 31) >> 5) * ((H + 31) >> 5), warps = (long long)num_sms * kCastCtas * kWarpsN;
    return tiles >= 3 * warps ? kCastLarge : (2 * tiles >= warps ? kCastMid : kCastSmall);
}

// Do nearly all bricks around a node hold occupied voxels (kClutter)?
__device__ __forceinline__ bool in_clutter(const LevelParams &p, const uint8_t *dist, const int4 nd) {
    const BrickDims n = brick_dims(p.grid.nx, p.grid.ny, p.grid.nz);
    return ld_dist(dist, (size_t)((nd.z >> 18) * n.nby + (nd.y >> 18)) * n.nbx + (nd.x >> 18) MIG_CHECKED(, &p)) & kClutter;
}

// The rays of a yaw's image from node nd.
struct CameraRays {
    const LevelParams &p;
    int4 nd;
    bool clutter;  // nearly all bricks around the node hold occupied voxels
    int ck, sk, W, H;
    // pixel (i, j)'s direction (Q30, unit) and its camera depth per unit length
    __device__ __forceinline__ int4 ray(int i, int j) const { return p.body[j * W + i]; }
    __device__ __forceinline__ void dir(const int4 &b, int &dx, int &dy, int &dz) const { ray_dir(b, ck, sk, dx, dy, dz); }
    // the beam of the 8x4 part at pixel (i0, j0)
    __device__ __forceinline__ float beam(const uint8_t *dist, int i0, int j0) const {
        if (i0 >= W || j0 >= H || clutter) return 0.0f;
        const int i1 = min(i0 + 7, W - 1), j1 = min(j0 + 3, H - 1);
        const float q30 = 9.31322574615478515625e-10f, c = (float)ck * q30, s = (float)sk * q30;
        float lo[3] = {1e30f, 1e30f, 1e30f}, hi[3] = {-1e30f, -1e30f, -1e30f};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int4 b = p.body[(t & 2 ? j1 : j0) * W + (t & 1 ? i1 : i0)];
            const float z = __fdividef(1.0f, (float)b.w), x = (float)b.x * z, y = (float)b.y * z;
            const float w[3] = {fmaf(c, x, -(s * y)), fmaf(s, x, c * y), (float)b.z * z};
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                lo[a] = fminf(lo[a], w[a]);
                hi[a] = fmaxf(hi[a], w[a]);
            }
        }
        // the largest camera depth of a unit ray: the part's pixel nearest the image centre on each axis
        const float a0 = ((float)i0 + 0.5f - 0.5f * (float)W) * p.ifx, a1 = ((float)i1 + 0.5f - 0.5f * (float)W) * p.ifx;
        const float b0 = ((float)j0 + 0.5f - 0.5f * (float)H) * p.ify, b1 = ((float)j1 + 0.5f - 0.5f * (float)H) * p.ify;
        const float am = a0 * a1 <= 0.0f ? 0.0f : fminf(fabsf(a0), fabsf(a1)), bm = b0 * b1 <= 0.0f ? 0.0f : fminf(fabsf(b0), fabsf(b1));
        const float s_end = q16f((int)p.Tq) * rsqrtf(1.0f + am * am + bm * bm) * 1.00001f;
        return beam_free(dist, p.grid.nx, p.grid.ny, p.grid.nz, nd.x, nd.y, nd.z, lo, hi, s_end MIG_CHECKED(, &p));
    }
};
// The time before which a ray of camera depth cz (Q30, per unit length) of a beam free to depth s
// meets no occupied voxel.
__device__ __forceinline__ float beam_time(float s, int cz) {
    return s > 0.0f ? fmaxf(0.0f, __fdividef(s * 1073741824.0f, (float)cz) * (1.0f - 1e-6f) - kCastEps) : 0.0f;
}

struct CastCnt {  // statistics
    uint32_t rays = 0, fine = 0, jump = 0;
};

// The rays of an image that a node's count casts, and the images' (tiles') number in the region.
__device__ __forceinline__ int image_width(const LevelParams &p) { return p.mode == MIG_MODE_PANORAMIC ? p.pano_A : p.W; }
__device__ __forceinline__ bool steps_ok(const LevelParams &p, const uint16_t *at) {
    return at_ok(p, at, (const uint16_t *)p.steps, (size_t)p.steps_cap * image_width(p) * p.H, kBoundsSteps);
}
__device__ __forceinline__ bool hz_ok(const LevelParams &p, const uint32_t *at) {
    return at_ok(p, at, (const uint32_t *)p.hz, (size_t)p.steps_cap * pyramid(image_width(p), p.H).n, kBoundsTiles);
}
__device__ __forceinline__ bool dpyr_ok(const LevelParams &p, const uint2 *at) {
    return p.arena_slots == 0 || at_ok(p, at, (const uint2 *)p.dpyr, (size_t)p.arena_slots * pyramid(p.W, p.H).n, kBoundsTiles);
}
__device__ __forceinline__ bool depth_ok(const LevelParams &p, const uint32_t *at) {
    return p.arena_slots == 0 || at_ok(p, at, (const uint32_t *)p.arena, (size_t)p.arena_slots * p.W * p.H, kBoundsDepth);
}
__device__ __forceinline__ bool queue_ok(const LevelParams &p, int i) { return at_ok(p, p.queue + i, (const BrickRec *)p.queue, p.queue_cap, kBoundsQueue); }

// What a pass keeps per ray and per tile: the cast the step index (16 bits, bounds packed as min |
// ~max << 16), the render the depth.
template <bool DEPTH>
struct CastOut {
    uint16_t *out;
    uint32_t *hz;
    uint32_t *depth;  // DEPTH: NULL for nodes that no descendant looks at
    static constexpr bool kDepth = DEPTH;
    static constexpr uint32_t kMin = 0xFFFFu;
    __device__ __forceinline__ bool stored() const { return false; }
    __device__ __forceinline__ uint32_t load(const LevelParams &, size_t) const { return 0u; }
    __device__ __forceinline__ uint32_t put(const LevelParams &p, size_t i, int dzc, uint32_t m, uint32_t ne, uint32_t ade) const {
        if (steps_ok(p, out + i)) out[i] = (uint16_t)m;
        if (DEPTH && depth && at_ok(p, depth + i, p.depths, (size_t)p.steps_cap * p.W * p.H, kBoundsSteps)) depth[i] = hit_depth(m != kNoHit, ne, ade, dzc, p.Tq);
        return m;
    }
    __device__ __forceinline__ void tile(const LevelParams &p, size_t i, uint32_t lo, uint32_t hi) const {
        if (hz_ok(p, hz + i)) hz[i] = lo | ((hi ^ 0xFFFFu) << 16);
    }
};
struct RenderOut {
    uint2 *pyr;  // NULL: not kept
    int slot;
    const uint32_t *src;  // NULL, or the depths that the cast stored
    static constexpr bool kDepth = true;
    static constexpr uint32_t kMin = 0xFFFFFFFFu;
    __device__ __forceinline__ bool stored() const { return src != nullptr; }
    __device__ __forceinline__ uint32_t load(const LevelParams &p, size_t i) const {
        const uint32_t D = at_ok(p, src + i, (const uint32_t *)p.depths, (size_t)p.steps_cap * p.W * p.H, kBoundsSteps) ? ld_written(src + i) : 0u;
        arena_store(p.arena, p.arena_slots, slot, i, (size_t)p.W * p.H, D, p.bounds_err);
        return D;
    }
    __device__ __forceinline__ uint32_t put(const LevelParams &p, size_t i, int dzc, uint32_t m, uint32_t ne, uint32_t ade) const {
        const uint32_t D = hit_depth(m != kNoHit, ne, ade, dzc, p.Tq);
        arena_store(p.arena, p.arena_slots, slot, i, (size_t)p.W * p.H, D, p.bounds_err);
        return D;
    }
    __device__ __forceinline__ void tile(const LevelParams &p, size_t i, uint32_t lo, uint32_t hi) const {
        if (pyr && dpyr_ok(p, pyr + i)) pyr[i] = make_uint2(lo, hi);
    }
};

// One ray, out of line: the layouts' loops keep their state in other registers than the walk's.
struct RayHit {
    uint32_t m, ne, ade;
};
template <bool STATS, bool DEPTH>
__device__ __noinline__ RayHit cast_ray(const uint64_t *om, const uint8_t *oct, int gnx, int gny, int gnz, int Px, int Py, int Pz,
                                       int dx, int dy, int dz, int Tq, float t0, int start, CastCnt *st MIG_CHECKED(, const LevelParams *lp)) {
    RayHit h{0, 0, 1};
    uint32_t fine = 0, jump = 0;
    h.m = cast_bricks<DEPTH, STATS>(om, oct, gnx, gny, gnz, Px, Py, Pz, dx, dy, dz, Tq, t0, h.ne, h.ade, fine, jump, start MIG_CHECKED(, lp));
    if constexpr (STATS) {
        st->fine += fine;
        st->jump += jump;
    }
    return h;
}

template <bool STATS>
__device__ __noinline__ NearWalk cast_near(const uint64_t *om, int gnx, int gny, int gnz, int Px, int Py, int Pz, int dx, int dy, int dz,
                                           int Tq, CastCnt *st MIG_CHECKED(, const LevelParams *lp)) {
    const NearWalk w = near_walk(om, gnx, gny, gnz, Px, Py, Pz, dx, dy, dz, Tq MIG_CHECKED(, lp));
    if constexpr (STATS) st->fine += w.steps + 1;
    return w;
}

// Casts the 8x4 part at pixel (i0, j0), lane l the pixel (l & 7, l >> 3); lo, hi gather its bounds.
template <bool STATS, class RAYS, class OUT>
__device__ __forceinline__ void cast_part(const LevelParams &p, const uint64_t *om, const uint8_t *dist, const RAYS &r,
                                          int i0, int j0, float beam, const OUT &o, int lane, uint32_t &lo, uint32_t &hi,
                                          CastCnt &st) {
    const int i = i0 + (lane & 7), j = j0 + (lane >> 3);
    if (i >= r.W || j >= r.H) return;
    const size_t at = (size_t)j * r.W + i;
    uint32_t v;
    if (o.stored()) {
        v = o.load(p, at);
    } else {
        RayHit hit{kNoHit, 0, 1};
        int dzc = 0;
        if (OUT::kDepth || beam < 1e29f) {
            const int4 b = r.ray(i, j);
            dzc = b.w;
            if (beam < 1e29f) {
                int dx, dy, dz;
                r.dir(b, dx, dy, dz);
                float t0 = beam_time(beam, b.w);
                int start = -1;
                bool on = true;
                if (r.clutter) {  // (the beam stops where it starts)
                    const NearWalk w = cast_near<STATS>(om, p.grid.nx, p.grid.ny, p.grid.nz, r.nd.x, r.nd.y, r.nd.z, dx, dy, dz, (int)p.Tq, &st
                                                        MIG_CHECKED(, &p));
                    if (w.hit != kNoHit) hit = RayHit{w.hit, w.en, w.ea};
                    on = w.brick >= 0;
                    start = w.brick;
                    t0 = w.t;
                }
                if (on) {
                    const uint8_t *oct = p.grid.g + oct_offset(p.grid.nx, p.grid.ny, p.grid.nz, octant_of(dx, dy, dz));
                    hit = cast_ray<STATS, OUT::kDepth>(om, oct, p.grid.nx, p.grid.ny, p.grid.nz, r.nd.x, r.nd.y, r.nd.z, dx, dy, dz, (int)p.Tq,
                                                       t0, start, &st MIG_CHECKED(, &p));
                }
            }
        }
        v = o.put(p, at, dzc, hit.m, hit.ne, hit.ade);
    }
    lo = min(lo, v);
    hi = max(hi, v);
    if constexpr (STATS) ++st.rays;
}

// The pixel of part t (0..7) of the 16x16 quadrant at (x0, y0): half t & 1 of 8x8 tile t >> 1.
__device__ __forceinline__ int2 part_at(int x0, int y0, int t) {
    return make_int2(x0 + ((t >> 1) & 1) * 8, y0 + (t >> 2) * 8 + (t & 1) * 4);
}

// One 16x16 quadrant by one warp, part t's beam in lane base + t of s; returns its bounds.
template <bool STATS, class RAYS, class OUT>
__device__ __forceinline__ uint2 cast_quad(const LevelParams &p, const uint64_t *om, const uint8_t *dist, const Pyramid &y,
                                           const RAYS &r, int x0, int y0, float s, int base, const OUT &o, int lane,
                                           CastCnt &st) {
    uint32_t lo = OUT::kMin, hi = 0u, lo16 = OUT::kMin, hi16 = 0u;
#pragma unroll 1
    for (int t = 0; t < 8; ++t) {
        const int2 at = part_at(x0, y0, t);
        const float beam = __shfl_sync(0xffffffffu, s, base + t);
        cast_part<STATS>(p, om, dist, r, at.x, at.y, beam, o, lane, lo, hi, st);
        __syncwarp();
        if (t & 1) {
            lo = __reduce_min_sync(0xffffffffu, lo);
            hi = __reduce_max_sync(0xffffffffu, hi);
            if (lane == 0 && at.x < r.W && at.y - 4 < r.H) o.tile(p, (size_t)(at.y >> 3) * y.w0 + (at.x >> 3), lo, hi);
            lo16 = min(lo16, lo);
            hi16 = max(hi16, hi);
            lo = OUT::kMin;
            hi = 0u;
        }
    }
    if (lane == 0 && x0 < r.W && y0 < r.H) o.tile(p, y.o1 + (size_t)(y0 >> 4) * y.w1 + (x0 >> 4), lo16, hi16);
    return make_uint2(lo16, hi16);
}

// One 32x32 tile at pixel (x0, y0) by one warp.
template <bool STATS, class RAYS, class OUT>
__device__ __forceinline__ void cast_large(const LevelParams &p, const uint64_t *om, const uint8_t *dist, const Pyramid &y,
                                           const RAYS &r, int x0, int y0, const OUT &o, int lane, CastCnt &st) {
    const int2 at = part_at(x0 + ((lane >> 3) & 1) * 16, y0 + (lane >> 4) * 16, lane & 7);
    const float s = r.beam(dist, at.x, at.y);
    uint2 b = make_uint2(OUT::kMin, 0u);
#pragma unroll 1
    for (int q = 0; q < 4; ++q) {
        const uint2 v = cast_quad<STATS>(p, om, dist, y, r, x0 + (q & 1) * 16, y0 + (q >> 1) * 16, s, 8 * q, o, lane, st);
        b = make_uint2(min(b.x, v.x), max(b.y, v.y));
    }
    if (lane == 0) o.tile(p, y.o2 + (size_t)(y0 >> 5) * y.w2 + (x0 >> 5), b.x, b.y);
}

// One 32x32 tile at pixel (x0, y0) by a CTA of 8 warps: warp w casts half of quadrant w >> 1.
template <bool STATS, class RAYS, class OUT>
__device__ __forceinline__ void cast_mid(const LevelParams &p, const uint64_t *om, const uint8_t *dist, const Pyramid &y,
                                         const RAYS &r, int x0, int y0, const OUT &o, uint2 *s_t, float *s_beam, int warp,
                                         int lane, CastCnt &st) {
    if (warp == 0) {
        const int2 at = part_at(x0 + ((lane >> 3) & 1) * 16, y0 + (lane >> 4) * 16, lane & 7);
        s_beam[lane] = r.beam(dist, at.x, at.y);
    }
    __syncthreads();
    const int qx = x0 + ((warp >> 1) & 1) * 16, qy = y0 + (warp >> 2) * 16;
    uint32_t lo = OUT::kMin, hi = 0u, lo2 = OUT::kMin, hi2 = 0u;
#pragma unroll 1
    for (int t = 4 * (warp & 1); t < 4 * (warp & 1) + 4; ++t) {
        const int2 at = part_at(qx, qy, t);
        cast_part<STATS>(p, om, dist, r, at.x, at.y, s_beam[8 * (warp >> 1) + t], o, lane, lo, hi, st);
        __syncwarp();
        if (t & 1) {
            lo = __reduce_min_sync(0xffffffffu, lo);
            hi = __reduce_max_sync(0xffffffffu, hi);
            if (lane == 0 && at.x < r.W && at.y - 4 < r.H) o.tile(p, (size_t)(at.y >> 3) * y.w0 + (at.x >> 3), lo, hi);
            lo2 = min(lo2, lo);
            hi2 = max(hi2, hi);
            lo = OUT::kMin;
            hi = 0u;
        }
    }
    if (lane == 0) s_t[warp] = make_uint2(lo2, hi2);
    __syncthreads();
    if (threadIdx.x < 4) {
        const uint2 a = s_t[2 * threadIdx.x], b = s_t[2 * threadIdx.x + 1];
        lo = min(a.x, b.x);
        hi = max(a.y, b.y);
        const int i0 = x0 + (threadIdx.x & 1) * 16, j0 = y0 + (threadIdx.x >> 1) * 16;
        if (i0 < r.W && j0 < r.H) o.tile(p, y.o1 + (size_t)(j0 >> 4) * y.w1 + (i0 >> 4), lo, hi);
        lo = __reduce_min_sync(0xfu, lo);
        hi = __reduce_max_sync(0xfu, hi);
        if (threadIdx.x == 0) o.tile(p, y.o2 + (size_t)(y0 >> 5) * y.w2 + (x0 >> 5), lo, hi);
    }
    __syncthreads();
}

// One 16x16 tile at pixel (x0, y0) by a CTA of 8 warps.
template <bool STATS, class RAYS, class OUT>
__device__ __forceinline__ void cast_small(const LevelParams &p, const uint64_t *om, const uint8_t *dist, const Pyramid &y,
                                            const RAYS &r, int x0, int y0, const OUT &o, uint2 *s_t, int warp, int lane,
                                            CastCnt &st) {
    uint32_t lo = OUT::kMin, hi = 0u;
    const int2 at = part_at(x0, y0, warp);
    cast_part<STATS>(p, om, dist, r, at.x, at.y, 0.0f, o, lane, lo, hi, st);
    __syncwarp();
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) s_t[warp] = make_uint2(lo, hi);
    __syncthreads();
    if (threadIdx.x < 4) {
        const uint2 a = s_t[2 * threadIdx.x], b = s_t[2 * threadIdx.x + 1];
        lo = min(a.x, b.x);
        hi = max(a.y, b.y);
        const int i0 = x0 + (threadIdx.x & 1) * 8, j0 = y0 + (threadIdx.x >> 1) * 8;
        if (i0 < r.W && j0 < r.H) o.tile(p, (size_t)(j0 >> 3) * y.w0 + (i0 >> 3), lo, hi);
        lo = __reduce_min_sync(0xfu, lo);
        hi = __reduce_max_sync(0xfu, hi);
        if (threadIdx.x == 0) o.tile(p, y.o1 + (size_t)(y0 >> 4) * y.w1 + (x0 >> 4), lo, hi);
    }
    __syncthreads();
}

constexpr int kMacX = 16, kMacZ = 8;
__host__ __device__ inline int mac_xy(int64_t Tq) { return (2 * ((int)(Tq >> 16) + 2)) / kMacX + 2; }
__host__ __device__ inline int mac_z(int64_t Tq) { return (2 * ((int)(Tq >> 16) + 2)) / kMacZ + 2; }

// Macro block mi of the mn (mxy by mxy columns) around node nd: is it inside the grid, the ball and the
// elevation band? (mX, mY, mZ): its place.
__device__ __forceinline__ bool macro_block(const LevelParams &p, const int4 nd, int mi, int mn, int mxy, int Rv, float R2, int &mX,
                                            int &mY, int &mZ) {
    if (mi >= mn) return false;
    const int a = mi / mxy;
    mX = (((nd.x >> 16) - Rv) >> 4) + (mi - a * mxy);
    mZ = (((nd.z >> 16) - Rv) >> 3) + a / mxy;
    mY = (((nd.y >> 16) - Rv) >> 4) + (a - (a / mxy) * mxy);
    if (mX < 0 || mY < 0 || mZ < 0 || 16 * mX >= p.grid.nx || 16 * mY >= p.grid.ny || 8 * mZ >= p.grid.nz) return false;
    const float cx = q16f(((16 * mX + 8) << 16) - nd.x), cy = q16f(((16 * mY + 8) << 16) - nd.y), cz = q16f(((8 * mZ + 4) << 16) - nd.z);
    const float dx = fmaxf(fabsf(cx) - 7.5f, 0.f), dy = fmaxf(fabsf(cy) - 7.5f, 0.f), dz = fmaxf(fabsf(cz) - 3.5f, 0.f);
    const float rho = sqrtf(cx * cx + cy * cy), r0 = fmaxf(rho - 10.7f, 0.f), r1 = rho + 10.7f;
    const float eps = 0.01f * (r1 + fabsf(cz) + 4.f) + 0.05f;
    return dx * dx + dy * dy + dz * dz <= R2 &&
           (p.band_thi >= 1e29f || cz - 3.5f <= p.band_thi * (p.band_thi > 0.f ? r1 : r0) + eps) &&
           (p.band_tlo <= -1e29f || cz + 3.5f >= p.band_tlo * (p.band_tlo < 0.f ? r1 : r0) - eps);
}

struct NodeAnc {
    int px, py, pz, yaw;
    const uint32_t *D;
    const uint2 *pyr;
    float U0, V0, Z0;  // the node in the ancestor's camera coordinates
    float err;         // 5e-7 of the node's largest offset from the ancestor
};

struct NodeCnt {  // statistics
    uint32_t cand = 0, unk = 0, visit = 0, anc = 0, reads = 0, smp = 0;
};

__device__ __forceinline__ uint64_t shfl64(uint64_t v, int src) {
    return (uint64_t)__shfl_sync(0xffffffffu, (unsigned long long)v, src);
}
__device__ __forceinline__ uint64_t or64(uint64_t v) {  // over the warp
    return (uint64_t)__reduce_or_sync(0xffffffffu, (unsigned)v) | ((uint64_t)__reduce_or_sync(0xffffffffu, (unsigned)(v >> 32)) << 32);
}

// Bounds of the step counts under a pixel box: min in the low half, ~max in the high half.
__device__ __forceinline__ uint32_t hz_box(const LevelParams &p, const uint32_t *hz, const Pyramid &y, int top, const BoxView &b) {
    int sh, off, w;
    pyramid_level(y, max(b.u1 - b.u0, b.v1 - b.v0), top, sh, off, w);
    const uint32_t *t = hz + off;
    uint32_t r = 0xFFFFFFFFu;
#pragma unroll 1
    for (int ty = b.v0 >> sh; ty <= (b.v1 >> sh); ++ty)
#pragma unroll 1
        for (int tx = b.u0 >> sh; tx <= (b.u1 >> sh); ++tx) r = __vminu2(r, hz_ok(p, t + ty * w + tx) ? ld_written(t + ty * w + tx) : 0u);
    return r;
}
// Bounds of the stored depths under a pixel box (the 32x32 level is not kept by every render).
__device__ __forceinline__ uint2 depth_box(const LevelParams &p, const uint2 *pyr, const Pyramid &y, const BoxView &b) {
    int sh, off, w;
    pyramid_level(y, max(b.u1 - b.u0, b.v1 - b.v0), 4, sh, off, w);
    const uint2 *t = pyr + off;
    uint2 r = make_uint2(0xFFFFFFFFu, 0u);
#pragma unroll 1
    for (int ty = b.v0 >> sh; ty <= (b.v1 >> sh); ++ty)
#pragma unroll 1
        for (int tx = b.u0 >> sh; tx <= (b.u1 >> sh); ++tx) {
            const uint2 v = dpyr_ok(p, t + ty * w + tx) ? ld_written(t + ty * w + tx) : make_uint2(0u, 0xFFFFFFFFu);
            r.x = min(r.x, v.x);
            r.y = max(r.y, v.y);
        }
    return r;
}
__device__ __forceinline__ bool box_lookup(const BoxView &b) {
    return b.zlo >= 0.5f && b.u1 - b.u0 <= kPyramidSpan && b.v1 - b.v0 <= kPyramidSpan;
}

// Float pixel of a voxel centre at camera depth >= 1/2. c = 5e-7 (largest offset + 1) bounds a row
// product's error per unit of the row's L1 norm, so eu = 2 c (norm_u + W norm_z) / Z + 1e-6 (W + 1)
// bounds the error of u for every pixel inside the image, and of an outside one by less than its
// distance to the image. su, sv: 2 c (norm + size norm_z).
struct PixelErr {
    float su, sv, bu, bv;
};
// 1: inside the image, pixel index pix; 0: outside; -1: undecided.
__device__ __forceinline__ int pixel_float(const PixelErr &e, float Z, float U, float V, float fW, float fH, int &pix) {
    const float kMagic = 12582912.0f;
    const float zi = __fdividef(1.0f, Z);
    const float u = fmaf(U, zi, -0.5f), v = fmaf(V, zi, -0.5f);
    const float fu = (u + kMagic) - kMagic, fv = (v + kMagic) - kMagic;  // floors: nearest integers of u - 1/2
    const bool sure = Z >= 0.5f && fmaf(zi, e.su, fabsf(u - fu)) <= e.bu && fmaf(zi, e.sv, fabsf(v - fv)) <= e.bv;
    pix = __float_as_int(fmaf(fv, fW, fu) + 8388608.0f) & 0x7FFFFF;
    if (!sure) return -1;
    return fu >= 0.0f && fu < fW && fv >= 0.0f && fv < fH;
}
// The exact pixel index (Eq. 5) in integers, or -1 outside the image; Z (Q32).
__device__ __forceinline__ int pixel_index(const int32_t *row, int rx, int ry, int rz, int W, int H, int64_t &Z) {
    Z = (int64_t)row[8] * rx + (int64_t)row[9] * ry + (int64_t)row[10] * rz;
    if (Z <= 0) return -1;
    const int64_t U = (int64_t)row[2] * rx + (int64_t)row[3] * ry + (int64_t)row[4] * rz;
    const int64_t V = (int64_t)row[5] * rx + (int64_t)row[6] * ry + (int64_t)row[7] * rz;
    const float zi = __fdividef(1.0f, (float)Z);
    int pu, pv;
    if (!pixel_in(U, Z, (float)U * zi, W, pu) || !pixel_in(V, Z, (float)V * zi, H, pv)) return -1;
    return pv * W + pu;
}
__device__ __noinline__ int pixel_exact(const int32_t *row, int rx, int ry, int rz, int W, int H) {
    int64_t Z;
    return pixel_index(row, rx, ry, rz, W, H, Z);
}
// The exact ancestor test (Sec. IV-B): inside the image and z <= D.
__device__ __noinline__ bool observed_exact(const int32_t *row, int rx, int ry, int rz, int W, int H, const uint32_t *D
                                              MIG_CHECKED(, const LevelParams *p)) {
    int64_t Z;
    const int pix = pixel_index(row, rx, ry, rz, W, H, Z);
#if MIG_DEBUG_BOUNDS
    if (pix >= 0 && !depth_ok(*p, D + pix)) return false;
#endif
    return pix >= 0 && Z < (((int64_t)ld_written(D + pix) + 1) << 16);
}
// The exact visit test of a voxel by its owner ray.
__device__ __noinline__ bool visit_exact(int Px, int Py, int Pz, int bx, int by, int bz, int ck, int sk, int x, int y, int z,
                                         int64_t Tq) {
    int dx, dy, dz;
    ray_dir(make_int4(bx, by, bz, 0), ck, sk, dx, dy, dz);
    return visit_index(Px, Py, Pz, dx, dy, dz, x, y, z, Tq) >= 0;
}

// Per-launch constants of the voxel stage.
struct VoxConst {
    float fW, fH, bu, bv, Tv, out2, inf2, l22;
};
__device__ __forceinline__ VoxConst vox_const(const LevelParams &p) {
    VoxConst c;
    c.fW = (float)p.W;
    c.fH = (float)p.H;
    c.bu = 0.5f - 1.0e-6f * (c.fW + 1.0f);
    c.bv = 0.5f - 1.0e-6f * (c.fH + 1.0f);
    c.Tv = q16f((int)p.Tq);
    // squared centre distances: no visit beyond out2; certain visits by the yaw's limit and by zl2
    c.out2 = (c.Tv + 0.88f) * (c.Tv + 0.88f);
    c.inf2 = fmaxf(c.Tv - 0.86f, 0.f) * fmaxf(c.Tv - 0.86f, 0.f);
    c.l22 = fmaxf(c.Tv - 0.02f, 0.f) * fmaxf(c.Tv - 0.02f, 0.f);
    return c;
}

// The ancestors of node n that the mode tests (Sec. IV-B), parent first; returns their number.
__device__ __forceinline__ int node_ancestors(const LevelParams &p, int n, NodeAnc *anc, size_t WH, int pyr_n, int lane) {
    const int2 ar = p.anc_range[n];
    int na = p.mode == MIG_MODE_ABSOLUTE ? 0 : (p.mode == MIG_MODE_SINGLE_PARENT ? min(ar.y, 1) : ar.y);
    na = min(na, p.max_anc);
    const int4 nd = p.node[n];
    __syncwarp();
    for (int t = lane; t < na; t += 32) {
        const int a = p.anc[ar.x + t];
        const int4 an = p.node[a];
        const int32_t *m = p.yawtab + p.sel_yaw[a] * 12 + 2;
        const int rx = nd.x - an.x, ry = nd.y - an.y, rz = nd.z - an.z;
        anc[t] = NodeAnc{an.x, an.y, an.z, p.sel_yaw[a], p.arena + (size_t)an.w * WH, p.dpyr + (size_t)an.w * pyr_n,
                         seg_coord(m, rx, ry, rz), seg_coord(m + 3, rx, ry, rz), seg_coord(m + 6, rx, ry, rz),
                         5e-7f * fmaxf(fmaxf(fabsf(q16f(rx)), fabsf(q16f(ry))), fabsf(q16f(rz)))};
    }
    __syncwarp();
    return na;
}

// Interval mode: no sample in the box of half extents (hx, hy, hz) about the offset (cx, cy, cz) from
// ancestor A's camera can fall in an observed portion of its buffer. A sample inside a portion
// projects into the image within the float error of seg_setup and seg_param, whose screen coordinates
// reach |U| / kZNear where the ray passes the camera plane: 6e-7 of that, plus one pixel, widens the
// image here; its depth is at most the range.
__device__ __forceinline__ bool iv_box_out(const YawRows &r, const NodeAnc &A, const int4 nd, float cx, float cy, float cz, float hx,
                                           float hy, float hz, float W, float H, float Tv) {
    const float reach = fmaxf(fmaxf(fabsf(q16f(A.px - nd.x)), fabsf(q16f(A.py - nd.y))), fabsf(q16f(A.pz - nd.z))) + Tv + 2.0f;
    const float mu = fmaf(6.2e-4f * r.u.w, reach, 1.0f), mv = fmaf(6.2e-4f * r.v.w, reach, 1.0f);
    const float Z = row_dot(r.z, cx, cy, cz), U = row_dot(r.u, cx, cy, cz), V = row_dot(r.v, cx, cy, cz);
    const float eZ = row_ext(r.z.x, r.z.y, r.z.z, hx, hy, hz) + 0.05f;
    // a half-space a Z + s m . r > 0: its value at the centre plus its largest change over the box
    auto out = [&](float a, float s, const float4 &m, float v) {
        return fmaf(a, Z, s * v) + row_ext(fmaf(a, r.z.x, s * m.x), fmaf(a, r.z.y, s * m.y), fmaf(a, r.z.z, s * m.z), hx, hy, hz) +
                   kBoxErr * fmaf(fabsf(a), r.z.w, m.w) <
               0.0f;
    };
    return Z + eZ < 0.0f || Z - eZ > Tv || out(mu, 1.0f, r.u, U) || out(W + mu, -1.0f, r.u, U) || out(mv, 1.0f, r.v, V) ||
           out(H + mv, -1.0f, r.v, V);
}

// The ancestors' test (Sec. IV-B) of a macro block's bricks (lane = brick (bx, by, bz) of unknown voxels
// U, first brick (X, Y, Z)), as whole bricks, for the lanes that want it: O = U where one ancestor
// observes the whole brick, left = the ancestors (bit = place in the node's list) to test voxel by voxel.
template <bool INTERVAL>
__device__ __forceinline__ void block_ancestors(const LevelParams &p, const YawRows *s_y, const NodeAnc *anc, int na, const int4 nd,
                                                const Pyramid &pyr, const VoxConst &vc, int X, int Y, int Z, int bx, int by, int bz,
                                                uint64_t U, bool want, int lane, uint64_t &O, uint64_t &left) {
    const int W = p.W, H = p.H;
#pragma unroll 1
    for (int ab = 0; ab < na; ab += 32) {
        bool rel = false;  // lane = ancestor: does it look at the block, not behind its depths?
        if (ab + lane < na) {
            const NodeAnc A = anc[ab + lane];
            const float ox = q16f(((4 * X + 8) << 16) - A.px), oy = q16f(((4 * Y + 8) << 16) - A.py),
                        oz = q16f(((4 * Z + 4) << 16) - A.pz);
            if (INTERVAL) {
                rel = !iv_box_out(s_y[A.yaw], A, nd, ox, oy, oz, 8.0f, 8.0f, 4.0f, vc.fW, vc.fH, vc.Tv);
            } else {
                const BoxView b = box_view<false>(s_y[A.yaw], ox, oy, oz, 7.5f, 7.5f, 3.5f, W, H);
                rel = b.in >= 0;
                if (rel && box_lookup(b)) {
                    const uint2 D = depth_box(p, A.pyr, pyr, b);
                    rel = b.zlo * (65536.0f * (1.0f - 1e-6f)) <= (float)D.y + 1.5f;
                }
            }
        }
#pragma unroll 1
        for (unsigned as = __ballot_sync(0xffffffffu, rel); as; as &= as - 1) {
            const int a = ab + __ffs(as) - 1;
            if (want && O != U) {
                const NodeAnc A = anc[a];
                const float ox = q16f(((4 * bx + 2) << 16) - A.px), oy = q16f(((4 * by + 2) << 16) - A.py),
                            oz = q16f(((4 * bz + 2) << 16) - A.pz);
                bool vox;
                if (INTERVAL) {
                    vox = !iv_box_out(s_y[A.yaw], A, nd, ox, oy, oz, 2.0f, 2.0f, 2.0f, vc.fW, vc.fH, vc.Tv);
                } else {
                    const BoxView b = box_view<true>(s_y[A.yaw], ox, oy, oz, 1.5f, 1.5f, 1.5f, W, H);
                    vox = b.in >= 0;
                    if (vox && box_lookup(b)) {
                        const uint2 D = depth_box(p, A.pyr, pyr, b);
                        if (b.zlo * (65536.0f * (1.0f - 1e-6f)) > (float)D.y + 1.5f) {
                            vox = false;
                        } else if (b.in > 0 && b.zhi * (65536.0f * (1.0f + 1e-6f)) < (float)D.x) {
                            O = U;
                            vox = false;
                        }
                    }
                }
                if (vox) left |= 1ull << a;
            }
        }
    }
}

// The exact test of a brick's voxels (lane = voxel (x, y, z0) and (x, y, z0 + 2)) against the ancestors
// `left`: O with the voxels of U that one of them observes. verr: the error of a row product per unit
// of the row's norm.
template <bool STATS>
__device__ __forceinline__ uint64_t voxel_ancestors(const LevelParams &p, const VoxConst &vc, const YawRows *s_y, const NodeAnc *anc,
                                                    const int4 nd, uint64_t left, uint64_t U, uint64_t O, int x, int y, int z0,
                                                    float verr, int lane, NodeCnt &st) {
    const int W = p.W, H = p.H;
    const float ex = q16f((x << 16) + 32768 - nd.x), ey = q16f((y << 16) + 32768 - nd.y), ez0 = q16f((z0 << 16) + 32768 - nd.z);
    for (uint64_t as = left; as && (U & ~O); as &= as - 1) {
        const NodeAnc &A = anc[__ffsll((long long)as) - 1];
        const float4 ru = s_y[A.yaw].u, rv = s_y[A.yaw].v, rz = s_y[A.yaw].z;
        // camera coordinates: the node's plus the rotated offset from the node
        const float Zxy = fmaf(rz.x, ex, fmaf(rz.y, ey, A.Z0)), Uxy = fmaf(ru.x, ex, fmaf(ru.y, ey, A.U0)),
                    Vxy = fmaf(rv.x, ex, fmaf(rv.y, ey, A.V0));
        const float c = verr + A.err;
        const PixelErr pe{2.0f * c * fmaf(vc.fW, rz.w, ru.w), 2.0f * c * fmaf(vc.fH, rz.w, rv.w), vc.bu, vc.bv};
        const float e_z = c * rz.w;
        const uint64_t rem = U & ~O;
        bool obs[2] = {false, false};
        int pix[2], in[2];
        float Zf[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float ez = ez0 + (float)(2 * h);
            Zf[h] = fmaf(rz.z, ez, Zxy);
            in[h] = pixel_float(pe, Zf[h], fmaf(ru.z, ez, Uxy), fmaf(rv.z, ez, Vxy), vc.fW, vc.fH, pix[h]);
            if (!((uint32_t)(rem >> (32 * h)) >> lane & 1)) in[h] = 0;
            if constexpr (STATS) st.anc += (uint32_t)(rem >> (32 * h)) >> lane & 1;
        }
        uint32_t D[2] = {0u, 0u};
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (in[h] > 0 && depth_ok(p, A.D + pix[h])) D[h] = ld_written(A.D + pix[h]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if constexpr (STATS) st.reads += in[h] > 0;
            // z <= D  <=>  Z < (D + 1) / 2^16 (voxels); lim within 2^-23 of that
            const float lim = ((float)D[h] + 1.0f) * (1.0f / 65536.0f);
            obs[h] = in[h] > 0 && Zf[h] + e_z < lim * (1.0f - 2.4e-7f);
            if (in[h] < 0 || (in[h] > 0 && !obs[h] && Zf[h] - e_z < lim * (1.0f + 2.4e-7f)))
                obs[h] = observed_exact(p.yawtab + A.yaw * 12, (x << 16) + 32768 - A.px, (y << 16) + 32768 - A.py,
                                        (z0 << 16) + 32768 + (h << 17) - A.pz, W, H, A.D MIG_CHECKED(, &p));
        }
        O |= (uint64_t)__ballot_sync(0xffffffffu, obs[0]) | ((uint64_t)__ballot_sync(0xffffffffu, obs[1]) << 32);
    }
    return O;
}

// CTAs for a cast of `images` images (an upper bound of the level's): one per 16x16 tile, at most as
// many as keep the kernel's loops short.
inline int cast_grid(long long images, int W, int H, int num_sms, int per_sm) {
    const long long tiles = images * ((W + 15) / 16) * ((H + 15) / 16);
    return (int)std::max<long long>(1, std::min<long long>(tiles, (long long)num_sms * per_sm));
}

// Shared memory of a CTA: the yaws' rows and each warp's ancestors.
inline size_t node_dyn_smem(int K, int max_anc) {
    return (size_t)K * sizeof(YawRows) + (size_t)kWarpsN * std::max(1, max_anc) * sizeof(NodeAnc);
}

}  // namespace

}  // namespace mig
