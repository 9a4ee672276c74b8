// The 4x4x4-brick view of a map and the exact steps that run on it, as plain functions of their
// arguments (callable from host code too): the cast of a ray to its first occupied voxel, and the
// tests that decide a whole brick of voxels, or one voxel, against a camera.
//
// After the voxel codes and the occupancy bytes (voxcount.cuh) a map carries, per 4x4x4 brick
// (x-fastest bricks; bit = (z & 3) * 16 + (y & 3) * 4 + (x & 3)):
//   umask  64 bits, 1 = unknown voxel;      omask  64 bits, 1 = occupied voxel;
//   oct    8 bytes (one array per octant of directions): the Chebyshev distance in bricks to the
//          nearest brick with an occupied voxel among those not behind this one along any axis (0 =
//          this one), capped at kDistCap: no occupied voxel lies in that many bricks ahead;
//   dist   1 byte, the least of the eight: the distance in any direction; with kClutter where the brick and
//          nearly all of those around it (22 of 27, or as many of those in the grid) hold occupied voxels.
// They are refreshed by every update for the bricks whose value it can change.
#pragma once

#include "voxcount.cuh"

namespace mig {
namespace dev {

constexpr int kDistCap = 15;  // bricks: one jump of the cast crosses at most 60 voxels of an axis
constexpr int kClutter = 128;

struct BrickDims {
    int nbx, nby, nbz;
};
MIG_HD BrickDims brick_dims(int nx, int ny, int nz) { return BrickDims{(nx + 3) >> 2, (ny + 3) >> 2, (nz + 3) >> 2}; }
MIG_HD size_t brick_count(int nx, int ny, int nz) {
    return (size_t)((nx + 3) >> 2) * (size_t)((ny + 3) >> 2) * (size_t)((nz + 3) >> 2);
}
MIG_HD size_t umask_offset(int nx, int ny, int nz) { return (occ_summary_end(nx, ny, nz) + 255) & ~(size_t)255; }
MIG_HD size_t omask_offset(int nx, int ny, int nz) {
    return umask_offset(nx, ny, nz) + ((8 * brick_count(nx, ny, nz) + 255) & ~(size_t)255);
}
MIG_HD size_t dist_offset(int nx, int ny, int nz) {
    return omask_offset(nx, ny, nz) + ((8 * brick_count(nx, ny, nz) + 255) & ~(size_t)255);
}
// the octants' distances (octant_of), then what only updates use: the distances within a z layer (four
// bytes a brick), a bit per brick with an occupied voxel, rows of bits_words words, and a map version
MIG_HD size_t brick_bytes_offset(int nx, int ny, int nz, int i) {
    return dist_offset(nx, ny, nz) + (size_t)i * ((brick_count(nx, ny, nz) + 255) & ~(size_t)255);
}
MIG_HD size_t oct_offset(int nx, int ny, int nz, int o) { return brick_bytes_offset(nx, ny, nz, 1 + o); }
MIG_HD size_t dist_xy_offset(int nx, int ny, int nz) { return brick_bytes_offset(nx, ny, nz, 9); }
MIG_HD size_t bits_offset(int nx, int ny, int nz) { return brick_bytes_offset(nx, ny, nz, 13); }
MIG_HD int bits_words(int nbx) { return (nbx + 31) >> 5; }
MIG_HD size_t brick_data_end(int nx, int ny, int nz) {
    const BrickDims n = brick_dims(nx, ny, nz);
    return bits_offset(nx, ny, nz) + (size_t)n.nby * n.nbz * bits_words(n.nbx) * 4 + 4;
}
MIG_HD size_t changed_offset(int nx, int ny, int nz) { return brick_data_end(nx, ny, nz) - 4; }
// The octant of a direction: a bit per axis that does not run backwards.
MIG_HD int octant_of(int dx, int dy, int dz) { return (dx >= 0 ? 1 : 0) | (dy >= 0 ? 2 : 0) | (dz >= 0 ? 4 : 0); }

MIG_HD uint64_t ld_u64(const uint64_t *p) {
#ifdef __CUDA_ARCH__
    return __ldg(reinterpret_cast<const unsigned long long *>(p));
#else
    return *p;
#endif
}

// Mask and distance of brick i; a checked build's skipped access reads an occupied brick.
MIG_HD uint64_t ld_mask(const uint64_t *m, size_t i MIG_CHECKED(, const LevelParams *p)) {
#if MIG_DEBUG_BOUNDS && defined(__CUDA_ARCH__)
    if (!at_ok(*p, m + i, m, brick_count(p->grid.nx, p->grid.ny, p->grid.nz), kBoundsBrick)) return ~0ull;
#endif
    return ld_u64(m + i);
}
MIG_HD int ld_dist(const uint8_t *d, size_t i MIG_CHECKED(, const LevelParams *p)) {
#if MIG_DEBUG_BOUNDS && defined(__CUDA_ARCH__)
    if (!at_ok(*p, d + i, d, brick_count(p->grid.nx, p->grid.ny, p->grid.nz), kBoundsBrick)) return 0;
#endif
    return ld_u8(d + i);
}

// ------------------------------------------------------------------------------------- cast
// Crossings of an axis (face distances n0 + k 2^16, speed ad) that start before the time ts (Q16
// voxel units along the ray), exactly.
MIG_HD int crossings_until(uint32_t n0, uint32_t ad, uint32_t ts) {
    const uint32_t lim = (uint32_t)(((uint64_t)ts * ad + ((1u << 30) - 1)) >> 30);
    return n0 >= lim ? 0 : (int)((lim - n0 + (kQ16 - 1)) >> 16);
}

// Slack of the cast's float times and positions (voxels): at most 1024 voxels from the origin every
// float step below is within 5e-4 of the exact value (5e-7 of the range at shorter ones; the cast takes
// 2e-6 of its range, so that few rays of a warp ever need the exact walk).
constexpr float kCastEps = 2e-3f;
// Relative error of the mask DDA's crossing times (4 roundings, then one per step of at most 10), with
// room to spare.
constexpr int kCastRounds = 2048;
constexpr float kFineErr = 4e-6f;
constexpr float kTimeErr = 8e-6f;  // of a time that the fine phase hands back

MIG_HD int float_bits(float v) {
#ifdef __CUDA_ARCH__
    return __float_as_int(v);
#else
    union { float f; int i; } u;
    u.f = v;
    return u.i;
#endif
}

// v as a float, 0 <= v < 2^23, without a conversion instruction.
MIG_HD float small_float(int v) {
#ifdef __CUDA_ARCH__
    return __int_as_float(0x4B000000 | v) - 8388608.0f;
#else
    return (float)v;
#endif
}

// The exact DDA from the voxel state at time ts (Q16; all crossings before it, in integers) up to the
// first brick face crossed at a time of at least tf.
struct ExactWalk {
    bool more;         // the ray goes on, in voxel v just entered at time t by the crossing (en / ea, axis)
    uint32_t hit;      // step index of an occupied voxel, entered by (en / ea), else kNoHit
    int vx, vy, vz, axis;
    uint32_t en, ea, steps;
    float t;
};
MIG_HD ExactWalk exact_walk(const uint64_t *om, int gnx, int gny, int gnz, int Px, int Py, int Pz, int dx, int dy, int dz, int64_t Tq,
                     uint32_t ts, float tf MIG_CHECKED(, const LevelParams *lp)) {
    int v0x, v0y, v0z, sx, sy, sz;
    uint32_t n0x, n0y, n0z, ax, ay, az;
    ray_axis(Px, dx, v0x, sx, n0x, ax);
    ray_axis(Py, dy, v0y, sy, n0y, ay);
    ray_axis(Pz, dz, v0z, sz, n0z, az);
    const int nbx = (gnx + 3) >> 2, nby = (gny + 3) >> 2;
    const int cx = crossings_until(n0x, ax, ts), cy = crossings_until(n0y, ay, ts), cz = crossings_until(n0z, az, ts);
    ExactWalk w;
    w.vx = v0x + sx * cx;
    w.vy = v0y + sy * cy;
    w.vz = v0z + sz * cz;
    w.hit = kNoHit;
    w.axis = 3;
    w.en = 0;
    w.ea = 1;
    w.steps = 0;
    w.t = 0.0f;
    w.more = true;
    uint32_t nx = n0x + ((uint32_t)cx << 16), ny = n0y + ((uint32_t)cy << 16), nz = n0z + ((uint32_t)cz << 16);
    uint64_t m = ld_mask(om, (size_t)((w.vz >> 2) * nby + (w.vy >> 2)) * nbx + (w.vx >> 2) MIG_CHECKED(, lp));
    bool walk = true;
    while (walk) {
        ++w.steps;
        if ((m >> (((w.vz & 3) << 4) | ((w.vy & 3) << 2) | (w.vx & 3))) & 1ull) {
            w.hit = (uint32_t)(abs(w.vx - v0x) + abs(w.vy - v0y) + abs(w.vz - v0z));
            walk = w.more = false;
        } else {
            const int a = ev_argmin3(nx, ax, ny, ay, nz, az);
            w.axis = a;
            w.en = a == 0 ? nx : (a == 1 ? ny : nz);
            w.ea = a == 0 ? ax : (a == 1 ? ay : az);
            w.vx += a == 0 ? sx : 0;
            w.vy += a == 1 ? sy : 0;
            w.vz += a == 2 ? sz : 0;
            nx += a == 0 ? kQ16 : 0u;
            ny += a == 1 ? kQ16 : 0u;
            nz += a == 2 ? kQ16 : 0u;
            const int v = a == 0 ? w.vx : (a == 1 ? w.vy : w.vz), s = a == 0 ? sx : (a == 1 ? sy : sz);  // the coordinate that moved
            if (((uint64_t)w.en << 30) >= (uint64_t)Tq * w.ea || (unsigned)v >= (unsigned)(a == 0 ? gnx : (a == 1 ? gny : gnz))) {
                walk = w.more = false;  // the crossing starts at or beyond the range, or leaves the grid
            } else if ((v & 3) == (s > 0 ? 0 : 3)) {  // entered another brick
                m = ld_mask(om, (size_t)((w.vz >> 2) * nby + (w.vy >> 2)) * nbx + (w.vx >> 2) MIG_CHECKED(, lp));
                // en / ea in voxels (Q16 over Q30)
                w.t = (float)w.en * fast_divf(16384.0f, (float)w.ea);
                walk = w.t < tf;
            }
        }
    }
    return w;
}

// The exact DDA from the start voxel through bricks with occupied voxels: to the first occupied voxel, to the
// ray's end, or to the first brick without one. For nodes in clutter (kClutter): most rays end here, after a few
// voxels and without the set-up of cast_bricks, which pays where rays pass whole bricks: 1000 nodes of
// 160x120x16 with 5 voxels of range among 50 % of occupied voxels 8.1 -> 4.9 ms, 400 of 320x240x8 with 20 voxels
// among 20 % 8.9 -> 6.0.
// (Where only the node's own brick had to hold an occupied voxel, rays along walls took this way too: cast of
// 150 nodes of 223x131x7 among rooms 14 % slower.) steps: voxels visited.
struct NearWalk {
    uint32_t hit;   // step index of the occupied voxel, entered by (en / ea), else kNoHit
    uint32_t en, ea, steps;
    int brick;      // -1, or the free brick just entered (x | y << 10 | z << 20), at time t
    float t;
};
MIG_HD NearWalk near_walk(const uint64_t *om, int gnx, int gny, int gnz, int Px, int Py, int Pz, int dx, int dy, int dz,
                          int64_t Tq MIG_CHECKED(, const LevelParams *lp)) {
    int v0x, v0y, v0z, sx, sy, sz;
    uint32_t n0x, n0y, n0z, ax, ay, az;
    ray_axis(Px, dx, v0x, sx, n0x, ax);
    ray_axis(Py, dy, v0y, sy, n0y, ay);
    ray_axis(Pz, dz, v0z, sz, n0z, az);
    // a crossing at face distance n along an axis is allowed iff n < l
    const uint32_t lx = n0x + ((uint32_t)allowed_crossings(v0x, sx, n0x, ax, gnx, Tq) << 16),
                   ly = n0y + ((uint32_t)allowed_crossings(v0y, sy, n0y, ay, gny, Tq) << 16),
                   lz = n0z + ((uint32_t)allowed_crossings(v0z, sz, n0z, az, gnz, Tq) << 16);
    const int nbx = (gnx + 3) >> 2, nby = (gny + 3) >> 2;
    int vx = v0x, vy = v0y, vz = v0z;
    uint32_t nx = n0x, ny = n0y, nz = n0z;
    NearWalk w{kNoHit, 0u, 1u, 0u, -1, 0.0f};
    uint64_t m = ld_mask(om, (size_t)((vz >> 2) * nby + (vy >> 2)) * nbx + (vx >> 2) MIG_CHECKED(, lp));
    for (bool walk = true; walk;) {
        if ((m >> (((vz & 3) << 4) | ((vy & 3) << 2) | (vx & 3))) & 1ull) {
            w.hit = w.steps;
            walk = false;
        } else {
            const int a = ev_argmin3(nx, ax, ny, ay, nz, az);
            w.en = a == 0 ? nx : (a == 1 ? ny : nz);
            w.ea = a == 0 ? ax : (a == 1 ? ay : az);
            walk = w.en < (a == 0 ? lx : (a == 1 ? ly : lz));  // else it leaves the grid or the range
            if (walk) {
                nx += a == 0 ? kQ16 : 0u;
                ny += a == 1 ? kQ16 : 0u;
                nz += a == 2 ? kQ16 : 0u;
                vx += a == 0 ? sx : 0;
                vy += a == 1 ? sy : 0;
                vz += a == 2 ? sz : 0;
                ++w.steps;
                if (((a == 0 ? vx : (a == 1 ? vy : vz)) & 3) == ((a == 0 ? sx : (a == 1 ? sy : sz)) > 0 ? 0 : 3)) {  // entered another brick
                    m = ld_mask(om, (size_t)((vz >> 2) * nby + (vy >> 2)) * nbx + (vx >> 2) MIG_CHECKED(, lp));
                    if (m == 0) {
                        w.brick = (vx >> 2) | ((vy >> 2) << 10) | ((vz >> 2) << 20);
                        w.t = (float)w.en * fast_divf(16384.0f, (float)w.ea);  // in voxels (Q16 over Q30)
                        walk = false;
                    }
                }
            }
        }
    }
    return w;
}

// Occupied voxels of a brick's mask m inside the box of local voxel coordinates [lo, hi] per axis.
MIG_HD bool mask_box(uint64_t m, int lx, int hx, int ly, int hy, int lz, int hz) {
    const uint32_t row = (2u << hx) - (1u << lx);                                    // 4 bits
    const uint32_t plane = row * ((0x1111u << (4 * ly)) & (0x1111u >> (4 * (3 - hy))));  // 16 bits, no carries
    const uint64_t z = m & (~0ull << (16 * lz)) & (~0ull >> (16 * (3 - hz)));
    return (((uint32_t)z | (uint32_t)(z >> 32)) & (plane | (plane << 16))) != 0;
}

// Step index of the first occupied voxel that the DDA (Sec. IV-B) visits, else kNoHit; the same
// value as the plain walk's. t0: a time up to which the caller knows that the ray meets no occupied
// voxel (0 if it knows nothing); start: -1, or the brick (near_walk) that it enters at t0. oct: the distances for the ray's octant (octant_of).
//
// The ray is in brick b, known exactly, at time t. If no occupied brick lies within the d bricks ahead
// of b along each axis (the octant distance, d >= 1), the ray moves to the brick beyond the face of
// that box which it crosses first. It also passes a brick with occupied voxels (d = 0) if none of them
// lies in the box of voxels between its entry and exit; otherwise it runs the DDA on the brick's
// 64-bit mask, by float times. Either way the new brick is exact as long as the floats decide: a jump's
// other two coordinates are floors of positions that must not lie within eps of a brick face, and two
// crossings of the mask's DDA must differ by more than their error. Where they do not decide, and near
// the range (0.2 to 0.4 % of the rays), the exact voxel state at a time in free space (all crossings
// before it, in integers) is rebuilt and the DDA runs with exactly compared crossings up to the next
// brick face (exact_walk). The loops have single exits (no return or break inside), so that a warp's rays
// meet again after each; the mask's DDA runs outside the jump loop, where the rays that need it run it
// together (inside it the cast took 9.3 instead of 8.0 ms at paper scale).
// Bound by instruction issue (about 65 % of the slots, 23 of 32 lanes active). Cast per replan at
// paper scale / on the large workload: 12.3 / 493 ms with 64-bit compared crossings, 8.2 / 219 ms with
// one distance for all directions, 8.0 / 208 ms without the box test of occupied bricks, 6.4 / 166 ms;
// 5.3 ms at paper scale with all levels in one launch, 4.8 / 148 ms with tiles taken one at a time by warps.
// The step index of a voxel is its Manhattan distance from the start voxel, so the walk need not
// count steps. With DEPTH, ne / ade return the face distance and speed of the hit voxel's entry
// (0 / 1 for the start voxel). fine, coarse: voxel steps and jumps taken (STATS).
template <bool DEPTH, bool STATS>
MIG_HD uint32_t cast_bricks(const uint64_t *om, const uint8_t *oct, int gnx, int gny, int gnz, int Px, int Py, int Pz,
                            int dx, int dy, int dz, int64_t Tq, float t0, uint32_t &ne, uint32_t &ade, uint32_t &fine,
                            uint32_t &coarse, int start = -1 MIG_CHECKED(, const LevelParams *lp = nullptr)) {
    const float q30 = 9.31322574615478515625e-10f, q16 = 1.52587890625e-5f, q18 = 3.814697265625e-6f;
    const int nbx = (gnx + 3) >> 2, nby = (gny + 3) >> 2, nbz = (gnz + 3) >> 2;
    const int b0x = Px >> 18, b0y = Py >> 18, b0z = Pz >> 18;
    const int sx = dx < 0 ? -1 : 1, sy = dy < 0 ? -1 : 1, sz = dz < 0 ? -1 : 1;
    // times per voxel along each axis; an axis that does not move gets a time beyond every range
    const float fx = fabsf((float)dx) * q30, fy = fabsf((float)dy) * q30, fz = fabsf((float)dz) * q30;
    const float ix = fx > 0.0f ? fast_divf(1.0f, fx) : 1e30f, iy = fy > 0.0f ? fast_divf(1.0f, fy) : 1e30f, iz = fz > 0.0f ? fast_divf(1.0f, fz) : 1e30f;
    const float T = (float)Tq * q16, eps = fmaf(T, 2e-6f, 3e-5f);
    float t_end = fminf(T, (float)(sx > 0 ? (gnx << 16) - Px : Px) * q16 * ix);
    t_end = fminf(t_end, (float)(sy > 0 ? (gny << 16) - Py : Py) * q16 * iy);
    t_end = fminf(t_end, (float)(sz > 0 ? (gnz << 16) - Pz : Pz) * q16 * iz);
    // brick coordinates relative to the start brick, as floats: position p0 + k t; the far face of the
    // d bricks from b on, at b + d or b - d + 1, is crossed at (b +- d + h) j
    const float gx = sx > 0 ? 1.0f : -1.0f, gy = sy > 0 ? 1.0f : -1.0f, gz = sz > 0 ? 1.0f : -1.0f;
    const float p0x = (float)(Px & 0x3FFFF) * q18, p0y = (float)(Py & 0x3FFFF) * q18, p0z = (float)(Pz & 0x3FFFF) * q18;
    const float kx = 0.25f * fx * gx, ky = 0.25f * fy * gy, kz = 0.25f * fz * gz;
    const float hx = (sx > 0 ? 0.0f : 1.0f) - p0x, hy = (sy > 0 ? 0.0f : 1.0f) - p0y, hz = (sz > 0 ? 0.0f : 1.0f) - p0z;
    const float jx = 4.0f * ix * gx, jy = 4.0f * iy * gy, jz = 4.0f * iz * gz;
    const float kR = 0.5f - 0.25f * eps, kMagic = 12582912.0f, t_sure = t_end - eps;
    uint32_t hit = kNoHit;
    int last = 3;  // the axis of the latest crossing (3: none yet); with DEPTH
    // the brick at time t0, and whether it is certain (p: position minus 1/2, m: nearest integers of p)
    float t = t0;
    float px = fmaf(kx, t, p0x) - 0.5f, py = fmaf(ky, t, p0y) - 0.5f, pz = fmaf(kz, t, p0z) - 0.5f;
    float bx = (px + kMagic) - kMagic, by = (py + kMagic) - kMagic, bz = (pz + kMagic) - kMagic;
    bool sure = t < t_sure && (t0 == 0.0f || fmaxf(fabsf(px - bx), fmaxf(fabsf(py - by), fabsf(pz - bz))) < kR);
    if (t0 == 0.0f) bx = by = bz = 0.0f;
    if (start >= 0) {
        bx = small_float(start & 1023) - small_float(b0x);
        by = small_float((start >> 10) & 1023) - small_float(b0y);
        bz = small_float(start >> 20) - small_float(b0z);
        sure = t < t_sure;
    }
    auto oct_at = [&]() {  // the distance at brick b; (int)b by the bits of a float whose unit is its last place
        const int ib = (b0z + float_bits(bz + kMagic) - 0x4B400000) * nby + (b0y + float_bits(by + kMagic) - 0x4B400000);
        return (size_t)ib * (size_t)nbx + (size_t)(b0x + float_bits(bx + kMagic) - 0x4B400000);
    };
    auto outside = [&]() {  // brick b is beyond the grid
        const int x = b0x + float_bits(bx + kMagic) - 0x4B400000, y = b0y + float_bits(by + kMagic) - 0x4B400000, z = b0z + float_bits(bz + kMagic) - 0x4B400000;
        return (unsigned)x >= (unsigned)nbx || (unsigned)y >= (unsigned)nby || (unsigned)z >= (unsigned)nbz;
    };
    size_t bi = 0;
    int d = 0;
    float r = 1.0f;
    if (sure) {
        bi = oct_at();
        d = ld_dist(oct, bi MIG_CHECKED(, lp));
    }
    int rounds = 0;  // every round passes a brick face; beyond kCastRounds the exact walk runs to the end
    for (bool more = true; more;) {
        bool dda = false;  // in a brick with an occupied voxel near the ray's way through it
        while (sure && !dda) {
            if constexpr (STATS) ++coarse;
            const float df = small_float(max(d, 1));
            const float tx = (fmaf(gx, df, bx) + hx) * jx, ty = (fmaf(gy, df, by) + hy) * jy, tz = (fmaf(gz, df, bz) + hz) * jz;
            const float t1 = fminf(tx, fminf(ty, tz));
            const bool ox = tx == t1, oy = !ox && ty == t1, oz = !ox && !oy;
            // floors of the positions (nearest integer of p - 1/2) and their distance from a brick's middle
            const float qx = fmaf(kx, t1, p0x) - 0.5f, qy = fmaf(ky, t1, p0y) - 0.5f, qz = fmaf(kz, t1, p0z) - 0.5f;
            const float mx = (qx + kMagic) - kMagic, my = (qy + kMagic) - kMagic, mz = (qz + kMagic) - kMagic;
            if (d == 0) {
                // the voxels between entry and exit, widened by e: local coordinates (minus 1/2, nearest integers)
                const float e = fmaf(t, kTimeErr, 2.0f * eps);
                auto at = [&](float v) { return float_bits(fminf(fmaxf(v, 0.0f), 3.0f) + kMagic) & 3; };
                const float cx = fmaf(-4.0f, bx, 1.5f), cy = fmaf(-4.0f, by, 1.5f), cz = fmaf(-4.0f, bz, 1.5f);
                dda = mask_box(ld_mask(om, bi MIG_CHECKED(, lp)), at(fmaf(4.0f, fminf(px, qx), cx - e)), at(fmaf(4.0f, fmaxf(px, qx), cx + e)),
                               at(fmaf(4.0f, fminf(py, qy), cy - e)), at(fmaf(4.0f, fmaxf(py, qy), cy + e)),
                               at(fmaf(4.0f, fminf(pz, qz), cz - e)), at(fmaf(4.0f, fmaxf(pz, qz), cz + e)));
            }
            if (!dda) {
                r = fmaxf(ox ? 0.0f : fabsf(qx - mx), fmaxf(oy ? 0.0f : fabsf(qy - my), oz ? 0.0f : fabsf(qz - mz)));
                t = t1;
                px = qx;
                py = qy;
                pz = qz;
                sure = t < t_sure && r < kR;
                bx = ox ? fmaf(gx, df, bx) : mx;
                by = oy ? fmaf(gy, df, by) : my;
                bz = oz ? fmaf(gz, df, bz) : mz;
                if constexpr (DEPTH) last = ox ? 0 : (oy ? 1 : 2);
                if (sure) {
                    bi = oct_at();
                    d = ld_dist(oct, bi MIG_CHECKED(, lp));
                }
            }
        }
        // free to the grid's edge: past it with a certain brick, every voxel before being in the free box
        if (!sure && r < kR && outside()) more = false;
        if (sure) {
            // DDA on the brick's mask: entry voxel (local coordinates l, not within e of an inner face of the
            // brick's voxels; the entry face itself is exact), next crossing times, and a packed state: bits
            // 0-5 the mask's bit (plus 64), above them a guard per axis whose third bit is set while the
            // coordinate is in 0..3
            const uint64_t m = ld_mask(om, bi MIG_CHECKED(, lp));
            const float e = fmaf(t, kTimeErr, eps);
            const float lx = fminf(fmaxf(4.0f * (px - bx) + 1.5f, -0.5f), 3.499f), ly = fminf(fmaxf(4.0f * (py - by) + 1.5f, -0.5f), 3.499f),
                        lz = fminf(fmaxf(4.0f * (pz - bz) + 1.5f, -0.5f), 3.499f);  // minus 1/2
            const float cx = fmaxf((lx + kMagic) - kMagic, 0.0f), cy = fmaxf((ly + kMagic) - kMagic, 0.0f), cz = fmaxf((lz + kMagic) - kMagic, 0.0f);
            // within e of an inner face: l - c = +-1/2, but not at the brick's own faces
            const float ux = fabsf(lx - 1.5f) > 1.9f ? 0.0f : fabsf(lx - cx), uy = fabsf(ly - 1.5f) > 1.9f ? 0.0f : fabsf(ly - cy),
                        uz = fabsf(lz - 1.5f) > 1.9f ? 0.0f : fabsf(lz - cz);
            float tx = (fmaf(0.25f, cx + (sx > 0 ? 1.0f : -4.0f), bx) + hx) * jx, ty = (fmaf(0.25f, cy + (sy > 0 ? 1.0f : -4.0f), by) + hy) * jy,
                  tz = (fmaf(0.25f, cz + (sz > 0 ? 1.0f : -4.0f), bz) + hz) * jz;
            const int vx = float_bits(cx + kMagic) & 3, vy = float_bits(cy + kMagic) & 3, vz = float_bits(cz + kMagic) & 3;
            int w = 64 + vx + 4 * vy + 16 * vz + ((vx + 4) << 8) + ((vy + 4) << 12) + ((vz + 4) << 16);
            const int wx = sx * 257, wy = sy * 4100, wz = sz * 65552;
            bool walk = fmaxf(ux, fmaxf(uy, uz)) < 0.5f - e, ox = false, oy = false, left = false, occ = false;
            sure = false;
            float mn = t;
            while (walk) {
                if constexpr (STATS) ++fine;
                occ = (m >> (w & 63)) & 1ull;
                mn = fminf(tx, fminf(ty, tz));
                const float lim = fmaf(mn, kFineErr, mn);
                ox = tx <= lim;
                oy = ty <= lim;
                const bool oz = tz <= lim;
                walk = !occ && !((ox && oy) || (ox && oz) || (oy && oz)) && mn < T - eps;
                if (walk) {
                    tx += ox ? ix : 0.0f;
                    ty += oy ? iy : 0.0f;
                    tz += oz ? iz : 0.0f;
                    w += ox ? wx : (oy ? wy : wz);
                    if constexpr (DEPTH) last = ox ? 0 : (oy ? 1 : 2);
                    left = (w & 0x44400) != 0x44400;
                    walk = !left;
                }
            }
            if (occ) {
                const int b4x = 4 * (b0x + float_bits(bx + kMagic) - 0x4B400000), b4y = 4 * (b0y + float_bits(by + kMagic) - 0x4B400000),
                          b4z = 4 * (b0z + float_bits(bz + kMagic) - 0x4B400000);
                const int cx_ = abs(b4x + (w & 3) - (Px >> 16)), cy_ = abs(b4y + ((w >> 2) & 3) - (Py >> 16)), cz_ = abs(b4z + ((w >> 4) & 3) - (Pz >> 16));
                hit = (uint32_t)(cx_ + cy_ + cz_);
                if constexpr (DEPTH) {
                    const int c = last == 0 ? cx_ : (last == 1 ? cy_ : cz_), P = last == 0 ? Px : (last == 1 ? Py : Pz),
                              dd = last == 0 ? dx : (last == 1 ? dy : dz);
                    int v0, s;
                    uint32_t n0;
                    ray_axis(P, dd, v0, s, n0, ade);
                    ne = n0 + ((uint32_t)(c - 1) << 16);
                    if (last == 3) {  // the start voxel
                        ne = 0;
                        ade = 1;
                    }
                }
                more = false;
            } else if (left) {  // into the next brick, across the face of the axis just crossed
                t = mn;
                bx += ox ? gx : 0.0f;
                by += !ox && oy ? gy : 0.0f;
                bz += !ox && !oy ? gz : 0.0f;
                px = fmaf(kx, t, p0x) - 0.5f;
                py = fmaf(ky, t, p0y) - 0.5f;
                pz = fmaf(kz, t, p0z) - 0.5f;
                more = !outside();
                sure = more && t < t_sure;
                r = 1.0f;
                if (sure) {
                    bi = oct_at();
                    d = ld_dist(oct, bi MIG_CHECKED(, lp));
                }
            } else if (mn > T + eps) {
                more = false;  // the next crossing is beyond the range
            }
        }
        // the ray is free of occupied voxels up to t: done if that is the range or the grid's edge
        more = more && t <= t_end + eps;
        if (more && !sure) {
            const float slack = fmaf(t, kTimeErr, eps);
            const ExactWalk w = exact_walk(om, gnx, gny, gnz, Px, Py, Pz, dx, dy, dz, Tq,
                                           (uint32_t)(int)(fmaxf(0.0f, fminf(t, t_end) - slack) * 65536.0f),
                                           ++rounds < kCastRounds ? t + slack : 1e30f MIG_CHECKED(, lp));
            if constexpr (STATS) fine += w.steps;
            if constexpr (DEPTH) {
                ne = w.en;
                ade = w.ea;
                last = w.axis;
            }
            hit = w.hit;
            more = w.more;
            if (more) {  // back to the jumps from the brick just entered, exactly known
                t = w.t;
                bx = small_float(w.vx >> 2) - small_float(Px >> 18);
                by = small_float(w.vy >> 2) - small_float(Py >> 18);
                bz = small_float(w.vz >> 2) - small_float(Pz >> 18);
                px = fmaf(kx, t, p0x) - 0.5f;
                py = fmaf(ky, t, p0y) - 0.5f;
                pz = fmaf(kz, t, p0z) - 0.5f;
                r = 1.0f;
                sure = t < t_sure;
                if (sure) {
                    bi = oct_at();
                    d = ld_dist(oct, bi MIG_CHECKED(, lp));
                }
            }
        }
    }
    if constexpr (DEPTH) {
        if (hit == kNoHit) {
            ne = 0;
            ade = 1;
        }
    }
    return hit;
}

// A tile of rays as one beam: the camera depth s up to which no ray of the tile meets an occupied
// voxel, or 1e30 if none meets one within its range. The rays of a tile, taken as points P + w s at
// camera depth s, have w between the corners' values on every axis, so at depth s they lie in a box
// whose edges move linearly from P. While that box stays inside the free box of 2 d - 1 bricks around
// its middle's brick (unbounded towards a side where that box reaches the grid's edge), the depth
// advances to where its first edge leaves it. w: the corner rays over their camera depth (world
// axes), s_end: the largest camera depth of a ray's range. The bounds are widened by 4e-6 of w (the
// rounding of w and of the positions) and the result is kCastEps short.
MIG_HD float beam_free(const uint8_t *dist, int gnx, int gny, int gnz, int Px, int Py, int Pz, const float wlo[3],
                       const float whi[3], float s_end MIG_CHECKED(, const LevelParams *lp)) {
    const int nb[3] = {(gnx + 3) >> 2, (gny + 3) >> 2, (gnz + 3) >> 2}, P[3] = {Px, Py, Pz};
    const float q18 = 3.814697265625e-6f;
    float p0[3], lo[3], hi[3];
    int b0[3], b[3];
    for (int a = 0; a < 3; ++a) {
        b0[a] = P[a] >> 18;
        b[a] = b0[a];
        p0[a] = (float)(P[a] & 0x3FFFF) * q18;
        lo[a] = 0.25f * (wlo[a] - 4e-6f * fabsf(wlo[a]) - 1e-7f);
        hi[a] = 0.25f * (whi[a] + 4e-6f * fabsf(whi[a]) + 1e-7f);
    }
    float s = 0.0f;
    for (bool go = true; go;) {
        const int d = ld_dist(dist, (size_t)(b[2] * nb[1] + b[1]) * nb[0] + b[0] MIG_CHECKED(, lp)) & 15;
        float s1 = 1e30f;
        bool in = d > 0;
        for (int a = 0; a < 3; ++a) {
            const float f_lo = b[a] - d + 1 <= 0 ? -1e30f : (float)(b[a] - d + 1 - b0[a]);
            const float f_hi = b[a] + d >= nb[a] ? 1e30f : (float)(b[a] + d - b0[a]);
            // an edge moving outwards limits the depth, one moving inwards must be inside already
            if (hi[a] > 0.0f) s1 = fminf(s1, fast_divf(f_hi - p0[a], hi[a]));
            else in = in && fmaf(hi[a], s, p0[a]) < f_hi;
            if (lo[a] < 0.0f) s1 = fminf(s1, fast_divf(f_lo - p0[a], lo[a]));
            else in = in && fmaf(lo[a], s, p0[a]) > f_lo;
        }
        s1 = s1 * (1.0f - 2e-6f) - kCastEps;
        go = in && s1 > s + 0.25f;
        if (go) {
            s = s1;
            for (int a = 0; a < 3; ++a)
                b[a] = max(0, min(b0[a] + (int)floorf(fmaf(0.5f * (lo[a] + hi[a]), fminf(s, 8192.0f), p0[a])), nb[a] - 1));
            if (s >= s_end) {
                s = 1e30f;
                go = false;
            }
        }
    }
    return s;
}

// ----------------------------------------------------------------------- the owner ray's visit
// A voxel's owner pixel holds its centre's projection, so the owner ray (through the pixel's
// centre) passes the voxel's centre within half a pixel. For a voxel near enough this alone puts
// the ray inside the voxel. With h_u = (1/2 + e_u) / f_x and h_v = (1/2 + e_v) / f_y (e: the
// rounding of the Q16 rows in pixels), the ray's point at the centre's depth z is at most z h_u
// along the camera's x axis and z h_v along its y axis from the centre, so
//   - z hypot(h_u, h_v) < 0.485: the ray's nearest point lies inside the voxel, at a distance along
//     the ray of at most |r| (depth limit zl2, the same for every yaw);
//   - z (h_u |ex_a| + h_v |ey_a|) < 0.485 for each world axis a: the point at depth z lies inside
//     it, at a distance of at most |r| + 0.85 (depth limit zinf of the yaw).
// Either visits the voxel if that distance is below the range (and the depth is at least 1/2). The
// 0.015 left to the voxel's faces covers the Q30 rounding of the ray and the float depth.
struct VisitLimits {
    float hu, hv, zl2;
};
inline VisitLimits visit_limits(double hfov_deg, double vfov_deg, int W, int H) {
    const double th = tan(hfov_deg * 0.5 * (3.14159265358979323846 / 180.0)), tv = tan(vfov_deg * 0.5 * (3.14159265358979323846 / 180.0));
    const double fx = W * 0.5 / th, fy = H * 0.5 / tv;
    const double S = 1.05 * sqrt(1.0 + th * th + tv * tv);  // |r| / z inside the frustum
    const double q = 7.62939453125e-06 * 1.7320508 * S;     // 2^-17 sqrt(3) |r| / z
    const double eu = 1.1 * q * (1.0 + W), ev = 1.1 * q * (1.0 + H);
    VisitLimits l;
    const double hu = (0.5 + eu) / fx, hv = (0.5 + ev) / fy;
    l.hu = (float)(hu * 1.001 * (1.0 + 4.0 * q));
    l.hv = (float)(hv * 1.001 * (1.0 + 4.0 * q));
    l.zl2 = (float)(0.485 / (sqrt(hu * hu + hv * hv) * 1.001 * (1.0 + 4.0 * q)));
    return l;
}

// Does the ray from the origin along (dx, dy, dz) (unit, float) visit the voxel whose centre is at
// (cx, cy, cz) before the range Tv? 1 = surely, 0 = surely not, -1 = too close to tell (the exact
// test decides). The ray's time inside the voxel shrunk (widened) by 1e-3 on every face: the float
// rounding of the centre, the direction and the quotients moves a face by less than 5e-4 voxel up to
// 1024 voxels from the origin. An axis slower than 2^-24 moves less than 1e-4 voxel over the range.
MIG_HD int visit_slab(float cx, float cy, float cz, float dx, float dy, float dz, float Tv) {
    const float m = 5.9604645e-8f;
    const float ix = fast_divf(1.0f, copysignf(fmaxf(fabsf(dx), m), dx)), iy = fast_divf(1.0f, copysignf(fmaxf(fabsf(dy), m), dy)),
                iz = fast_divf(1.0f, copysignf(fmaxf(fabsf(dz), m), dz));
    const float tx = cx * ix, ty = cy * iy, tz = cz * iz;
    const float hx = fabsf(ix), hy = fabsf(iy), hz = fabsf(iz);
    const float lo = fmaxf(fmaf(-0.499f, hx, tx), fmaxf(fmaf(-0.499f, hy, ty), fmaf(-0.499f, hz, tz)));
    const float hi = fminf(fmaf(0.499f, hx, tx), fminf(fmaf(0.499f, hy, ty), fmaf(0.499f, hz, tz)));
    if (lo <= hi && hi >= 1e-3f && lo < Tv - 1e-3f) return 1;
    const float lo2 = fmaxf(fmaf(-0.501f, hx, tx), fmaxf(fmaf(-0.501f, hy, ty), fmaf(-0.501f, hz, tz)));
    const float hi2 = fminf(fmaf(0.501f, hx, tx), fminf(fmaf(0.501f, hy, ty), fmaf(0.501f, hz, tz)));
    if (lo2 > hi2 || hi2 < -1e-3f || lo2 > Tv + 1e-3f) return 0;
    return -1;
}

// -------------------------------------------------------------------------- camera against a box
// A yaw's projection rows in floats (mu, mv, mz / 2^16) for tests of boxes of voxel centres.
// For a box of half extents (hx, hy, hz) about r, a linear form m . r varies by at most
// |m_x| hx + |m_y| hy + |m_z| hz; kBoxErr of the row's L1 norm covers the float rounding (the
// centre's offset and the products, up to 1030 voxels from the camera).
struct YawRows {
    float4 u, v, z;  // mu, mv, mz; w = L1 norm
    float4 x;        // zinf (the depth limit of the certain visit for this yaw), cos, sin of the yaw, -
    float4 e;        // half ranges over a brick's voxel centres: of U, V, Z and W Z - U
    float4 f;        // of H Z - V; -
};
constexpr float kBoxErr = 5e-4f;

MIG_HD YawRows yaw_rows(const int32_t *y /* ck sk mu mv mz */, int W, int H, float hu, float hv, float ifx, float ify) {
    const float s = 1.0f / 65536.0f, q30 = 9.31322574615478515625e-10f;
    YawRows r;
    r.u = make_float4((float)y[2] * s, (float)y[3] * s, (float)y[4] * s, 0.f);
    r.v = make_float4((float)y[5] * s, (float)y[6] * s, (float)y[7] * s, 0.f);
    r.z = make_float4((float)y[8] * s, (float)y[9] * s, (float)y[10] * s, 0.f);
    r.u.w = fabsf(r.u.x) + fabsf(r.u.y) + fabsf(r.u.z);
    r.v.w = fabsf(r.v.x) + fabsf(r.v.y) + fabsf(r.v.z);
    r.z.w = fabsf(r.z.x) + fabsf(r.z.y) + fabsf(r.z.z);
    // camera axes from the rows: ex = (mu - W/2 mz) / f_x, ey = (mv - H/2 mz) / f_y
    const float cw = 0.5f * (float)W, ch = 0.5f * (float)H;
    const float a = hu * fabsf((r.u.x - cw * r.z.x) * ifx) + hv * fabsf((r.v.x - ch * r.z.x) * ify);
    const float b = hu * fabsf((r.u.y - cw * r.z.y) * ifx) + hv * fabsf((r.v.y - ch * r.z.y) * ify);
    const float c = hu * fabsf((r.u.z - cw * r.z.z) * ifx) + hv * fabsf((r.v.z - ch * r.z.z) * ify);
    r.x = make_float4(0.484f / fmaxf(fmaxf(a, b), fmaxf(c, 1e-12f)), (float)y[0] * q30, (float)y[1] * q30, 0.f);
    const float fW = (float)W, fH = (float)H;
    const float nR = fabsf(fmaf(fW, r.z.x, -r.u.x)) + fabsf(fmaf(fW, r.z.y, -r.u.y)) + fabsf(fmaf(fW, r.z.z, -r.u.z));
    const float nB = fabsf(fmaf(fH, r.z.x, -r.v.x)) + fabsf(fmaf(fH, r.z.y, -r.v.y)) + fabsf(fmaf(fH, r.z.z, -r.v.z));
    const float h = 1.5f + kBoxErr;
    r.e = make_float4(h * r.u.w, h * r.v.w, h * r.z.w, 1.5f * nR + kBoxErr * fmaf(fW, r.z.w, r.u.w));
    r.f = make_float4(1.5f * nB + kBoxErr * fmaf(fH, r.z.w, r.v.w), 0.f, 0.f, 0.f);
    return r;
}

MIG_HD float row_dot(const float4 &m, float x, float y, float z) { return fmaf(m.x, x, fmaf(m.y, y, m.z * z)); }
MIG_HD float row_ext(float a, float b, float c, float hx, float hy, float hz) {
    return fmaf(fabsf(a), hx, fmaf(fabsf(b), hy, fabsf(c) * hz));
}

// The box of voxel centres of half extents (hx, hy, hz) about the offset (cx, cy, cz) from a camera
// against its image (Eq. 5: Z > 0, 0 <= U < W Z, 0 <= V < H Z).
//   in:    -1 = no centre projects into the image, 1 = every centre does, 0 = undecided
//   zlo, zhi: bounds of the centres' camera depth; u0..u1, v0..v1: bounds of their pixels inside the
//   image (valid when zlo >= 1/2 and in >= 0).
struct BoxView {
    int in;
    float zlo, zhi;
    int u0, u1, v0, v1;
};
// BRICK: the box is a brick's 4x4x4 centres (half extents 1.5), whose ranges the rows carry.
template <bool BRICK>
MIG_HD BoxView box_view(const YawRows &r, float cx, float cy, float cz, float hx, float hy, float hz, int W, int H) {
    BoxView b;
    const float fW = (float)W, fH = (float)H;
    const float Z = row_dot(r.z, cx, cy, cz), U = row_dot(r.u, cx, cy, cz), V = row_dot(r.v, cx, cy, cz);
    const float R = fmaf(fW, Z, -U), B = fmaf(fH, Z, -V);
    float eZ = r.e.z, eU = r.e.x, eV = r.e.y, eR = r.e.w, eB = r.f.x;
    if (!BRICK) {
        eZ = row_ext(r.z.x, r.z.y, r.z.z, hx, hy, hz) + kBoxErr * r.z.w;
        eU = row_ext(r.u.x, r.u.y, r.u.z, hx, hy, hz) + kBoxErr * r.u.w;
        eV = row_ext(r.v.x, r.v.y, r.v.z, hx, hy, hz) + kBoxErr * r.v.w;
        eR = row_ext(fmaf(fW, r.z.x, -r.u.x), fmaf(fW, r.z.y, -r.u.y), fmaf(fW, r.z.z, -r.u.z), hx, hy, hz) +
             kBoxErr * fmaf(fW, r.z.w, r.u.w);
        eB = row_ext(fmaf(fH, r.z.x, -r.v.x), fmaf(fH, r.z.y, -r.v.y), fmaf(fH, r.z.z, -r.v.z), hx, hy, hz) +
             kBoxErr * fmaf(fH, r.z.w, r.v.w);
    }
    b.zlo = Z - eZ;
    b.zhi = Z + eZ;
    if (b.zhi < 0.f || U + eU < 0.f || V + eV < 0.f || R + eR < 0.f || B + eB < 0.f) {
        b.in = -1;
        return b;
    }
    b.in = b.zlo > 0.f && U - eU > 0.f && V - eV > 0.f && R - eR > 0.f && B - eB > 0.f;
    // pixel bounds: over the box, U/Z - u = ((mu - u mz) . delta) / Z with u the centre's U/Z
    const float zi = fast_divf(1.0f, Z), zli = fast_divf(1.0f, fmaxf(b.zlo, 0.25f));
    const float u = U * zi, v = V * zi;
    const float du = (row_ext(fmaf(-u, r.z.x, r.u.x), fmaf(-u, r.z.y, r.u.y), fmaf(-u, r.z.z, r.u.z), hx, hy, hz) +
                      kBoxErr * fmaf(fabsf(u), r.z.w, r.u.w)) * zli + 0.01f;
    const float dv = (row_ext(fmaf(-v, r.z.x, r.v.x), fmaf(-v, r.z.y, r.v.y), fmaf(-v, r.z.z, r.v.z), hx, hy, hz) +
                      kBoxErr * fmaf(fabsf(v), r.z.w, r.v.w)) * zli + 0.01f;
    b.u0 = (int)fminf(fmaxf(floorf(u - du), 0.0f), fW - 1.0f);
    b.u1 = (int)fminf(fmaxf(floorf(u + du), 0.0f), fW - 1.0f);
    b.v0 = (int)fminf(fmaxf(floorf(v - dv), 0.0f), fH - 1.0f);
    b.v1 = (int)fminf(fmaxf(floorf(v + dv), 0.0f), fH - 1.0f);
    return b;
}

// ---------------------------------------------------------------------------------- pyramids
// Minimum and maximum of an image over 8x8, 16x16 and 32x32 pixel tiles (three levels, one after
// the other), so that the values under a box's pixels are bounded by a few reads.
struct Pyramid {
    int w0, w1, w2;  // tiles per row of each level
    int o1, o2, n;   // offsets of the second and third level, total entries
};
MIG_HD Pyramid pyramid(int W, int H) {
    Pyramid y;
    y.w0 = (W + 7) >> 3;
    y.w1 = (W + 15) >> 4;
    y.w2 = (W + 31) >> 5;
    y.o1 = y.w0 * ((H + 7) >> 3);
    y.o2 = y.o1 + y.w1 * ((H + 15) >> 4);
    y.n = y.o2 + y.w2 * ((H + 31) >> 5);
    return y;
}
// The level whose tiles cover a box `span` pixels wide in at most 2 x 2 of them; the coarsest one
// kept (top: 4 = 16x16, 5 = 32x32) for wider boxes.
MIG_HD void pyramid_level(const Pyramid &y, int span, int top, int &sh, int &off, int &w) {
    sh = span < 8 ? 3 : (span < 16 ? 4 : top);
    off = sh == 3 ? 0 : (sh == 4 ? y.o1 : y.o2);
    w = sh == 3 ? y.w0 : (sh == 4 ? y.w1 : y.w2);
}
constexpr int kPyramidSpan = 160;  // boxes wider than this many pixels are not looked up

}  // namespace dev
}  // namespace mig
