// The 4x4x4-brick view of a map and the exact steps that run on it, as plain functions of their
// arguments (callable from host code too): the cast of a ray to its first occupied voxel, and the
// tests that decide a whole brick of voxels, or one voxel, against a camera.
//
// After the voxel codes and the occupancy bytes (voxcount.cuh) a map carries, per 4x4x4 brick
// (x-fastest bricks; bit = (z & 3) * 16 + (y & 3) * 4 + (x & 3)):
//   umask  64 bits, 1 = unknown voxel;      omask  64 bits, 1 = occupied voxel;
//   dist   1 byte, the Chebyshev distance in bricks to the nearest brick that holds an occupied
//          voxel (0 = this one), capped at kDistCap.
// They are refreshed by every update for the bricks whose value it can change.
#pragma once

#include "voxcount.cuh"

namespace mig {
namespace dev {

constexpr int kDistCap = 15;  // bricks: one jump of the cast crosses at most 60 voxels of an axis

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
// two byte arrays the distance passes work in, one after the other
MIG_HD size_t dist_scratch_offset(int nx, int ny, int nz, int i) {
    return dist_offset(nx, ny, nz) + (size_t)(1 + i) * ((brick_count(nx, ny, nz) + 255) & ~(size_t)255);
}
MIG_HD size_t brick_data_end(int nx, int ny, int nz) { return dist_scratch_offset(nx, ny, nz, 2); }

MIG_HD uint64_t ld_u64(const uint64_t *p) {
#ifdef __CUDA_ARCH__
    return __ldg(reinterpret_cast<const unsigned long long *>(p));
#else
    return *p;
#endif
}

// ------------------------------------------------------------------------------------- cast
// Crossings of an axis (face distances n0 + k 2^16, speed ad) that start before the time ts (Q16
// voxel units along the ray), exactly.
MIG_HD int crossings_until(uint32_t n0, uint32_t ad, uint32_t ts) {
    const uint32_t lim = (uint32_t)(((uint64_t)ts * ad + ((1u << 30) - 1)) >> 30);
    return n0 >= lim ? 0 : (int)((lim - n0 + (kQ16 - 1)) >> 16);
}

// Slack of the cast's float times and positions (voxels): at most 1024 voxels from the origin every
// float step below is within 5e-4 of the exact value.
constexpr float kCastEps = 2e-3f;
// Voxel steps after which the fine phase rebuilds its float times, and their relative error by then
// (the division and product 4 roundings, one per step).
constexpr int kCastRounds = 2048;
constexpr int kFineSteps = 48;
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

// Occupied voxels of a brick's mask m inside the box of local voxel coordinates [lo, hi] per axis.
MIG_HD bool mask_box(uint64_t m, int lx, int hx, int ly, int hy, int lz, int hz) {
    const uint32_t row = (2u << hx) - (1u << lx);                                    // 4 bits
    const uint32_t plane = row * ((0x1111u << (4 * ly)) & (0x1111u >> (4 * (3 - hy))));  // 16 bits, no carries
    const uint64_t z = m & (~0ull << (16 * lz)) & (~0ull >> (16 * (3 - hz)));
    return (((uint32_t)z | (uint32_t)(z >> 32)) & (plane | (plane << 16))) != 0;
}

// Step index of the first occupied voxel that the DDA (Sec. IV-B) visits, else kNoHit; the same
// value as the plain walk's. t0: a time up to which the caller knows that the ray meets no occupied
// voxel (0 if it knows nothing). Two alternating phases, each a single-exit loop (no return or break
// inside, so that a warp's rays meet again after each phase):
//   jump - the ray is in brick b, known exactly, and crosses the box of 2 d - 1 bricks around it that
//          holds no occupied voxel (d bricks to the nearest occupied one), or, in a brick with occupied
//          voxels (d = 0), that brick if none of them lies in the box of voxels between the ray's entry
//          and exit. It moves to the brick beyond the face that it crosses first. That brick's
//          coordinate along the crossed axis is exact; the other two are floors of float positions, and
//          where one lies within kCastEps of a brick face the jump is not taken (fine phase instead).
//   fine - the exact voxel state at a time ts in free space (all crossings before ts, in integers) is
//          rebuilt and the DDA runs voxel by voxel, reading one 64-bit occupancy mask per brick. The
//          next crossing is chosen by float times where they differ by more than their error, else by
//          the exact comparison of n / |d|; the voxel position is exact throughout.
// The step index of a voxel is its Manhattan distance from the start voxel, so the walk need not
// count steps. With DEPTH, ne / ade return the face distance and speed of the hit voxel's entry
// (0 / 1 for the start voxel). fine, coarse: voxel steps and jumps taken (STATS).
template <bool DEPTH, bool STATS>
MIG_HD uint32_t cast_bricks(const uint64_t *om, const uint8_t *dist, int gnx, int gny, int gnz, int Px, int Py, int Pz,
                            int dx, int dy, int dz, int64_t Tq, float t0, uint32_t &ne, uint32_t &ade, uint32_t &fine,
                            uint32_t &coarse) {
    int v0x, v0y, v0z, sx, sy, sz;
    uint32_t n0x, n0y, n0z, ax, ay, az;
    ray_axis(Px, dx, v0x, sx, n0x, ax);
    ray_axis(Py, dy, v0y, sy, n0y, ay);
    ray_axis(Pz, dz, v0z, sz, n0z, az);
    const float q30 = 9.31322574615478515625e-10f, q16 = 1.52587890625e-5f, q18 = 3.814697265625e-6f;
    const int nbx = (gnx + 3) >> 2, nby = (gny + 3) >> 2;
    const int b0x = v0x >> 2, b0y = v0y >> 2, b0z = v0z >> 2;
    // times per voxel along each axis; an axis that does not move gets a time beyond every range
    const float fx = (float)ax * q30, fy = (float)ay * q30, fz = (float)az * q30;
    const float ix = ax ? fast_divf(1.0f, fx) : 1e30f, iy = ay ? fast_divf(1.0f, fy) : 1e30f, iz = az ? fast_divf(1.0f, fz) : 1e30f;
    const float T = (float)Tq * q16;
    float t_end = T;
    t_end = fminf(t_end, (float)(sx > 0 ? (gnx << 16) - Px : Px) * q16 * ix);
    t_end = fminf(t_end, (float)(sy > 0 ? (gny << 16) - Py : Py) * q16 * iy);
    t_end = fminf(t_end, (float)(sz > 0 ? (gnz << 16) - Pz : Pz) * q16 * iz);
    // brick coordinates relative to the start brick, as floats: position p0 + k t; the far face of the
    // box of brick b, at b + d or b - d + 1, is crossed at (b +- d + h) j
    const float gx = sx > 0 ? 1.0f : -1.0f, gy = sy > 0 ? 1.0f : -1.0f, gz = sz > 0 ? 1.0f : -1.0f;
    const float p0x = (float)(Px & 0x3FFFF) * q18, p0y = (float)(Py & 0x3FFFF) * q18, p0z = (float)(Pz & 0x3FFFF) * q18;
    const float kx = 0.25f * fx * gx, ky = 0.25f * fy * gy, kz = 0.25f * fz * gz;
    const float hx = (sx > 0 ? 0.0f : 1.0f) - p0x, hy = (sy > 0 ? 0.0f : 1.0f) - p0y, hz = (sz > 0 ? 0.0f : 1.0f) - p0z;
    const float jx = 4.0f * ix * gx, jy = 4.0f * iy * gy, jz = 4.0f * iz * gz;
    if constexpr (DEPTH) {
        ne = 0;
        ade = 1;
    }
    const float kR = 0.5f - 0.25f * kCastEps, kMagic = 12582912.0f;
    // the brick at time t0, and whether it is certain
    float t = t0;
    float px = fmaf(kx, t, p0x) - 0.5f, py = fmaf(ky, t, p0y) - 0.5f, pz = fmaf(kz, t, p0z) - 0.5f;
    float bx = (px + kMagic) - kMagic, by = (py + kMagic) - kMagic, bz = (pz + kMagic) - kMagic;
    bool sure = t < t_end - kCastEps && (t0 == 0.0f || fmaxf(fabsf(px - bx), fmaxf(fabsf(py - by), fabsf(pz - bz))) < kR);
    if (t0 == 0.0f) bx = by = bz = 0.0f;
    uint32_t hit = kNoHit;
    int rounds = 0;  // every round passes a brick face; beyond kCastRounds one fine phase runs to the end
    for (bool more = true; more;) {
        while (sure) {
            // (int)b and (float)d by the bits of floats whose unit is their last place, without conversions
            const int ib = (b0z + float_bits(bz + kMagic) - 0x4B400000) * nby + (b0y + float_bits(by + kMagic) - 0x4B400000);
            const size_t bi = (size_t)ib * (size_t)nbx + (size_t)(b0x + float_bits(bx + kMagic) - 0x4B400000);
            const int d = ld_u8(dist + bi);
            if constexpr (STATS) ++coarse;
            const float df = small_float(max(d, 1));
            const float tx = (fmaf(gx, df, bx) + hx) * jx, ty = (fmaf(gy, df, by) + hy) * jy, tz = (fmaf(gz, df, bz) + hz) * jz;
            const float t1 = fminf(tx, fminf(ty, tz));
            const bool ox = tx == t1, oy = !ox && ty == t1, oz = !ox && !oy;
            // floors of the positions (nearest integer of p - 1/2) and their distance from a brick's middle
            const float qx = fmaf(kx, t1, p0x) - 0.5f, qy = fmaf(ky, t1, p0y) - 0.5f, qz = fmaf(kz, t1, p0z) - 0.5f;
            const float mx = (qx + kMagic) - kMagic, my = (qy + kMagic) - kMagic, mz = (qz + kMagic) - kMagic;
            const float r = fmaxf(ox ? 0.0f : fabsf(qx - mx), fmaxf(oy ? 0.0f : fabsf(qy - my), oz ? 0.0f : fabsf(qz - mz)));
            bool ok = true;
            if (d == 0) {  // an occupied voxel between the entry and the exit?
                const float e = fmaf(t, kTimeErr, 2.0f * kCastEps);
                const float fx_ = bx - 0.5f, fy_ = by - 0.5f, fz_ = bz - 0.5f;
                const int lx = max(0, (int)floorf(4.0f * (fminf(px, qx) - fx_) - e)), ux = min(3, (int)floorf(4.0f * (fmaxf(px, qx) - fx_) + e));
                const int ly = max(0, (int)floorf(4.0f * (fminf(py, qy) - fy_) - e)), uy = min(3, (int)floorf(4.0f * (fmaxf(py, qy) - fy_) + e));
                const int lz = max(0, (int)floorf(4.0f * (fminf(pz, qz) - fz_) - e)), uz = min(3, (int)floorf(4.0f * (fmaxf(pz, qz) - fz_) + e));
                ok = !mask_box(ld_u64(om + bi), min(lx, 3), max(ux, 0), min(ly, 3), max(uy, 0), min(lz, 3), max(uz, 0));
            }
            if (ok) {
                t = t1;
                bx = ox ? fmaf(gx, df, bx) : mx;
                by = oy ? fmaf(gy, df, by) : my;
                bz = oz ? fmaf(gz, df, bz) : mz;
                px = qx;
                py = qy;
                pz = qz;
            }
            sure = ok && t < t_end - kCastEps && r < kR;
        }
        // the ray is free of occupied voxels up to t: done if that is the range or the grid's edge
        more = t <= t_end + kCastEps;
        const float slack = fmaf(t, kTimeErr, kCastEps);
        const float tf = ++rounds < kCastRounds ? t + slack : 1e30f;  // the fine phase runs at least to here
        const uint32_t ts = (uint32_t)(int)(fmaxf(0.0f, fminf(t, t_end) - slack) * 65536.0f);
        const int cx = crossings_until(n0x, ax, ts), cy = crossings_until(n0y, ay, ts), cz = crossings_until(n0z, az, ts);
        int vx = v0x + sx * cx, vy = v0y + sy * cy, vz = v0z + sz * cz;
        // next crossing times, advanced by additions: within 2^-24 t per step, hence kFineSteps and kFineErr
        float tx = (float)(n0x + ((uint32_t)cx << 16)) * q16 * ix, ty = (float)(n0y + ((uint32_t)cy << 16)) * q16 * iy,
              tz = (float)(n0z + ((uint32_t)cz << 16)) * q16 * iz;
        uint64_t m = more ? ld_u64(om + ((size_t)((vz >> 2) * nby + (vy >> 2)) * nbx + (vx >> 2))) : 0ull;
        int left = kFineSteps;
        bool walk = more;
        while (walk) {
            if constexpr (STATS) ++fine;
            const float mn = fminf(tx, fminf(ty, tz));
            const float lim = fmaf(mn, kFineErr, mn);
            bool ox = tx <= lim, oy = ty <= lim, oz = tz <= lim;
            const bool occ = (m >> (((vz & 3) << 4) | ((vy & 3) << 2) | (vx & 3))) & 1ull;
            if (occ) hit = (uint32_t)(abs(vx - v0x) + abs(vy - v0y) + abs(vz - v0z));
            walk = !occ;
            // two crossings too close to tell, or one near the range: the exact order and range test
            if ((ox && oy) || (ox && oz) || (oy && oz) || lim >= T * (1.0f - kFineErr)) {
                const uint32_t nx = n0x + ((uint32_t)abs(vx - v0x) << 16), ny = n0y + ((uint32_t)abs(vy - v0y) << 16),
                               nz = n0z + ((uint32_t)abs(vz - v0z) << 16);
                const int a = ev_argmin3(nx, ax, ny, ay, nz, az);
                ox = a == 0;
                oy = a == 1;
                oz = a == 2;
                const uint32_t nc = ox ? nx : (oy ? ny : nz), ac = ox ? ax : (oy ? ay : az);
                walk = walk && ((uint64_t)nc << 30) < (uint64_t)Tq * ac;
            }
            if (walk) {
                if constexpr (DEPTH) {
                    ne = ox ? n0x + ((uint32_t)abs(vx - v0x) << 16) : (oy ? n0y + ((uint32_t)abs(vy - v0y) << 16) : n0z + ((uint32_t)abs(vz - v0z) << 16));
                    ade = ox ? ax : (oy ? ay : az);
                }
                tx += ox ? ix : 0.0f;
                ty += oy ? iy : 0.0f;
                tz += oz ? iz : 0.0f;
                vx += ox ? sx : 0;
                vy += oy ? sy : 0;
                vz += oz ? sz : 0;
                --left;
                const int v = ox ? vx : (oy ? vy : vz), s = ox ? sx : (oy ? sy : sz);  // the coordinate that moved
                if ((v & 3) == (s > 0 ? 0 : 3) || left <= 0) {  // entered another brick
                    // beyond the grid: in a brick of its own, or in the last, partial brick (no bit there)
                    walk = (unsigned)v < (unsigned)(ox ? gnx : (oy ? gny : gnz));
                    more = walk;
                    if (walk) {
                        m = ld_u64(om + ((size_t)((vz >> 2) * nby + (vy >> 2)) * nbx + (vx >> 2)));
                        t = mn;
                        walk = mn < tf && left > 0;
                    }
                }
            } else {
                more = false;
            }
        }
        // back to the jumps from the brick just entered, exactly known
        bx = small_float(vx >> 2) - small_float(b0x);
        by = small_float(vy >> 2) - small_float(b0y);
        bz = small_float(vz >> 2) - small_float(b0z);
        px = fmaf(kx, t, p0x) - 0.5f;
        py = fmaf(ky, t, p0y) - 0.5f;
        pz = fmaf(kz, t, p0z) - 0.5f;
        sure = more && t < t_end - kCastEps;
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
                       const float whi[3], float s_end) {
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
        const int d = ld_u8(dist + ((size_t)(b[2] * nb[1] + b[1]) * nb[0] + b[0]));
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
