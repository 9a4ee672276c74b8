// Panoramic mode by 4x4x4 bricks: the counts of pano.cu's ray-by-ray kernel by owned voxels.
//
//   pano_cast_kernel   - the A x H rays of every node run to their first occupied voxel (cast_bricks) and
//                        store its step index with the minimum and maximum of every pixel tile, column
//                        along the row: one image of A x H per node where the pinhole modes have K of W x H.
//   pano_node_kernel   - every node's range ball, 32 bricks at a time, lane = brick: bricks above or below
//                        the strips' rows or behind every ray's first hit are dropped; the others go to a
//                        queue with what could be decided for the brick as a whole (all rows in the image,
//                        all before the hit, all visited for certain; observed by one ancestor).
//   pano_brick_kernel  - one warp per record, lane = the brick's voxel column pair: a voxel's azimuth gives
//                        its wedge, and each counted voxel adds to its wedge's pair of counts.
//   pano_window_kernel - each yaw's counts, the sums over its Wc columns.
//
// A voxel is tested once per node here, not once per yaw, so the undecided work is small and the cast and
// the ancestors' tests dominate: 1.9 and 2.0 ms of 4.2 ms for 500 nodes of A = 640, H = 120 at 0.1 m, range
// 6 m (the ray-by-ray kernel: 13.7 ms in all, bound by its chain of voxel loads); with the tree cast by
// one launch 1.5 and 2.0 of 3.7 ms. Every decision is conservative with an exact integer fallback (the
// wedge's cross products, the strip's rows, visit_index), so the counts equal the ray-by-ray kernel's.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "launch.cuh"
#include "nodecount.cuh"
#include "pano.h"
#include "voxcount.h"

namespace mig {

namespace {

// The nodes [q0, q1) of the level that this chunk takes.
struct NodeRange {
    int l0, q0, q1;
};
// (with p.tree: of the tree, in the cast, where lvl is the number of levels)
__device__ __forceinline__ NodeRange node_range(const LevelParams &p, bool cast = false) {
    if (p.tree && cast) return NodeRange{0, 0, min(p.tree, p.level_off[p.lvl])};
    const int l0 = p.level_off[p.lvl], n = p.level_off[p.lvl + 1] - l0;
    return NodeRange{l0, p.q0, min(p.q1, n)};
}

// The rays of a node's panorama; pixel (i, j) = (column, row).
struct PanoRays {
    const LevelParams &p;
    int4 nd;
    bool clutter;  // as of CameraRays
    int W, H;
    // w: at least the horizontal part of the unit ray (Q30)
    __device__ __forceinline__ int4 ray(int i, int j) const {
        int4 d = p.pano_dir[(size_t)i * H + j];
        d.w = (int)fminf(sqrtf((float)d.x * (float)d.x + (float)d.y * (float)d.y) * 1.000001f, 1.0737418e9f) + 1;
        return d;
    }
    __device__ __forceinline__ void dir(const int4 &b, int &dx, int &dy, int &dz) const {
        dx = b.x;
        dy = b.y;
        dz = b.z;
    }
    // The beam of the 8x4 part at pixel (i0, j0), by depth along the azimuth m in the middle of its columns:
    // at unit depth its rays' horizontal parts lie on a line, and their heights between z / h and
    // z / (h cos) of the outermost columns. A unit ray's depth is at most h.
    __device__ __forceinline__ float beam(const uint8_t *dist, int i0, int j0) const {
        if (i0 >= W || j0 >= H || W < 64 || clutter) return 0.0f;  // 8 columns: at most 45 degrees
        const int i1 = min(i0 + 7, W - 1), j1 = min(j0 + 3, H - 1);
        const int4 a = p.pano_dir[(size_t)i0 * H + j0], b = p.pano_dir[(size_t)i1 * H + j0], d = p.pano_dir[(size_t)i0 * H + j1];
        const float ha = sqrtf((float)a.x * (float)a.x + (float)a.y * (float)a.y), ia = 1.0f / ha;
        const float hd = sqrtf((float)d.x * (float)d.x + (float)d.y * (float)d.y);
        const float ax = (float)a.x * ia, ay = (float)a.y * ia, bx = (float)b.x * ia, by = (float)b.y * ia;
        const float mx = ax + bx, my = ay + by, mi = rsqrtf(mx * mx + my * my);
        const float ic = 1.0f / ((ax * mx + ay * my) * mi);  // 1 / cos of the outermost columns
        const float z0 = (float)a.z * ia, z1 = (float)d.z / hd;
        const float lo[3] = {fminf(ax, bx) * ic, fminf(ay, by) * ic, fminf(fminf(z0, z1), fminf(z0, z1) * ic)};
        const float hi[3] = {fmaxf(ax, bx) * ic, fmaxf(ay, by) * ic, fmaxf(fmaxf(z0, z1), fmaxf(z0, z1) * ic)};
        const float zm = z0 * z1 <= 0.0f ? 0.0f : fminf(fabsf(z0), fabsf(z1));
        const float s_end = q16f((int)p.Tq) * rsqrtf(1.0f + zm * zm) * 1.00001f;
        return beam_free(dist, p.grid.nx, p.grid.ny, p.grid.nz, nd.x, nd.y, nd.z, lo, hi, s_end MIG_CHECKED(, &p));
    }
};

__global__ void __launch_bounds__(kWarpsN * 32, kCastCtas) pano_cast_kernel(const LevelParams p, int num_sms) {
    __shared__ uint2 s_t[kWarpsN];
    __shared__ float s_beam[32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    wait_previous();
    if (blockIdx.x == 0 && threadIdx.x < 3) p.vctr[threadIdx.x] = 0;  // the counters of the passes that follow
    const NodeRange nr = node_range(p, true);
    if (nr.q0 >= nr.q1) return;
    const int A = p.pano_A, H = p.H;
    const CastLayout lay = cast_layout(p.tree ? p.tree : nr.q1 - nr.q0, A, H, num_sms);
    const int T = lay == kCastSmall ? 16 : 32;
    const int tx = (A + T - 1) / T, ty = (H + T - 1) / T;
    const size_t AH = (size_t)A * H;
    const Pyramid y = pyramid(A, H);
    const uint64_t *om = grid_omask(p.grid);
    const uint8_t *dist = p.grid.g + dist_offset(p.grid.nx, p.grid.ny, p.grid.nz);
    CastCnt st;
    const long long items = (long long)(nr.q1 - nr.q0) * tx * ty;
    const bool dyn = lay == kCastLarge;  // tile by tile, as in cast_kernel
    long long it = dyn ? __shfl_sync(0xffffffffu, lane == 0 ? atomicAdd(p.work, 1) : 0, 0) : (long long)blockIdx.x;
    while (it < items) {
        int more = 0;
        if (dyn && lane == 0) more = atomicAdd(p.work, 1);
        const int tile = (int)(it % (tx * ty)), ln = (int)(it / (tx * ty));
        const int n = p.level_nodes[nr.l0 + nr.q0 + ln];
        const int4 nd = p.node[n];
        const PanoRays rays{p, nd, in_clutter(p, dist, nd), A, H};
        const CastOut<false> o{p.steps + (size_t)ln * AH, p.hz + (size_t)ln * y.n, nullptr};
        const int x0 = tile % tx * T, y0 = tile / tx * T;
        if (y0 == 0) {  // the first row of tiles clears its columns' counts
            const int c = x0 + (lay == kCastLarge ? lane : (int)threadIdx.x);
            if (c < min(x0 + T, A)) reinterpret_cast<unsigned long long *>(p.pano_cnt)[(size_t)n * A + c] = 0ull;
        }
        if (lay == kCastLarge) {
            cast_large<false>(p, om, dist, y, rays, x0, y0, o, lane, st);
        } else if (lay == kCastMid) {
            cast_mid<false>(p, om, dist, y, rays, x0, y0, o, s_t, s_beam, warp, lane, st);
        } else {
            cast_small<false>(p, om, dist, y, rays, x0, y0, o, s_t, warp, lane, st);
        }
        it = dyn ? __shfl_sync(0xffffffffu, more, 0) : it + gridDim.x;
    }
}

// Per-launch constants.
struct PanoConst {
    float a2c;   // columns per radian
    float fA, fH, fy, cosw;
    float cerr;  // columns: the error of a voxel's azimuth in columns
    float verr;  // rows: the error of the exact test's Q16 rows
    float bv, nv;
};
// cerr: atan2f (3 ulp), the offsets and the product, 2.6e-7 of a turn's columns together.
// verr: 2^-17 per coefficient of a row, sqrt(3) |r| / Z inside a strip, (1 + H) for the quotient.
__device__ __forceinline__ PanoConst pano_const(const LevelParams &p) {
    PanoConst c;
    c.fA = (float)p.pano_A;
    c.fH = (float)p.H;
    c.a2c = c.fA * 0.15915494f;
    c.fy = 1.0f / p.ify;
    const float w = 3.1415927f / c.fA, tv = 0.5f * c.fH * p.ify;
    c.cosw = cosf(w) * 0.999999f;
    const float cw = fmaxf(c.cosw, 1e-3f);
    c.cerr = 6e-7f * c.fA + 1e-5f;
    c.verr = 2e-5f * sqrtf(1.0f / (cw * cw) + tv * tv) * (1.0f + c.fH) + 0.01f;
    c.bv = 0.5f - 1.0e-6f * (c.fH + 1.0f);
    c.nv = 1.001f * (0.7072f * c.fH + c.fy);  // at least a strip row's L1 norm
    return c;
}

// A brick in a node's panorama: the columns [c0, c1] (modulo A) and rows [r0, r1] that its voxels' centres
// can fall in. (cx, cy, cz): the brick's centre from the node. The extents 1.5 are widened by 0.05.
struct PanoBox {
    int in;  // 1: every centre inside the rows, -1: none, 0: undecided
    bool look;  // the tile bounds can be looked up
    int c0, c1, r0, r1;
    float zlo, zhi;  // strip depths
};
__device__ __forceinline__ PanoBox pano_box(const PanoConst &c, float cx, float cy, float cz, int A, int H) {
    const float kR = 2.1921f;  // 1.55 sqrt(2)
    PanoBox b;
    const float rho = sqrtf(fmaf(cx, cx, cy * cy)), h0 = rho - kR;
    b.in = 0;
    b.look = false;
    b.c0 = b.c1 = b.r0 = b.r1 = 0;
    b.zhi = rho + kR;
    b.zlo = h0 * c.cosw;
    if (h0 > 0.0f && b.zlo >= 0.5f) {
        const float zt = cz + 1.55f, zb = cz - 1.55f;
        const float v0 = 0.5f * c.fH - c.fy * __fdividef(zt, zt > 0.0f ? b.zlo : b.zhi) - c.verr;
        const float v1 = 0.5f * c.fH - c.fy * __fdividef(zb, zb > 0.0f ? b.zhi : b.zlo) + c.verr;
        b.in = v1 < 0.0f || v0 > c.fH ? -1 : (v0 >= 0.0f && v1 <= c.fH ? 1 : 0);
        b.r0 = (int)floorf(fminf(fmaxf(v0, 0.0f), c.fH - 1.0f));
        b.r1 = (int)floorf(fminf(fmaxf(v1, 0.0f), c.fH - 1.0f));
        float az = atan2f(cy, cx) * c.a2c;
        az += az < 0.0f ? c.fA : 0.0f;
        const float d = fmaf(asinf(kR / rho), c.a2c, 0.02f + c.cerr);
        b.c0 = (int)floorf(az - d);
        b.c1 = (int)floorf(az + d);
        b.look = b.c1 - b.c0 <= min(kPyramidSpan, A - 1) && b.r1 - b.r0 <= kPyramidSpan;
    }
    return b;
}
// Bounds of the step counts under a box (hz_box), over the seam between the last and the first column.
__device__ __forceinline__ uint32_t pano_hz(const LevelParams &p, const uint32_t *hz, const Pyramid &y, int top, const PanoBox &b, int A) {
    BoxView v;
    v.v0 = b.r0;
    v.v1 = b.r1;
    v.u0 = max(b.c0, 0);
    v.u1 = min(b.c1, A - 1);
    uint32_t r = hz_box(p, hz, y, top, v);
    if (b.c0 < 0) {
        v.u0 = b.c0 + A;
        v.u1 = A - 1;
        r = __vminu2(r, hz_box(p, hz, y, top, v));
    } else if (b.c1 >= A) {
        v.u0 = 0;
        v.u1 = b.c1 - A;
        r = __vminu2(r, hz_box(p, hz, y, top, v));
    }
    return r;
}

// The wedge that holds the horizontal offset (rx, ry) by its exact test (x0 >= 0 and x1 < 0), near the
// guess c, or -1 (the offset 0).
__device__ __noinline__ int wedge_exact(const int2 *bc, int A, int c, int rx, int ry) {
    int col = -1;
    for (int i = -1; i <= 1; ++i) {
        const int k = c + i < 0 ? c + i + A : (c + i >= A ? c + i - A : c + i);
        const int2 b0 = bc[k], b1 = bc[k + 1 == A ? 0 : k + 1];
        if ((int64_t)b0.x * ry - (int64_t)b0.y * rx >= 0 && (int64_t)b1.x * ry - (int64_t)b1.y * rx < 0) col = k;
    }
    return col;
}
// The strip's exact row of a voxel centre, or -1.
__device__ __noinline__ int row_exact(const int4 m0, const int4 m1, int rx, int ry, int rz, int H) {
    const int64_t Z = (int64_t)m0.w * rx + (int64_t)m1.x * ry + (int64_t)m1.y * rz;
    const int64_t V = (int64_t)m0.x * rx + (int64_t)m0.y * ry + (int64_t)m0.z * rz;
    if (Z <= 0 || V < 0 || V >= (int64_t)H * Z) return -1;
    return (int)(V / Z);
}

// One record (lane = voxel of the brick's lower and upper half): the ancestor tests left, then each
// voxel's wedge, row, reach and visit.
__device__ __forceinline__ void count_pano_brick(const LevelParams &p, const VoxConst &vc, const PanoConst &pc, const YawRows *s_y,
                                                 const NodeAnc *anc, int n, const int4 nd, const uint16_t *steps, const BrickRec &r,
                                                 int lane) {
    const int A = p.pano_A, H = p.H;
    const int x = 4 * (int)(r.brick & 1023) + (lane & 3), y = 4 * (int)((r.brick >> 10) & 1023) + ((lane >> 2) & 3),
              z0 = 4 * (int)(r.brick >> 20) + (lane >> 4);
    const uint64_t U = r.U;
    const int rx = (x << 16) + 32768 - nd.x, ry = (y << 16) + 32768 - nd.y, rz0 = (z0 << 16) + 32768 - nd.z;
    const float ex = q16f(rx), ey = q16f(ry), ez[2] = {q16f(rz0), q16f(rz0 + 131072)};
    const float rinf = fmaxf(fmaxf(fabsf(ex), fabsf(ey)), fabsf(ez[0])) + 8.0f;
    const float verr = 5e-7f * (__uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(rinf))) + 1.0f);
    NodeCnt st;
    const uint64_t O = voxel_ancestors<false>(p, vc, s_y, anc, nd, r.anc, U, r.O, x, y, z0, verr, lane, st);
    bool c[2] = {((uint32_t)U >> lane & 1) != 0, ((uint32_t)(U >> 32) >> lane & 1) != 0};
    // ---- the wedge, the same for the lane's two voxels
    int col = -1;
    if (c[0] || c[1]) {
        float af = atan2f(ey, ex) * pc.a2c;
        af += af < 0.0f ? pc.fA : 0.0f;
        const float ff = floorf(af), fr = af - ff;
        col = min((int)ff, A - 1);
        if (fr < pc.cerr || fr > 1.0f - pc.cerr || ff >= pc.fA) col = wedge_exact(p.pano_bc, A, col, rx, ry);
    }
    c[0] = c[0] && col >= 0;
    c[1] = c[1] && col >= 0;
    if (!r.all) {
        const float exy2 = fmaf(ex, ex, ey * ey);
        const int mxy = abs(x - (nd.x >> 16)) + abs(y - (nd.y >> 16));
        int4 m0 = make_int4(0, 0, 0, 0), m1 = m0;
        if (c[0] || c[1]) {
            m0 = p.pano_row[2 * col];
            m1 = p.pano_row[2 * col + 1];
        }
        const float Z = fmaf(q16f(m0.w), ex, q16f(m1.x) * ey), zi = __fdividef(1.0f, Z);
        const float Vxy = fmaf(q16f(m0.x), ex, q16f(m0.y) * ey), vz = q16f(m0.z);
        const float sv = 2.0f * verr * fmaf(pc.fH, 1.4143f, pc.nv);
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            const float e = h ? ez[1] : ez[0];
            const float r2 = fmaf(e, e, exy2);
            bool in = (h ? c[1] : c[0]) && r2 < vc.out2;
            const float kMagic = 12582912.0f;
            const float v = fmaf(fmaf(vz, e, Vxy), zi, -0.5f), fv = (v + kMagic) - kMagic;
            const bool sure = Z >= 0.5f && fmaf(zi, sv, fabsf(v - fv)) <= pc.bv;
            int row = -1;
            if (in) {
                if (sure) row = fv >= 0.0f && fv < pc.fH ? (int)fv : -1;
                else row = row_exact(m0, m1, rx, ry, rz0 + (h << 17), H);
                in = row >= 0;
            }
            if (in && r.rch) {
                const uint16_t *s = steps + (size_t)row * A + col;
                in = steps_ok(p, s) && mxy + abs(z0 + 2 * h - (nd.z >> 16)) < (int)ld_written(s);
            }
            if (in && r.vis && !(Z >= 0.5f && r2 < vc.l22 && Z < p.vis_zl2)) {
                const int4 d = p.pano_dir[(size_t)col * H + row];
                const float q30 = 9.31322574615478515625e-10f;
                const int t = visit_slab(ex, ey, e, (float)d.x * q30, (float)d.y * q30, (float)d.z * q30, vc.Tv);
                in = t > 0 || (t < 0 && visit_index(nd.x, nd.y, nd.z, d.x, d.y, d.z, x, y, z0 + 2 * h, p.Tq) >= 0);
            }
            c[0] = h ? c[0] : in;
            c[1] = h ? in : c[1];
        }
    }
    const bool o0 = (uint32_t)O >> lane & 1, o1 = (uint32_t)(O >> 32) >> lane & 1;
    unsigned v = (unsigned)c[0] + (unsigned)c[1] + ((unsigned)(c[0] && !o0) << 16) + ((unsigned)(c[1] && !o1) << 16);
    // lanes l and l + 16 hold the same voxel column; then neighbours along x of one wedge
    v += __shfl_xor_sync(0xffffffffu, v, 16);
    col = max(col, __shfl_xor_sync(0xffffffffu, col, 16));
    const unsigned w = __shfl_down_sync(0xffffffffu, v, 1);
    const int cw = __shfl_down_sync(0xffffffffu, col, 1);
    const bool lead = !(lane & 1);
    const bool pair = cw == col || w == 0;  // of an even lane and the odd one after it
    const bool taken = __shfl_up_sync(0xffffffffu, (int)pair, 1) && !lead;
    if (lead && pair) v += w;
    if (lane < 16 && v && !taken)
        atomicAdd(reinterpret_cast<unsigned long long *>(p.pano_cnt) + (size_t)n * A + col,
                  (unsigned long long)(v & 0xFFFFu) | ((unsigned long long)(v >> 16) << 32));
}

__global__ void __launch_bounds__(kWarpsN * 32, 3) pano_node_kernel(const LevelParams p, int num_sms) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    YawRows *s_y = reinterpret_cast<YawRows *>(s_dyn);
    NodeAnc *anc = reinterpret_cast<NodeAnc *>(s_y + p.K) + warp * p.max_anc;
    for (int k = threadIdx.x; k < p.K; k += blockDim.x)
        s_y[k] = yaw_rows(p.yawtab + k * 12, p.W, p.H, p.vis_hu, p.vis_hv, p.ifx, p.ify);
    wait_previous();
    if (blockIdx.x == 0 && threadIdx.x == 0) p.work[0] = 0;  // the next cast's tiles
    __syncthreads();
    const NodeRange nr = node_range(p);
    const int nn = nr.q1 - nr.q0;
    if (nn <= 0) return;
    const int base = p.tree ? nr.l0 + nr.q0 : 0;  // the chunk's first node in the step counts and bounds
    const int A = p.pano_A, H = p.H;
    const size_t WH = (size_t)p.W * H, AH = (size_t)A * H;
    const Pyramid pyr = pyramid(p.W, H), ppyr = pyramid(A, H);
    const int top = cast_layout(p.tree ? p.tree : nn, A, H, num_sms) == kCastSmall ? 4 : 5;  // the bounds the cast kept
    const BrickDims bd = brick_dims(p.grid.nx, p.grid.ny, p.grid.nz);
    const uint64_t *umask = grid_umask(p.grid);
    const VoxConst vc = vox_const(p);
    const PanoConst pc = pano_const(p);
    const float R2 = (vc.Tv + 1.0f) * (vc.Tv + 1.0f);
    const int Rv = (int)(p.Tq >> 16) + 2;
    const int mxy = mac_xy(p.Tq), mn = mxy * mxy * mac_z(p.Tq);
    // macro blocks per work item: enough items for every warp to get several, at most one per lane
    const int group = (int)max(1ll, min(32ll, (long long)nn * mn / ((long long)gridDim.x * kWarpsN * 8)));
    const int gpn = (mn + group - 1) / group;
    int cur = -1, na = 0;
    for (;;) {
        int it = 0;
        if (lane == 0) it = atomicAdd(p.vctr, 1);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= nn * gpn) break;
        const int ln = it / gpn, g0 = (it - ln * gpn) * group;
        const int n = p.level_nodes[nr.l0 + nr.q0 + ln];
        const int4 nd = p.node[n];
        const int v0x = nd.x >> 16, v0y = nd.y >> 16, v0z = nd.z >> 16;
        int mX = 0, mY = 0, mZ = 0;
        const bool live = lane < group && macro_block(p, nd, g0 + lane, mn, mxy, Rv, R2, mX, mY, mZ);
        unsigned todo = __ballot_sync(0xffffffffu, live);
        if (todo && n != cur) {
            cur = n;
            na = node_ancestors(p, n, anc, WH, pyr.n, lane);
        }
        const uint32_t *hz = p.hz + (size_t)(base + ln) * ppyr.n;
#pragma unroll 1
        for (; todo; todo &= todo - 1) {
            const int src = __ffs(todo) - 1;
            const int X = __shfl_sync(0xffffffffu, mX, src) * 4, Y = __shfl_sync(0xffffffffu, mY, src) * 4,
                      Z = __shfl_sync(0xffffffffu, mZ, src) * 2;  // the block's first brick
            const int bx = X + (lane & 3), by = Y + ((lane >> 2) & 3), bz = Z + (lane >> 4);
            uint64_t U = 0;
            if (bx < bd.nbx && by < bd.nby && bz < bd.nbz) U = ld_mask(umask, (size_t)(bz * bd.nby + by) * bd.nbx + bx MIG_CHECKED(, &p));
            const float cx = q16f(((4 * bx + 2) << 16) - nd.x), cy = q16f(((4 * by + 2) << 16) - nd.y),
                        cz = q16f(((4 * bz + 2) << 16) - nd.z);
            float far;
            {
                const float dx = fmaxf(fabsf(cx) - 1.5f, 0.f), dy = fmaxf(fabsf(cy) - 1.5f, 0.f), dz = fmaxf(fabsf(cz) - 1.5f, 0.f);
                if (dx * dx + dy * dy + dz * dz > R2) U = 0;
                const float ex = fabsf(cx) + 1.5f, ey = fabsf(cy) + 1.5f, ez = fabsf(cz) + 1.5f;
                far = sqrtf(ex * ex + ey * ey + ez * ez);
            }
            bool want = false, reach = false, sure = false, in = false;  // reach, sure: of every voxel
            if (U) {
                const PanoBox b = pano_box(pc, cx, cy, cz, A, H);
                want = b.in >= 0;
                in = b.in > 0;
                if (want && b.look) {
                    // Manhattan distances (step indices) of the brick's voxels from the start voxel
                    const int ax = 4 * bx - v0x, ay = 4 * by - v0y, az = 4 * bz - v0z;
                    const int man0 = max(max(ax, -ax - 3), 0) + max(max(ay, -ay - 3), 0) + max(max(az, -az - 3), 0);
                    const int man1 = max(abs(ax), abs(ax + 3)) + max(abs(ay), abs(ay + 3)) + max(abs(az), abs(az + 3));
                    const uint32_t hm = pano_hz(p, hz, ppyr, top, b, A);
                    want = man0 < (int)((hm >> 16) ^ 0xFFFFu);
                    reach = man1 < (int)(hm & 0xFFFFu);
                }
                sure = b.zlo >= 0.5f && b.zhi < p.vis_zl2 && far + 0.02f < vc.Tv;
            }
            const unsigned recs = __ballot_sync(0xffffffffu, want);
            if (!recs) continue;
            uint64_t O = 0, left = 0;  // observed voxels; ancestors undecided for the brick
            block_ancestors<false>(p, s_y, anc, na, nd, pyr, vc, X, Y, Z, bx, by, bz, U, want, lane, O, left);
            if (O == U) left = 0;
            int at = 0;
            if (lane == 0) at = atomicAdd(p.vctr + 1, __popc(recs));
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(recs & ((1u << lane) - 1u));
            BrickRec r{U, O, left, in && reach && sure, 0ull, !reach, !sure, (uint32_t)bx | ((uint32_t)by << 10) | ((uint32_t)bz << 20),
                       (uint32_t)ln};
            if (want && at < p.queue_cap && queue_ok(p, at)) p.queue[at] = r;
#pragma unroll 1
            for (unsigned full = __ballot_sync(0xffffffffu, want && at >= p.queue_cap); full; full &= full - 1) {
                const int s = __ffs(full) - 1;
                BrickRec q{shfl64(r.U, s), shfl64(r.O, s), shfl64(r.anc, s), shfl64(r.all, s), 0ull,
                           shfl64(r.rch, s), shfl64(r.vis, s), __shfl_sync(0xffffffffu, r.brick, s), r.node};
                count_pano_brick(p, vc, pc, s_y, anc, n, nd, p.steps + (size_t)(base + ln) * AH, q, lane);
            }
        }
    }
}

// The queue's records, one warp each, in slices of consecutive records (mostly of one node).
__global__ void __launch_bounds__(kWarpsN * 32, 4) pano_brick_kernel(const LevelParams p) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    YawRows *s_y = reinterpret_cast<YawRows *>(s_dyn);
    NodeAnc *anc = reinterpret_cast<NodeAnc *>(s_y + p.K) + warp * p.max_anc;
    for (int k = threadIdx.x; k < p.K; k += blockDim.x)
        s_y[k] = yaw_rows(p.yawtab + k * 12, p.W, p.H, p.vis_hu, p.vis_hv, p.ifx, p.ify);
    wait_previous();
    __syncthreads();
    const NodeRange nr = node_range(p);
    if (nr.q1 <= nr.q0) return;
    const int base = p.tree ? nr.l0 + nr.q0 : 0;
    const int total = min(p.vctr[1], p.queue_cap);
    const int slice = max(1, min(64, total / (int)(gridDim.x * kWarpsN * 8)));
    if (blockIdx.x * kWarpsN * slice >= total) return;
    const size_t WH = (size_t)p.W * p.H, AH = (size_t)p.pano_A * p.H;
    const int pyr_n = pyramid(p.W, p.H).n;
    const VoxConst vc = vox_const(p);
    const PanoConst pc = pano_const(p);
    uint32_t cur = 0xFFFFFFFFu;
    int n = 0;
    int4 nd = make_int4(0, 0, 0, 0);
    for (;;) {
        int i = 0;
        if (lane == 0) i = atomicAdd(p.vctr + 2, slice);
        i = __shfl_sync(0xffffffffu, i, 0);
        if (i >= total) break;
        const int end = min(i + slice, total);
#pragma unroll 1
        for (; i < end; ++i) {
            if (!queue_ok(p, i)) continue;
            const BrickRec r = p.queue[i];
            if (r.node != cur) {
                cur = r.node;
                n = p.level_nodes[nr.l0 + nr.q0 + (int)cur];
                nd = p.node[n];
                node_ancestors(p, n, anc, WH, pyr_n, lane);
            }
            count_pano_brick(p, vc, pc, s_y, anc, n, nd, p.steps + (size_t)(base + (int)cur) * AH, r, lane);
        }
    }
}

}  // namespace

void set_pano_visit(LevelParams &p, int A, float vfov_deg) {
    p.vis_zl2 = visit_limits(360.0 / A, vfov_deg, 1, p.H).zl2;
}

void launch_pano_cast_chunk(const LevelParams &c, int num_sms, cudaStream_t s) {
    launch_behind(pano_cast_kernel, cast_grid(c.q1 - c.q0, c.pano_A, c.H, num_sms, 64), kWarpsN * 32, 0, s, c, num_sms);
}

void launch_pano_tree_cast(const LevelParams &p, int levels, int num_sms, cudaStream_t s) {
    LevelParams c = p;
    c.lvl = levels;
    c.q0 = 0;
    c.q1 = p.tree;
    launch_pano_cast_chunk(c, num_sms, s);
}

void launch_pano_voxel_chunk(const LevelParams &c, int num_sms, cudaStream_t s) {
    const int g = node_grid((long long)(c.q1 - c.q0) * node_items(c.Tq), num_sms * 3, c.crowd);
    const size_t smem = node_dyn_smem(c.K, c.max_anc);
    launch_behind(pano_node_kernel, g, kWarpsN * 32, smem, s, c, num_sms);
    launch_behind(pano_brick_kernel, brick_grid(c.q1 - c.q0, c.Tq, num_sms, c.crowd), kWarpsN * 32, smem, s, c);
}

void pano_bricks_init() {
    const int smem = (int)node_dyn_smem(MIG_MAX_YAW_BINS, MIG_MAX_DEPTH);
    cudaFuncSetAttribute(pano_node_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    cudaFuncSetAttribute(pano_brick_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

}  // namespace mig
