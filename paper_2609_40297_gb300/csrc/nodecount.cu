// The owned-voxel count of one tree level by 4x4x4 bricks, and the depth-buffer render.
//
//   cast_kernel   - every pixel ray of every (node, yaw) pair runs to its first occupied voxel
//                   (cast_bricks, bricks.cuh) and stores that voxel's step index (uint16; kNoHit if
//                   none), with the minimum and maximum of every 8x8, 16x16 and 32x32 pixel tile.
//                   A small tree's images are all cast by one launch (p.tree), else a level's or a chunk's.
//   node_kernel   - every node's range ball is enumerated once for all yaws, 32 bricks of 64 voxels
//                   at a time. A brick's unknown voxels are one 64-bit mask. Against each yaw, and each
//                   ancestor's depth buffer, a brick is decided as a whole where it can be (all in the
//                   image, all before the first hit of their pixels' rays, all visited for certain; or
//                   none of them), so a yaw's counts are mostly sums of population counts of masks.
//   brick_kernel  - the bricks left undecided, voxel by voxel.
//   render_kernel - the yaw selection, and the depth buffer of each internal node's selected yaw
//                   (Sec. IV-A) with the same tile bounds.
// Every whole-brick decision is conservative (boxes widened by proven rounding bounds) and every
// undecided voxel takes the exact integer tests of Sec. IV-B, so the counts equal the ray-by-ray
// walk's and the oracle's bit for bit.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdint>

#include "bricks.cuh"
#include "interval.cuh"
#include "kernels.h"
#include "launch.cuh"
#include "mig.h"
#include "nodecount.cuh"
#include "voxcount.h"

namespace mig {

namespace {

using namespace dev;

template <bool STATS, bool DEPTH>
__global__ void __launch_bounds__(kWarpsN * 32, kCastCtas) cast_kernel(const LevelParams p, int num_sms) {
    __shared__ uint2 s_t[kWarpsN];
    __shared__ float s_beam[32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    wait_previous();
    if (blockIdx.x == 0 && threadIdx.x < 3) p.vctr[threadIdx.x] = 0;  // the counters of the passes that follow
    int l0 = 0, q0 = 0, q1 = 0;
    if (p.tree) {  // lvl: the number of levels
        q1 = min(p.tree, p.level_off[p.lvl]) * p.K;
    } else {
        const StepRange step = step_range(p);
        l0 = step.l0;
        q0 = step.q0;
        q1 = step.q1;
    }
    if (q0 >= q1) return;
    const CastLayout lay = cast_layout(p.tree ? (long long)p.tree * p.K : q1 - q0, p.W, p.H, num_sms);
    const int T = lay == kCastSmall ? 16 : 32;
    const int tx = (p.W + T - 1) / T, ty = (p.H + T - 1) / T;
    const size_t WH = (size_t)p.W * p.H;
    const Pyramid y = pyramid(p.W, p.H);
    const uint64_t *om = grid_omask(p.grid);
    const uint8_t *dist = p.grid.g + dist_offset(p.grid.nx, p.grid.ny, p.grid.nz);
    CastCnt st;
    const long long items = (long long)(q1 - q0) * tx * ty;
    // large: a warp takes the next tile when it is done with one (asked for a tile's time ahead), so that
    // no warp waits for its CTA's slowest: 5.3 -> 4.8 ms at paper scale, 165 -> 148 ms on the large workload
    const bool dyn = lay == kCastLarge;
    long long it = dyn ? __shfl_sync(0xffffffffu, lane == 0 ? atomicAdd(p.work, 1) : 0, 0) : (long long)blockIdx.x;
    while (it < items) {
        int more = 0;
        if (dyn && lane == 0) more = atomicAdd(p.work, 1);
        const int tile = (int)(it % (tx * ty)), ql = (int)(it / (tx * ty));
        const int q = q0 + ql;
        const int4 nd = p.node[p.level_nodes[l0 + q / p.K]];
        const int32_t *yk = p.yawtab + (q % p.K) * 12;
        const CameraRays rays{p, nd, in_clutter(p, dist, nd), yk[0], yk[1], p.W, p.H};
        const CastOut<DEPTH> o{p.steps + (size_t)ql * WH, p.hz + (size_t)ql * y.n,
                               DEPTH && nd.w >= 0 ? p.depths + (size_t)ql * WH : nullptr};
        const int x0 = tile % tx * T, y0 = tile / tx * T;
        if (lay == kCastLarge) {
            cast_large<STATS>(p, om, dist, y, rays, x0, y0, o, lane, st);
        } else if (lay == kCastMid) {
            cast_mid<STATS>(p, om, dist, y, rays, x0, y0, o, s_t, s_beam, warp, lane, st);
        } else {
            cast_small<STATS>(p, om, dist, y, rays, x0, y0, o, s_t, warp, lane, st);
        }
        it = dyn ? __shfl_sync(0xffffffffu, more, 0) : it + gridDim.x;
    }
    if constexpr (STATS) {
        atomicAdd(p.stats + 8, (unsigned long long)st.rays);
        atomicAdd(p.stats + 9, (unsigned long long)st.fine);
        atomicAdd(p.stats + 10, (unsigned long long)st.jump);
    }
}

// Yaw selection (select_node's rule) of one node by a warp; returns the yaw.
__device__ __forceinline__ int select_warp(const LevelParams &p, int n, bool write, int lane) {
    const int2 *c = reinterpret_cast<const int2 *>(p.cnt) + (size_t)n * p.K;  // (abs, marginal)
    int best = 0x7fffffff, bm = -1, amax = 0;
    for (int k = lane; k < p.K; k += 32) {
        const int2 v = c[k];
        best = v.y > bm ? k : best;
        bm = max(bm, v.y);
        amax = max(amax, v.x);
    }
    const int m = __reduce_max_sync(0xffffffffu, bm);
    best = __reduce_min_sync(0xffffffffu, bm == m ? best : 0x7fffffff);
    amax = __reduce_max_sync(0xffffffffu, amax);
    if (write && lane == 0) {
        p.sel_yaw[n] = best;
        p.out_abs[n] = amax;
        p.out_marg[n] = m;
        p.out_yaw[n] = best;
    }
    return best;
}

// The yaw selection of the level's nodes, and the depth buffer of the selected yaw (Sec. IV-A): per
// pixel ray, camera z of the entry point of the first occupied voxel, else of the range endpoint. Only
// nodes with children (the level's first level_int nodes) are rendered; descendants read them in the
// ancestor test. Each tile's warps select their node's yaw themselves (one load and three reductions),
// which saves a level one launch of its chain: 4 to 5 us.
template <bool STATS>
__global__ void __launch_bounds__(kWarpsN * 32, kCastCtas) render_kernel(const LevelParams p, int num_sms) {
    __shared__ uint2 s_t[kWarpsN];
    __shared__ float s_beam[32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    wait_previous();
    if (p.tree && blockIdx.x == 0 && threadIdx.x < 3) p.vctr[threadIdx.x] = 0;  // for the next level's count
    int lvl = p.lvl;
    if (p.cursor) {
        const StepRange r = step_range(p);
        // the next step: the level's next chunk, the next level, or (past the deepest node) here again
        // with nothing to do
        if (blockIdx.x == 0 && threadIdx.x == 0)
            p.cursor[1] = r.q1 <= r.q0 ? make_int2(r.lvl, r.q0 / p.K) : (r.ends ? make_int2(r.lvl + 1, 0) : make_int2(r.lvl, r.q1 / p.K));
        if (!r.ends || r.q1 <= r.q0) return;
        lvl = r.lvl;
    }
    const int l0 = p.level_off[lvl], Li = p.level_int[lvl], L = p.level_off[lvl + 1] - l0;
    for (int li = Li + blockIdx.x * kWarpsN + warp; li < L; li += gridDim.x * kWarpsN)
        select_warp(p, p.level_nodes[l0 + li], true, lane);
    const CastLayout lay = cast_layout(Li, p.W, p.H, num_sms);
    const int T = lay == kCastSmall ? 16 : 32;
    const int tx = (p.W + T - 1) / T, ty = (p.H + T - 1) / T;
    const int items = Li * tx * ty;
    const Pyramid y = pyramid(p.W, p.H);
    const uint64_t *om = grid_omask(p.grid);
    const uint8_t *dist = p.grid.g + dist_offset(p.grid.nx, p.grid.ny, p.grid.nz);
    CastCnt st;
    const int per = lay == kCastLarge ? kWarpsN : 1, mine = lay == kCastLarge ? warp : 0;  // items at a time per CTA
    for (int it = blockIdx.x * per + mine; it < items; it += gridDim.x * per) {
        const int tile = it % (tx * ty);
        const int n = p.level_nodes[l0 + it / (tx * ty)];
        const int4 nd = p.node[n];
        const int k = select_warp(p, n, tile == 0 && (lay == kCastLarge || warp == 0), lane);
        const int32_t *yk = p.yawtab + k * 12;
        if (nd.w < 0) continue;  // uniform over the warps of the item
        const CameraRays rays{p, nd, in_clutter(p, dist, nd), yk[0], yk[1], p.W, p.H};
        const RenderOut o{p.dpyr ? p.dpyr + (size_t)nd.w * y.n : nullptr, nd.w,
                          p.depths ? p.depths + ((size_t)(l0 + it / (tx * ty)) * p.K + k) * ((size_t)p.W * p.H) : nullptr};
        const int x0 = tile % tx * T, y0 = tile / tx * T;
        if (lay == kCastLarge) {
            cast_large<STATS>(p, om, dist, y, rays, x0, y0, o, lane, st);
        } else if (lay == kCastMid) {
            cast_mid<STATS>(p, om, dist, y, rays, x0, y0, o, s_t, s_beam, warp, lane, st);
        } else {
            cast_small<STATS>(p, om, dist, y, rays, x0, y0, o, s_t, warp, lane, st);
        }
    }
    if constexpr (STATS) {
        atomicAdd(p.stats + 6, (unsigned long long)st.rays);
        atomicAdd(p.stats + 7, (unsigned long long)(st.fine + st.jump));
    }
}

// ---------------------------------------------------------------------------- the per-node count
// Two kernels per chunk of nodes. node_kernel takes macro blocks of 16x16x8 voxels, 4x4x2 bricks, one
// brick per lane, and decides whole bricks against every yaw and ancestor; what it cannot decide as a
// whole it appends to a queue, one record per brick. brick_kernel takes the records, one warp each,
// one voxel of the brick's lower and upper half per lane. (As one kernel the two stages' code, 4300
// instructions, did not fit the instruction cache, and a warp's block took 10 to 100 times as long as
// another's: 338 ms on the large workload.)
// Both are bound by instruction issue. node_kernel: 46 ms on the large workload (1.7 G (brick, yaw) pairs),
// 1.1 ms at paper scale; 60 % of the slots, 13 of 32 lanes (bricks without unknown voxels idle).
// brick_kernel: 165 and 2.3 ms (114 M records with about 4 undecided yaws each; 2 M); 82 % of the
// slots, 25 of 32 lanes. The row-by-row per-node pass before: 947 and 12.6 ms.

// Interval mode: is the sample of voxel (x, y, z) on its owner ray (body-frame ray b, yaw cos ck, sin sk)
// observed by one of the ancestors `left`? The ray's crossings that enter and leave the voxel are the
// last entering and the first leaving event in the DDA's order (visit_index).
__device__ __forceinline__ bool iv_observed(const LevelParams &p, const NodeAnc *anc, uint64_t left, const int4 nd, const int4 b, int ck,
                                            int sk, int x, int y, int z) {
    int dx, dy, dz;
    ray_dir(b, ck, sk, dx, dy, dz);
    uint32_t n[3], ad[3], en = 0, eA = 1, xn = 0, xA = 1;
    int c[3], ea = -1;
    {
        const int P[3] = {nd.x, nd.y, nd.z}, d[3] = {dx, dy, dz}, v[3] = {x, y, z};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            int v0, s;
            ray_axis(P[a], d[a], v0, s, n[a], ad[a]);
            c[a] = s * (v[a] - v0);
            if (c[a] >= 1) {
                const uint32_t na = n[a] + ((uint32_t)(c[a] - 1) << 16);
                if (ea < 0 || ev_lt(en, eA, ea, na, ad[a], a)) {
                    ea = a;
                    en = na;
                    eA = ad[a];
                }
            }
        }
        const uint32_t l0 = n[0] + ((uint32_t)c[0] << 16), l1 = n[1] + ((uint32_t)c[1] << 16), l2 = n[2] + ((uint32_t)c[2] << 16);
        const int a = ev_argmin3(l0, ad[0], l1, ad[1], l2, ad[2]);
        xn = a == 0 ? l0 : (a == 1 ? l1 : l2);
        xA = a == 0 ? ad[0] : (a == 1 ? ad[1] : ad[2]);
    }
    const float zf = fmul(__ll2float_rn(p.Tq), 1.52587890625e-05f);     // range, voxel units
    const float T = fmul(__ll2float_rn(p.Tq), 9.313225746154785e-10f);  // range, crossing units
    const float lam = sample_lambda(en, eA, xn, xA, T);
    const int Ex = nd.x + (int)(((int64_t)p.Tq * dx) >> 30), Ey = nd.y + (int)(((int64_t)p.Tq * dy) >> 30),
              Ez = nd.z + (int)(((int64_t)p.Tq * dz) >> 30);
    bool obs = false;
    for (; left && !obs; left &= left - 1) {
        const NodeAnc &A = anc[__ffsll((long long)left) - 1];
        Seg g;
        float s;
        obs = seg_setup(p.yawtab + A.yaw * 12 + 2, A.U0, A.V0, A.Z0, make_int3(Ex - A.px, Ey - A.py, Ez - A.pz), zf, p.W, p.H, lam, g) &&
              seg_param(g, lam, s) && seg_lookup(g, p.W, p.H, A.D, s MIG_CHECKED(, &p));
    }
    return obs;
}

// One undecided brick (warp-uniform record r; lane = voxel of its lower and upper half): the
// ancestor tests left, then each yaw's counts into c_abs / c_mrg of lane (yaw - first) % 32, slot
// (yaw - first) / 32.
template <bool STATS, bool INTERVAL>
__device__ __forceinline__ void count_brick(const LevelParams &p, const VoxConst &vc, const YawRows *s_y, const NodeAnc *anc,
                                            const int4 nd, const uint16_t *steps, const BrickRec &r, int lane, int c_abs[2],
                                            int c_mrg[2], NodeCnt &st) {
    const int W = p.W, H = p.H, kb = (int)(r.node >> kRecNodeBits) * 64;
    const size_t WH = (size_t)W * H;
    const int x = 4 * (int)(r.brick & 1023) + (lane & 3), y = 4 * (int)((r.brick >> 10) & 1023) + ((lane >> 2) & 3),
              z0 = 4 * (int)(r.brick >> 20) + (lane >> 4);
    const uint64_t U = r.U;
    uint64_t O = r.O;
    const int rx = (x << 16) + 32768 - nd.x, ry = (y << 16) + 32768 - nd.y, rz0 = (z0 << 16) + 32768 - nd.z;
    const float rinf = fmaxf(fmaxf(fabsf(q16f(rx)), fabsf(q16f(ry))), fabsf(q16f(rz0))) + 8.0f;
    // error of a row product per unit of the row's norm, for every voxel of the brick
    const float verr = 5e-7f * (__uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(rinf))) + 1.0f);
    // ---- the ancestors that were not decided for the whole brick
    if (!INTERVAL) O = voxel_ancestors<STATS>(p, vc, s_y, anc, nd, r.anc, U, O, x, y, z0, verr, lane, st);
    // ---- yaws that count every unknown voxel (interval mode: their samples differ by yaw, see below)
    if (!INTERVAL) {
        const int cu = __popcll(U), cm = __popcll(U & ~O);
#pragma unroll
        for (int i = 0; i < 2; ++i)
            if ((uint32_t)(r.all >> (32 * i)) >> lane & 1) {
                c_abs[i] += cu;
                c_mrg[i] += cm;
                if constexpr (STATS) st.visit += cu;
            }
    }
    // ---- yaws that left the brick undecided
    const float ex = q16f(rx), ey = q16f(ry), ez[2] = {q16f(rz0), q16f(rz0 + 131072)};
    const float exy2 = fmaf(ex, ex, ey * ey);
    const int v0z = nd.z >> 16, mxy = abs(x - (nd.x >> 16)) + abs(y - (nd.y >> 16));
    bool has[2], near_inf[2], near_l2[2];
    int man[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float r2 = fmaf(ez[h], ez[h], exy2);
        has[h] = ((uint32_t)(U >> (32 * h)) >> lane & 1) && r2 < vc.out2;
        near_inf[h] = r2 < vc.inf2;
        near_l2[h] = r2 < vc.l22;
        man[h] = mxy + abs(z0 + 2 * h - v0z);
    }
    const uint64_t rv64 = r.rch | r.vis;
    for (uint64_t ks = INTERVAL ? r.part | r.all : r.part; ks; ks &= ks - 1) {
        const int j = __ffsll((long long)ks) - 1, k = kb + j;
        const float4 ru = s_y[k].u, rv = s_y[k].v, rz = s_y[k].z;
        const float Zxy = fmaf(rz.x, ex, rz.y * ey), Uxy = fmaf(ru.x, ex, ru.y * ey), Vxy = fmaf(rv.x, ex, rv.y * ey);
        const int32_t *row = p.yawtab + k * 12;
        bool c[2] = {false, false};
        int pix[2] = {0, 0};
        if (!INTERVAL && !((rv64 >> j) & 1)) {
            // every voxel is reached and visited: only the image test, without the pixel
            const float cz = verr * rz.w, cu = verr * ru.w, cv = verr * rv.w, cr = fmaf(vc.fW, cz, cu), cb = fmaf(vc.fH, cz, cv);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float Zf = fmaf(rz.z, ez[h], Zxy), Uf = fmaf(ru.z, ez[h], Uxy), Vf = fmaf(rv.z, ez[h], Vxy);
                const float Rf = fmaf(vc.fW, Zf, -Uf), Bf = fmaf(vc.fH, Zf, -Vf);
                const bool in = fminf(fminf(Uf - cu, Vf - cv), fminf(Rf - cr, Bf - cb)) > 0.0f;
                const bool out = fminf(fminf(Uf + cu, Vf + cv), fminf(Rf + cr, Bf + cb)) < 0.0f;
                c[h] = has[h] && in;
                if (has[h] && !in && !out) c[h] = pixel_exact(row, rx, ry, rz0 + (h << 17), W, H) >= 0;
            }
            if constexpr (STATS) st.visit += (int)c[0] + (int)c[1];
        } else {
            const PixelErr pe{2.0f * verr * fmaf(vc.fW, rz.w, ru.w), 2.0f * verr * fmaf(vc.fH, rz.w, rv.w), vc.bu, vc.bv};
            const bool nr = (r.rch >> j) & 1, nv = (r.vis >> j) & 1;
            const uint16_t *stp = steps + (size_t)k * WH;
            float Zf[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                Zf[h] = fmaf(rz.z, ez[h], Zxy);
                const int in = pixel_float(pe, Zf[h], fmaf(ru.z, ez[h], Uxy), fmaf(rv.z, ez[h], Vxy), vc.fW, vc.fH, pix[h]);
                c[h] = has[h] && in > 0;
                if (has[h] && in < 0) {
                    pix[h] = pixel_exact(row, rx, ry, rz0 + (h << 17), W, H);
                    c[h] = pix[h] >= 0;
                }
            }
            if (nr) {  // before the owner ray's hit
                int m[2] = {0, 0};
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (c[h] && steps_ok(p, stp + pix[h])) m[h] = ld_written(stp + pix[h]);
                c[0] = man[0] < m[0];
                c[1] = man[1] < m[1];
            }
            if constexpr (STATS) st.visit += (int)c[0] + (int)c[1];
            if (nv) {  // the owner ray visits the voxel
                const float4 rq = s_y[k].x;
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (c[h] && !(Zf[h] >= 0.5f && ((near_inf[h] && Zf[h] < rq.x) || (near_l2[h] && Zf[h] < p.vis_zl2)))) {
                        const int4 b = p.body[pix[h]];
                        const float q30 = 9.31322574615478515625e-10f;
                        const float bxf = (float)b.x * q30, byf = (float)b.y * q30;
                        const int d = visit_slab(ex, ey, ez[h], fmaf(rq.y, bxf, -(rq.z * byf)), fmaf(rq.z, bxf, rq.y * byf),
                                                 (float)b.z * q30, vc.Tv);
                        c[h] = d > 0;
                        if (d < 0) c[h] = visit_exact(nd.x, nd.y, nd.z, b.x, b.y, b.z, row[0], row[1], x, y, z0 + 2 * h, p.Tq);
                    }
            }
        }
        if (INTERVAL && r.anc) {  // the sample on this yaw's owner ray
            bool obs[2] = {false, false};
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                bool o = false;
                if (h ? c[1] : c[0]) o = iv_observed(p, anc, r.anc, nd, p.body[h ? pix[1] : pix[0]], row[0], row[1], x, y, z0 + 2 * h);
                obs[0] = h ? obs[0] : o;
                obs[1] = h ? o : obs[1];
            }
            O = (uint64_t)__ballot_sync(0xffffffffu, obs[0]) | ((uint64_t)__ballot_sync(0xffffffffu, obs[1]) << 32);
        }
        const unsigned m0 = __ballot_sync(0xffffffffu, c[0]), m1 = __ballot_sync(0xffffffffu, c[1]);
        if (lane == (j & 31)) {
            const int a = __popc(m0) + __popc(m1), m = __popc(m0 & ~(unsigned)O) + __popc(m1 & ~(unsigned)(O >> 32));
            c_abs[0] += j < 32 ? a : 0;
            c_mrg[0] += j < 32 ? m : 0;
            c_abs[1] += j < 32 ? 0 : a;
            c_mrg[1] += j < 32 ? 0 : m;
        }
    }
}

// Adds a warp's counts of node n's yaws [kb, kb + 64) to the level's counters and clears them: one
// 64-bit addition for the (abs, marginal) pair, whose halves stay below 2^31.
template <bool STATS>
__device__ __forceinline__ void flush_counts(const LevelParams &p, int n, int kb, int lane, int c_abs[2], int c_mrg[2], NodeCnt &st) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int k = kb + 32 * i + lane;
        if (k < p.K && (c_abs[i] | c_mrg[i]))
            atomicAdd(reinterpret_cast<unsigned long long *>(p.cnt) + (size_t)n * p.K + k,
                      (unsigned long long)(unsigned)c_abs[i] | ((unsigned long long)(unsigned)c_mrg[i] << 32));
        if constexpr (STATS) st.smp += c_abs[i];
        c_abs[i] = c_mrg[i] = 0;
    }
}

template <bool STATS>
__device__ __forceinline__ void add_stats(const LevelParams &p, const NodeCnt &st) {
    if constexpr (STATS) {
        const uint32_t v[6] = {st.cand, st.unk, st.visit, st.smp, st.anc, st.reads};
        for (int i = 0; i < 6; ++i) atomicAdd(p.stats + 11 + i, (unsigned long long)v[i]);
    }
}

constexpr int kNodeSplit = 8;  // parts of the yaws at most
template <bool STATS, bool INTERVAL>
__global__ void __launch_bounds__(kWarpsN * 32, 3) node_kernel(const LevelParams p, int num_sms) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int K = p.K;
    YawRows *s_y = reinterpret_cast<YawRows *>(s_dyn);
    NodeAnc *anc = reinterpret_cast<NodeAnc *>(s_y + K) + warp * p.max_anc;
    for (int k = threadIdx.x; k < K; k += blockDim.x)
        s_y[k] = yaw_rows(p.yawtab + k * 12, p.W, p.H, p.vis_hu, p.vis_hv, p.ifx, p.ify);
    wait_previous();
    if (blockIdx.x == 0 && threadIdx.x == 0) p.work[0] = 0;  // the next cast's tiles
    __syncthreads();
    const StepRange step = step_range(p);
    const int l0 = step.l0, nb0 = step.q0 / K, nn = step.q1 / K - nb0;
    if (nn <= 0) return;
    const int base = p.tree ? l0 + nb0 : 0;  // the chunk's first node in the step counts and bounds
    const int W = p.W, H = p.H;
    const size_t WH = (size_t)W * H;
    const Pyramid pyr = pyramid(W, H);
    const int top = cast_layout((long long)(p.tree ? p.tree : nn) * K, W, H, num_sms) == kCastSmall ? 4 : 5;  // the bounds the cast kept
    const BrickDims bd = brick_dims(p.grid.nx, p.grid.ny, p.grid.nz);
    const uint64_t *umask = grid_umask(p.grid);
    const VoxConst vc = vox_const(p);
    const float R2 = (vc.Tv + 1.0f) * (vc.Tv + 1.0f);
    const int Rv = (int)(p.Tq >> 16) + 2;
    const int mxy = mac_xy(p.Tq), mn = mxy * mxy * mac_z(p.Tq);
    // macro blocks per work item: enough items for every warp to get several, at most one per lane
    const int group = (int)max(1ll, min(32ll, (long long)nn * mn / ((long long)gridDim.x * kWarpsN * 8)));
    // too few blocks to fill the GPU: an item takes every split-th yaw of a block, so that every warp gets
    // one or two (node and brick pass of 9 levels of 11 nodes: 389 us with 8 parts below half that size
    // and a warp per block, 313 so, 329 with twice, 343 with half as many)
    const int split = (int)max(1ll, min((long long)min(K, kNodeSplit), 2ll * gridDim.x * kWarpsN / ((long long)nn * mn)));
    const int gpn = (mn + group - 1) / group * split;
    NodeCnt st;
    int cur = -1, cur_kb = 0, na = 0;
    int c_abs[2] = {0, 0}, c_mrg[2] = {0, 0};  // node cur, yaws cur_kb + lane and cur_kb + 32 + lane
    for (;;) {
        int it = 0;
        if (lane == 0) it = atomicAdd(p.vctr, 1);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= nn * gpn) break;
        const int ln = it / gpn, sub = (it - ln * gpn) % split, g0 = (it - ln * gpn) / split * group;
        const int n = p.level_nodes[l0 + nb0 + ln];
        const int4 nd = p.node[n];
        const int v0x = nd.x >> 16, v0y = nd.y >> 16, v0z = nd.z >> 16;
        // lane = macro block of the item: inside the grid, the ball and the elevation band?
        int mX = 0, mY = 0, mZ = 0;
        const bool live = lane < group && macro_block(p, nd, g0 + lane, mn, mxy, Rv, R2, mX, mY, mZ);
        unsigned todo = __ballot_sync(0xffffffffu, live);
        if (todo && n != cur) {
            if (cur >= 0) flush_counts<STATS>(p, cur, cur_kb, lane, c_abs, c_mrg, st);
            cur = n;
            na = node_ancestors(p, n, anc, WH, pyr.n, lane);
        }
        const uint32_t *hz = p.hz + (size_t)(base + ln) * K * pyr.n;
#pragma unroll 1
        for (; todo; todo &= todo - 1) {
            const int src = __ffs(todo) - 1;
            const int X = __shfl_sync(0xffffffffu, mX, src) * 4, Y = __shfl_sync(0xffffffffu, mY, src) * 4,
                      Z = __shfl_sync(0xffffffffu, mZ, src) * 2;  // the block's first brick
            // ---- lane = brick
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
            if (!__any_sync(0xffffffffu, U != 0)) continue;
            // Manhattan distances (step indices) of the brick's voxels from the start voxel
            int man0, man1;
            {
                const int ax = 4 * bx - v0x, ay = 4 * by - v0y, az = 4 * bz - v0z;
                man0 = max(max(ax, -ax - 3), 0) + max(max(ay, -ay - 3), 0) + max(max(az, -az - 3), 0);
                man1 = max(abs(ax), abs(ax + 3)) + max(abs(ay), abs(ay + 3)) + max(abs(az), abs(az + 3));
            }
            const float gx = q16f(((4 * X + 8) << 16) - nd.x), gy = q16f(((4 * Y + 8) << 16) - nd.y),
                        gz = q16f(((4 * Z + 4) << 16) - nd.z);  // the block's centre
            const int mac_man0 = __reduce_min_sync(0xffffffffu, U ? man0 : 0x7fffffff);
#pragma unroll 1
            for (int kb = 0; kb < K; kb += 64) {
                // ---- lane = yaw: which yaws may count a voxel of the block?
                uint64_t yaws = 0;
#pragma unroll 1
                for (int i = 0; i < 64 && kb + i < K; i += 32) {
                    bool may = false;
                    const int k = kb + i + lane;
                    if (k < K && k % split == sub) {
                        const BoxView b = box_view<false>(s_y[k], gx, gy, gz, 7.5f, 7.5f, 3.5f, W, H);
                        may = b.in >= 0;
                        if (may && box_lookup(b)) {
                            const uint32_t hm = hz_box(p, hz + (size_t)k * pyr.n, pyr, top, b);
                            may = mac_man0 < (int)((hm >> 16) ^ 0xFFFFu);  // else every ray stops before the block
                        }
                    }
                    yaws |= (uint64_t)__ballot_sync(0xffffffffu, may) << i;
                }
                // ---- lane = brick against each of them
                uint64_t all = 0, part = 0, rch = 0, vis = 0;  // bit k - kb
#pragma unroll 1
                for (uint64_t ks = yaws; ks; ks &= ks - 1) {
                    const int j = __ffsll((long long)ks) - 1;
                    if (U) {
                        const BoxView b = box_view<true>(s_y[kb + j], cx, cy, cz, 1.5f, 1.5f, 1.5f, W, H);
                        bool some = b.in >= 0, reach = false, sure = false;  // all reached; all visited for certain
                        if constexpr (STATS) {
                            st.cand += 64;
                            st.unk += __popcll(U);
                        }
                        if (some && b.zlo >= 0.5f) {
                            if (box_lookup(b)) {
                                const uint32_t hm = hz_box(p, hz + (size_t)(kb + j) * pyr.n, pyr, top, b);
                                some = man0 < (int)((hm >> 16) ^ 0xFFFFu);
                                reach = man1 < (int)(hm & 0xFFFFu);
                            }
                            sure = (b.zhi < s_y[kb + j].x.x && far + 0.86f < vc.Tv) || (b.zhi < p.vis_zl2 && far + 0.02f < vc.Tv);
                        }
                        if (some) {
                            const uint64_t bit = 1ull << j;
                            const bool whole = b.in > 0 && reach && sure;
                            all |= whole ? bit : 0ull;
                            part |= whole ? 0ull : bit;
                            rch |= reach ? 0ull : bit;
                            vis |= sure ? 0ull : bit;
                        }
                    }
                }
                const bool want = (all | part) != 0;
                if (!__any_sync(0xffffffffu, want)) continue;
                // ---- the ancestors' test (Sec. IV-B) of the bricks some yaw may count
                uint64_t O = 0, left = 0;  // observed voxels; ancestors undecided for the brick
                block_ancestors<INTERVAL>(p, s_y, anc, na, nd, pyr, vc, X, Y, Z, bx, by, bz, U, want, lane, O, left);
                if (O == U) left = 0;
                if (kb != cur_kb) {
                    flush_counts<STATS>(p, cur, cur_kb, lane, c_abs, c_mrg, st);
                    cur_kb = kb;
                }
                // ---- decided bricks: population counts; lane j % 32 keeps the counts of yaw kb + j
                const bool rec = part != 0 || (all != 0 && left != 0);
                const unsigned pc = (unsigned)__popcll(U) | ((unsigned)__popcll(U & ~O) << 16);
#pragma unroll 1
                for (uint64_t ks = or64(rec ? 0ull : all); ks; ks &= ks - 1) {
                    const int j = __ffsll((long long)ks) - 1;
                    const unsigned v = __reduce_add_sync(0xffffffffu, !rec && ((all >> j) & 1) ? pc : 0u);
                    if (lane == (j & 31)) {
                        const int i = j >> 5;
                        c_abs[0] += i ? 0 : (int)(v & 0xFFFF);
                        c_mrg[0] += i ? 0 : (int)(v >> 16);
                        c_abs[1] += i ? (int)(v & 0xFFFF) : 0;
                        c_mrg[1] += i ? (int)(v >> 16) : 0;
                        if constexpr (STATS) st.visit += v & 0xFFFF;
                    }
                }
                // ---- undecided bricks: to the queue (counted here if it is full)
                const unsigned recs = __ballot_sync(0xffffffffu, rec);
                if (recs) {
                    int at = 0;
                    if (lane == 0) at = atomicAdd(p.vctr + 1, __popc(recs));
                    at = __shfl_sync(0xffffffffu, at, 0) + __popc(recs & ((1u << lane) - 1u));
                    BrickRec r{U, O, left, all, part, rch, vis, (uint32_t)bx | ((uint32_t)by << 10) | ((uint32_t)bz << 20),
                               (uint32_t)ln | ((uint32_t)(kb >> 6) << kRecNodeBits)};
                    if (rec && at < p.queue_cap && queue_ok(p, at)) p.queue[at] = r;
#pragma unroll 1
                    for (unsigned full = __ballot_sync(0xffffffffu, rec && at >= p.queue_cap); full; full &= full - 1) {
                        const int s = __ffs(full) - 1;
                        BrickRec q{shfl64(r.U, s), shfl64(r.O, s), shfl64(r.anc, s), shfl64(r.all, s), shfl64(r.part, s),
                                   shfl64(r.rch, s), shfl64(r.vis, s), __shfl_sync(0xffffffffu, r.brick, s), r.node};
                        count_brick<STATS, INTERVAL>(p, vc, s_y, anc, nd, p.steps + (size_t)(base + ln) * K * WH, q, lane, c_abs, c_mrg, st);
                    }
                }
            }
        }
    }
    if (cur >= 0) flush_counts<STATS>(p, cur, cur_kb, lane, c_abs, c_mrg, st);
    add_stats<STATS>(p, st);
}

// The queue's records, one warp each, in slices of consecutive records (mostly of one node).
template <bool STATS, bool INTERVAL>
__global__ void __launch_bounds__(kWarpsN * 32, 4) brick_kernel(const LevelParams p) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int K = p.K;
    YawRows *s_y = reinterpret_cast<YawRows *>(s_dyn);
    NodeAnc *anc = reinterpret_cast<NodeAnc *>(s_y + K) + warp * p.max_anc;
    for (int k = threadIdx.x; k < K; k += blockDim.x)
        s_y[k] = yaw_rows(p.yawtab + k * 12, p.W, p.H, p.vis_hu, p.vis_hv, p.ifx, p.ify);
    wait_previous();
    __syncthreads();
    const StepRange step = step_range(p);
    const int l0 = step.l0, nb0 = step.q0 / K;
    if (step.q1 <= step.q0) return;
    const int base = p.tree ? l0 + nb0 : 0;
    const int total = min(p.vctr[1], p.queue_cap);
    const int slice = max(1, min(64, total / (int)(gridDim.x * kWarpsN * 8)));
    if (blockIdx.x * kWarpsN * slice >= total) return;
    const size_t WH = (size_t)p.W * p.H;
    const int pyr_n = pyramid(p.W, p.H).n;
    const VoxConst vc = vox_const(p);
    NodeCnt st;
    uint32_t cur = 0xFFFFFFFFu;
    int n = 0, c_abs[2] = {0, 0}, c_mrg[2] = {0, 0};
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
                if (cur != 0xFFFFFFFFu) flush_counts<STATS>(p, n, (int)(cur >> kRecNodeBits) * 64, lane, c_abs, c_mrg, st);
                cur = r.node;
                n = p.level_nodes[l0 + nb0 + (int)(cur & ((1u << kRecNodeBits) - 1))];
                nd = p.node[n];
                node_ancestors(p, n, anc, WH, pyr_n, lane);
            }
            count_brick<STATS, INTERVAL>(p, vc, s_y, anc, nd, p.steps + (size_t)(base + (int)(cur & ((1u << kRecNodeBits) - 1))) * K * WH, r, lane, c_abs,
                               c_mrg, st);
        }
    }
    if (cur != 0xFFFFFFFFu) flush_counts<STATS>(p, n, (int)(cur >> kRecNodeBits) * 64, lane, c_abs, c_mrg, st);
    add_stats<STATS>(p, st);
}

}  // namespace

size_t hz_entries(int W, int H) { return (size_t)pyramid(W, H).n; }

void set_visit_params(LevelParams &p, float hfov_deg, float vfov_deg) {
    const VisitLimits l = visit_limits(hfov_deg, vfov_deg, p.W, p.H);
    p.vis_hu = l.hu;
    p.vis_hv = l.hv;
    p.vis_zl2 = l.zl2;
    p.ifx = (float)(std::tan(hfov_deg * 0.5 * (3.14159265358979323846 / 180.0)) / (p.W * 0.5));
    p.ify = (float)(std::tan(vfov_deg * 0.5 * (3.14159265358979323846 / 180.0)) / (p.H * 0.5));
}

void launch_cast_chunk(const LevelParams &c, int num_sms, cudaStream_t s) {
    const int g = cast_grid(c.q1 - c.q0, c.W, c.H, num_sms, 64);
    if (c.stats) launch_behind(c.depths ? cast_kernel<true, true> : cast_kernel<true, false>, g, kWarpsN * 32, 0, s, c, num_sms);
    else launch_behind(c.depths ? cast_kernel<false, true> : cast_kernel<false, false>, g, kWarpsN * 32, 0, s, c, num_sms);
}

void launch_tree_cast(const LevelParams &p, int levels, int num_sms, cudaStream_t s) {
    LevelParams c = p;
    c.lvl = levels;
    c.q0 = 0;
    c.q1 = p.tree * p.K;
    launch_cast_chunk(c, num_sms, s);
}

void launch_select_render(const LevelParams &p, int nodes, int num_sms, cudaStream_t s) {
    const int g = cast_grid(nodes, p.W, p.H, num_sms, 16);
    if (p.stats) launch_behind(render_kernel<true>, g, kWarpsN * 32, 0, s, p, num_sms);
    else launch_behind(render_kernel<false>, g, kWarpsN * 32, 0, s, p, num_sms);
}

int node_ctas_per_sm() {
    // the most yaws and the deepest tree: 120 KiB
    const int smem = (int)node_dyn_smem(MIG_MAX_YAW_BINS, MIG_MAX_DEPTH);
    cudaFuncSetAttribute(node_kernel<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    cudaFuncSetAttribute(node_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    cudaFuncSetAttribute(node_kernel<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    cudaFuncSetAttribute(brick_kernel<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    cudaFuncSetAttribute(brick_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    cudaFuncSetAttribute(brick_kernel<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    int a = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, node_kernel<false, false>, kWarpsN * 32, node_dyn_smem(36, 16));
    cudaGetLastError();
    return std::max(1, a);
}

// Macro blocks of a node's range ball (its bounding box): the node pass's items per node.
long long node_items(int64_t Tq) { return (long long)mac_xy(Tq) * mac_xy(Tq) * mac_z(Tq); }

// Bricks that a node's range ball can touch.
static long long node_bricks(int64_t Tq) {
    const double r = ((double)Tq / 65536.0 + 1.0) / 4.0 + 1.74;
    return (long long)(4.19 * r * r * r) + 1;
}

// The CTAs of a node pass of `items` work items, and of the brick pass that follows it for `nodes` nodes (and
// groups of 64 yaws). A tree alone takes every SM it can use, down to one item per warp. Among others a
// small level takes several items per warp instead, since its CTAs that find little to do, and the next
// launch's that wait for it, keep the others' from the SMs: 9 trees of 10 to 78 nodes of 43x24x8 in one batch
// 995 -> 750 us (935 row by row), while one of them alone takes 325 us with one item per warp, 329 with 8.
int node_grid(long long items, int most, int crowd) {
    const long long per_cta = kWarpsN * std::max(1, std::min(crowd, 8));
    return (int)std::max<long long>(1, std::min<long long>((items + per_cta - 1) / per_cta, most));
}
int brick_grid(long long nodes, int64_t Tq, int num_sms, int crowd) {
    const long long most = num_sms * 4;
    return (int)(crowd > 1 ? std::max<long long>(1, std::min<long long>(most, nodes * node_bricks(Tq) / (4 * kWarpsN))) : most);
}

void launch_node_chunk(const LevelParams &c, int num_sms, int node_ctas, cudaStream_t s) {
    // a warp per macro block, or per block and eighth of the yaws where the blocks alone leave SMs idle (split)
    const int nodes = (c.q1 - c.q0) / c.K;
    const int g = node_grid((long long)nodes * node_items(c.Tq) * std::min(c.K, kNodeSplit), num_sms * node_ctas, c.crowd);
    const size_t smem = node_dyn_smem(c.K, c.max_anc);
    const int gb = brick_grid((long long)nodes * ((c.K + 63) / 64), c.Tq, num_sms, c.crowd);
    if (c.mode == MIG_MODE_INTERVAL) {
        launch_behind(node_kernel<false, true>, g, kWarpsN * 32, smem, s, c, num_sms);
        launch_behind(brick_kernel<false, true>, gb, kWarpsN * 32, smem, s, c);
    } else if (c.stats) {
        launch_behind(node_kernel<true, false>, g, kWarpsN * 32, smem, s, c, num_sms);
        launch_behind(brick_kernel<true, false>, gb, kWarpsN * 32, smem, s, c);
    } else {
        launch_behind(node_kernel<false, false>, g, kWarpsN * 32, smem, s, c, num_sms);
        launch_behind(brick_kernel<false, false>, gb, kWarpsN * 32, smem, s, c);
    }
}

// The share of them that a chunk's queue has room for (measured with up to 64 yaws: up to 0.27 of a node's bricks
// are left undecided as a whole; every further 64 yaws queue a brick again). A fuller queue only sends its last
// bricks through the slower path inside node_kernel.
constexpr double kQueueShare = 0.3;
constexpr double kQueueShareInterval = 0.7;  // there every counted brick that an ancestor looks at
constexpr double kQueueSharePano = 0.5;      // every brick that a ray can reach
constexpr long long kQueueMax = 8ll << 20;  // records (512 MB)

static double queue_share(int mode) {
    return mode == MIG_MODE_INTERVAL ? kQueueShareInterval : (mode == MIG_MODE_PANORAMIC ? kQueueSharePano : kQueueShare);
}

// The offsets of a region of L.cap pairs and L.queue_cap records.
static void place(StepsLayout &L, const SensorDims &d) {
    auto align = [](size_t b) { return (b + 255) & ~(size_t)255; };
    L.o_ctr = align((size_t)L.cap * d.W * d.H * sizeof(uint16_t));
    L.o_hz = L.o_ctr + 256;
    L.o_queue = align(L.o_hz + (size_t)L.cap * hz_entries(d.W, d.H) * sizeof(uint32_t));
    L.o_depths = align(L.o_queue + (size_t)L.queue_cap * sizeof(BrickRec));
    L.bytes = L.o_depths + (L.depths ? (size_t)L.cap * d.W * d.H * sizeof(uint32_t) : 0);
}

StepsLayout steps_layout(const SensorDims &d, int n, int max_nodes, size_t budget_bytes, size_t tree_bytes, bool node_pass, int mode) {
    StepsLayout L{};
    const long long pairs = (long long)std::max(1, max_nodes) * d.K;
    L.cap = (int)std::min<size_t>(steps_pairs(pairs, d.W, d.H, budget_bytes), (size_t)1 << 30);
    const long long per_node = (long long)(queue_share(mode) * (double)node_bricks(d.Tq)) + 1;
    if (node_pass && L.cap >= d.K) {  // whole nodes, as many as the queue has room for
        const long long nodes = std::max<long long>(1, std::min<long long>(L.cap / d.K, kQueueMax / per_node));
        L.cap = (int)nodes * d.K;
        L.queue_cap = (int)std::min(kQueueMax, std::max<long long>(nodes * per_node, 1ll << 16));
        // all of a small tree's nodes, if one level's work items stay below 2^30
        const double images = (double)n * d.K, bytes = images * d.W * d.H * sizeof(uint16_t);
        if (bytes <= (double)std::min(budget_bytes, tree_bytes) && images * (double)hz_entries(d.W, d.H) <= (double)tree_bytes &&
            nodes >= max_nodes && (double)n * (double)node_items(d.Tq) * d.K < (double)(1ll << 30)) {
            L.tree = n;
            L.cap = n * d.K;
            L.depths = mode != MIG_MODE_PANORAMIC && 2.0 * bytes <= (double)kTreeDepths;
        }
    }
    place(L, d);
    return L;
}

StepsLayout steps_layout_in(const SensorDims &d, int n, int max_nodes, size_t bytes, bool with_depths) {
    // per node: its step counts, their bounds and 0.7 of the usual queue (a full queue only slows the
    // bricks beyond it), so that a fixed region holds more nodes at a time
    const size_t recs = (size_t)(0.7 * kQueueShare * (double)node_bricks(d.Tq)) + 1;
    const size_t node = (size_t)d.K * ((size_t)d.W * d.H * sizeof(uint16_t) + hz_entries(d.W, d.H) * sizeof(uint32_t)) +
                        recs * sizeof(BrickRec);
    const size_t fixed = 4 * 256;  // the counters and the alignment of the parts
    StepsLayout L{};
    if (bytes < fixed + node) return L;
    const long long nodes = std::min<long long>(std::min<long long>(max_nodes, (1 << kRecNodeBits) - 1), (long long)((bytes - fixed) / node));
    L.cap = (int)std::min<long long>(nodes, INT_MAX / d.K) * d.K;
    L.queue_cap = (int)std::min<long long>(kQueueMax, (long long)(L.cap / d.K) * recs);
    // room for the whole tree: one cast
    if (nodes == n && (double)nodes * (double)node_items(d.Tq) * d.K < (double)(1ll << 30)) L.tree = n;
    place(L, d);
    const size_t depths = (size_t)L.cap * d.W * d.H * sizeof(uint32_t);
    if (L.tree && with_depths && depths <= kTreeDepths && L.bytes + depths <= bytes) {
        L.depths = true;
        place(L, d);
    }
    return L;
}

StepsLayout steps_pairs_in(const SensorDims &d, size_t max_pairs, size_t bytes) {
    const size_t pair = (size_t)d.W * d.H * sizeof(uint16_t) + hz_entries(d.W, d.H) * sizeof(uint32_t), fixed = 4 * 256;
    StepsLayout L{};
    if (bytes < fixed + pair) return L;
    L.cap = (int)std::min({(bytes - fixed) / pair, max_pairs, (size_t)1 << 30});
    place(L, d);
    return L;
}

void set_steps(LevelParams &p, void *base, const StepsLayout &L) {
    char *b = static_cast<char *>(base);
    p.steps = reinterpret_cast<uint16_t *>(b);
    p.vctr = reinterpret_cast<int32_t *>(b + L.o_ctr);
    p.hz = reinterpret_cast<uint32_t *>(b + L.o_hz);
    p.queue = reinterpret_cast<BrickRec *>(b + L.o_queue);
    p.queue_cap = L.queue_cap;
    p.steps_cap = L.cap;
    p.tree = L.tree;
    p.depths = L.depths ? reinterpret_cast<uint32_t *>(b + L.o_depths) : nullptr;
}

}  // namespace mig
