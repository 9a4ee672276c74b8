// Interval-mode count pass, ray by ray (where the per-node pass of nodecount.cu does not apply or is the
// slower one): the paper's screen-space overlap test (Sec. IV-B, Eq. 5-7).
//
// For every candidate ray the 3D DDA (Sec. IV-B) visits voxels exactly as in the sample mode;
// each owned unknown voxel (its centre projects into the ray's pixel) counts as absolute gain and
// becomes a sample at the midpoint of the ray's traversal of it. A sample is excluded from the
// marginal gain when it lies in the union of the ancestors' overlap intervals of the ray. For
// each ancestor the ray is
//   1. taken to the ancestor's camera as projective image coordinates (U, V, Z), exact integers
//      from the Q16 projection rows, then IEEE single precision in voxel units;
//   2. clipped to the valid depth range [Z_NEAR, range];
//   3. projected (Eq. 5) and clipped to the buffer [0, W] x [0, H] (Liang-Barsky);
//   4. walked pixel by pixel (2D DDA); each visited pixel holds one portion of the segment, whose
//      depth sample at the portion's midpoint (inverse depth linear in the screen parameter,
//      Eq. 6) is compared with the stored depth, "smaller or equal" => observed, in inverse depth
//      (w D >= 1); boundary crossings use one reciprocal of the segment's screen extent.
// A sample belongs to the first portion, in walk order, that contains its perspective-correct
// screen parameter. Every floating-point step is one correctly rounded single-precision
// operation (__fadd_rn and friends: no contraction), in a fixed order, so the counts are
// reproducible bit for bit.
//
// The walk is not stepped pixel by pixel here: its portion boundaries are a fixed function of the
// boundary index (the same rounded operations as the walk), non-decreasing along it, so the
// portion that contains a sample is found directly by counting the column and row crossings at or
// before the sample's screen parameter (seg_lookup). The result is the walk's, bit for bit.
//
// Layout: one warp per work item (node, yaw, tile of rays), taken from the level's atomic work
// counter; a lane takes the tile's next ray as soon as its ray ends. Owned samples go to a
// per-warp queue as the crossings that bound their voxel and their pixel; each full batch of 32 is
// tested against the ancestors with one sample per lane, which is also where each sample's ray
// fraction is computed.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "dev_path.cuh"
#include "interval.cuh"
#include "interval.h"
#include "kernels.h"
#include "mig.h"

namespace mig {

namespace {

using namespace dev;

// minimum resident interval-kernel CTAs per SM requested from the register allocator
#ifndef MIG_IV_MINB
#define MIG_IV_MINB 4
#endif

constexpr int kIvWarps = 8;
constexpr int kIvThreads = kIvWarps * 32;
// an ancestor as the interval walk needs it: position (Q16), selected yaw, the node in its camera's
// coordinates (every ray's origin), depth buffer
struct IvAnc {
    int px, py, pz, yaw;
    float U0, V0, Z0;
    const uint32_t *D;
};

// A queued sample: the face distances of the crossings that enter and leave its voxel (Q16), and
// which of the ray's direction components |d_x|, |d_y|, |d_z| each is divided by (code 3: the
// ray's start, entry at t = 0 written as 0 / 1), with the pixel. The ray fraction is computed from
// it when the sample is tested, one sample per lane, not in the divergent DDA loop.
__device__ __forceinline__ uint32_t speed_code(uint32_t ad, const RayIn &r) {
    return ad == r.adx ? 0u : (ad == r.ady ? 1u : (ad == r.adz ? 2u : 3u));
}
__device__ __forceinline__ uint32_t speed_of(uint32_t code, uint32_t adx, uint32_t ady, uint32_t adz) {
    return code == 0u ? adx : (code == 1u ? ady : (code == 2u ? adz : 1u));
}

// Is the queued sample e (ray through pixel e.z >> 4, yaw ck / sk, origin P) inside an ancestor's
// observed portions? Ancestors parent first; the ray's set-up is rebuilt per sample.
template <bool STATS>
__device__ bool iv_observed(const LevelParams &p, const IvAnc *anc, int na, const int P[3], int ck, int sk,
                            float zf, float T, const uint4 e, uint32_t &st_seg) {
    const int pix = (int)(e.z >> 4);
    const int4 b = p.body[pix];
    int dx, dy, dz;
    ray_dir(b, ck, sk, dx, dy, dz);
    const uint32_t adx = (uint32_t)(dx < 0 ? -dx : dx), ady = (uint32_t)(dy < 0 ? -dy : dy),
                   adz = (uint32_t)(dz < 0 ? -dz : dz);
    const float lam = sample_lambda(e.x, speed_of(e.z & 3u, adx, ady, adz), e.y, speed_of((e.z >> 2) & 3u, adx, ady, adz), T);
    const int E[3] = {P[0] + (int)(((int64_t)p.Tq * dx) >> 30), P[1] + (int)(((int64_t)p.Tq * dy) >> 30),
                      P[2] + (int)(((int64_t)p.Tq * dz) >> 30)};
    for (int a = 0; a < na; ++a) {
        const IvAnc &A = anc[a];
        Seg g;
        if constexpr (STATS) ++st_seg;
        const int32_t *m = p.yawtab + A.yaw * 12 + 2;
        if (!seg_setup(m, A.U0, A.V0, A.Z0, make_int3(E[0] - A.px, E[1] - A.py, E[2] - A.pz), zf, p.W, p.H, lam, g)) continue;
        float s;
        if (seg_param(g, lam, s) && seg_lookup(g, p.W, p.H, A.D, s MIG_CHECKED(, &p))) return true;
    }
    return false;
}

template <bool STATS>
__global__ void __launch_bounds__(kIvThreads, MIG_IV_MINB) interval_count_kernel(const LevelParams p) {
    extern __shared__ IvAnc s_iv_anc[];
    __shared__ uint4 s_q[kIvWarps][64];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    IvAnc *anc = s_iv_anc + warp * p.max_anc;
    uint4 *q = s_q[warp];
    const int l0 = p.level_off[p.lvl];
    const int L = p.level_off[p.lvl + 1] - l0;
    const int items = L * p.K * p.tiles;
    const float zf = fmul(__ll2float_rn(p.Tq), 1.52587890625e-05f);   // range, voxel units
    const float T = fmul(__ll2float_rn(p.Tq), 9.313225746154785e-10f);  // range, crossing units
    uint32_t st_rays = 0, st_steps = 0, st_unk = 0, st_seg = 0;
    for (;;) {
        int c = 0;
        if (lane == 0) c = atomicAdd(p.work + p.lvl, 1);
        c = __shfl_sync(0xffffffffu, c, 0);
        if (c >= items) break;
        int li, k, tile;
        decode_item(p, c, li, k, tile);
        const int n = p.level_nodes[l0 + li];
        const int4 nd = p.node[n];
        const int2 ar = p.anc_range[n];
        const int na = min(ar.y, p.max_anc);
        __syncwarp();
        for (int t = lane; t < na; t += 32) {
            const int a = p.anc[ar.x + t];
            const int4 an = p.node[a];
            IvAnc rec;
            rec.px = an.x;
            rec.py = an.y;
            rec.pz = an.z;
            rec.yaw = p.sel_yaw[a];
            const int32_t *m = p.yawtab + rec.yaw * 12 + 2;
            const int rx = nd.x - an.x, ry = nd.y - an.y, rz = nd.z - an.z;
            rec.U0 = seg_coord(m, rx, ry, rz);
            rec.V0 = seg_coord(m + 3, rx, ry, rz);
            rec.Z0 = seg_coord(m + 6, rx, ry, rz);
            rec.D = p.arena + (size_t)an.w * p.W * p.H;
            anc[t] = rec;
        }
        __syncwarp();
        const int32_t *yk = p.yawtab + k * 12;
        const int ck = yk[0], sk = yk[1];
        const int P[3] = {nd.x, nd.y, nd.z};
        const int tx0 = (tile % p.tiles_x) * p.tile_w, ty0 = (tile / p.tiles_x) * p.tile_h;
        const int tile_rays = p.tile_w * p.tile_h;
        int next = 0, ti = 0, tj = 0, qn = 0, c_abs = 0, c_mrg = 0;
        bool have = false;
        RayIn r;
        uint32_t ne = 0, ade = 1;
        for (;;) {
            // lanes without a ray take the tile's next rays in order
            const unsigned need = __ballot_sync(0xffffffffu, !have);
            if (need && next < tile_rays) {
                const int idx = next + __popc(need & lt_mask);
                next += __popc(need);
                if (!have && idx < tile_rays) {
                    ti = tx0 + idx % p.tile_w;
                    tj = ty0 + idx / p.tile_w;
                    if (ti < p.W && tj < p.H) {
                        const int4 b = p.body[tj * p.W + ti];
                        int dx, dy, dz;
                        ray_dir(b, ck, sk, dx, dy, dz);
                        ray_init(r, p.grid, nd.x, nd.y, nd.z, dx, dy, dz, p.Tq);
                        ne = 0;
                        ade = 1;
                        have = true;
                        if constexpr (STATS) ++st_rays;
                    }
                }
            }
            if (!__any_sync(0xffffffffu, have)) {
                if (next >= tile_rays) break;
                continue;
            }
            bool owned = false;
            uint4 key = make_uint4(0u, 0u, 0u, 0u);
            if (have) {
                const uint8_t code = load_code(p.grid.g, r.addr, p.grid, p.bounds_err);
                if constexpr (STATS) ++st_steps;
                if (code == kOcc) {
                    have = false;
                } else {
                    if (code == kUnknown) {
                        if constexpr (STATS) ++st_unk;
                        // owner test: the voxel centre projects into pixel (ti, tj)
                        const int rx = voxel_offset(r.nx, r.sx), ry = voxel_offset(r.ny, r.sy),
                                  rz = voxel_offset(r.nz, r.sz);
                        const int64_t Z = (int64_t)yk[8] * rx + (int64_t)yk[9] * ry + (int64_t)yk[10] * rz;
                        const int64_t U = (int64_t)yk[2] * rx + (int64_t)yk[3] * ry + (int64_t)yk[4] * rz;
                        const int64_t iZ = (int64_t)ti * Z;
                        if (Z > 0 && U >= iZ && U < iZ + Z) {
                            const int64_t V = (int64_t)yk[5] * rx + (int64_t)yk[6] * ry + (int64_t)yk[7] * rz;
                            const int64_t jZ = (int64_t)tj * Z;
                            owned = V >= jZ && V < jZ + Z;
                        }
                    }
                    uint32_t nx = 0, adx = 1;
                    const bool more = ray_step<true>(r, nx, adx);  // nx / adx: this voxel's exit crossing
                    if (owned)
                        key = make_uint4(ne, nx, speed_code(ade, r) | (speed_code(adx, r) << 2) |
                                                     ((uint32_t)(tj * p.W + ti) << 4), 0u);
                    ne = nx;
                    ade = adx;
                    have = more;
                }
            }
            c_abs += owned;
            const unsigned bal = __ballot_sync(0xffffffffu, owned);
            if (bal) {
                if (owned) q[qn + __popc(bal & lt_mask)] = key;
                qn += __popc(bal);
                if (qn >= 32) {  // a full batch: every lane tests one sample against the ancestors
                    __syncwarp();
                    c_mrg += !iv_observed<STATS>(p, anc, na, P, ck, sk, zf, T, q[lane], st_seg);
                    __syncwarp();
                    if (lane < qn - 32) q[lane] = q[lane + 32];
                    __syncwarp();
                    qn -= 32;
                }
            }
        }
        __syncwarp();
        if (lane < qn) {
            c_mrg += !iv_observed<STATS>(p, anc, na, P, ck, sk, zf, T, q[lane], st_seg);
        }
        c_abs = __reduce_add_sync(0xffffffffu, c_abs);
        c_mrg = __reduce_add_sync(0xffffffffu, c_mrg);
        if (lane == 0 && (c_abs | c_mrg)) {
            atomicAdd(p.cnt + ((size_t)n * p.K + k) * 2, c_abs);
            atomicAdd(p.cnt + ((size_t)n * p.K + k) * 2 + 1, c_mrg);
        }
        if constexpr (STATS) {
            if (lane == 0) atomicAdd(p.stats + 3, (unsigned long long)(uint32_t)c_abs);
        }
        __syncwarp();
    }
    if constexpr (STATS) {
        st_rays = __reduce_add_sync(0xffffffffu, st_rays);
        st_steps = __reduce_add_sync(0xffffffffu, st_steps);
        st_unk = __reduce_add_sync(0xffffffffu, st_unk);
        st_seg = __reduce_add_sync(0xffffffffu, st_seg);
        if (lane == 0) {
            atomicAdd(p.stats + 0, (unsigned long long)st_rays);
            atomicAdd(p.stats + 1, (unsigned long long)st_steps);
            atomicAdd(p.stats + 2, (unsigned long long)st_unk);
            atomicAdd(p.stats + 4, (unsigned long long)st_seg);
        }
    }
}

}  // namespace

// dynamic shared memory: the warps' ancestor records, up to MIG_MAX_DEPTH each
constexpr size_t kIvMaxDyn = (size_t)kIvWarps * MIG_MAX_DEPTH * sizeof(IvAnc);

void launch_count_interval(const LevelParams &p, int grid, cudaStream_t s) {
    const size_t smem = (size_t)kIvWarps * (size_t)std::max(1, p.max_anc) * sizeof(IvAnc);
    if (p.stats) interval_count_kernel<true><<<grid, kIvThreads, smem, s>>>(p);
    else interval_count_kernel<false><<<grid, kIvThreads, smem, s>>>(p);
}

// Resident CTAs per SM (for the grid cap); also lifts the kernels' dynamic shared-memory limit to
// the deepest tree's ancestor records. Called once per context, before any launch.
int count_interval_ctas_per_sm() {
    cudaFuncSetAttribute(interval_count_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kIvMaxDyn);
    cudaFuncSetAttribute(interval_count_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kIvMaxDyn);
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, interval_count_kernel<false>, kIvThreads,
                                                  (size_t)kIvWarps * 16 * sizeof(IvAnc));
    return std::max(1, n);
}

}  // namespace mig
