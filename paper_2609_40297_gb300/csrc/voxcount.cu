// Owned-voxel count of one tree level (Sec. IV-B, the counts of Eq. 1 and Eq. 2 by depth
// buffers), per chunk of (node, yaw) pairs: the cast and the per-node count are in nodecount.cu;
//   voxel_kernel - the count of single (node, yaw) pairs, for chunks that do not hold whole nodes
//                  (or when asked for): for every pair, the voxels within range of the node are enumerated slice by
//                  slice (z), rows clipped to the camera frustum; each unknown voxel goes to the
//                  pixel that owns it (its centre's projection) and counts as absolute gain iff
//                  that pixel's DDA reaches it before the range and before its first occupied
//                  voxel; counted voxels are tested against the ancestors' depth buffers
//                  (marginal gain). Each test stage runs on full warps: the voxels that pass one
//                  stage wait in a per-warp queue until 32 of them are ready for the next.
// Results are identical to the ray-by-ray count kernel (and the CPU oracle) bit for bit.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "kernels.h"
#include "mig.h"
#include "voxcount.h"
#include "voxitems.cuh"

namespace mig {

namespace {

using namespace dev;

constexpr int kVoxWarps = 8;

__device__ __forceinline__ int level_pairs(const LevelParams &p) {
    return (p.level_off[p.lvl + 1] - p.level_off[p.lvl]) * p.K;
}

// ----------------------------------------------------------------------------- voxel kernel
// Per-warp queues between the test stages: unknown voxels of the slice (x | y << 12), voxels whose
// owner pixel's ray may reach them (x | y << 12 | pixel << 24), counted samples (x | y << 16 |
// z << 32). Each holds fewer than 64 entries: a stage runs whenever 32 are waiting.
struct VoxQueues {
    unsigned long long unk[64], own[64], smp[64];
};


// Warp work item = (pair q of the chunk, slice z of the node's range ball). Lanes take 32 rows
// (y) of the slice at a time, clip each row to the frustum and the ball, and then load the rows'
// voxels 32 at a time (flattened over the rows with a warp prefix sum).
template <bool STATS>
__global__ void __launch_bounds__(kVoxWarps * 32, 3) voxel_kernel(const LevelParams p) {
    extern __shared__ AncRec s_anc_dyn[];
    __shared__ VoxQueues s_vq[kVoxWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    AncRec *anc = s_anc_dyn + warp * p.max_anc;
    VoxQueues &Q = s_vq[warp];
    if (blockIdx.x == 0 && threadIdx.x == 0) p.work[0] = 0;  // the next cast's tiles
    const int l0 = p.level_off[p.lvl];
    const int q1 = min(p.q1, level_pairs(p));
    if (p.q0 >= q1) return;
    const int Rv = (int)(p.Tq >> 16) + 2;    // voxels: every visited voxel's centre is nearer than T + 1
    const int slices = 2 * Rv + 1;
    const int npairs = q1 - p.q0;
    const int items = npairs * slices;
    const float R = (float)p.Tq * (1.0f / 65536.0f) + 1.0f, R2 = R * R;
    const int gnx = p.grid.nx, gny = p.grid.ny, gnz = p.grid.nz;
    const size_t WH = (size_t)p.W * p.H;
    uint32_t st_cand = 0, st_unk = 0, st_visit = 0, st_anc = 0, st_reads = 0;
    int cur_node = -1, na = 0;
    // items are handed out one at a time from the launch's counter, in groups of pairs whose step
    // counts stay in L2 together; within a group every pair's slice at the node's own height first,
    // then outwards alternately above and below
    const int grp = (int)max((size_t)1, min((size_t)npairs, kStepsGroupBytes / (WH * sizeof(uint16_t))));
    for (;;) {
        int it = 0;
        if (lane == 0) it = atomicAdd(p.vctr, 1);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= items) break;
        const int g = it / (grp * slices), r = it - g * grp * slices;
        const int gsz = min(grp, npairs - g * grp);
        const int rank = r / gsz, ql = g * grp + r % gsz;
        const int zi = Rv + ((rank & 1) ? (rank + 1) >> 1 : -(rank >> 1));
        const int qq = p.q0 + ql;
        const int n = p.level_nodes[l0 + qq / p.K], k = qq % p.K;
        const int4 nd = p.node[n];
        const int z = (nd.z >> 16) - Rv + zi;
        if (z < 0 || z >= gnz) continue;
        const float Pzf = (float)nd.z * (1.0f / 65536.0f) - 0.5f;  // centre of voxel z at offset z - Pzf
        const float rz = small_int_to_float(z) - Pzf;
        const float h2 = R2 - rz * rz;
        if (h2 < 0.f) continue;
        if (n != cur_node) {  // the node's ancestors (Sec. IV-B), parent first
            const int2 ar = p.anc_range[n];
            na = ar.y;
            if (p.mode == MIG_MODE_ABSOLUTE) na = 0;
            else if (p.mode == MIG_MODE_SINGLE_PARENT) na = min(na, 1);
            na = min(na, p.max_anc);
            fill_anc_records(p, ar, na, anc, lane);
            cur_node = n;
        }
        const int32_t *yk = p.yawtab + k * 12;
        const int ck = yk[0], sk = yk[1];
        const int mu0 = yk[2], mu1 = yk[3], mu2 = yk[4], mv0 = yk[5], mv1 = yk[6], mv2 = yk[7];
        const int mz0 = yk[8], mz1 = yk[9], mz2 = yk[10];
        const float s16 = 1.0f / 65536.0f;
        const float Pxf = (float)nd.x * s16 - 0.5f, Pyf = (float)nd.y * s16 - 0.5f;
        HalfSpace hs[5];
        frustum_half_spaces(mu0, mu1, mu2, mv0, mv1, mv2, mz0, mz1, mz2, p.W, p.H, hs);
        const uint16_t *steps = p.steps + (size_t)ql * WH;
        const int v0x = nd.x >> 16, v0y = nd.y >> 16, v0z = nd.z >> 16;
        const int zq = (z << 16) + 32768 - nd.z;
        int c_abs = 0, c_mrg = 0, nu = 0, no = 0, ns = 0;

        // stage 2: owner pixel of 32 unknown voxel centres (Eq. 5), and the cheap reach test: a voxel
        // is the (|x - x0| + |y - y0| + |z - z0|)-th of any ray that visits it, so it is reached only
        // if that index is below the owner ray's first occupied voxel
        auto owner_stage = [&](bool full) {
            const bool have = full || lane < nu;
            const unsigned long long e = full ? q_pop32(Q.unk, nu, lane) : Q.unk[lane];
            bool keep = false;
            int pix = 0;
            if (have) {
                const int x = (int)(e & 0xFFF), y = (int)((e >> 12) & 0xFFF);
                const int rx = (x << 16) + 32768 - nd.x, ry = (y << 16) + 32768 - nd.y;
                const int64_t Z = (int64_t)mz0 * rx + (int64_t)mz1 * ry + (int64_t)mz2 * zq;
                const int64_t U = (int64_t)mu0 * rx + (int64_t)mu1 * ry + (int64_t)mu2 * zq;
                const int64_t V = (int64_t)mv0 * rx + (int64_t)mv1 * ry + (int64_t)mv2 * zq;
                if (Z > 0) {
                    const float fxr = small_int_to_float(x) - Pxf, fyr = small_int_to_float(y) - Pyf;
                    const float zi_ = __fdividef(1.0f, fmaf(hs[0].a, fxr, fmaf(hs[0].b, fyr, hs[0].c * rz)));
                    const float uf = fmaf(hs[1].a, fxr, fmaf(hs[1].b, fyr, hs[1].c * rz)) * zi_;
                    const float vf = fmaf(hs[3].a, fxr, fmaf(hs[3].b, fyr, hs[3].c * rz)) * zi_;
                    int pu, pv;
                    if (pixel_in(U, Z, uf, p.W, pu) && pixel_in(V, Z, vf, p.H, pv)) {
                        pix = pv * p.W + pu;
                        const int man = abs(x - v0x) + abs(y - v0y) + abs(z - v0z);
                        keep = at_ok(p, steps + pix, (const uint16_t *)p.steps, (size_t)p.steps_cap * p.W * p.H, kBoundsSteps) &&
                               man < (int)ld_written(steps + pix);
                    }
                }
            }
            if (!full) nu = 0;
            q_push(Q.own, no, keep, (e & 0xFFFFFFull) | ((unsigned long long)pix << 24), lt_mask);
        };
        // stage 3: the exact visit test by the owner ray (event order of its DDA, range)
        auto visit_stage = [&](bool full) {
            const bool have = full || lane < no;
            const unsigned long long e = full ? q_pop32(Q.own, no, lane) : Q.own[lane];
            bool counted = false;
            int x = 0, y = 0;
            if (have) {
                if constexpr (STATS) ++st_visit;
                x = (int)(e & 0xFFF);
                y = (int)((e >> 12) & 0xFFF);
                const int pix = (int)(e >> 24);
                int dx, dy, dz;
                ray_dir(p.body[pix], ck, sk, dx, dy, dz);
                counted = visit_index(nd.x, nd.y, nd.z, dx, dy, dz, x, y, z, p.Tq) >= 0;
            }
            if (!full) no = 0;
            c_abs += counted;
            q_push(Q.smp, ns, counted,
                   (unsigned long long)x | ((unsigned long long)y << 16) | ((unsigned long long)z << 32), lt_mask);
        };
        // stage 4: the ancestor test of 32 counted samples (Sec. IV-B)
        auto ancestor_stage = [&](bool full) {
            const bool have = full || lane < ns;
            const unsigned long long sm = full ? q_pop32(Q.smp, ns, lane) : Q.smp[lane];
            if (have)
                c_mrg += !observed<STATS>(HotDirect{p}, anc, na, (int)(sm & 0xFFFF), (int)((sm >> 16) & 0xFFFF),
                                          (int)(sm >> 32), st_anc, st_reads);
            if (!full) ns = 0;
        };

        const float hy = sqrtf(h2);
        const int ylo = max(0, (int)floorf(Pyf - hy) - 1), yhi = min(gny - 1, (int)ceilf(Pyf + hy) + 1);
        for (int yb = ylo; yb <= yhi; yb += 32) {
            // this lane's row: x range of the centres inside the ball and the frustum
            const int y = yb + lane;
            int xa = 0, len = 0;
            if (y <= yhi) row_span(hs, Pxf, small_int_to_float(y) - Pyf, rz, h2, gnx, xa, len);
            int incl = len;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, d);
                if (lane >= d) incl += v;
            }
            const int tot = __shfl_sync(0xffffffffu, incl, 31);
            for (int base = 0; base < tot; base += 32) {
                const int f = base + lane;
                // the row holding flat index f: the first lane whose inclusive sum exceeds f
                int r = 0;
#pragma unroll
                for (int s = 16; s >= 1; s >>= 1) {
                    const int cv = __shfl_sync(0xffffffffu, incl, r + s - 1);
                    if (cv <= f) r += s;
                }
                r = min(r, 31);
                const int rxa = __shfl_sync(0xffffffffu, xa, r);
                const int rstart = __shfl_sync(0xffffffffu, incl - len, r);
                bool unk = false;
                int x = 0;
                if (f < tot) {
                    x = rxa + (f - rstart);
                    if constexpr (STATS) ++st_cand;
                    const uint32_t addr = ((uint32_t)z * (uint32_t)gny + (uint32_t)(yb + r)) * (uint32_t)gnx + (uint32_t)x;
                    unk = load_code(p.grid.g, addr, p.grid, p.bounds_err) == kUnknown;
                    if constexpr (STATS) st_unk += unk;
                }
                q_push(Q.unk, nu, unk, (unsigned long long)x | ((unsigned long long)(yb + r) << 12), lt_mask);
                if (nu >= 32) {
                    owner_stage(true);
                    if (no >= 32) {
                        visit_stage(true);
                        if (ns >= 32) ancestor_stage(true);
                    }
                }
            }
        }
        // the slice's partial batches, stage by stage
        if (nu > 0) owner_stage(false);
        while (no >= 32) {
            visit_stage(true);
            if (ns >= 32) ancestor_stage(true);
        }
        if (no > 0) visit_stage(false);
        while (ns >= 32) ancestor_stage(true);
        if (ns > 0) ancestor_stage(false);
        c_abs = __reduce_add_sync(0xffffffffu, c_abs);
        c_mrg = __reduce_add_sync(0xffffffffu, c_mrg);
        if (lane == 0 && (c_abs | c_mrg)) {
            atomicAdd(p.cnt + ((size_t)n * p.K + k) * 2, c_abs);
            atomicAdd(p.cnt + ((size_t)n * p.K + k) * 2 + 1, c_mrg);
            if constexpr (STATS) atomicAdd(p.stats + 14, (unsigned long long)(uint32_t)c_abs);
        }
        __syncwarp();
    }
    if constexpr (STATS) {
        st_cand = __reduce_add_sync(0xffffffffu, st_cand);
        st_unk = __reduce_add_sync(0xffffffffu, st_unk);
        st_visit = __reduce_add_sync(0xffffffffu, st_visit);
        st_anc = __reduce_add_sync(0xffffffffu, st_anc);
        st_reads = __reduce_add_sync(0xffffffffu, st_reads);
        if (lane == 0) {
            atomicAdd(p.stats + 11, (unsigned long long)st_cand);
            atomicAdd(p.stats + 12, (unsigned long long)st_unk);
            atomicAdd(p.stats + 13, (unsigned long long)st_visit);
            atomicAdd(p.stats + 15, (unsigned long long)st_anc);
            atomicAdd(p.stats + 16, (unsigned long long)st_reads);
        }
    }
}

}  // namespace

size_t vox_dyn_smem(int max_anc) { return (size_t)kVoxWarps * (size_t)std::max(1, max_anc) * sizeof(AncRec); }

int vox_ctas_per_sm() {
    int a = 0, b = 0;
    const size_t smem = vox_dyn_smem(MIG_MAX_DEPTH);
    cudaFuncSetAttribute(voxel_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(voxel_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, voxel_kernel<false>, kVoxWarps * 32, vox_dyn_smem(16));
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, voxel_kernel<true>, kVoxWarps * 32, vox_dyn_smem(16));
    cudaGetLastError();
    return std::max(1, std::min(a, b));
}

size_t steps_pairs(long long pairs, int W, int H, size_t budget_bytes) {
    const size_t per = (size_t)W * H * sizeof(uint16_t);
    const size_t cap = std::max<size_t>(1, budget_bytes / per);
    return (size_t)std::max<long long>(1, std::min<long long>(pairs, (long long)cap));
}

void launch_voxel_chunk(const LevelParams &c, int num_sms, int vox_ctas, cudaStream_t s) {
    const long long vitems = (long long)(c.q1 - c.q0) * (2 * ((int)(c.Tq >> 16) + 2) + 1);
    const int vg = (int)std::max<long long>(1, std::min<long long>((vitems + kVoxWarps - 1) / kVoxWarps,
                                                                    (long long)num_sms * vox_ctas));
    const size_t smem = vox_dyn_smem(c.max_anc);
    if (c.stats) voxel_kernel<true><<<vg, kVoxWarps * 32, smem, s>>>(c);
    else voxel_kernel<false><<<vg, kVoxWarps * 32, smem, s>>>(c);
}

// The per-node pass, when a chunk holds whole nodes (all their yaws).
bool node_pass(const LevelParams &p) { return p.steps_cap >= p.K && p.voxel_pass != MIG_COUNT_PAIRS; }

// Pairs per launch: within the step-count buffer, and few enough that the launch's work items
// (pairs x slices, or nodes x macro blocks) stay below 2^30 for the 32-bit work counter.
int vox_chunk_pairs(const LevelParams &p) {
    const long long slices = 2 * ((long long)(p.Tq >> 16) + 2) + 1;
    const long long lim = 1ll << 30;
    if (node_pass(p)) {
        const long long nodes = std::min<long long>(p.steps_cap / p.K, lim / node_items(p.Tq));
        return (int)std::max<long long>(1, nodes) * p.K;
    }
    return (int)std::max<long long>(1, std::min<long long>(p.steps_cap, lim / slices));
}

void launch_vox_level(const LevelParams &p, long long pairs, int num_sms, int vox_ctas, int node_ctas, cudaStream_t s) {
    const int cap = vox_chunk_pairs(p);
    for (long long q0 = 0; q0 < pairs; q0 += cap) {
        LevelParams c = p;
        c.q0 = (int)q0;
        c.q1 = (int)std::min<long long>(pairs, q0 + cap);
        if (!p.tree) launch_cast_chunk(c, num_sms, s);
        if (node_pass(p)) launch_node_chunk(c, num_sms, node_ctas, s);
        else launch_voxel_chunk(c, num_sms, vox_ctas, s);
    }
}

}  // namespace mig
