// Device kernels: fused per-level count (3D DDA + owner test + ancestor depth test + integer
// reductions), yaw selection, device planning.
//
// All result-deciding arithmetic is integer (the fixed-point reading of Sec. IV-A..C):
// positions Q16 voxel units, ray directions Q30, projection rows Q16, depths Q16.16.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "dev_path.cuh"
#include "kernels.h"
#include "launch.cuh"
#include "mig.h"

namespace mig {

namespace {

using namespace dev;

template <bool STATS>
__global__ void __launch_bounds__(kWarps * 32, MIG_COUNT_MINB) count_kernel(const LevelParams p) {
    // ancestor records: p.max_anc per warp, sized at launch from the tree's depth (dynamic shared
    // memory), so that the rest of the unified L1/shared storage serves the voxel gathers
    extern __shared__ AncRec s_anc_dyn[];
    __shared__ unsigned long long s_q[kWarps][kQueue];
    __shared__ int4 s_cam[kWarps][4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int l0 = p.level_off[p.lvl];
    const int L = p.level_off[p.lvl + 1] - l0;
    const int chunks = L * p.K * p.tiles;
    for (;;) {
        int c = 0;
        if (lane == 0) c = atomicAdd(p.work + p.lvl, 1);
        c = __shfl_sync(0xffffffffu, c, 0);
        if (c >= chunks) break;
        count_chunk<STATS>(p, HotDirect{p}, l0, c, s_anc_dyn + warp * p.max_anc, s_q[warp], s_cam[warp], lane);
    }
}

// ------------------------------------------------------------------------------ select kernel
// Yaw selection (Sec. III-B): lowest k with the largest marginal count (absolute count in the
// absolute mode, where both counts are equal); g_abs = max over yaws of the absolute count. For levels
// without internal nodes; the others select in the render's launch (launch_select_render).
__global__ void select_kernel(const LevelParams p) {
    wait_previous();
    if (p.tree && blockIdx.x == 0 && threadIdx.x < 3) p.vctr[threadIdx.x] = 0;  // for the next level's count
    const int lvl = p.lvl;
    const int l0 = p.level_off[lvl];
    const int L = p.level_off[lvl + 1] - l0;
    for (int li = blockIdx.x * blockDim.x + threadIdx.x; li < L; li += gridDim.x * blockDim.x)
        select_node(p, p.level_nodes[l0 + li]);
}

// ----------------------------------------------------------------------------- device plan
__global__ void plan_depth_kernel(const DevPlanParams p) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < p.n; i += gridDim.x * blockDim.x) {
        int d = 0, q = p.parent[i];
        bool bad = false;
        if (q == -1) atomicAdd(p.roots, 1);
        while (q != -1) {
            if (q < 0 || q >= p.n || d >= p.max_depth) {
                bad = true;
                break;
            }
            p.anc[(size_t)i * p.max_depth + d] = q;
            ++d;
            q = p.parent[q];
        }
        if (bad) {
            atomicOr(p.err, 1);
            d = 0;
        }
        p.depth[i] = d;
        p.anc_range[i] = make_int2(i * p.max_depth, d);
        const int pa = p.parent[i];
        if (!bad && pa >= 0) p.has_child[pa] = 1;
        // quantised position, round half to even (the same IEEE double steps as the host)
        const float pos3[3] = {p.pos[3 * (size_t)i], p.pos[3 * (size_t)i + 1], p.pos[3 * (size_t)i + 2]};
        const float org[3] = {p.ox, p.oy, p.oz};
        const int dims[3] = {p.nx, p.ny, p.nz};
        int P[3];
        for (int a = 0; a < 3; ++a) {
            const double qd = __dmul_rn(__ddiv_rn(__dsub_rn((double)pos3[a], (double)org[a]), (double)p.voxel), 65536.0);
            if (!(qd > -1.0 && qd < (double)dims[a] * 65536.0)) {
                atomicOr(p.err, 2);
                P[a] = 0;
                continue;
            }
            const long long v = __double2ll_rn(qd);
            if (v < 0 || v >= (long long)dims[a] * 65536) {
                atomicOr(p.err, 2);
                P[a] = 0;
            } else {
                P[a] = (int)v;
            }
        }
        p.node[i] = make_int4(P[0], P[1], P[2], -1);
        atomicAdd(p.level_cnt + d, 1);
    }
}

__global__ void plan_slot_kernel(const DevPlanParams p) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < p.n; i += gridDim.x * blockDim.x) {
        if (p.has_child[i]) {
            p.node[i].w = atomicAdd(p.slot_cnt, 1);
            atomicAdd(p.level_icnt + p.depth[i], 1);
        }
    }
}

__global__ void plan_scan_kernel(const DevPlanParams p) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    if (p.n > 0 && *p.roots != 1) atomicOr(p.err, 4);
    const bool bad = *p.err != 0;
    int acc = 0;
    for (int d = 0; d <= p.max_depth; ++d) {
        p.level_off[d] = bad ? 0 : acc;
        p.level_int[d] = bad ? 0 : p.level_icnt[d];
        acc += p.level_cnt[d];
    }
    p.level_off[p.max_depth + 1] = bad ? 0 : acc;
    if (bad) atomicOr(p.ctx_err, *p.err);
}

__global__ void plan_scatter_kernel(const DevPlanParams p) {
    const bool bad = *p.err != 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < p.n; i += gridDim.x * blockDim.x) {
        if (bad) {
            p.out_abs[i] = -1;
            p.out_marg[i] = -1;
            p.out_yaw[i] = -1;
            continue;
        }
        const int d = p.depth[i];
        int idx;
        if (p.has_child[i]) idx = p.level_off[d] + atomicAdd(p.level_cur2 + 2 * d, 1);
        else idx = p.level_off[d] + p.level_icnt[d] + atomicAdd(p.level_cur2 + 2 * d + 1, 1);
        p.level_nodes[idx] = i;
    }
}

}  // namespace

size_t count_dyn_smem(int max_anc) { return (size_t)kWarps * (size_t)std::max(1, max_anc) * sizeof(AncRec); }

void launch_count(const LevelParams &p, int grid, cudaStream_t s) {
    const size_t smem = count_dyn_smem(p.max_anc);
    if (p.stats) count_kernel<true><<<grid, kWarps * 32, smem, s>>>(p);
    else count_kernel<false><<<grid, kWarps * 32, smem, s>>>(p);
}

int count_ctas_per_sm() {
    int a = 0, b = 0;
    const size_t smem = count_dyn_smem(MIG_MAX_DEPTH);  // the worst case
    cudaFuncSetAttribute(count_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(count_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, count_kernel<false>, kWarps * 32, smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, count_kernel<true>, kWarps * 32, smem);
    cudaGetLastError();
    return std::max(1, std::min(a, b));
}
void launch_select(const LevelParams &p, int grid, cudaStream_t s) { launch_behind(select_kernel, grid, 128, 0, s, p); }
void launch_plan(const DevPlanParams &p, cudaStream_t s) {
    const int grid = std::max(1, std::min((p.n + 255) / 256, 1024));
    plan_depth_kernel<<<grid, 256, 0, s>>>(p);
    plan_slot_kernel<<<grid, 256, 0, s>>>(p);
    plan_scan_kernel<<<1, 32, 0, s>>>(p);
    plan_scatter_kernel<<<grid, 256, 0, s>>>(p);
}

}  // namespace mig
