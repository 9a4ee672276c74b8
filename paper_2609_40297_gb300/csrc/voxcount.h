// Launchers of the owned-voxel count kernels (voxcount.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

#include "kernels.h"

namespace mig {

// (node, yaw) pairs per chunk of the owned-voxel count: all `pairs` of a level, or as many as a
// step-count buffer of budget_bytes holds (W * H uint16 per pair), at least 1.
size_t steps_pairs(long long pairs, int W, int H, size_t budget_bytes);
// Entries of one image's tile bounds (bricks.cuh, Pyramid).
size_t hz_entries(int W, int H);
// The device region of an owned-voxel count of a tree of n nodes with levels of at most max_nodes: the step counts of
// `cap` pairs, the counters, the counts' tile bounds and the per-node pass's queue. The panoramic mode
// has one image of A x H per node: W = A, K = 1.
struct SensorDims {
    int W, H, K;
    int64_t Tq;
};
struct StepsLayout {
    int cap;        // pairs per chunk (0: the ray-by-ray count, an empty region)
    int tree;       // 0, or the tree's nodes: the region holds all of them (cap = tree * K)
    int queue_cap;  // records
    bool depths;    // the tree's depth buffers, all yaws
    size_t o_ctr, o_hz, o_queue, o_depths, bytes;
};
// tree_bytes: the most step counts for the whole tree (0: level by level)
StepsLayout steps_layout(const SensorDims &d, int n, int max_nodes, size_t budget_bytes, size_t tree_bytes, bool node_pass, int mode);
// The same for as many whole nodes as fit in a region of at most `bytes` bytes, and for single pairs (without a
// queue) as many as fit (cap 0: not one does). with_depths: also a whole tree's depth buffers, where they fit.
StepsLayout steps_layout_in(const SensorDims &d, int n, int max_nodes, size_t bytes, bool with_depths);
StepsLayout steps_pairs_in(const SensorDims &d, size_t max_pairs, size_t bytes);
void set_steps(LevelParams &p, void *base, const StepsLayout &L);  // the region's fields
// Step-count buffer budget per evaluation (device bytes).
constexpr size_t kStepsBudget = (size_t)1 << 30;
// A tree whose step counts stay below this is cast by one launch instead of level by level: a level's cast
// needs nothing of the levels above it, and each level's cast ends with SMs idle. Cast times of 20 nodes
// of 36x24x8: 89 -> 30 us, 100 of 48x28x8: 188 -> 76 us, 500 of 160x120x16 (307 MB, beyond L2): 6.4 -> 5.3
// ms with an unchanged voxel stage. Larger trees have levels of several ms of cast each.
constexpr size_t kTreeSteps = (size_t)512 << 20;
// A tree whose depth buffers, those of every yaw of its nodes, stay below this has them stored by the cast,
// and its levels' renders are copies: 63 -> 34 us of render for 20 nodes of 36x24x8 (4 levels), 145 -> 74 for
// 100 of 48x28x8 (9), the cast within 10 us. For larger trees the stores cost more than they save: the cast
// of 500 nodes of 160x120x16 5.3 -> 5.9 ms, the render 0.43 -> 0.28.
constexpr size_t kTreeDepths = (size_t)64 << 20;
// One level's count for the sample modes (marginal, single parent, absolute): for each chunk of
// p.steps_cap pairs of the first `pairs` (node, yaw) pairs, a cast launch and a voxel launch. The
// kernels read the level's true size from p.level_off and skip pairs beyond it, so `pairs` may be
// an upper bound.
// When every chunk holds whole nodes (all K yaws), the voxel pass runs once per node over all its
// yaws (node_kernel); otherwise once per (node, yaw) pair (voxel_kernel).
void launch_vox_level(const LevelParams &p, long long pairs, int num_sms, int vox_ctas, int node_ctas, cudaStream_t s);
// The launches of one chunk [c.q0, c.q1) (launch_vox_level runs them for every chunk).
void launch_cast_chunk(const LevelParams &c, int num_sms, cudaStream_t s);
// The cast of all nodes of a tree of `levels` levels (p.tree > 0), before its levels are counted.
void launch_tree_cast(const LevelParams &p, int levels, int num_sms, cudaStream_t s);
void launch_voxel_chunk(const LevelParams &c, int num_sms, int vox_ctas, cudaStream_t s);
void launch_node_chunk(const LevelParams &c, int num_sms, int node_ctas, cudaStream_t s);
bool node_pass(const LevelParams &p);  // whole nodes per chunk: the per-node pass
int vox_chunk_pairs(const LevelParams &p);  // pairs per chunk (a multiple of K for the per-node pass)
int node_ctas_per_sm();
int vox_ctas_per_sm();
int node_grid(long long items, int most, int crowd);  // CTAs of the node and the brick pass
int brick_grid(long long nodes, int64_t Tq, int num_sms, int crowd);
long long node_items(int64_t Tq);  // work items of one node of the per-node pass

}  // namespace mig
