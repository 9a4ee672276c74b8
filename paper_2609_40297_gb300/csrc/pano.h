// Panoramic-mode passes (internal): one 360-degree cast per node, then per-yaw window sums.
#pragma once

#include <cuda_runtime.h>

#include "kernels.h"

namespace mig {

// Per-(node, column) absolute and marginal counts of one level into p.pano_cnt (work items from
// p.work[p.lvl]); then each yaw's window sums into p.cnt, ready for launch_select.
void launch_pano_count(const LevelParams &p, int grid, cudaStream_t s);
void launch_pano_window(const LevelParams &p, int grid, cudaStream_t s);
// The same counts by owned voxels (panocount.cu), for the nodes [c.q0, c.q1) of the level, at most
// steps_cap: the cast, then the per-node and the brick pass. The cast clears their column counts.
void launch_pano_cast_chunk(const LevelParams &c, int num_sms, cudaStream_t s);
void launch_pano_tree_cast(const LevelParams &p, int levels, int num_sms, cudaStream_t s);  // launch_tree_cast
void launch_pano_voxel_chunk(const LevelParams &c, int num_sms, cudaStream_t s);
void set_pano_visit(LevelParams &p, int A, float vfov_deg);  // vis_zl2 of a strip's cells
void pano_bricks_init();  // lifts the kernels' dynamic shared-memory limit; call once
int pano_ctas_per_sm();  // also lifts the count kernel's dynamic shared-memory limit; call once

}  // namespace mig
