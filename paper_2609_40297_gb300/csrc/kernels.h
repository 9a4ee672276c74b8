// Device kernels of the marginal-gain path and their launch parameters (internal).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace mig {

constexpr int kStatsCounters = 20;

struct GridView {
    const uint8_t *g;  // voxel codes (x-fastest rows), then what bricks.cuh lists
    int nx, ny, nz;
};

// A brick that the per-node pass leaves to its voxel stage: unknown voxels, those an ancestor is known
// to observe, the ancestors (bit = place in the node's list) still to test, and by yaw (bit = yaw -
// first) those that count every unknown voxel, those undecided, and of these the ones whose voxels
// need the test against the owner ray's first hit, and against the owner ray itself. brick: x | y << 10 |
// z << 20 (4x4x4 bricks); node: its place in the chunk | first yaw / 64 << kRecNodeBits.
struct BrickRec {
    uint64_t U, O, anc, all, part, rch, vis;
    uint32_t brick, node;
};
constexpr int kRecNodeBits = 27;

// One tree level's work (Sec. IV-C): the nodes level_nodes[level_off[lvl] ..), the first
// level_int[lvl] of which have children and need their depth buffer rendered.
struct LevelParams {
    GridView grid;
    const int4 *body;        // H*W: body-frame ray (Q30) and camera z (Q30)
    const int32_t *yawtab;   // K*12: ck, sk, mu[3], mv[3], mz[3] (Q30, Q16)
    const float *yawf;       // K*9: mu, mv, mz as floats / 2^16 (estimates only)
    int W, H, K;
    int64_t Tq;              // range, Q16 voxel units
    int tile_w, tile_h, tiles_x, tiles;  // count-pass tile (rays per warp work item)
    const int32_t *level_off;   // device, levels + 1
    const int32_t *level_int;   // device, levels
    const int32_t *level_nodes; // device, n
    const int4 *node;           // device, n: Px, Py, Pz (Q16), arena slot
    const int2 *anc_range;      // device, n: (offset into anc, ancestor count = depth)
    const int32_t *anc;         // device: ancestors, parent first
    int32_t *sel_yaw;           // device, n (written by select)
    uint32_t *arena;            // device, slots * W * H depth buffers
    int32_t *cnt;               // device, n*K*2 (abs, excl) counts
    int32_t *work;              // device, levels: count-pass work counters (zeroed); [0] also the cast's
    int32_t *out_abs, *out_marg, *out_yaw;  // device, n
    int mode;                   // mig_mode
    int lvl;
    unsigned long long *stats;  // NULL, or kStatsCounters counters (instrumented pass)
    int max_anc;                // ancestor records per warp (>= the deepest node's depth, <= 64)
    // panoramic mode: A wedges ("columns") of `pano_step` per yaw bin, Wc columns per yaw window
    int pano_A, pano_Wc, pano_step;
    const int2 *pano_bc;        // A: wedge boundary cos, sin (Q30)
    const int4 *pano_dir;       // A*H: ray of cell (column, row) (Q30), pad
    const int4 *pano_row;       // A*2: strip rows (mv0 mv1 mv2 mz0) (mz1 mz2 - -) (Q16)
    int32_t *pano_cnt;          // n*A*2 (abs, excl) per column
    // checked builds (MIG_DEBUG_BOUNDS=1): out-of-buffer indices are or-ed into *bounds_err (NULL:
    // not recorded) and the access is skipped; arena_slots = depth buffers in the arena (0: unchecked)
    int32_t *bounds_err;
    int arena_slots;
    int bounds_half;  // checked builds: kinds of buffers that count as half as large (a test of the checks)
    // owned-voxel count (voxcount.cu): per-ray DDA step counts of a chunk of (node, yaw) pairs
    // [q0, q1) of the level, steps_cap pairs of W * H each; NULL = the ray-by-ray count kernel
    uint16_t *steps;
    int32_t *vctr;  // [0] work counter of the voxel pass, [1] records queued, [2] records handed out
                    // (zeroed by the cast launch before it)
    int steps_cap;
    int q0, q1;
    // per-node voxel pass: the frustum's elevation band (tangents) and azimuth half-width
    float band_tlo, band_thi, az_half;
    int voxel_pass;  // MIG_COUNT_AUTO, MIG_COUNT_PAIRS or MIG_COUNT_NODES
    // bounds of the step counts (hz, pairs of the chunk) and of the depth buffers (dpyr, arena slots)
    // over pixel tiles, hz_entries(W, H) each; dpyr NULL: not kept
    uint32_t *hz;
    uint2 *dpyr;
    // NULL, or the place in the tree where this step's launches begin: (level, first node of the level).
    // The step takes one chunk of steps_cap pairs; a step that ends its level selects and renders it, and
    // select writes the next step's place to cursor[1]. Used where the host does not know the levels'
    // sizes: q0 and q1 are then taken from here (step_range), and lvl is the number of levels.
    int2 *cursor;
    BrickRec *queue;  // per-node pass: undecided bricks of the chunk
    int queue_cap;
    // 0, or the tree's nodes: all of them were cast by one launch, and the step counts and bounds of the
    // i-th of level_nodes are the buffers' i-th (else a chunk's nodes are, from 0)
    int tree;
    // NULL, or the depth buffers of all the tree's (node, yaw) pairs of internal nodes, stored by the cast:
    // W * H per pair, in the step counts' order. The render then copies the selected yaw's.
    uint32_t *depths;
    // per-node pass: half a pixel at unit depth along the image axes, the depth below which the owner
    // ray certainly visits its voxel, and the reciprocal focal lengths (set_visit_params)
    float vis_hu, vis_hv, vis_zl2, ifx, ify;
    int crowd;  // trees whose launches run beside these (batches, servers), with this one; 0: alone
};

void launch_count(const LevelParams &p, int grid, cudaStream_t s);
int count_ctas_per_sm();  // resident CTAs per SM of the count kernel
void launch_select(const LevelParams &p, int grid, cudaStream_t s);  // a level without internal nodes
// Selects the yaws of the level's nodes and renders its internal ones (`nodes`: at least their number).
void launch_select_render(const LevelParams &p, int nodes, int num_sms, cudaStream_t s);
void set_visit_params(LevelParams &p, float hfov_deg, float vfov_deg);  // the vis_* fields, from p.W and p.H
// Writes a box of voxel codes into a grid of nx * ny * nz (box NULL: they are in place) and refreshes the
// occupancy bytes, masks and distances that depend on it (mapwrite.cu). version: the map's after this write, or
// 0 for its first.
void launch_map_write(uint8_t *grid, int nx, int ny, int nz, const uint8_t *box, int x0, int y0, int z0, int dx, int dy, int dz,
                      uint32_t version, cudaStream_t s);
// device bytes of an nx*ny*nz grid's voxel codes and occupancy bytes
size_t map_codes_bytes(int nx, int ny, int nz);
// device bytes of an nx*ny*nz grid with the masks and distances of its bricks
size_t map_layout_bytes(int nx, int ny, int nz);

// Device planning (tree on the device): depth, levels, ancestors, slots, quantised positions.
struct DevPlanParams {
    int n, max_depth;
    const int32_t *parent;
    const float *pos;
    float ox, oy, oz, voxel;
    int nx, ny, nz;
    int32_t *depth;        // n
    int32_t *level_cnt;    // max_depth + 1 (zeroed)
    int32_t *level_icnt;   // max_depth + 1 (zeroed)
    int32_t *level_off;    // max_depth + 2
    int32_t *level_int;    // max_depth + 1
    int32_t *has_child;    // n (zeroed)
    int32_t *level_nodes;  // n
    int2 *anc_range;       // n: (n * max_depth, depth)
    int32_t *anc;          // n * max_depth
    int32_t *level_cur2;   // 2 * (max_depth + 1) (zeroed): internal / leaf scatter cursors
    int32_t *roots;        // 1 (zeroed)
    int4 *node;            // n
    int32_t *slot_cnt;     // 1 (zeroed)
    int32_t *err;          // device error word of this call
    int32_t *ctx_err;      // context error word (read by mig_ctx_sync)
    int32_t *out_abs, *out_marg, *out_yaw;
};
void launch_plan(const DevPlanParams &p, cudaStream_t s);

}  // namespace mig
