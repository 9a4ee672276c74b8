// Writing a map: a box of voxel codes, and what is derived from them (voxcount.cuh, bricks.cuh) wherever the
// box can change it. Three launches, the second and third behind the one before (launch.cuh):
//   map_write_kernel - one warp per row of 8 bricks (4x4x4 voxels each) that the box touches: the codes, the
//                      bricks' masks and a bit per brick with an occupied voxel, and per four rows the
//                      occupancy bytes of the 8x8x8 bricks they make up;
//   dist_xy_kernel   - per brick, the distances to the occupied bricks of its own z layer; the occupancy bytes
//                      of the 32x32x32 super-bricks;
//   dist_z_kernel    - the octant distances and their minimum, from the layers ahead and behind; the clutter bit.
// An update of a few voxels is a chain of launches and of dependent loads, so both are few: every kernel
// issues its loads together, before any store, and a brick's row of neighbours is three words of bits. Codes,
// two summaries, masks and three distance passes as seven launches took 75 us per mig_map_update of one voxel
// of a 400x400x100 map (96 of 40x40x20 voxels, 75 of one voxel of 800x800x200); this takes 30 (43, 30) where no
// brick is emptied or first occupied, which ends the second and third launch at once, and 37 (54, 40) else.
// Codes and summaries alone took 36 (51, 35).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "bricks.cuh"
#include "kernels.h"
#include "launch.cuh"

namespace mig {

namespace {

using namespace dev;

// The words of the occupied-brick bits of row (by, bz): bit bx & 31 of word bx >> 5.
__device__ __forceinline__ uint32_t *brick_bits(uint8_t *grid, int nx, int ny, int nz, int by, int bz) {
    const BrickDims n = brick_dims(nx, ny, nz);
    return reinterpret_cast<uint32_t *>(grid + bits_offset(nx, ny, nz)) + ((size_t)bz * n.nby + by) * bits_words(n.nbx);
}

// The version of the map whose write last emptied or occupied a brick: another one leaves distances and
// super-bricks as they are.
__device__ __forceinline__ uint32_t *changed_flag(uint8_t *grid, int nx, int ny, int nz) {
    return reinterpret_cast<uint32_t *>(grid + changed_offset(nx, ny, nz));
}

// A CTA's four warps take the brick rows (2 Y + (warp & 1), 2 Z + (warp >> 1)), lane = x. box NULL: the codes
// are in place.
__global__ void __launch_bounds__(128) map_write_kernel(uint8_t *grid, int nx, int ny, int nz, const uint8_t *box, int x0, int y0,
                                                        int z0, int dx, int dy, int dz, uint32_t version) {
    __shared__ uint32_t s_occ[4];
    wait_previous();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sx = (x0 >> 5) + blockIdx.x, Y = (y0 >> 3) + blockIdx.y, Z = (z0 >> 3) + blockIdx.z;
    const int x = 32 * sx + lane, by = 2 * Y + (warp & 1), bz = 2 * Z + (warp >> 1);
    const BrickDims nb = brick_dims(nx, ny, nz);
    uint32_t occ = 0;
    if (by < nb.nby && bz < nb.nbz) {
        uint8_t *bits = reinterpret_cast<uint8_t *>(brick_bits(grid, nx, ny, nz, by, bz)) + sx, c[16];
        const uint32_t before = *bits;
        uint32_t in = 0;  // bit i: voxel i of the lane's column is in the box
        uint8_t *first = grid + ((size_t)(4 * bz) * ny + 4 * by) * nx + x;
#pragma unroll
        for (int i = 0; i < 16; ++i) {  // all loads, then all stores
            const int y = 4 * by + (i & 3), z = 4 * bz + (i >> 2);
            const bool b = box && (unsigned)(x - x0) < (unsigned)dx && (unsigned)(y - y0) < (unsigned)dy && (unsigned)(z - z0) < (unsigned)dz;
            const uint8_t *from = b ? box + (((size_t)(z - z0) * dy + (y - y0)) * dx + (x - x0)) : first + ((size_t)(i >> 2) * ny + (i & 3)) * nx;
            c[i] = 3;  // beyond the grid: neither unknown nor occupied
            if (x < nx && y < ny && z < nz) c[i] = *from;
            in |= b ? 1u << i : 0u;
        }
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (in >> i & 1) first[((size_t)(i >> 2) * ny + (i & 3)) * nx] = c[i];
        uint64_t u = 0, o = 0;  // of brick `lane` of the row, lanes 0 to 7
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const uint32_t mu = __ballot_sync(0xffffffffu, c[i] == kUnknown), mo = __ballot_sync(0xffffffffu, c[i] == kOcc);
            u |= (uint64_t)((mu >> (4 * (lane & 7))) & 15u) << (4 * i);
            o |= (uint64_t)((mo >> (4 * (lane & 7))) & 15u) << (4 * i);
        }
        if (lane < 8 && 8 * sx + lane < nb.nbx) {
            const size_t b = ((size_t)bz * nb.nby + by) * nb.nbx + 8 * sx + lane;
            reinterpret_cast<uint64_t *>(grid + umask_offset(nx, ny, nz))[b] = u;
            reinterpret_cast<uint64_t *>(grid + omask_offset(nx, ny, nz))[b] = o;
        }
        occ = __ballot_sync(0xffffffffu, o != 0) & 255u;
        if (lane == 0 && occ != before) {
            *bits = (uint8_t)occ;
            *changed_flag(grid, nx, ny, nz) = version;
        }
    }
    if (lane == 0) s_occ[warp] = occ;
    __syncthreads();
    const int X = 4 * sx + (int)threadIdx.x, nbx = (nx + 7) >> 3, nby = (ny + 7) >> 3;
    if (threadIdx.x < 4 && X < nbx)
        grid[bocc_offset(nx, ny, nz) + ((size_t)Z * nby + Y) * nbx + X] =
            ((s_occ[0] | s_occ[1] | s_occ[2] | s_occ[3]) >> (2 * threadIdx.x)) & 3 ? 1 : 0;
}

// The bricks of a pass from (ax, ay, az) on: blocks of 32x4x1, one thread each.
struct BrickBox {
    int ax, ay, az, wx, wy, wz;
};
constexpr int kDistY = 4;

// One-sided distances d = min over j >= 0 of max(j, the previous axis' distance j bricks ahead), capped at
// kDistCap, as bytes: here the four combinations of directions along x (bit 0) and y (bit 1). The block
// layers from box.wz on take the occupancy bytes of the super-bricks from (sx, sy, sz) on.
__global__ void __launch_bounds__(32 * kDistY) dist_xy_kernel(uint8_t *grid, int nx, int ny, int nz, const BrickBox box, const BrickBox supers,
                                                              uint32_t version) {
    wait_previous();
    if (version && *changed_flag(grid, nx, ny, nz) != version) return;
    const BrickDims n = brick_dims(nx, ny, nz);
    if ((int)blockIdx.z >= box.wz) {  // a byte of the bits for each of 8x8 brick rows, two per lane
        const int lane = threadIdx.x;
        int i = (((blockIdx.z - box.wz) * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) * kDistY + threadIdx.y;
        if (i >= supers.wx * supers.wy * supers.wz) return;
        const int sx = supers.ax + i % supers.wx;
        i /= supers.wx;
        const int sy = supers.ay + i % supers.wy, sz = supers.az + i / supers.wy;
        uint32_t any = 0;
        for (int r = lane; r < 64; r += 32) {
            const int by = 8 * sy + (r & 7), bz = 8 * sz + (r >> 3);
            if (by < n.nby && bz < n.nbz) any |= reinterpret_cast<const uint8_t *>(brick_bits(grid, nx, ny, nz, by, bz))[sx];
        }
        any = __any_sync(0xffffffffu, any != 0);
        if (lane == 0) grid[sbocc_offset(nx, ny, nz) + ((size_t)sz * ((ny + 31) >> 5) + sy) * ((nx + 31) >> 5) + sx] = any ? 1 : 0;
        return;
    }
    const int ix = blockIdx.x * 32 + threadIdx.x, iy = blockIdx.y * kDistY + threadIdx.y;
    if (ix >= box.wx || iy >= box.wy) return;
    const int bx = box.ax + ix, by = box.ay + iy, bz = box.az + blockIdx.z;
    const int words = bits_words(n.nbx), w = bx >> 5, sh = bx & 31;
    // distances back (low byte) and ahead along the row of bits: the words around the brick, from its bit
    auto along_x = [&](const uint32_t *row) {
        const uint32_t m = row[w], before = w > 0 ? row[w - 1] : 0u, after = w + 1 < words ? row[w + 1] : 0u;
        const uint32_t back = __funnelshift_l(before, m, 31 - sh), ahead = __funnelshift_r(m, after, sh);
        return (uint32_t)min(__clz((int)back), kDistCap) | ((uint32_t)min(__clz((int)__brev(ahead)), kDistCap) << 8);
    };
    const uint32_t *row = brick_bits(grid, nx, ny, nz, by, bz);
    uint32_t d = kDistCap * 0x01010101u;
#pragma unroll
    for (int j = 0; j < kDistCap; ++j) {
        const uint32_t lo = j <= by ? along_x(row - j * words) : kDistCap * 0x0101u;
        const uint32_t hi = by + j < n.nby ? along_x(row + j * words) : kDistCap * 0x0101u;
        d = __vminu4(d, __vmaxu4(lo | (hi << 16), j * 0x01010101u));
    }
    reinterpret_cast<uint32_t *>(grid + dist_xy_offset(nx, ny, nz))[((size_t)bz * n.nby + by) * n.nbx + bx] = d;
}

// ... and along z: the eight octants (octant_of) and their minimum. Lets no launch start early: what follows
// reads the map through the read-only path.
__global__ void __launch_bounds__(32 * kDistY) dist_z_kernel(uint8_t *grid, int nx, int ny, int nz, const BrickBox box, uint32_t version) {
    cudaGridDependencySynchronize();
    if (version && *changed_flag(grid, nx, ny, nz) != version) return;
    const BrickDims n = brick_dims(nx, ny, nz);
    const int ix = blockIdx.x * 32 + threadIdx.x, iy = blockIdx.y * kDistY + threadIdx.y;
    if (ix >= box.wx || iy >= box.wy) return;
    const int bx = box.ax + ix, by = box.ay + iy, bz = box.az + blockIdx.z, layer = n.nbx * n.nby;
    const size_t at = ((size_t)bz * n.nby + by) * n.nbx + bx;
    const uint32_t *xy = reinterpret_cast<const uint32_t *>(grid + dist_xy_offset(nx, ny, nz)) + at;
    // occupied bricks among the 27 around it, loaded with the rest
    const int words = bits_words(n.nbx), w = bx >> 5, sh = bx & 31;
    const uint32_t *row = brick_bits(grid, nx, ny, nz, by, bz) + w;
    int occ = 0;
#pragma unroll
    for (int r = 0; r < 9; ++r) {
        const int dy = r % 3 - 1, dz = r / 3 - 1;
        if ((unsigned)(by + dy) < (unsigned)n.nby && (unsigned)(bz + dz) < (unsigned)n.nbz) {
            const uint32_t *q = row + (ptrdiff_t)(dz * n.nby + dy) * words;
            const uint32_t before = sh == 0 && w > 0 ? q[-1] >> 31 : 0u, after = sh == 31 && w + 1 < words ? q[1] << 31 : 0u;
            occ += __popc(sh == 0 ? (before | (*q << 1)) & 7u : ((*q >> (sh - 1)) & (sh == 31 ? 3u : 7u)) | (after >> 29));
        }
    }
    uint32_t lo = kDistCap * 0x01010101u, hi = lo;
#pragma unroll
    for (int j = 0; j < kDistCap; ++j) {
        if (j <= bz) lo = __vminu4(lo, __vmaxu4(xy[-(ptrdiff_t)j * layer], j * 0x01010101u));
        if (bz + j < n.nbz) hi = __vminu4(hi, __vmaxu4(xy[(ptrdiff_t)j * layer], j * 0x01010101u));
    }
    uint32_t least = kDistCap;
    const size_t plane = oct_offset(nx, ny, nz, 1) - oct_offset(nx, ny, nz, 0);
    uint8_t *dist = grid + dist_offset(nx, ny, nz) + at;  // then the octants, a plane each
#pragma unroll
    for (int o = 0; o < 8; ++o) {
        const uint32_t v = ((o < 4 ? lo : hi) >> (8 * (o & 3))) & 255u;
        dist[(o + 1) * plane] = (uint8_t)v;
        least = min(least, v);
    }
    const int in = (min(bx + 1, n.nbx - 1) - max(bx - 1, 0) + 1) * (min(by + 1, n.nby - 1) - max(by - 1, 0) + 1) *
                   (min(bz + 1, n.nbz - 1) - max(bz - 1, 0) + 1);
    *dist = (uint8_t)(least | (least == 0 && 27 * occ >= 22 * in ? kClutter : 0));
}

}  // namespace

size_t map_codes_bytes(int nx, int ny, int nz) { return occ_summary_end(nx, ny, nz); }
size_t map_layout_bytes(int nx, int ny, int nz) { return brick_data_end(nx, ny, nz); }

void launch_map_write(uint8_t *grid, int nx, int ny, int nz, const uint8_t *box, int x0, int y0, int z0, int dx, int dy, int dz,
                      uint32_t version, cudaStream_t s) {
    const int x1 = x0 + dx - 1, y1 = y0 + dy - 1, z1 = z0 + dz - 1;
    const dim3 rows((unsigned)((x1 >> 5) - (x0 >> 5) + 1), (unsigned)((y1 >> 3) - (y0 >> 3) + 1), (unsigned)((z1 >> 3) - (z0 >> 3) + 1));
    map_write_kernel<<<rows, 128, 0, s>>>(grid, nx, ny, nz, box, x0, y0, z0, dx, dy, dz, version);
    // a brick's distances depend on the bricks up to kDistCap - 1 away along each axis
    const BrickDims n = brick_dims(nx, ny, nz);
    const int first[3] = {x0 >> 2, y0 >> 2, z0 >> 2}, last[3] = {x1 >> 2, y1 >> 2, z1 >> 2}, nb[3] = {n.nbx, n.nby, n.nbz};
    int a[3], w[3];
    for (int i = 0; i < 3; ++i) {
        a[i] = std::max(0, first[i] - (kDistCap - 1));
        w[i] = std::min(nb[i] - 1, last[i] + (kDistCap - 1)) - a[i] + 1;
    }
    const BrickBox xy{a[0], a[1], first[2], w[0], w[1], last[2] - first[2] + 1}, all{a[0], a[1], a[2], w[0], w[1], w[2]};
    const BrickBox supers{x0 >> 5, y0 >> 5, z0 >> 5, (x1 >> 5) - (x0 >> 5) + 1, (y1 >> 5) - (y0 >> 5) + 1, (z1 >> 5) - (z0 >> 5) + 1};
    auto blocks = [](const BrickBox &b) { return dim3((unsigned)(b.wx + 31) / 32, (unsigned)(b.wy + kDistY - 1) / kDistY, (unsigned)b.wz); };
    dim3 g = blocks(xy);
    const unsigned per_layer = g.x * g.y * kDistY;
    g.z += ((unsigned)(supers.wx * supers.wy * supers.wz) + per_layer - 1) / per_layer;
    launch_behind(dist_xy_kernel, g, dim3(32, kDistY), 0, s, grid, nx, ny, nz, xy, supers, version);
    launch_behind(dist_z_kernel, blocks(all), dim3(32, kDistY), 0, s, grid, nx, ny, nz, all, version);
}

}  // namespace mig
