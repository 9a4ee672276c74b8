"""The work that a planner has this library do, as measurable cases.

Each case is one call (or one replanning step) of the public Python binding on a seeded synthetic
map and planning tree. The maps are made here with the structure of a robot's map: rooms with
walls, doors, pillars and furniture, or terrain with boxes, unknown except for what a few scans from
poses around the robot saw. The trees are RRTs grown from the latest scan pose.

Sizes are those of the repository's own workloads (tiny, paper scale, large, batched, serving), of
the method's published table (87x58 degrees, 10 degrees nose down, 5 m, the depth-buffer size rule
at 0.2 m and 0.1 m), and of odd sensors in between.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2609_40297_gb300 as mig

FREE, OCCUPIED = 1, 2
MODES = {"marginal": mig.MODE_MARGINAL, "single_parent": mig.MODE_SINGLE_PARENT, "absolute": mig.MODE_ABSOLUTE,
         "interval": mig.MODE_INTERVAL, "panoramic": mig.MODE_PANORAMIC}
RAY_GRIDS = [(64, 48), (96, 72), (128, 96), (160, 120), (240, 180), (320, 240)]


def _case(name, call, world, dims, voxel, nodes, depth, step, image, range_m, yaws, fov=(90.0, 60.0), pitch=0.0,
          mode="marginal", outputs="gains", trees=1, maps=1):
    c = {"call": call, "world": world, "nx": dims[0], "ny": dims[1], "nz": dims[2], "voxel": voxel, "nodes": nodes,
         "depth": depth, "step": step, "width": image[0], "height": image[1], "range": range_m, "yaws": yaws,
         "hfov": fov[0], "vfov": fov[1], "pitch": pitch, "mode": mode, "outputs": outputs, "trees": trees, "maps": maps}
    return {"name": name, **c} if name else c


ROOMS_FINE, ROOMS_COARSE = (400, 400, 100), (200, 200, 50)


def listed():
    return [
        # a short-horizon replan of a few nodes from host arrays: latency and launches count
        _case("tiny", "host", "boxes", (64, 64, 32), 0.2, 20, 4, 1.5, (36, 24), 4.0, 8),
        # the published table's coarse row (0.2 m), with every diagnostic output
        _case("table_coarse", "host", "rooms", ROOMS_COARSE, 0.2, 100, 8, 1.5, (48, 28), 5.0, 8, (87.0, 58.0), 10.0,
              outputs="all"),
        # the published table's fine row (0.1 m), tree and results on the device
        _case("table_fine", "device", "rooms", ROOMS_FINE, 0.1, 1000, 12, 1.5, (95, 56), 5.0, 16, (87.0, 58.0), 10.0),
        # the paper-scale tree, device arrays: a planner that keeps its tree on the GPU
        _case("paper", "device", "rooms", ROOMS_FINE, 0.1, 500, 10, 1.5, (160, 120), 6.0, 16),
        # one replanning step of a robot: 10 % of the map updated, a tree evaluated from host arrays, its paths scored
        _case("replan", "replan", "rooms", ROOMS_FINE, 0.1, 200, 10, 1.5, (160, 120), 6.0, 16),
        # the paper's own screen-space overlap test on the paper-scale tree, with every yaw's counts
        _case("interval", "host", "rooms", ROOMS_FINE, 0.1, 500, 10, 1.5, (160, 120), 6.0, 16, mode="interval",
              outputs="counts"),
        # one 360-degree cast per node on the paper-scale tree, with every yaw's counts
        _case("panoramic", "host", "rooms", ROOMS_FINE, 0.1, 500, 10, 1.5, (160, 120), 6.0, 16, mode="panoramic",
              outputs="counts"),
        # the single-parent gain with an odd image, an odd number of yaws and a pitched camera
        _case("single_parent_odd", "host", "rooms", ROOMS_FINE, 0.1, 150, 6, 1.2, (223, 131), 6.5, 7, (75.0, 50.0), -5.0,
              mode="single_parent", outputs="counts"),
        # a real-time control loop that may not allocate: fixed scratch, the largest paper-scale tree it holds
        _case("noalloc", "noalloc", "rooms", ROOMS_FINE, 0.1, 500, 10, 1.5, (160, 120), 6.0, 16),
        # many independent trees of mixed sizes and ray grids in one call
        _case("batch", "batch", "rooms", ROOMS_FINE, 0.1, 800, 12, 1.5, (320, 240), 6.0, 16, trees=12, maps=4),
        # robots on shared maps, each request after its map update, through the continuous-batching server
        _case("serving", "serving", "rooms", ROOMS_FINE, 0.1, 600, 10, 1.5, (160, 120), 6.0, 16, trees=8, maps=2),
        # the largest replan: 0.05 m, 320x240 rays, 36 yaws, 8 m
        _case("large", "device", "terrain", (800, 800, 200), 0.05, 2000, 15, 2.0, (320, 240), 8.0, 36),
    ]


def draw(rng):
    """One more case: a call and mode drawn evenly, sizes spread over the logarithm of their range."""
    def logint(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    call, mode = rng.choice([("host", "marginal"), ("host", "absolute"), ("host", "single_parent"), ("host", "interval"),
                             ("host", "panoramic"), ("device", "marginal"), ("device", "marginal"), ("replan", "marginal"),
                             ("noalloc", "marginal"), ("batch", "marginal"), ("serving", "marginal")])
    world, dims, voxel, range_m = rng.choice([("boxes", (64, 64, 32), 0.2, 4.0), ("rooms", ROOMS_COARSE, 0.2, 5.0),
                                              ("rooms", ROOMS_FINE, 0.1, 6.0), ("rooms", ROOMS_FINE, 0.1, 5.0),
                                              ("rooms", (313, 277, 61), 0.13, 6.0),
                                              ("terrain", (800, 800, 200), 0.05, 8.0)])
    if world == "terrain" and call in ("batch", "serving"):
        world, dims, voxel, range_m = "rooms", ROOMS_FINE, 0.1, 6.0
    dims = tuple(d - rng.randrange(0, 8) for d in dims)
    range_m = round(range_m * rng.uniform(0.75, 1.0), 2)
    w = logint(36, 320)
    h = max(20, int(w * rng.uniform(0.55, 0.8)))
    fov = (rng.choice([90.0, 87.0, round(rng.uniform(60.0, 110.0), 1)]), rng.choice([60.0, 58.0, round(rng.uniform(40.0, 75.0), 1)]))
    pitch = 0.0 if mode == "panoramic" else rng.choice([0.0, 0.0, 10.0, round(rng.uniform(-20.0, 20.0), 1)])
    yaws = rng.choice([4, 8, 12, 16, 16, rng.randrange(5, 37)])
    nodes = logint(20, 1500)
    depth = rng.randrange(4, 16)
    most = {"interval": 2.5e8, "panoramic": 1.0e9}.get(mode, 1.5e9)
    if call == "noalloc":
        nodes = min(nodes, int(48e6 / (w * h * 4 + yaws * 8 + 400)))
        most = 4.0e8
    if call in ("batch", "serving"):
        most /= 8
    nodes = max(20, min(nodes, int(most / (yaws * w * h)), sum(6 ** d for d in range(depth + 1)) // 2))
    trees = rng.randrange(4, 13) if call in ("batch", "serving") else 1
    return _case(None, call, world, dims, voxel, nodes, depth, rng.choice([1.0, 1.5, 2.0]), (w, h), range_m, yaws, fov,
                 pitch, mode, "gains" if call != "host" else "all" if nodes * w * h < 3e6 else "counts", trees=trees,
                 maps=min(trees, rng.randrange(2, 4)))


# ------------------------------------------------------------------------------------------ worlds
def _rooms(rng, nx, ny, nz, v):
    """Floor and ceiling, a jittered grid of walls with doors, pillars and furniture: about 10 % occupied."""
    occ = np.zeros((nz, ny, nx), bool)
    slab = max(1, round(0.2 / v))
    occ[:slab] = True
    occ[nz - slab:] = True
    door = min(nz - slab - 1, round(2.4 / v))

    def cuts(n):
        at, x = [], int(rng.uniform(3.0, 6.0) / v)
        while x < n - int(2.0 / v):
            at.append(x)
            x += int(rng.uniform(5.5, 9.5) / v)
        return at

    xc, yc = cuts(nx), cuts(ny)
    for axis, planes, others, n in ((2, xc, yc, ny), (1, yc, xc, nx)):
        ends = [0] + others + [n]
        for c in planes:
            wall = [slice(None)] * 3
            wall[axis] = slice(c, c + slab)
            occ[tuple(wall)] = True
            for a, b in zip(ends[:-1], ends[1:]):
                if b - a > int(2.0 / v):
                    wide = min(int(rng.uniform(1.0, 1.7) / v), b - a - 6)
                    s = int(rng.integers(a + 3, b - wide - 2))
                    gap = [slice(slab, slab + door), slice(None), slice(None)]
                    gap[axis] = slice(c, c + slab)
                    gap[3 - axis] = slice(s, s + wide)
                    occ[tuple(gap)] = False
    count, total = int(np.count_nonzero(occ)), occ.size
    pillar = max(1, round(0.4 / v))
    while count < 0.10 * total:
        if rng.random() < 0.5:
            x, y = int(rng.integers(0, nx - pillar)), int(rng.integers(0, ny - pillar))
            part = occ[:, y:y + pillar, x:x + pillar]
        else:
            ex, ey, ez = (max(2, int(rng.uniform(a, b) / v)) for a, b in ((0.6, 3.0), (0.6, 3.0), (0.4, 1.5)))
            x, y = int(rng.integers(0, nx - ex)), int(rng.integers(0, ny - ey))
            part = occ[slab:slab + ez, y:y + ey, x:x + ex]
        count += part.size - int(np.count_nonzero(part))
        part[...] = True
    return torch.from_numpy(occ).cuda()


def _boxes(occ, rng, frac, lo, hi):
    """Random boxes with edges lo..hi voxels added until about `frac` of the voxels are occupied."""
    nz, ny, nx = occ.shape
    left = frac * occ.numel()
    while left > 0:
        ex, ey, ez = (min(int(e), d) for e, d in zip(rng.integers(lo, hi + 1, 3), (nx, ny, nz)))
        x, y, z = (int(rng.integers(0, d - e + 1)) for e, d in ((ex, nx), (ey, ny), (ez, nz)))
        occ[z:z + ez, y:y + ey, x:x + ex] = True
        left -= ex * ey * ez
    return occ


def _terrain(rng, nx, ny, nz):
    """A rough height field (four octaves of smooth noise) with boxes: about 12 % occupied."""
    gen = torch.Generator().manual_seed(int(rng.integers(1 << 31)))
    h = torch.zeros(1, 1, ny, nx)
    for o in range(4):
        cells = max(2, round(max(nx, ny) * 2 ** o / 160))
        grid = torch.rand(1, 1, cells + 3, cells + 3, generator=gen)
        h += 0.5 ** o * torch.nn.functional.interpolate(grid, size=(ny, nx), mode="bicubic", align_corners=True)
    h = (h - h.min()) / (h.max() - h.min())
    h = (h * 0.5 + 0.25)[0, 0].cuda()
    h = h * (0.095 * nz / h.mean())
    occ = torch.arange(nz, device="cuda").view(-1, 1, 1) < h
    return _boxes(occ, rng, 0.025, 8, 60), h


def _explored(truth, v, poses, range_m):
    """The robot's map: unknown except for what 360x60 degree scans from the poses saw."""
    nz, ny, nx = truth.shape
    flat = truth.reshape(-1)
    grid = torch.zeros(flat.shape, dtype=torch.uint8, device="cuda")
    az = torch.deg2rad(torch.arange(0.0, 360.0, 0.5, device="cuda", dtype=torch.float64))
    el = torch.deg2rad(torch.arange(-30.0, 30.01, 0.5, device="cuda", dtype=torch.float64))
    A, E = torch.meshgrid(az, el, indexing="ij")
    d = torch.stack([E.cos() * A.cos(), E.cos() * A.sin(), E.sin()], -1).reshape(-1, 1, 3)
    t = 0.5 * torch.arange(math.ceil(2.0 * range_m / v), device="cuda", dtype=torch.float64).view(1, -1, 1)
    size = torch.tensor([nx, ny, nz], device="cuda")
    for p in poses:
        for part in d.split(20000):
            at = (torch.as_tensor(p / v, device="cuda") + t * part).floor().long()
            inside = ((at >= 0) & (at < size)).all(-1)
            lin = ((at[..., 2] * ny + at[..., 1]) * nx + at[..., 0]).masked_fill(~inside, 0)
            stop = flat[lin] | ~inside
            before = stop.long().cumsum(1) - stop.long()
            seen = (before == 0) & inside
            grid[lin[seen & ~stop]] = FREE
            grid[lin[seen & stop]] = OCCUPIED
    return grid.view(nz, ny, nx)


def _pose(rng, truth, v, height, around, spread):
    """A spot `height` voxels up (an array: above the ground there) with a little clearance."""
    nz, ny, nx = truth.shape
    for _ in range(4000):
        x, y = (int(np.clip(rng.integers(c - s, c + s + 1), 6, n - 7)) for c, s, n in zip(around, spread, (nx, ny)))
        z = min(nz - 6, int(height[y, x]) if isinstance(height, np.ndarray) else height)
        if not truth[z - 1:z + 2, y - 3:y + 4, x - 3:x + 4].any():
            return np.array([x + 0.5, y + 0.5, z + 0.5]) * v
    raise RuntimeError("no free spot")


def _world(case, rng):
    """(map codes on the host, ground truth on the host, scan poses) of a case's world."""
    nx, ny, nz, v = case["nx"], case["ny"], case["nz"], case["voxel"]
    if case["world"] == "boxes":
        truth = _boxes(torch.zeros(nz, ny, nx, dtype=torch.bool, device="cuda"), rng, 0.15, 1, 8)
        pose = np.array([nx, ny, nz]) / 2.0 * v
        z, y, x = (torch.arange(n, device="cuda") + 0.5 for n in (nz, ny, nx))
        near = ((z - nz / 2) ** 2).view(-1, 1, 1) + ((y - ny / 2) ** 2).view(1, -1, 1) + (x - nx / 2) ** 2 <= (3.0 / v) ** 2
        grid = truth.to(torch.uint8) * OCCUPIED
        grid[near] = FREE
        return grid.cpu().numpy(), (truth & ~near).cpu().numpy(), [pose]
    if case["world"] == "terrain":
        truth, h = _terrain(rng, nx, ny, nz)
        height = (h.ceil() + 1.5 / v).cpu().numpy()
    else:
        truth, height = _rooms(rng, nx, ny, nz, v), round(1.5 / v)
    host = truth.cpu().numpy()
    poses = [_pose(rng, host, v, height, (nx // 2, ny // 2), (nx // 10, ny // 10))]
    centre = [int(c / v) for c in poses[0][:2]]
    spread = int((6.0 if case["world"] == "terrain" else 8.0) / v)
    while len(poses) < 5:
        poses.append(_pose(rng, host, v, height, centre, (spread, spread)))
    return _explored(truth, v, poses, max(6.0, case["range"])).cpu().numpy(), host, poses


def _tree(rng, grid, v, root, nodes, depth, step, half, down, up):
    """An RRT in a box around its root: uniform samples, nearest node that may take a child (at most 6), edges of at
    most `step` metres that cross no occupied voxel. Returns (parent int32, position float32)."""
    size = np.array(grid.shape[::-1]) * v
    lo = np.maximum(v, root - [half, half, down])
    hi = np.minimum(size - v, root + [half, half, up])
    pos, parent = np.zeros((nodes, 3)), np.full(nodes, -1, np.int32)
    level, kids = np.zeros(nodes, np.int32), np.zeros(nodes, np.int32)
    open_ = np.zeros(nodes, bool)
    pos[0], n, open_[0] = root, 1, True
    while n < nodes:
        s = lo + rng.random(3) * (hi - lo)
        d2 = np.where(open_[:n], ((pos[:n] - s) ** 2).sum(1), np.inf)
        j = int(d2.argmin())
        dist = math.sqrt(d2[j])
        if not 1e-6 < dist < 1e30:
            continue
        q = pos[j] + (s - pos[j]) * min(1.0, step / dist)
        along = np.linspace(0.0, 1.0, max(2, math.ceil(min(step, dist) / (0.25 * v)) + 1))[:, None]
        c = ((pos[j] + along * (q - pos[j])) / v).astype(np.int64)
        if (grid[c[:, 2], c[:, 1], c[:, 0]] == OCCUPIED).any():
            continue
        pos[n], parent[n], level[n] = q, j, level[j] + 1
        open_[n] = level[n] < depth
        kids[j] += 1
        open_[j] = kids[j] < 6
        n += 1
    return parent, pos.astype(np.float32)


def _update_box(rng, truth, v):
    """A map update: a box of 10 % of the voxels, relabelled as a scan would see it."""
    nz, ny, nx = truth.shape
    side = min(nx, ny, round(math.sqrt(0.10 * nx * ny)))
    x, y = int(rng.integers(0, nx - side + 1)), int(rng.integers(0, ny - side + 1))
    return x, y, 0, np.where(truth[:, y:y + side, x:x + side], OCCUPIED, FREE).astype(np.uint8)


# ------------------------------------------------------------------------------------- the cases
class _State:
    """What a planner keeps: its context, maps, trees and (where it has one) its server."""

    def __init__(self):
        self.ctx, self.maps, self.server = None, [], None

    def __del__(self):
        if self.server is not None:
            self.server.close()
        for m in self.maps:
            m.close()
        if self.ctx is not None:
            self.ctx.close()


def _problem(case, rng, grid, poses, i):
    """(parent, pos, sensor) of the case's i-th tree; the sizes of several trees are spread over their range by i."""
    nodes, w, h = case["nodes"], case["width"], case["height"]
    if case["trees"] > 1:
        nodes = max(10, round(nodes * (0.08 + 0.92 * (i * 7 % case["trees"]) / (case["trees"] - 1))))
    if case["call"] == "batch":
        grids = [g for g in RAY_GRIDS if g[0] <= w] + [(w, h)]
        w, h = grids[i * 5 % len(grids)]
    half, down, up = (10.0, 1.5, 2.5) if case["world"] == "terrain" else (8.0, 1.0, 1.5)
    parent, pos = _tree(rng, grid, case["voxel"], poses[i // case["maps"] % len(poses)], nodes, case["depth"], case["step"], half, down, up)
    return parent, pos, mig.Sensor(case["hfov"], case["vfov"], w, h, case["range"], case["yaws"], case["pitch"])


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    s = _State()
    s.case = case
    worlds = [_world(case, rng) for _ in range(case["maps"])]
    s.updates = []
    if case["call"] in ("replan", "serving"):  # the maps as after the updates, so that every pass meets the same ones
        for i in range(case["trees"]):
            grid, truth, _ = worlds[i % len(worlds)]
            x, y, z, box = _update_box(rng, truth, case["voxel"])
            s.updates.append((x, y, z, box))
            grid[z:z + box.shape[0], y:y + box.shape[1], x:x + box.shape[2]] = box
    s.problems = [_problem(case, rng, worlds[i % len(worlds)][0], worlds[i % len(worlds)][2], i)
                  for i in range(case["trees"])]
    # batches and servers run on a stream of their own (a captured graph needs one)
    stream = torch.cuda.Stream() if case["call"] in ("batch", "serving") else None
    s.ctx = mig.Context(0, stream=stream)
    s.maps = [mig.Map(s.ctx, grid, case["voxel"]) for grid, _, _ in worlds]
    if case["call"] == "serving":
        s.server = mig.Server(s.ctx, arena_budget_bytes=8 << 30)
    if case["call"] in ("device", "noalloc"):
        parent, pos, _ = s.problems[0]
        s.depth = int(mig.tree_check(parent)[1])
        s.parent, s.pos = torch.from_numpy(parent).cuda(), torch.from_numpy(pos).cuda()
        s.out = {k: torch.empty(len(parent), dtype=torch.int32, device="cuda") for k in ("abs", "marg", "yaw")}
    return s


def run(s):
    c, call = s.case, s.case["call"]
    parent, pos, sensor = s.problems[0]
    if call == "device":
        mig.tree_eval_device(s.maps[0], s.parent, s.pos, sensor, s.depth, s.out["abs"], s.out["marg"], s.out["yaw"])
        return s.out
    if call == "noalloc":
        mig.tree_eval_device_noalloc(s.maps[0], s.parent, s.pos, sensor, s.depth, s.out["abs"], s.out["marg"], s.out["yaw"])
        return s.out
    if call == "host":
        return mig.tree_eval(s.maps[0], parent, pos, sensor, mode=MODES[c["mode"]], want_counts=c["outputs"] != "gains",
                             want_depth=c["outputs"] == "all")
    if call == "replan":
        s.maps[0].update(*s.updates[0])
        got = mig.tree_eval(s.maps[0], parent, pos, sensor)
        got["cost"], got["objective"], got["best"] = mig.tree_score(s.ctx, parent, pos, got["marg"], c["voxel"])
        return got
    on = [s.maps[i % len(s.maps)] for i in range(len(s.problems))]
    if call == "batch":
        return mig.tree_eval_batch(s.ctx, s.problems, on)
    tickets = []
    for m, update, (parent, pos, sensor) in zip(on, s.updates, s.problems):
        s.server.map_update(m, *update)
        tickets.append(s.server.submit(m, parent, pos, sensor))
    for ticket, _ in tickets:
        while not s.server.poll(ticket, timeout_us=10_000_000):
            pass
    return [out for _, out in tickets]


def work(case):
    """Bytes: the maps (one byte a voxel), trees and results once each, with the updates and diagnostic outputs where the
    case has them. Operations: each ray's direction (8: the yaw rotation) and one comparison for each voxel of its way."""
    trees, maps = case["trees"], case["maps"]
    nodes = case["nodes"] * (0.54 if trees > 1 else 1.0) * trees
    voxels = case["nx"] * case["ny"] * case["nz"]
    rays = nodes * case["yaws"] * case["width"] * case["height"] * (0.35 if case["call"] == "batch" else 1.0)
    b = maps * voxels + nodes * (16 + 12)
    if case["call"] in ("replan", "serving"):
        b += trees * 0.1 * voxels
    if case["outputs"] != "gains":
        b += nodes * 8 * case["yaws"]
    if case["outputs"] == "all":
        b += nodes * 4 * case["width"] * case["height"]
    return {"bytes": b, "flops": rays * (8 + case["range"] / case["voxel"])}


def exact(case, seed):
    """Of the computed numbers only a path's length does not hang on counts: the counts are whole numbers, and the
    objective is a sum over them. So: the cost of each node, the rest None."""
    if case["call"] != "replan":
        return None
    rng = np.random.default_rng(seed)
    grid, truth, poses = _world(case, rng)
    x, y, z, box = _update_box(rng, truth, case["voxel"])
    grid[z:z + box.shape[0], y:y + box.shape[1], x:x + box.shape[2]] = box
    parent, pos, _ = _problem(case, rng, grid, poses, 0)
    pos, cost = pos.astype(np.float64), np.zeros(len(parent))
    for i in range(1, len(parent)):  # parents come before their children
        cost[i] = cost[parent[i]] + np.linalg.norm(pos[i] - pos[parent[i]])
    return {"abs": None, "marg": None, "yaw": None, "cost": cost, "objective": None, "best": None}
