"""The workloads the framework's speed is measured on.

Each case is one kind of work a program hands to the library, through the
binding's entry points, on seeded synthetic frames made on the GPU: a box room
(walls, floor and ceiling in 1 m panels) with boxes and ellipsoids, seen from
a camera walking a closed path, 1 % depth noise and 1 % holes, the largest
visible objects as masks, patch tokens as a per-object mean plus noise.

A map is in use while it is timed: every pass takes the next frames of the
path, and each lap of the path is shifted by a few voxels (the odometry's
drift), so that passes keep finding new voxels beside the ones the map already
holds.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2603_03935_gb300 import (DiscGroup, DiscMap, DiscServer, binding, device_frame, host_frame, query_heatmap,
                                    token_stats_static)

LAPS = 24    # laps of a path before its frames come back at the poses of the first
DRIFT = 0.6  # voxels from lap to lap, along one direction
PRECISION = {"fp32": 0, "bf16": 1, "fp8": 2}
STAT_COLUMNS = [i for i, (k, _) in enumerate(binding.Stats._fields_) if k != "max_probe"]
# (max_probe, the longest hash probe, depends on the order in which threads claim slots)
ROWS = dict(frame=1 << 11, calls=1 << 12, stream=1 << 15, group=1 << 13, scan=1 << 10)
VOXELS = 1 << 20  # voxels that a scan reads out at most


def listed():
    return [
        # the smallest call: one 64x48 frame of the Tiny configuration, a low-resolution sensor's live frame
        dict(name="frame-tiny", kind="frame", width=64, height=48, masks=8, grid_h=6, grid_w=8, dim=512, voxel_mm=50,
             frames=1, dtype="f32", precision="fp32", host=False),
        # a live camera: one 640x480 frame per call, straight from pinned host memory
        dict(name="frame-live", kind="frame", width=640, height=480, masks=40, grid_h=24, grid_w=24, dim=768,
             voxel_mm=25, frames=1, dtype="f32", precision="fp32", host=True),
        # the headline: a Room-scale trajectory streamed in asynchronous 32-frame calls, inputs on the device
        dict(name="stream-room", kind="stream", width=640, height=480, masks=40, grid_h=24, grid_w=24, dim=768,
             voxel_mm=25, frames=32, calls=4, dtype="f32", precision="fp32"),
        # a large building: 100 masks, 5 cm voxels, depth to 20 m, bf16 tokens, BF16 pooling and scoring
        dict(name="stream-building", kind="stream", width=640, height=480, masks=100, grid_h=24, grid_w=24, dim=768,
             voxel_mm=50, frames=32, calls=2, dtype="bf16", precision="bf16"),
        # many robots at once: maps of uneven frame sizes and mask counts, a few frames of each per group call
        dict(name="group-mixed", kind="group", width=640, height=480, masks=60, grid_h=24, grid_w=24, dim=768,
             voxel_mm=25, frames=4, calls=2, maps=16, dtype="bf16", precision="fp32"),
        # serving: integrate and query requests of concurrent maps, host inputs read in place, FP8 pooling and scoring
        dict(name="served-fp8", kind="served", width=640, height=480, masks=40, grid_h=24, grid_w=24, dim=768,
             voxel_mm=25, frames=3, maps=12, dtype="bf16", precision="fp8"),
        # the DBSCAN noise filter before voxelisation, on a ragged frame and grid, one synchronous call
        dict(name="denoise", kind="calls", width=561, height=421, masks=33, grid_h=23, grid_w=29, dim=514, voxel_mm=25,
             frames=12, dtype="f32", precision="fp32", dbscan=True),
        # two encoders: a second (24x32x1024) token grid drives association
        dict(name="two-encoders", kind="calls", width=640, height=480, masks=40, grid_h=24, grid_w=24, dim=768,
             voxel_mm=25, frames=16, dtype="f32", precision="fp32", grid2_h=24, grid2_w=32, dim2=1024),
        # the neighbourhood overlap: a segment voxel also overlaps what labels its 26 neighbours
        dict(name="neighbourhood", kind="calls", width=640, height=480, masks=40, grid_h=24, grid_w=24, dim=768,
             voxel_mm=25, frames=16, dtype="f32", precision="fp32", neighbours=True),
        # a whole scan: a new map, its frames, the end-of-trajectory step, the voxels and instances read out
        dict(name="scan", kind="scan", width=160, height=120, masks=24, grid_h=12, grid_w=16, dim=512, voxel_mm=50,
             frames=24, dtype="f32", precision="fp32"),
        # retrieval: a list of text queries against every instance, and the instances at a cloud of points
        dict(name="query", kind="query", dim=768, instances=4000, queries=64, top=10, points=100000),
        # one image's heatmap for a text query, and its distinctiveness map
        dict(name="heatmap", kind="heatmap", grid_h=37, grid_w=37, dim=1024, dtype="bf16"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "stream", "group", "served", "calls", "calls", "scan", "query", "heatmap"])
    if kind == "query":
        return dict(kind=kind, dim=_log(rng, 128, 1024), instances=_log(rng, 200, 6000), queries=_log(rng, 1, 100),
                    top=rng.randint(1, 20), points=_log(rng, 100, 200000))
    if kind == "heatmap":
        return dict(kind=kind, grid_h=rng.randint(6, 64), grid_w=rng.randint(6, 64), dim=_log(rng, 64, 1536),
                    dtype=rng.choice(["f32", "bf16"]))
    small = kind == "scan"
    w = _log(rng, 48, 200 if small else 640)
    c = dict(kind=kind, width=w, height=max(32, w * rng.randint(55, 80) // 100), masks=_log(rng, 4, 100),
             grid_h=rng.randint(6, 24), grid_w=rng.randint(6, 32), dim=_log(rng, 128, 1024),
             voxel_mm=rng.choice([25, 40, 50]), frames=1, dtype=rng.choice(["f32", "bf16"]),
             precision=rng.choice(["fp32", "bf16", "fp8"]))
    if kind == "frame":
        c["host"] = rng.choice([True, False])
    elif kind == "stream":
        c.update(frames=rng.randint(5, 32), calls=rng.randint(1, 4))
    elif kind == "group":
        c.update(frames=rng.randint(1, 4), calls=rng.randint(1, 2), maps=rng.randint(2, 16))
    elif kind == "served":
        c.update(frames=rng.randint(1, 4), maps=rng.randint(2, 12))
    elif kind == "calls":
        c.update(frames=rng.randint(2, 16))
        option = rng.choice(["none", "dbscan", "second", "neighbours"])
        if option == "dbscan":
            c["dbscan"] = True
        elif option == "second":
            c.update(grid2_h=rng.randint(8, 24), grid2_w=rng.randint(8, 32), dim2=_log(rng, 128, 1024))
        elif option == "neighbours":
            c["neighbours"] = True
    else:
        c["frames"] = rng.randint(8, 24)
    return c


# ---- seeded scenes and frames ----------------------------------------------------


def _rotations(eyes, targets):
    """camera->world rotations (x right, y down, z forward) [n, 3, 3]."""
    z = targets - eyes
    z /= np.linalg.norm(z, axis=1, keepdims=True)
    x = np.cross(z, np.array([0.0, 0.0, 1.0]))
    x /= np.linalg.norm(x, axis=1, keepdims=True)
    return np.stack([x, np.cross(z, x), z], axis=2)


def _scene(rng, building):
    """Room size and primitives (kind, centre, half extent) off the voxel grid, clear of the camera's path."""
    size = np.array([30.0, 20.0, 3.0] if building else [10.0, 8.0, 3.0])
    mid = size / 2
    prims = []
    for _ in range(150 if building else 60):
        half = rng.uniform(0.1, 0.6, 3)
        c = np.array([rng.uniform(0.5, size[0] - 0.5), rng.uniform(0.5, size[1] - 0.5), half[2]])
        # the path runs on an ellipse at 0.6 of the half extents
        r = math.hypot((c[0] - mid[0]) / (0.6 * mid[0]), (c[1] - mid[1]) / (0.6 * mid[1]))
        if abs(r - 1.0) * 0.6 * min(mid[0], mid[1]) < 1.0:
            c[2] = size[2] - half[2]  # hangs from the ceiling
            half[2] = min(half[2], 0.3)
        prims.append((int(rng.uniform() < 0.35), c + 0.0071, half))
    return size, prims


def _path(n, size):
    s = 2 * np.pi * np.arange(n) / n
    mid = size / 2
    eyes = np.stack([mid[0] * (1 + 0.6 * np.cos(s)), mid[1] * (1 + 0.6 * np.sin(s)), np.full(n, 1.2)], 1)
    targets = np.stack([mid[0] * (1 + 0.5 * np.cos(s + 1.4)), mid[1] * (1 + 0.5 * np.sin(s + 1.4)),
                        np.full(n, 0.7)], 1)
    return eyes, _rotations(eyes, targets)


def _render(size, prims, eyes, rot, width, height, focal, gen):
    """Depth [n, H, W] and object ids [n, H, W] (panel ids after the primitives')."""
    dev = torch.device("cuda")
    n = len(eyes)
    u = (torch.arange(width, device=dev, dtype=torch.float32) + 0.5 - width / 2) / focal
    v = (torch.arange(height, device=dev, dtype=torch.float32) + 0.5 - height / 2) / focal
    cam = torch.stack([u.expand(height, width), v[:, None].expand(height, width),
                       torch.ones(height, width, device=dev)]).reshape(3, 1, -1)
    r = torch.tensor(rot, dtype=torch.float32, device=dev).permute(1, 2, 0)  # [3, 3, n]
    o = torch.tensor(eyes, dtype=torch.float32, device=dev).t()[:, :, None]  # [3, n, 1]
    d = r[:, 0, :, None] * cam[0] + r[:, 1, :, None] * cam[1] + r[:, 2, :, None] * cam[2]  # [3, n, HW]
    d = torch.where(d.abs() < 1e-9, torch.full_like(d, 1e-9), d)
    inv = 1.0 / d
    hi = torch.tensor(size, dtype=torch.float32, device=dev)[:, None, None] - 0.0071
    t, axis = torch.where(d > 0, (hi - o) * inv, (-0.0071 - o) * inv).min(0)
    p = o + t * d
    nx, ny, nz = (int(math.ceil(x)) + 1 for x in size)
    q = [p[a].floor().long().clamp(0, m) for a, m in enumerate((nx, ny, nz))]
    b0, b1 = torch.where(axis == 0, q[1], q[0]), torch.where(axis == 2, q[1], q[2])
    side = (d.gather(0, axis[None])[0] > 0).long()
    ids = len(prims) + 1 + ((axis * 2 + side) * 64 + b0) * 32 + b1
    for i, (kind, c, h) in enumerate(prims):
        c = torch.tensor(c, dtype=torch.float32, device=dev)[:, None, None]
        h = torch.tensor(h, dtype=torch.float32, device=dev)[:, None, None]
        if kind == 0:
            a, b = (c - h - o) * inv, (c + h - o) * inv
            near, far = torch.minimum(a, b).amax(0), torch.maximum(a, b).amin(0)
            hit = (near <= far) & (near > 0.05) & (near < t)
        else:
            e, f = (o - c) / h, d / h
            qa, qb, qc = (f * f).sum(0), (e * f).sum(0), (e * e).sum(0) - 1.0
            disc = qb * qb - qa * qc
            near = (-qb - disc.clamp(min=0).sqrt()) / qa
            hit = (disc > 0) & (near > 0.05) & (near < t)
        t = torch.where(hit, near, t)
        ids = torch.where(hit, torch.full_like(ids, i + 1), ids)
    t = t * (1.0 + 0.01 * torch.randn(t.shape, device=dev, generator=gen))
    t = torch.where(torch.rand(t.shape, device=dev, generator=gen) < 0.01, torch.zeros_like(t), t)
    return t.reshape(n, height, width).contiguous(), ids.reshape(n, height, width)


def _masks(ids, count):
    """Labels [n, H, W] (1..count, largest objects first; ties by id) and masks per frame."""
    n = ids.shape[0]
    top = int(ids.max()) + 1
    hist = torch.zeros(n, top, dtype=torch.int64, device=ids.device)
    hist.scatter_add_(1, ids.reshape(n, -1), torch.ones_like(ids.reshape(n, -1)))
    order = (hist * (top + 1) + torch.arange(top, 0, -1, device=ids.device)).topk(min(count, top), dim=1).indices
    present = hist.gather(1, order) > 0
    lut = torch.zeros(n, top, dtype=torch.int64, device=ids.device)
    lut.scatter_(1, order, torch.arange(1, order.shape[1] + 1, device=ids.device) * present)
    labels = lut.gather(1, ids.reshape(n, -1)).reshape(ids.shape).to(torch.int16)
    return labels.contiguous(), present.sum(1).tolist()


def _tokens(ids, grid_h, grid_w, dim, dtype, gen):
    n, height, width = ids.shape
    v = ((torch.arange(grid_h, device=ids.device) * 2 + 1) * height) // (2 * grid_h)
    u = ((torch.arange(grid_w, device=ids.device) * 2 + 1) * width) // (2 * grid_w)
    at = ids[:, v][:, :, u].reshape(n, -1)
    mean = torch.randn(int(ids.max()) + 1, dim, device=ids.device, generator=gen)
    out = mean[at]
    out += 0.1 * torch.randn(out.shape, device=ids.device, generator=gen)
    return out.to(torch.bfloat16 if dtype == "bf16" else torch.float32).contiguous()


class _Frames:
    """A ring of frames, each batch of them as ctypes arrays for every lap."""

    def __init__(self, case, seed, batch, batches, width=None, height=None, masks=None, host=False):
        rng = np.random.default_rng(seed)
        gen = torch.Generator(device="cuda").manual_seed(seed)
        n = batch * batches
        width, height = width or case["width"], height or case["height"]
        building = case["masks"] >= 90
        size, prims = _scene(rng, building)
        self.size = size
        self.z_max = 20.0 if building else 10.0
        # the first n frames of a loop of 512 (a scan walks one loop whole)
        eyes, rot = _path(n if case["kind"] == "scan" else max(n, 512), size)
        eyes, rot = eyes[:n], rot[:n]
        focal = 525.0 * width / 640.0
        step = max(1, 12_000_000 // (width * height))
        depth, ids = (torch.cat(x) for x in zip(*[_render(size, prims, eyes[i:i + step], rot[i:i + step], width, height,
                                                          focal, gen) for i in range(0, n, step)]))
        labels, counts = _masks(ids, masks or case["masks"])
        tokens = _tokens(ids, case["grid_h"], case["grid_w"], case["dim"], case["dtype"], gen)
        second = None
        if case.get("dim2"):
            second = _tokens(ids, case["grid2_h"], case["grid2_w"], case["dim2"], case["dtype"], gen)
        self.poses = np.tile(np.eye(4), (n, 1, 1))
        self.poses[:, :3, :3] = rot
        self.poses[:, :3, 3] = eyes
        self.intr = (focal, focal, width / 2.0, height / 2.0)
        self.depth, self.labels, self.tokens, self.counts, self.second = depth, labels, tokens, counts, second
        self.frames = []
        if host:
            pin = [x.cpu().pin_memory() for x in (depth, labels, tokens.view(torch.int16) if case["dtype"] == "bf16"
                                                  else tokens)]
            self.keep = pin
            hd, hl, ht = pin[0].numpy(), pin[1].numpy().view(np.uint16), pin[2].numpy()
            ht = ht.view(np.uint16) if case["dtype"] == "bf16" else ht
            self.frames = [host_frame(hd[i], hl[i], ht[i], self.poses[i], self.intr, counts[i]) for i in range(n)]
        else:
            self.frames = [device_frame(depth[i], labels[i], tokens[i], self.poses[i], self.intr, counts[i],
                                        assoc_tokens=None if second is None else second[i]) for i in range(n)]
        drift = np.arange(LAPS)[:, None] * np.array([0.8, 0.52, 0.3]) * 1e-3 * DRIFT * case["voxel_mm"]
        at = binding.Frame.T_world_cam.offset
        one = ctypes.sizeof(binding.Frame)
        ring = (binding.Frame * n)()
        for i, (f, _) in enumerate(self.frames):
            ring[i] = f
        raw = np.frombuffer(ring, np.uint8).reshape(n, one)
        self.batches = []
        for lap in range(LAPS):
            a = (binding.Frame * n)()
            w = np.frombuffer(a, np.uint8).reshape(n, one)
            w[:] = raw
            pose = w[:, at:at + 128].copy().view(np.float64)
            pose[:, 3:12:4] += drift[lap]
            w[:, at:at + 128] = pose.view(np.uint8)
            for b in range(batches):
                self.batches.append((binding.Frame * batch).from_buffer(a, b * batch * one))
        self.batch, self.at = batch, 0

    def next(self):
        b = self.batches[self.at]
        self.at = (self.at + 1) % len(self.batches)
        return b


def _min_pixels(case, width, height):
    """Masks smaller than this are ignored: with many masks a frame, those of a patch or two only."""
    return width * height // (200 if case["masks"] >= 90 else 400)


def _config(case, frames, width=None, height=None, masks=None, **more):
    width, height = width or case["width"], height or case["height"]
    c = dict(voxel_size=case["voxel_mm"] / 1000.0, z_min=0.1, z_max=frames.z_max, embed_dim=case["dim"],
             patch_h=case["grid_h"], patch_w=case["grid_w"], max_width=width, max_height=height,
             max_masks=masks or case["masks"], min_mask_pixels=_min_pixels(case, width, height), max_load=0.5,
             voxel_capacity=1 << 22, instance_capacity=1 << 12, precision=PRECISION[case["precision"]])
    if case.get("dbscan"):
        c.update(dbscan_eps=0.05, dbscan_min_pts=10)
    if case.get("neighbours"):
        c["overlap_dilation"] = 1
    if case.get("dim2"):
        c.update(assoc_dim=case["dim2"], assoc_patch_h=case["grid2_h"], assoc_patch_w=case["grid2_w"])
    c.update(more)
    return c


class _Table:
    """Host arrays that a map's instance table is read into: as many rows as the map will ever hand out ids, zero past
    the last one."""

    def __init__(self, rows, case):
        self.out = dict(parent=np.zeros(rows, np.int32), count=np.zeros(rows, np.int64), Q=np.zeros(rows, np.float32),
                        E=np.zeros((rows, case["dim"]), np.float32), n_obs=np.zeros(rows, np.int32))
        if case.get("dim2"):
            self.out["A"] = np.zeros((rows, case["dim2"]), np.float32)
        self.rows = rows

    def read(self, gmap):
        o, lib = self.out, binding.lib()
        rc = lib.disc_map_export_instances(gmap._h, *[o[k].ctypes.data for k in ("parent", "count", "Q", "E", "n_obs")],
                                           self.rows)
        if rc == 0 and "A" in o:
            rc = lib.disc_map_export_assoc(gmap._h, o["A"].ctypes.data, self.rows)
        if rc:
            raise RuntimeError(f"the instance table was not read out: {rc}")
        return o


def _stats(*arrays):
    """The per-frame counters of the calls [frames, counters]."""
    n = len(binding.Stats._fields_)
    return np.concatenate([np.frombuffer(a, np.int32).reshape(-1, n) for a in arrays])[:, STAT_COLUMNS]


# ---- the cases ---------------------------------------------------------------------


def prepare(case, seed):
    kind = case["kind"]
    if kind == "heatmap":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        p, d = case["grid_h"] * case["grid_w"], case["dim"]
        objects = torch.randn(24, d, device="cuda", generator=gen)
        rows = torch.arange(p, device="cuda") // case["grid_w"] // 6 * 4 + torch.arange(p, device="cuda") % case["grid_w"] // 10
        tokens = objects[rows % 24] + 0.1 * torch.randn(p, d, device="cuda", generator=gen)
        query = objects[5] + 0.3 * torch.randn(d, device="cuda", generator=gen)
        if case["dtype"] == "bf16":
            tokens = tokens.to(torch.bfloat16)
        return dict(kind=kind, tokens=tokens.contiguous(), query=query.contiguous())
    if kind == "query":
        return _prepare_query(case, seed)
    if kind == "group":
        sizes = ((1.0, 1.0), (0.75, 0.75), (0.5, 0.5), (0.877, 0.879))
        limits = (1.0, 0.1, 0.67, 0.42, 0.25, 0.84)
        rings, maps = [], []
        for g in range(case["maps"]):
            w, h = (max(32, int(case["width"] * sizes[g % 4][0])), max(24, int(case["height"] * sizes[g % 4][1])))
            m = max(2, int(case["masks"] * limits[g % 6]))
            rings.append(_Frames(case, seed * 131 + g, case["frames"], 2, w, h, m))
            maps.append(DiscMap(**_config(case, rings[-1], w, h, m, voxel_capacity=1 << 21)))
        group = DiscGroup(max_maps=case["maps"], frames_per_map=case["frames"], embed_dim=case["dim"],
                          patch_h=case["grid_h"], patch_w=case["grid_w"], max_width=case["width"],
                          max_height=case["height"], max_masks=max(2, case["masks"]))
        return dict(kind=kind, group=group, maps=maps, rings=rings, calls=case["calls"], frames=case["frames"],
                    tables=[_Table(ROWS[kind], case) for _ in maps])
    if kind == "served":
        sizes = ((1.0, 1.0), (0.5, 0.5), (0.75, 0.75))
        server = DiscServer(64 << 30, max_queue=4096, workers=2, max_maps=case["maps"], frames_per_map=case["frames"],
                            embed_dim=case["dim"], patch_h=case["grid_h"], patch_w=case["grid_w"],
                            max_width=case["width"], max_height=case["height"], max_masks=case["masks"])
        rings, ids, queries = [], [], []
        for g in range(case["maps"]):
            w, h = (max(32, int(case["width"] * sizes[g % 3][0])), max(24, int(case["height"] * sizes[g % 3][1])))
            rings.append(_Frames(case, seed * 137 + g, case["frames"], 2, w, h, host=True))
            ids.append(server.open_map(**_config(case, rings[-1], w, h, voxel_capacity=1 << 21)))
            queries.append(rings[-1].tokens[0, :4].float().cpu().numpy())
        return dict(kind=kind, server=server, rings=rings, ids=ids, queries=queries)
    if kind == "scan":
        ring = _Frames(case, seed, case["frames"], 1)
        return dict(kind=kind, ring=ring, config=_config(case, ring, voxel_capacity=1 << 16, instance_capacity=256),
                    keys=np.zeros(VOXELS, np.uint64), ids=np.zeros(VOXELS, np.int32), case=case)
    calls = case.get("calls", 1)
    ring = _Frames(case, seed, case["frames"], 16 if kind == "frame" else max(4 * calls, 4), host=case.get("host", False))
    table = 1 << (25 if case["frames"] * calls * case["width"] * case["height"] > 8_000_000 else 22)
    gmap = DiscMap(**_config(case, ring, voxel_capacity=table))
    return dict(kind=kind, ring=ring, map=gmap, calls=calls, frames=case["frames"], table=_Table(ROWS[kind], case))


def run(state):
    kind = state["kind"]
    if kind == "frame":
        stats = state["map"].integrate((state["ring"].next()[0], None))
        del stats["max_probe"]
        return [stats, state["table"].read(state["map"])]
    if kind == "calls":
        n = state["frames"]
        stats = (binding.Stats * n)()
        rc = state["map"].integrate_frames_raw(state["ring"].next(), n, stats)
        return [rc, _stats(stats), state["table"].read(state["map"])]
    if kind == "stream":
        n = state["frames"]
        stats = [(binding.Stats * n)() for _ in range(state["calls"])]
        for s in stats:
            rc = state["map"].integrate_frames_async_raw(state["ring"].next(), n, s)
            if rc:
                break
        rc = rc or state["map"].wait()
        return [rc, _stats(*stats), state["table"].read(state["map"])]
    if kind == "group":
        maps, n = state["maps"], state["frames"]
        stats = []
        for _ in range(state["calls"]):
            stats.append([(binding.Stats * n)() for _ in maps])
            rc = state["group"].integrate_async_raw(maps, [r.next() for r in state["rings"]], [n] * len(maps), stats[-1])
            if rc:
                break
        rc = rc or state["group"].wait()
        tables = [t.read(m) for t, m in zip(state["tables"], maps)]
        # (64 outputs at most: the embeddings one by one, the small columns side by side)
        return [rc, _stats(*[s for call in stats for s in call]), [t["E"] for t in tables],
                {k: np.stack([t[k] for t in tables]) for k in ("parent", "count", "Q", "n_obs")}]
    if kind == "served":
        server = state["server"]
        batches = [r.next() for r in state["rings"]]
        tickets = [server.submit_frame_borrowed(i, (f, None)) for j in range(len(batches[0]))
                   for i, f in zip(state["ids"], [b[j] for b in batches])]
        asked = [server.submit_query(i, q, 5) for i, q in zip(state["ids"], state["queries"])]
        stats = [server.wait_frame(t) for t in tickets]
        found = [server.wait_query(t) for t in asked]
        names = [k for k in stats[0] if k not in ("max_probe", "latency_ms")]
        return [np.array([[s[k] for k in names] for s in stats]), np.stack([f[1] for f in found]),
                np.stack([f[2] for f in found])]
    if kind == "scan":
        gmap = DiscMap(**state["config"])
        stats = (binding.Stats * state["ring"].batch)()
        rc = gmap.integrate_frames_raw(state["ring"].next(), state["ring"].batch, stats)
        report = gmap.finalize(20)
        keys, ids = state["keys"], state["ids"]
        voxels, _ = gmap.counts()
        rc = rc or binding.lib().disc_map_export_voxels(gmap._h, keys.ctypes.data, ids.ctypes.data, len(keys))
        keys[voxels:], ids[voxels:] = 0, 0
        table = _Table(ROWS[kind], state["case"]).read(gmap)
        gmap.close()
        return [rc, _stats(stats), report, keys, ids, table]
    if kind == "query":
        ids, scores = state["map"].query_topk(state["queries"], state["top"])
        return [ids, scores, state["map"].query_points(state["points"])]
    dp, cosg = token_stats_static(state["tokens"])
    return [query_heatmap(state["tokens"], state["query"]), dp, cosg]


# ---- retrieval: a map of known instances ---------------------------------------------
# One frame per block of instances: a wall at 2 m cut into 8x8-pixel masks, each
# frame 40 m from the last, so every mask opens an instance of its own.

_CELLS = (12, 8)  # masks across and down
_W, _H = _CELLS[0] * 8, _CELLS[1] * 8


def _query_inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    per = _CELLS[0] * _CELLS[1]
    n = -(-case["instances"] // per)
    tokens = torch.randn(n, per, case["dim"], device="cuda", generator=gen)
    picks = torch.randint(0, n * per, (case["queries"],), device="cuda", generator=gen)
    queries = tokens.reshape(-1, case["dim"])[picks]
    queries = queries + 0.5 * torch.randn(queries.shape, device="cuda", generator=gen)
    xyz = torch.rand(case["points"], 3, device="cuda", generator=gen)
    frame = torch.randint(0, n, (case["points"],), device="cuda", generator=gen)
    # points in a slab around the walls: most on a mapped voxel's layer, some beside it
    xyz = torch.stack([(xyz[:, 0] - 0.5) * 2.4 + 40.0 * frame, (xyz[:, 1] - 0.5) * 1.6, 1.95 + 0.1 * xyz[:, 2]], 1)
    return tokens, queries, xyz, n, per


def _prepare_query(case, seed):
    tokens, queries, xyz, n, per = _query_inputs(case, seed)
    depth = torch.full((_H, _W), 2.0, device="cuda")
    v, u = torch.arange(_H, device="cuda")[:, None] // 8, torch.arange(_W, device="cuda")[None, :] // 8
    labels = (v * _CELLS[0] + u + 1).to(torch.int16).contiguous()
    gmap = DiscMap(voxel_size=0.025, embed_dim=case["dim"], patch_h=_CELLS[1], patch_w=_CELLS[0], max_width=_W,
                   max_height=_H, max_masks=per, min_mask_pixels=1, voxel_capacity=1 << 20, max_load=0.5,
                   instance_capacity=1 << 13)
    frames = []
    for i in range(n):
        pose = np.eye(4)
        pose[0, 3] = 40.0 * i
        frames.append(device_frame(depth, labels, tokens[i], pose, (80.0, 80.0, _W / 2.0, _H / 2.0), per))
    torch.cuda.synchronize()
    gmap.integrate_frames(frames)
    return dict(kind="query", map=gmap, queries=queries.cpu().numpy(), points=xyz.cpu().numpy(), top=case["top"])


def work(case):
    kind = case["kind"]
    if kind == "query":
        n, q, d = case["instances"], case["queries"], case["dim"]
        return dict(bytes=4 * d * (n + q) + 8 * q * case["top"] + 28 * case["points"], flops=2 * n * q * d)
    size = 2 if case["dtype"] == "bf16" else 4
    p = case["grid_h"] * case["grid_w"]
    if kind == "heatmap":  # two calls on the same grid
        return dict(bytes=2 * p * case["dim"] * size + 12 * p, flops=2 * 8 * p * case["dim"])
    scale = {"group": 0.65, "served": 0.6}.get(kind, 1.0)  # frames of uneven size
    px = case["width"] * case["height"] * scale
    n = case["frames"] * case.get("calls", 1) * case.get("maps", 1)
    tokens = p * case["dim"]
    pooled = 2 * case["masks"] * tokens
    grid2 = case.get("grid2_h", 0) * case.get("grid2_w", 0) * case.get("dim2", 0)
    pooled += 2 * case["masks"] * grid2
    return dict(bytes=int(n * (6 * px + size * (tokens + grid2))), flops=int(n * (pooled + 8 * tokens + 60 * px)))


# ---- the same results in 64 bits -------------------------------------------------------


def _distinctiveness(tokens, query=None):
    """Eq. 1's D_p and each token's cosine with the query (default: the mean token)."""
    f = tokens.double()
    mean = f.mean(0)
    norm = (f - mean).norm(dim=1)
    g = mean if query is None else query.double()
    return norm / (norm.mean() + 1e-6), (f @ g) / (f.norm(dim=1) * g.norm())


def exact(case, seed):
    kind = case["kind"]
    if kind == "heatmap":
        s = prepare(case, seed)
        dp, cosg = _distinctiveness(s["tokens"])
        return [dp * _distinctiveness(s["tokens"], s["query"])[1], dp, cosg]
    if kind == "query":
        # every mask covers one patch: its embedding is that patch's token
        tokens, queries, _, _, _ = _query_inputs(case, seed)
        e, q = tokens.reshape(-1, case["dim"]).double(), queries.double()
        scores = (q @ e.t()) / (q.norm(dim=1)[:, None] * e.norm(dim=1))
        return [None, scores.topk(case["top"], dim=1).values.cpu(), None]
    if kind == "frame":
        return _exact_frame(case, seed)
    return None  # what a map of many frames holds follows its integer decisions frame by frame


def _exact_frame(case, seed):
    """The first frame's instances: every mask with a voxel opens one, in mask order."""
    s = prepare(case, seed)
    r = s["ring"]
    depth, labels, tokens = r.depth[0], r.labels[0].long(), r.tokens[0].double()
    height, width = depth.shape
    masks = r.counts[0]
    gh, gw = case["grid_h"], case["grid_w"]
    dp, _ = _distinctiveness(tokens)
    v = torch.arange(height, device="cuda")[:, None].expand(height, width) * gh // height
    u = torch.arange(width, device="cuda")[None, :].expand(height, width) * gw // width
    cov = torch.zeros((masks + 1) * gh * gw, dtype=torch.float64, device="cuda")
    inside = torch.where(labels <= masks, labels, torch.zeros_like(labels))
    cov.scatter_add_(0, (inside * gh * gw + v * gw + u).reshape(-1), torch.ones(height * width, dtype=torch.float64,
                                                                                device="cuda"))
    cov = cov.reshape(masks + 1, -1)[1:]
    weights = cov * dp
    pooled = (weights / weights.sum(1, keepdim=True).clamp(min=1e-300)) @ tokens
    pixels = cov.sum(1)
    seen = torch.zeros(masks + 1, dtype=torch.bool, device="cuda")
    seen[labels[(depth >= 0.1) & (depth <= r.z_max)]] = True
    keep = (pixels >= max(1, _min_pixels(case, width, height))) & seen[1:]
    out = torch.zeros(ROWS["frame"], case["dim"], dtype=torch.float64)
    out[:int(keep.sum())] = pooled[keep].cpu()
    return [None, dict(E=out)]
