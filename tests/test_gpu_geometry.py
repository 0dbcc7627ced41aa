"""Back-projection records and their gathering into (segment, voxel) entries,
at the edges of the partitions: every frame's voxel sets, normals (S_angle)
and counters equal the oracle's bit for bit."""
import ctypes

import numpy as np
import pytest

import oracle
from tests import common

pytestmark = pytest.mark.gpu

W, H, GRID, DIM = 64, 48, (6, 8), 32
MASK64 = (1 << 64) - 1


def _mix64(z):
    z = (z + 0x9E3779B97F4A7C15) & MASK64
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & MASK64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & MASK64
    return z ^ (z >> 31)


def _wall(width, height, z, tilt, voxel, f=50.0):
    """Depth of a tilted wall and the voxel key of every pixel (fp32, as the library computes it)."""
    u, v = np.meshgrid(np.arange(width, dtype=np.float32), np.arange(height, dtype=np.float32))
    depth = (z + tilt * (u + 0.37 * v)).astype(np.float32)
    inv_f, inv_s = np.float32(1) / np.float32(f), np.float32(1) / np.float32(voxel)
    x = ((u + np.float32(0.5) - np.float32(width / 2)) * depth) * inv_f
    y = ((v + np.float32(0.5) - np.float32(height / 2)) * depth) * inv_f
    k = [np.floor(a * inv_s).astype(np.int64) + (1 << 17) for a in (x, y, depth)]
    return depth, (k[0] << 36) | (k[1] << 18) | k[2]


def _one_partition(keys, parts, masks):
    """Labels that send every pixel's record to partition 0 (the key's top hash bits), so that it holds the whole
    frame: more records than its region and more distinct keys than one walk takes."""
    labels = np.zeros(keys.shape, np.uint16)
    for i, key in enumerate(keys.reshape(-1).tolist()):
        for m in range(1, masks + 1):
            m = (m + 7 * i) % masks + 1
            if ((_mix64((m << 54) | key) >> 32) * parts) >> 32 == 0:
                labels.reshape(-1)[i] = m
                break
    assert (labels > 0).mean() > 0.99
    return labels


@pytest.mark.parametrize("case", ["one_voxel", "few_voxels", "rows", "distinct", "one_partition", "ragged", "smallest"])
def test_records_at_the_partition_edges(case):
    import torch
    from paper_2603_03935_gb300 import DiscMap, device_frame
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(3)
    width, height, masks, voxel, z, tilt = W, H, 8, 0.02, 2.0, 0.004
    if case == "one_voxel":      # every pixel of a tile in a voxel or two: tiles merge
        voxel, z, tilt = 0.8, 0.3, 0.0
    elif case == "few_voxels":   # merged tiles, voxels crossing tiles
        voxel, z = 0.2, 1.0
    elif case == "rows":         # half the pixels share their row neighbour's voxel: the merge rule's line
        voxel, z, tilt = 0.08, 2.0, 0.0
    elif case == "ragged":
        width, height = 61, 35
    elif case == "smallest":
        width, height, masks = 3, 2, 2
    elif case == "one_partition":
        masks = 60
    depth, keys = _wall(width, height, z, tilt, voxel)
    if case == "one_partition":
        labels = _one_partition(keys, -(-width * height // 512), masks)
    else:
        labels = ((np.arange(height)[:, None] // 6 + np.arange(width)[None, :] // 9) % masks + 1).astype(np.uint16)
        depth[rng.uniform(size=depth.shape) < 0.03] = 0.0  # holes
    tokens = rng.normal(size=(GRID[0] * GRID[1], DIM)).astype(np.float32)
    cfg = dict(voxel_size=voxel, embed_dim=DIM, patch_h=GRID[0], patch_w=GRID[1], max_width=width, max_height=height,
               max_masks=masks, min_mask_pixels=1, voxel_capacity=1 << 14, max_load=0.5, instance_capacity=256,
               z_min=0.1, z_max=10.0, eps=1e-6, tau_cos=0.75, lambda_size=3.3, ov_num=1, ov_den=5)
    gmap, omap = DiscMap(**cfg), oracle.OracleMap(**common.to_oracle_cfg(cfg))
    intr = (50.0, 50.0, width / 2.0, height / 2.0)
    for i in range(2):  # the second frame reuses the slot
        pose = np.eye(4)
        pose[0, 3] = 0.013 * i
        fr = device_frame(torch.from_numpy(depth).to(dev), torch.from_numpy(labels.view(np.int16)).to(dev),
                          torch.from_numpy(tokens).to(dev), pose, intr, masks)
        st = gmap.integrate(fr)
        o = omap.integrate(depth, labels, tokens, pose, intr, masks)
        common.compare_frame(st, gmap.last_frame(), o, ctx=f"{case} frame {i}")
    common.compare_maps(gmap, omap, ctx=case)
    if case == "distinct":
        assert st["unique_seg_voxels"] > 0.9 * st["valid_pixels"]
    if case in ("one_voxel", "few_voxels"):
        assert st["unique_seg_voxels"] < 0.2 * st["valid_pixels"]
    gmap.close()


@pytest.mark.parametrize("probe_width", [1, 2, 8])
def test_skewed_voxel_tables_use_every_slot(probe_width):
    """Voxels two apart share one place of their blocks' eight slots: a table at 3/4 load has to place most of them
    in the other places, and every lookup has to find them there."""
    import torch
    from paper_2603_03935_gb300 import DiscMap, device_frame
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(5)
    cfg = dict(voxel_size=0.02, embed_dim=DIM, patch_h=GRID[0], patch_w=GRID[1], max_width=W, max_height=H, max_masks=8,
               min_mask_pixels=1, voxel_capacity=1 << 12, max_load=0.9, instance_capacity=64, z_min=0.1, z_max=10.0,
               eps=1e-6, tau_cos=0.75, lambda_size=3.3, ov_num=1, ov_den=5)
    gmap, omap = DiscMap(**cfg), oracle.OracleMap(**common.to_oracle_cfg(cfg))
    gmap.set_schedule(probe_width=probe_width)
    depth = np.full((H, W), 2.0, np.float32)
    labels = ((np.arange(H)[:, None] // 12 + np.arange(W)[None, :] // 16) % 8 + 1).astype(np.uint16)
    tokens = rng.normal(size=(GRID[0] * GRID[1], DIM)).astype(np.float32)
    intr = (50.0, 50.0, W / 2 - 0.25, H / 2 - 0.25)  # 0.04 m from pixel to pixel, each in the middle of its voxel
    for i in range(3):
        pose = np.eye(4)
        pose[2, 3] = 0.01
        pose[0, 3] = (0.0, 0.64, 0.0)[i]  # the second frame covers half of the first and new voxels
        st = gmap.integrate(device_frame(torch.from_numpy(depth).to(dev), torch.from_numpy(labels.view(np.int16)).to(dev),
                                         torch.from_numpy(tokens).to(dev), pose, intr, 8))
        o = omap.integrate(depth, labels, tokens, pose, intr, 8)
        common.compare_frame(st, gmap.last_frame(), o, ctx=f"frame {i}")
        if i == 0:
            assert st["unique_seg_voxels"] == W * H and gmap.cfg["voxel_capacity"] == 1 << 12
    common.compare_maps(gmap, omap, ctx="skewed")
    keys, ids = gmap.voxels()
    k = [((keys >> np.uint64(s)).astype(np.int64) & 0x3ffff) - (1 << 17) for s in (36, 18, 0)]
    xyz = (np.stack(k, 1) + 0.5) * 0.02
    assert np.array_equal(gmap.query_points(xyz.astype(np.float32)), ids)
    gmap.close()


def _sparse(kind, depth, labels):
    """Every other column, a checkerboard, every other row, or every other column of every fourth row of depth, or two
    labels in a checkerboard."""
    v, u = np.meshgrid(np.arange(depth.shape[0]), np.arange(depth.shape[1]), indexing="ij")
    if kind == "labels":
        return depth, np.where((u + v) % 2 == 1, (labels - 1) // 2 * 2 + 1, (labels - 1) // 2 * 2 + 2).astype(np.uint16)
    keep = {"columns": u % 2 == 0, "checker": (u + v) % 2 == 0, "rows": v % 2 == 1,
            "beams": (u % 2 == 0) & (v % 4 == 0)}[kind]
    return np.where(keep, depth, 0.0).astype(np.float32), labels


@pytest.mark.parametrize("kind", ["columns", "checker", "rows", "beams", "labels"])
@pytest.mark.parametrize("voxel", [0.01, 0.06, 0.9])
def test_sparse_frames_equal_the_oracle(kind, voxel):
    import torch
    from paper_2603_03935_gb300 import DiscMap, device_frame
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(9)
    width, height, masks = 131, 75, 6
    depth, _ = _wall(width, height, 1.5, 0.002, voxel)
    labels = ((np.arange(height)[:, None] // 20 + np.arange(width)[None, :] // 30) % masks + 1).astype(np.uint16)
    depth, labels = _sparse(kind, depth, labels)
    tokens = rng.normal(size=(GRID[0] * GRID[1], DIM)).astype(np.float32)
    cfg = dict(voxel_size=voxel, embed_dim=DIM, patch_h=GRID[0], patch_w=GRID[1], max_width=width, max_height=height,
               max_masks=masks, min_mask_pixels=1, voxel_capacity=1 << 15, max_load=0.5, instance_capacity=256,
               z_min=0.1, z_max=10.0, eps=1e-6, tau_cos=0.75, lambda_size=3.3, ov_num=1, ov_den=5)
    gmap, omap = DiscMap(**cfg), oracle.OracleMap(**common.to_oracle_cfg(cfg))
    intr = (50.0, 50.0, width / 2.0, height / 2.0)
    st = gmap.integrate(device_frame(torch.from_numpy(depth).to(dev), torch.from_numpy(labels.view(np.int16)).to(dev),
                                     torch.from_numpy(tokens).to(dev), np.eye(4), intr, masks))
    o = omap.integrate(depth, labels, tokens, np.eye(4), intr, masks)
    common.compare_frame(st, gmap.last_frame(), o, ctx=f"{kind}, voxels of {voxel}")
    common.compare_maps(gmap, omap, ctx=kind)
    gmap.close()


@pytest.mark.parametrize("kind", ["columns", "checker", "labels"])
def test_holes_do_not_cost_more_than_the_pixels_they_replace(kind):
    # Coarse voxels: nearly every pixel shares its voxel with its tile's others, and has to be merged with them
    # whatever lies between them. Half the pixels (or as many, under two labels) take no more than twice the time of
    # all of them; unmerged, a voxel's records pile up in one partition (over ten times).
    import torch
    from paper_2603_03935_gb300 import DiscMap, device_frame
    dev = torch.device("cuda:0")
    width, height, masks, n = 640, 480, 8, 16
    dense, _ = _wall(width, height, 2.0, 0.001, 0.5, f=525.0)
    whole = ((np.arange(height)[:, None] // 240 + np.arange(width)[None, :] // 160 * 2) % masks + 1).astype(np.uint16)
    tokens = torch.randn(GRID[0] * GRID[1], DIM, device=dev)
    intr = (525.0, 525.0, width / 2.0, height / 2.0)
    ms = []
    for depth, labels in ((dense, whole), _sparse(kind, dense, whole)):
        gmap = DiscMap(voxel_size=0.5, embed_dim=DIM, patch_h=GRID[0], patch_w=GRID[1], max_width=width,
                       max_height=height, max_masks=masks, min_mask_pixels=1, voxel_capacity=1 << 14, max_load=0.5,
                       instance_capacity=1024, z_min=0.1, z_max=10.0, batch_frames=n)
        fr = device_frame(torch.from_numpy(depth).to(dev), torch.from_numpy(labels.view(np.int16)).to(dev), tokens,
                          np.eye(4), intr, masks)
        best = 1e9
        for _ in range(4):
            gmap.set_phase_timing(True)
            gmap.integrate_frames([fr] * n)
            ph = gmap.phase_times()
            best = min(best, ph["backproject"]["ms"] + ph["entries"]["ms"])
        ms.append(best)
        gmap.close()
    assert ms[1] < 2 * ms[0], ms


@pytest.mark.parametrize("probe_width", [1, 2, 4, 8])
@pytest.mark.parametrize("capacity,first,more,place", [(64, 20, 12, 5), (256, 100, 60, 0), (512, 250, 90, 7)])
def test_more_voxels_of_one_place_than_groups(capacity, first, more, place, probe_width):
    """Voxels picked by the table's own hash: more of them have their home in one place of their groups of eight than
    there are groups, so the probe sequence has to go once round and on to the next place; then the table grows."""
    import torch
    from paper_2603_03935_gb300 import DiscMap, binding, device_frame
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(capacity)
    cfg = dict(voxel_size=0.02, embed_dim=DIM, patch_h=GRID[0], patch_w=GRID[1], max_width=W, max_height=H, max_masks=8,
               min_mask_pixels=1, voxel_capacity=capacity, max_load=0.7, instance_capacity=64, z_min=0.1, z_max=10.0,
               eps=1e-6, tau_cos=0.75, lambda_size=3.3, ov_num=1, ov_den=5)
    gmap, omap = DiscMap(**cfg), oracle.OracleMap(**common.to_oracle_cfg(cfg))
    gmap.set_schedule(probe_width=probe_width)
    cx, cy = W / 2 - 0.25, H / 2 - 0.25  # 0.04 m from pixel to pixel, each in the middle of its voxel
    u, v = np.meshgrid(np.arange(W), np.arange(H))
    kx, ky = (np.floor((a + 0.5 - c) * 0.04 / 0.02).astype(np.int64) + (1 << 17) for a, c in ((u, cx), (v, cy)))
    keys = (kx << 36) | (ky << 18) | (int(2.01 / 0.02) + (1 << 17))
    low = (1 << 36) | (1 << 18) | 1

    def home(key):  # the key's place in its group: parities, permuted by the block's hash
        local = ((key >> 34) & 4) | ((key >> 17) & 2) | (key & 1)
        return local ^ (_mix64(key & ~low) >> 61)

    same = np.array([home(int(k)) == place for k in keys.reshape(-1)])
    pick = rng.permutation(np.where(same)[0])
    assert len(pick) > first and first > capacity // 8
    labels = (np.arange(H)[:, None] // 24 * 4 + np.arange(W)[None, :] // 16 + 1).astype(np.uint16)
    tokens = rng.normal(size=(GRID[0] * GRID[1], DIM)).astype(np.float32)
    pose = np.eye(4)
    pose[2, 3] = 0.01
    probes = []
    for take in (pick[:first], pick[first // 2:first], pick[first // 3:first + more]):
        depth = np.zeros(H * W, np.float32)
        depth[take] = 2.0
        depth = depth.reshape(H, W)
        st = gmap.integrate(device_frame(torch.from_numpy(depth).to(dev), torch.from_numpy(labels.view(np.int16)).to(dev),
                                         torch.from_numpy(tokens).to(dev), pose, (50.0, 50.0, cx, cy), 8))
        o = omap.integrate(depth, labels, tokens, pose, (50.0, 50.0, cx, cy), 8)
        common.compare_frame(st, gmap.last_frame(), o, ctx=f"{len(take)} voxels of {capacity} slots")
        probes.append(st["max_probe"])
    got, ids = gmap.voxels()
    assert set(got.tolist()) == set(keys.reshape(-1)[pick[:first + more]].tolist())
    assert probes[1] >= capacity // 8  # found past a whole round
    now = binding.Config()
    assert binding.lib().disc_map_get_config(gmap._h, ctypes.byref(now)) == 0 and now.voxel_capacity > capacity
    common.compare_maps(gmap, omap, ctx="one place")
    k = [((got >> np.uint64(s)).astype(np.int64) & 0x3ffff) - (1 << 17) for s in (36, 18, 0)]
    assert np.array_equal(gmap.query_points(((np.stack(k, 1) + 0.5) * 0.02).astype(np.float32)), ids)
    gmap.close()
