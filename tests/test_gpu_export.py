"""Sorted voxel export against the oracle's, from one voxel to boxes too large
for the bitmap (which sort on the host), and with a buffer one row short."""
import numpy as np
import pytest

import oracle
from tests import common

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offsets", [[(0, 0, 0)], [(0, 0, 0), (1.3, 0, 0), (0, -2.7, 5.1)], [(0, 0, 0), (300.0, 0, 0)],
                                     [(0, 0, 0), (0, 900.0, -1200.0)], [(-900.0, 800.0, 1200.0), (900.0, -850.0, -1000.0)]])
@pytest.mark.parametrize("width,height", [(1, 1), (48, 36)])
def test_export_is_sorted_and_complete(offsets, width, height):
    import torch
    from paper_2603_03935_gb300 import DiscMap, binding, device_frame
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(len(offsets) + width)
    cfg = dict(voxel_size=0.02, embed_dim=16, patch_h=2, patch_w=3, max_width=width, max_height=height, max_masks=3,
               min_mask_pixels=1, voxel_capacity=1 << 10, max_load=0.5, instance_capacity=16, z_min=0.1, z_max=10.0,
               eps=1e-6, tau_cos=0.75, lambda_size=3.3, ov_num=1, ov_den=5)
    gmap, omap = DiscMap(**cfg), oracle.OracleMap(**common.to_oracle_cfg(cfg))
    intr = (50.0, 50.0, width / 2.0, height / 2.0)
    for t in offsets:
        depth = rng.uniform(0.5, 3.0, (height, width)).astype(np.float32)
        labels = rng.integers(1, 4, (height, width)).astype(np.uint16)
        tokens = rng.normal(size=(6, 16)).astype(np.float32)
        pose = np.eye(4)
        pose[:3, 3] = t
        gmap.integrate(device_frame(torch.from_numpy(depth).to(dev), torch.from_numpy(labels.view(np.int16)).to(dev),
                                    torch.from_numpy(tokens).to(dev), pose, intr, 3))
        omap.integrate(depth, labels, tokens, pose, intr, 3)
        common.compare_maps(gmap, omap, ctx=str(t))
    n, _ = gmap.counts()
    keys, ids = np.zeros(n, np.uint64), np.zeros(n, np.int32)
    lib = binding.lib()
    assert lib.disc_map_export_voxels(gmap._h, keys.ctypes.data, ids.ctypes.data, n - 1) == -1
    assert lib.disc_map_export_voxels(gmap._h, keys.ctypes.data, ids.ctypes.data, n + 5) == 0
    assert (np.diff(keys.astype(np.int64)) > 0).all()
    gmap.close()


@pytest.mark.parametrize("nid,nq,k,dim", [(3, 1, 5, 7), (96, 9, 20, 64), (97, 8, 1, 1030), (700, 17, 96, 60)])
def test_topk_at_tile_edges(nid, nq, k, dim):
    """Scores within fp32 rounding of float64, ids ordered by (score, id); dead instances and padding at the end."""
    import torch
    from paper_2603_03935_gb300 import DiscMap, device_frame
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(nid + dim)
    per = min(nid, 96)
    frames, made = [], 0
    gmap = DiscMap(voxel_size=0.025, embed_dim=dim, patch_h=8, patch_w=12, max_width=96, max_height=64, max_masks=96,
                   min_mask_pixels=1, voxel_capacity=1 << 16, max_load=0.5, instance_capacity=128)
    v, u = torch.arange(64, device=dev)[:, None] // 8, torch.arange(96, device=dev)[None, :] // 8
    while made < nid:
        n = min(per, nid - made)
        labels = (v * 12 + u + 1).clamp(max=97)
        labels = torch.where(labels <= n, labels, torch.zeros_like(labels)).to(torch.int16).contiguous()
        pose = np.eye(4)
        pose[0, 3] = 40.0 * len(frames)
        tokens = torch.randn(96, dim, device=dev, generator=gen)
        frames.append(device_frame(torch.full((64, 96), 2.0, device=dev), labels, tokens, pose, (80.0, 80.0, 48.0, 32.0), n))
        made += n
    gmap.integrate_frames(frames)
    E = gmap.instances()["E"]
    assert len(E) == nid
    if dim % 2 == 0:
        q = E[:nq] + 0.1 * np.random.default_rng(1).normal(size=(nq, dim)).astype(np.float32)
    else:
        q = np.repeat(E[:1], nq, 0)  # equal queries: equal answers
    ids, sc = gmap.query_topk(q, k)
    e64, q64 = E.astype(np.float64), q.astype(np.float64)
    want = q64 @ e64.T / (np.linalg.norm(q64, axis=1)[:, None] * np.linalg.norm(e64, axis=1))
    m = min(k, nid)
    assert (ids[:, m:] == -1).all() and np.isneginf(sc[:, m:]).all()
    assert np.abs(np.take_along_axis(want, ids[:, :m], 1) - sc[:, :m]).max() <= 3 * dim * 2.0 ** -24 + 2.0 ** -22
    assert all(len(set(r)) == m for r in ids[:, :m].tolist())
    for r, s in zip(ids[:, :m], sc[:, :m]):
        assert all(s[i] > s[i + 1] or (s[i] == s[i + 1] and r[i] < r[i + 1]) for i in range(m - 1))
    best = -np.sort(-want, axis=1)[:, :m]
    assert np.abs(best - sc[:, :m]).max() <= 3 * dim * 2.0 ** -24 + 2.0 ** -22
    gmap.close()


@pytest.mark.parametrize("dim,per", [(7, 3), (64, 96), (4096, 90)])
def test_instance_table_read_again_and_again(dim, per):
    """The first read of a map's table, later ones through pinned memory and tables too large for it are the same
    bytes; short buffers are refused and NULL arrays left out by all of them."""
    import torch
    from paper_2603_03935_gb300 import DiscMap, binding, device_frame
    dev = torch.device("cuda:0")
    lib = binding.lib()
    gen = torch.Generator(device=dev).manual_seed(dim)
    cfg = dict(voxel_size=0.025, embed_dim=dim, patch_h=8, patch_w=12, max_width=96, max_height=64, max_masks=96,
               min_mask_pixels=1, voxel_capacity=1 << 16, max_load=0.5, instance_capacity=64)
    again, empty = DiscMap(**cfg), DiscMap(**cfg)
    for _ in range(3):
        assert lib.disc_map_export_instances(empty._h, None, None, None, None, None, 0) == 0
    v, u = torch.arange(64, device=dev)[:, None] // 8, torch.arange(96, device=dev)[None, :] // 8
    labels = (v * 12 + u + 1).clamp(max=97)
    labels = torch.where(labels <= per, labels, torch.zeros_like(labels)).to(torch.int16).contiguous()
    frames = []
    for t in range(4):  # 4 x 90 rows of 4096 floats: 5.9 MB, above the pinned buffer's bound
        pose = np.eye(4)
        pose[0, 3] = 40.0 * t
        tokens = torch.randn(96, dim, device=dev, generator=gen)
        frames.append(device_frame(torch.full((64, 96), 2.0, device=dev), labels, tokens, pose,
                                   (80.0, 80.0, 48.0, 32.0), per))
        again.integrate(frames[-1])
        once = DiscMap(**cfg)
        for f in frames:
            once.integrate(f)
        want = once.instances()
        n = len(want["parent"])
        assert n == per * (t + 1)
        for _ in range(2):
            got = again.instances()
            assert sorted(got) == sorted(want)
            for k in want:
                assert np.array_equal(np.asarray(got[k]).view(np.uint8), np.asarray(want[k]).view(np.uint8)), (k, t)
        count = np.full(n, -1, np.int64)
        assert lib.disc_map_export_instances(again._h, None, count.ctypes.data, None, None, None, n - 1) == -1
        assert (count == -1).all()
        assert lib.disc_map_export_instances(again._h, None, count.ctypes.data, None, None, None, n + 7) == 0
        assert np.array_equal(count, want["count"])
        once.close()
    again.close()
    empty.close()


def test_a_large_export_gives_its_memory_back():
    # 17 million voxels too far apart for the bitmap (the host sorts them): the list of their slots goes back; and an
    # export beside a large query scratch leaves that as it is
    import torch
    from paper_2603_03935_gb300 import DiscMap, device_frame
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(2)
    width, height = 2048, 1536
    gmap = DiscMap(voxel_size=0.02, embed_dim=16, patch_h=4, patch_w=4, max_width=width, max_height=height, max_masks=2,
                   min_mask_pixels=1, voxel_capacity=1 << 26, max_load=0.5, instance_capacity=64, z_min=0.1, z_max=1e4,
                   batch_frames=1)
    labels = torch.ones(height, width, dtype=torch.int16, device=dev)
    tokens = torch.randn(16, 16, device=dev)
    intr = (1000.0, 1000.0, width / 2.0, height / 2.0)

    def frame():
        depth = 500.0 * (0.2 + torch.rand(height, width, device=dev, generator=gen))
        gmap.integrate(device_frame(depth, labels, tokens, np.eye(4), intr, 1))

    def export():
        n, _ = gmap.counts()
        keys, ids = gmap.voxels()
        assert len(keys) == n and (np.diff(keys.astype(np.int64)) > 0).all() and (ids >= 0).all()

    for _ in range(6):
        frame()
    assert gmap.counts()[0] > 17e6
    before = gmap.device_bytes()  # no query scratch yet; an export may leave 64 MB of it
    export()
    assert gmap.device_bytes() <= before + (64 << 20)
    gmap.query_points(np.zeros((9_000_000, 3), np.float32))  # 144 MB of query scratch
    held = gmap.device_bytes()
    export()
    assert gmap.device_bytes() == held
    gmap.close()
