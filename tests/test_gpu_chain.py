"""One batch of more frames than the association kernel stages at once, with
segments that split and join again: merges and better views change instances'
embeddings inside the batch, so gates taken at its start have to be taken
again; every counter and the final map equal the oracle's."""
import numpy as np
import pytest

import oracle
import synth
from tests import common

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_embeddings_changed_inside_a_long_batch(precision):
    import torch
    from paper_2603_03935_gb300 import DiscMap, device_frame
    dev = torch.device("cuda:0")
    sc = synth.tiny_scene(num_frames=70)
    fr = sc.render(range(70))
    masks = sc.max_masks + 2
    cfg = common.disc_cfg(sc, max_masks=masks, batch_frames=128, precision=precision)
    gmap, omap = DiscMap(**cfg), oracle.OracleMap(**common.to_oracle_cfg(cfg))
    gmap.set_schedule(batch_split=1)
    frames, counts = [], []
    for i in range(70):
        lab, n = fr.labels[i], int(fr.num_masks[i])
        if i % 4 != 0:  # the two largest masks cut in half
            for k in (1, 2):
                u = np.where((lab == k).any(axis=0))[0]
                half = lab[:, (u[0] + u[-1]) // 2:]
                half[half == k] = n + k
            n += 2
        counts.append(n)
        frames.append(device_frame(torch.from_numpy(fr.depth[i]).to(dev), torch.from_numpy(lab.view(np.int16)).to(dev),
                                   torch.from_numpy(fr.tokens[i]).to(dev), fr.poses[i], (sc.fx, sc.fy, sc.cx, sc.cy), n))
    stats, done, rc = gmap.integrate_frames(frames)
    assert rc == 0 and done == 70
    for i in range(70):
        o = omap.integrate(fr.depth[i], fr.labels[i], fr.tokens[i], fr.poses[i], (sc.fx, sc.fy, sc.cx, sc.cy), counts[i])
        for gk, ok in common.COUNT_FIELDS:
            assert stats[i][gk] == o[ok], f"frame {i} {gk}: {stats[i][gk]} vs {o[ok]}"
    common.compare_maps(gmap, omap, ctx="chain")
    assert sum(s["merges"] for s in stats) > 0
    assert sum(s["embedding_copies"] for s in stats) > sum(s["new_instances"] for s in stats)
    gmap.close()


@pytest.mark.parametrize("capacity", [1, 4, 8, 1 << 12])
@pytest.mark.parametrize("at", [(0, 0, 0), (2621.3, -2621.3, -2623.4), (-2621.3, 2621.3, 2619.9)])
def test_neighbourhood_at_table_and_key_edges(capacity, at):
    """The 26 neighbours in tables smaller than a block of slots, crowded tables, and at the ends of the key range on
    every axis (part of the pixels fall outside): counters and map equal the oracle's."""
    import torch
    from paper_2603_03935_gb300 import DiscMap, device_frame
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(capacity)
    for width, height in ((1, 1), (37, 29)):
        cfg = dict(voxel_size=0.02, embed_dim=16, patch_h=2, patch_w=3, max_width=width, max_height=height, max_masks=5,
                   min_mask_pixels=1, voxel_capacity=capacity, max_load=0.9, instance_capacity=16, z_min=0.1,
                   z_max=10.0, eps=1e-6, tau_cos=0.75, lambda_size=3.3, ov_num=1, ov_den=5, overlap_dilation=1)
        gmap, omap = DiscMap(**cfg), oracle.OracleMap(**common.to_oracle_cfg(cfg))
        intr = (400.0, 400.0, width / 2.0, height / 2.0)
        tokens = rng.normal(size=(6, 16)).astype(np.float32)
        for t in range(4):
            depth = (2.0 + 0.01 * rng.integers(0, 4, (height, width))).astype(np.float32)
            labels = np.tile((1 + np.arange(width) * 5 // width).astype(np.uint16), (height, 1))
            pose = np.eye(4)
            pose[:3, 3] = np.array(at) + 0.03 * t
            s = gmap.integrate(device_frame(torch.from_numpy(depth).to(dev),
                                            torch.from_numpy(labels.view(np.int16)).to(dev),
                                            torch.from_numpy(tokens).to(dev), pose, intr, 5))
            o = omap.integrate(depth, labels, tokens, pose, intr, 5)
            for gk, ok in common.COUNT_FIELDS:
                assert s[gk] == o[ok], f"frame {t} {gk}: {s[gk]} vs {o[ok]}"
            common.compare_maps(gmap, omap, ctx=f"{width}x{height} {t}")
        gmap.close()


def _crowd(blocks, n, dim, grid, dim2=0, width=160, height=120, drift=0.011, seed=5):
    """n frames of a wall cut into blocks[0] x blocks[1] masks, the camera drifting along it: each segment overlaps the
    instances of its neighbours, views improve and get worse."""
    rng = np.random.default_rng(seed)
    v, u = np.meshgrid(np.arange(height), np.arange(width), indexing="ij")
    label = (v * blocks[1] // height) * blocks[0] + u * blocks[0] // width + 1
    mean = rng.normal(size=(label.max() + 1, dim + dim2)).astype(np.float32)
    out = []
    for i in range(n):
        depth = (2.0 + 0.003 * u + 0.002 * rng.normal(size=u.shape)).astype(np.float32)
        at = label[((2 * np.arange(grid[0]) + 1) * height) // (2 * grid[0])][:, ((2 * np.arange(grid[1]) + 1) * width) // (2 * grid[1])]
        tok = mean[at.reshape(-1)] + rng.normal(size=(at.size, dim + dim2)).astype(np.float32) * rng.uniform(0.1, 0.8)
        pose = np.eye(4)
        pose[:2, 3] = drift * i, 0.7 * drift * i
        out.append((depth, label.astype(np.uint16), np.ascontiguousarray(tok[:, :dim], np.float32), pose,
                    np.ascontiguousarray(tok[:, dim:], np.float32) if dim2 else None))
    return out, int(label.max())


@pytest.mark.parametrize("cluster", [0, 1, 2, 8])
@pytest.mark.parametrize("precision,dim2", [(0, 0), (1, 0), (2, 0), (0, 48), (2, 50)])
def test_many_pairs_left_to_score_and_copy(cluster, precision, dim2):
    import torch
    from paper_2603_03935_gb300 import DiscMap, device_frame
    dev = torch.device("cuda:0")
    frames, masks = _crowd((16, 12), 14, 64, (24, 32), dim2)
    intr = (100.0, 100.0, 80.0, 60.0)
    cfg = dict(voxel_size=0.05, embed_dim=64, patch_h=24, patch_w=32, max_width=160, max_height=120, max_masks=masks,
               min_mask_pixels=2, voxel_capacity=1 << 16, max_load=0.5, instance_capacity=8192, z_min=0.1, z_max=10.0,
               eps=1e-6, tau_cos=0.75, lambda_size=30.0, ov_num=1, ov_den=5, precision=precision, batch_frames=32)
    if dim2:
        cfg.update(assoc_dim=dim2, assoc_patch_h=24, assoc_patch_w=32)
    gmap, omap = DiscMap(**cfg), oracle.OracleMap(**common.to_oracle_cfg(cfg))
    gmap.set_schedule(batch_split=1, assoc_cluster=cluster)
    up = [device_frame(torch.from_numpy(d).to(dev), torch.from_numpy(l.view(np.int16)).to(dev), torch.from_numpy(t).to(dev),
                       p, intr, masks, assoc_tokens=None if a is None else torch.from_numpy(a).to(dev))
          for d, l, t, p, a in frames]
    copies = 0
    for lo, hi in ((0, 1), (1, 11), (11, 14)):
        stats, done, rc = gmap.integrate_frames(up[lo:hi])
        assert rc == 0 and done == hi - lo
        for st, (d, l, t, p, a) in zip(stats, frames[lo:hi]):
            o = omap.integrate(d, l, t, p, intr, masks, **({} if a is None else {"assoc_tokens": a}))
            for gk, ok in common.COUNT_FIELDS:
                assert st[gk] == o[ok], (gk, st[gk], o[ok])
            copies = max(copies, st["embedding_copies"])
    assert copies > 60  # (48 are worth the cluster's help)
    common.compare_maps(gmap, omap, ctx=f"{masks} masks, cluster {cluster}, precision {precision}")
    gmap.close()


def test_a_crowded_frames_association_costs_no_more_than_its_pairs():
    # 240 masks in the place of 40, instances changing under them: the work that is left for the frame's turn is spread
    # over a cluster. (One CTA took over four times the time of 40 masks.)
    import torch
    from paper_2603_03935_gb300 import DiscMap, device_frame
    dev = torch.device("cuda:0")
    ms = []
    for blocks in ((8, 5), (16, 15)):
        frames, masks = _crowd(blocks, 17, 768, (24, 24), width=640, height=480, drift=0.013)
        up = [device_frame(torch.from_numpy(d).to(dev), torch.from_numpy(l.view(np.int16)).to(dev),
                           torch.from_numpy(t).to(dev), p, (525.0, 525.0, 320.0, 240.0), masks) for d, l, t, p, _ in frames]
        best = 1e9
        for _ in range(3):
            gmap = DiscMap(voxel_size=0.025, embed_dim=768, patch_h=24, patch_w=24, max_width=640, max_height=480,
                           max_masks=256, min_mask_pixels=50, voxel_capacity=1 << 20, max_load=0.5, z_min=0.1, z_max=10.0,
                           instance_capacity=1 << 14, batch_frames=16, lambda_size=30.0)
            gmap.set_phase_timing(True)
            gmap.integrate_frames(up[:1])
            gmap.set_phase_timing(True)
            gmap.integrate_frames(up[1:])
            best = min(best, gmap.phase_times()["associate"]["ms"])
            gmap.close()
        ms.append(best)
    assert ms[1] < 3 * ms[0], ms


@pytest.mark.parametrize("cluster", [0, 1, 4])
@pytest.mark.parametrize("precision", [0, 2])
def test_more_edges_than_shared_memory_holds(cluster, precision):
    # 512 instances (each half of the wall as 256 narrow masks), then 256 wide masks over two of them each: every wide
    # one joins both, 512 edges of 512 instances in one frame, past the shared arrays
    import torch
    from paper_2603_03935_gb300 import DiscMap, device_frame
    dev = torch.device("cuda:0")
    frames, masks = _crowd((16, 16), 8, 64, (24, 32), seed=8)
    v, u = np.meshgrid(np.arange(120), np.arange(160), indexing="ij")
    for i in range(2):
        narrow = (v * 16 // 120) * 16 + (u - 80 * i) * 32 // 160 + 1
        d, _, t, _, a = frames[i]
        frames[i] = d, np.where((u >= 80 * i) & (u < 80 * (i + 1)), narrow, 0).astype(np.uint16), t, np.eye(4), a
    intr = (100.0, 100.0, 80.0, 60.0)
    cfg = dict(voxel_size=0.05, embed_dim=64, patch_h=24, patch_w=32, max_width=160, max_height=120, max_masks=masks,
               min_mask_pixels=2, voxel_capacity=1 << 16, max_load=0.5, instance_capacity=8192, z_min=0.1, z_max=10.0,
               eps=1e-6, tau_cos=0.5, lambda_size=30.0, ov_num=1, ov_den=5, precision=precision, batch_frames=32)
    gmap, omap = DiscMap(**cfg), oracle.OracleMap(**common.to_oracle_cfg(cfg))
    gmap.set_schedule(batch_split=1, assoc_cluster=cluster)
    stats, done, rc = gmap.integrate_frames([
        device_frame(torch.from_numpy(d).to(dev), torch.from_numpy(l.view(np.int16)).to(dev), torch.from_numpy(t).to(dev),
                     p, intr, masks) for d, l, t, p, _ in frames])
    assert rc == 0 and done == 8
    for st, (d, l, t, p, _) in zip(stats, frames):
        o = omap.integrate(d, l, t, p, intr, masks)
        for gk, ok in common.COUNT_FIELDS:
            assert st[gk] == o[ok], (gk, st[gk], o[ok])
    assert stats[2]["active_instances"] > 256 and stats[2]["merges"] > 200
    common.compare_maps(gmap, omap, ctx=f"cluster {cluster}, precision {precision}")
    gmap.close()
