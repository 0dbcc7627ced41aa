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
