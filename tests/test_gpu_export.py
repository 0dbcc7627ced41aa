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
