"""Token statistics, coverage and exact pooling at the edges of their tiles:
column groups, patch blocks, unaligned rows and bases, narrow and one-row
frames; bit for bit against the oracle."""
import numpy as np
import pytest

import oracle
from tests import common

pytestmark = pytest.mark.gpu

#        width height  grid     dim   masks bf16   offset (elements the token buffer starts off its alignment)
CASES = [(16, 12, (1, 1), 1, 2, False, 0), (16, 12, (1, 3), 5, 2, False, 1), (64, 48, (3, 11), 257, 5, False, 0),
         (40, 30, (4, 8), 256, 7, True, 2), (61, 35, (5, 7), 259, 9, True, 1), (33, 65, (31, 1), 1024, 3, False, 3),
         (1, 40, (8, 4), 64, 2, False, 0), (1400, 3, (2, 33), 60, 12, True, 0), (48, 36, (6, 11), 4096, 4, False, 0)]


@pytest.mark.parametrize("width,height,grid,dim,masks,bf16,offset", CASES)
def test_feature_kernels_at_tile_edges(width, height, grid, dim, masks, bf16, offset):
    import torch
    from paper_2603_03935_gb300 import DiscMap, device_frame
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(dim + masks)
    P = grid[0] * grid[1]
    tokens = rng.normal(size=(P, dim)).astype(np.float32)
    if P * dim > 64:
        tokens.reshape(-1)[::37] *= 300.0  # products leave the 32-bit range
        tokens = np.clip(tokens, -1000.0, 1000.0)  # the library takes |token| <= 1024
    buf = torch.zeros(P * dim + 8, dtype=torch.bfloat16 if bf16 else torch.float32, device=dev)
    t = buf[offset:offset + P * dim].view(P, dim)
    t.copy_(torch.from_numpy(tokens))
    tokens = t.float().cpu().numpy()
    depth = rng.uniform(1.0, 2.0, (height, width)).astype(np.float32)
    labels = rng.integers(0, masks + 2, (height, max(1, width // 4) + 1)).repeat(4, axis=1)[:, :width]
    labels = np.ascontiguousarray(labels).astype(np.uint16)  # label masks + 1 counts as background
    cfg = dict(voxel_size=0.05, embed_dim=dim, patch_h=grid[0], patch_w=grid[1], max_width=width, max_height=height,
               max_masks=masks, min_mask_pixels=2, voxel_capacity=1 << 14, max_load=0.5, instance_capacity=64,
               z_min=0.1, z_max=10.0, eps=1e-6, tau_cos=0.75, lambda_size=3.3, ov_num=1, ov_den=5)
    gmap, omap = DiscMap(**cfg), oracle.OracleMap(**common.to_oracle_cfg(cfg))
    intr = (50.0, 50.0, width / 2.0, height / 2.0)
    st = gmap.integrate(device_frame(torch.from_numpy(depth).to(dev), torch.from_numpy(labels.view(np.int16)).to(dev), t,
                                     np.eye(4), intr, masks))
    o = omap.integrate(depth, labels, tokens, np.eye(4), intr, masks)
    common.compare_frame(st, gmap.last_frame(), o, ctx=f"dim {dim}")
    gmap.close()


def test_a_nan_token_among_finite_ones_fails_the_frame():
    import torch
    from paper_2603_03935_gb300 import DiscError, token_stats_static
    for k in range(4):
        t = torch.ones(9, 12, device="cuda:0")
        t[7, 4 + k] = float("nan")
        with pytest.raises(DiscError):
            token_stats_static(t)
