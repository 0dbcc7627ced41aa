"""The tensor-core pooled embedding at the edges of its tiles and of the split
of the patches over a cluster: against the exact one, within 1e-5 of its norm
per mask at FP32 precision and within the bound the gate uses at BF16 and FP8."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# patches: 1, 4, 8 and 32 chunks of 32 patches (clusters of 1, 1, 2 and 8), ragged ones among them
@pytest.mark.parametrize("masks", [1, 17, 64, 65, 130, 256])
@pytest.mark.parametrize("grid,dim,frames", [((4, 5), 60, 1), ((11, 11), 128, 1), ((16, 16), 129, 2), ((32, 31), 300, 1),
                                             ((16, 16), 4096, 7)])
def test_pool_gemm_within_its_bound(masks, grid, dim, frames):
    import torch
    from paper_2603_03935_gb300 import DiscMap, device_frame
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(masks * 7 + dim)
    P, W, H = grid[0] * grid[1], 96, 64
    bf16 = masks % 2 == 0
    tokens = torch.randn(P, dim, device=dev, generator=gen)
    if bf16:
        tokens = tokens.to(torch.bfloat16)
    labels = torch.randint(0, masks + 1, (H // 2, W // 2), device=dev, generator=gen).repeat_interleave(2, 0)
    labels = labels.repeat_interleave(2, 1).to(torch.int16).contiguous()
    depth = torch.full((H, W), 2.0, device=dev)
    for precision in (0, 1, 2):
        m = DiscMap(voxel_size=0.05, embed_dim=dim, patch_h=grid[0], patch_w=grid[1], max_width=W, max_height=H,
                    max_masks=masks, min_mask_pixels=1, voxel_capacity=1 << 16, max_load=0.5, instance_capacity=1024,
                    precision=precision)
        fr = device_frame(depth, labels, tokens, np.eye(4), (50.0, 50.0, W / 2.0, H / 2.0), masks)
        m.integrate_frames([fr] * frames)
        r = m.last_frame()
        live = r["npix"] > 0
        err = np.linalg.norm(r["E_fast"].astype(np.float64) - r["E"], axis=1)[live]
        if precision == 0:
            assert (err <= 1e-5 * np.linalg.norm(r["E"].astype(np.float64), axis=1)[live]).all()
        assert (err <= r["E_bound"][live]).all(), f"precision {precision}"
        m.close()
