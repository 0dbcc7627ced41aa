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


@pytest.mark.parametrize("precision", [0, 2])
def test_calls_on_an_sm_partition_smaller_than_a_cluster_wants(precision):
    # 128 of 152 SMs for the frame chain: the pooling GEMM of 250 masks (one
    # CTA per SM at FP32) runs on what is left
    import torch
    from paper_2603_03935_gb300 import DiscMap, device_frame
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(3)
    W, H, masks, dim = 160, 96, 250, 512
    maps = []
    for sms in (0, 128):
        maps.append(DiscMap(voxel_size=0.05, embed_dim=dim, patch_h=32, patch_w=32, max_width=W, max_height=H,
                            max_masks=masks, min_mask_pixels=1, voxel_capacity=1 << 18, max_load=0.5,
                            instance_capacity=4096, precision=precision, serial_sms=sms, batch_frames=2))
    frames = []
    for i in range(8):
        tokens = torch.randn(32 * 32, dim, device=dev, generator=gen)
        labels = torch.randint(0, masks + 1, (H // 4, W // 4), device=dev, generator=gen).repeat_interleave(4, 0)
        labels = labels.repeat_interleave(4, 1).to(torch.int16).contiguous()
        depth = torch.rand(H, W, device=dev, generator=gen) * 0.2 + 2.0
        frames.append(device_frame(depth, labels, tokens, np.eye(4), (50.0, 50.0, W / 2.0, H / 2.0), masks))
    for lo, hi in ((0, 2), (2, 3), (3, 8)):  # one batch (asynchronous), one frame, three batches
        for m in maps:
            _, done, rc = m.integrate_frames_async(frames[lo:hi]).result()
            assert rc == 0 and done == hi - lo
        r = [m.last_frame() for m in maps]
        live = r[0]["npix"] > 0
        assert np.array_equal(r[0]["E"], r[1]["E"]) and np.array_equal(r[0]["rep"], r[1]["rep"])
        for x in r:
            err = np.linalg.norm(x["E_fast"].astype(np.float64) - x["E"], axis=1)[live]
            assert (err <= x["E_bound"][live]).all()
    assert all(np.array_equal(a, b) for a, b in zip(maps[0].voxels(), maps[1].voxels()))
    for m in maps:
        m.close()


# patches: 8, 5, 31 and 3 chunks (4, 2, 8 and 1 groups)
@pytest.mark.parametrize("masks,precision,bf16", [(20, 0, False), (100, 1, True), (200, 0, False), (250, 2, True),
                                                  (130, 1, False)])
@pytest.mark.parametrize("grid,dim", [((16, 16), 200), ((12, 13), 128), ((32, 31), 700), ((9, 9), 64)])
def test_the_pooled_embedding_does_not_depend_on_the_batch(grid, dim, masks, precision, bf16):
    # the same frame last in batches of 1 to 64 frames, in smaller batches and
    # on an SM partition: the same bits
    import torch
    from paper_2603_03935_gb300 import DiscMap, device_frame
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(masks)
    W, H, P = 128, 96, grid[0] * grid[1]
    frames = []
    for i in range(2):
        tokens = torch.randn(P, dim, device=dev, generator=gen)
        labels = torch.randint(0, masks + 1, (H // 2, W // 2), device=dev, generator=gen).repeat_interleave(2, 0)
        labels = labels.repeat_interleave(2, 1).to(torch.int16).contiguous()
        depth = torch.full((H, W), 2.0, device=dev)
        frames.append(device_frame(depth, labels, tokens.bfloat16() if bf16 else tokens, np.eye(4),
                                   (50.0, 50.0, W / 2.0, H / 2.0), masks))
    first = None
    for n, split, sms in ((1, 0, 0), (3, 0, 0), (7, 0, 0), (14, 1, 0), (30, 1, 0), (64, 1, 0), (64, 8, 0), (16, 0, 64)):
        m = DiscMap(voxel_size=0.05, embed_dim=dim, patch_h=grid[0], patch_w=grid[1], max_width=W, max_height=H,
                    max_masks=masks, min_mask_pixels=1, voxel_capacity=1 << 16, max_load=0.5, instance_capacity=1024,
                    precision=precision, batch_frames=64, serial_sms=sms)
        m.set_schedule(batch_split=split)
        m.integrate_frames([frames[0]] * (n - 1) + [frames[1]])
        r = m.last_frame()
        if first is None:
            first = r["E_fast"], r["E_bound"]
            assert np.abs(first[0]).max() > 0
        assert np.array_equal(r["E_fast"], first[0]) and np.array_equal(r["E_bound"], first[1]), (n, split, sms)
        m.close()
