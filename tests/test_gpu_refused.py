"""What a refused call leaves behind: output buffers as they were, and a frame
report without the failed frame's voxels."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("where", ["tokens", "query"])
def test_a_refused_heatmap_leaves_its_output_as_it_was(where):
    import torch
    from paper_2603_03935_gb300 import binding, query_heatmap
    dev = torch.device("cuda:0")
    tokens, query = torch.randn(300, 96, device=dev), torch.randn(96, device=dev)
    query_heatmap(tokens, query)  # an earlier call's cosines stay in the working set
    (tokens if where == "tokens" else query).view(-1)[41] = 2000.0  # |value| <= 1024 is accepted
    heat = torch.arange(300, dtype=torch.float32, device=dev) + 0.5
    before = heat.clone()
    rc = binding.lib().disc_query_heatmap(tokens.data_ptr(), 0, 300, 96, query.data_ptr(), 1e-6, heat.data_ptr(),
                                          torch.cuda.current_stream().cuda_stream)
    assert binding.STATUS[rc] == "DISC_ERR_RANGE"
    assert torch.equal(heat, before)


@pytest.mark.parametrize("dilation", [0, 1])
def test_a_failed_frames_report_holds_no_voxels(dilation):
    import synth
    import torch
    from paper_2603_03935_gb300 import DiscMap, device_frame
    from tests import common
    dev = torch.device("cuda:0")
    sc = synth.tiny_scene(num_frames=2)
    fr = sc.render(range(2))
    gmap = DiscMap(**common.disc_cfg(sc, overlap_dilation=dilation))
    fr.tokens[1][3, 5] = 2000.0  # out of the accepted range: the second frame fails
    for i in range(2):
        frame = device_frame(torch.from_numpy(fr.depth[i]).to(dev), torch.from_numpy(fr.labels[i].view("int16")).to(dev),
                             torch.from_numpy(fr.tokens[i]).to(dev), fr.poses[i], (sc.fx, sc.fy, sc.cx, sc.cy),
                             int(fr.num_masks[i]))
        stats, done, rc = gmap.integrate_frames([frame], check=False)
        rep = gmap.last_frame()
        if i == 0:
            assert rc == 0 and done == 1 and rep["nvox"].sum() > 0 and (rep["S"][:, 1] > 0).any()
    assert rc != 0 and done == 0
    assert all(stats[0][k] == 0 for k in ("valid_pixels", "unique_seg_voxels", "new_voxels", "live_segments"))
    assert (rep["nvox"] == 0).all() and (rep["S"][:, [1, 4]] == 0).all() and (rep["rep"] == -1).all()
    gmap.close()


@pytest.mark.parametrize("bad_grid", ["second", "first", "both"])
def test_a_token_out_of_range_in_either_grid_fails_its_frame_alone(bad_grid):
    # the grids' kernels run side by side and share the frame's error word
    import numpy as np
    import oracle
    import synth
    import torch
    from paper_2603_03935_gb300 import DiscMap, device_frame
    from tests import common
    dev = torch.device("cuda:0")
    sc = synth.tiny_scene(num_frames=12)
    fr = sc.render(range(12))
    at = fr.assoc_tokens(5, 7, 96)
    cfg = common.disc_cfg(sc, assoc_dim=96, assoc_patch_h=5, assoc_patch_w=7)
    gmap, omap = DiscMap(**cfg), oracle.OracleMap(**common.to_oracle_cfg(cfg))

    def frame(i, bad):
        first, second = fr.tokens[i].copy(), at[i].copy()
        if bad:
            for g, t in (("first", first), ("second", second)):
                if bad_grid in (g, "both"):
                    t.reshape(-1)[i * 7 % t.size] = 1500.0
        return device_frame(torch.from_numpy(fr.depth[i]).to(dev), torch.from_numpy(fr.labels[i].view(np.int16)).to(dev),
                            torch.from_numpy(first).to(dev), fr.poses[i], (sc.fx, sc.fy, sc.cx, sc.cy),
                            int(fr.num_masks[i]), assoc_tokens=torch.from_numpy(second).to(dev))

    for i in range(0, 12, 4):
        # the call stops at its third frame; the rest is given again without the bad token
        stats, done, rc = gmap.integrate_frames([frame(i + j, j == 2) for j in range(4)], check=False)
        assert rc != 0 and done == 2 and stats[2]["status"] == rc and stats[2]["new_voxels"] == 0
        _, done, rc = gmap.integrate_frames([frame(i + j, False) for j in (2, 3)])
        assert rc == 0 and done == 2
        for j in range(4):
            omap.integrate(*oracle.frame_args(fr, i + j), assoc_tokens=at[i + j])
    common.compare_maps(gmap, omap, ctx=f"{bad_grid} grid out of range")
    gmap.close()
