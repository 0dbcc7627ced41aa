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
