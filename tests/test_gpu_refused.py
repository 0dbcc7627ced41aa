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
