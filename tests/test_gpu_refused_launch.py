"""A launch that the runtime refuses: the call says so, counts nothing for it and leaves no error behind."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    from paper_2609_32197_b200 import binding as b
    b.lib()
    return b


def test_a_refused_launch_is_an_error_of_its_own_call_only(binding):
    """More heads than a grid has places in its third dimension (one token each): the runtime refuses the score kernel before
    it starts.  Of the launches of that call one, the pooling, has happened; the next call of another kind succeeds."""
    H, d = 65536, 64
    shape = binding.make_shape(H, d, (1, 1, 1), 0, 64)
    ws = binding.make_workspace(shape, 2)
    Q = torch.ones(H, 1, d, dtype=torch.bfloat16, device="cuda")
    mask = torch.zeros(1, H, 1, 1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    before = binding.sparsp_launch_count()
    with pytest.raises(binding.SparspError) as e:
        binding.sparsp_block_mask(shape, Q, Q, 1, mask, None, None, None, None, ws)
    assert e.value.code == binding.SPARSP_ERR_CUDA
    refused = binding.sparsp_launch_count()
    rank = torch.zeros(1, dtype=torch.int32, device="cuda")
    hist = torch.ones(1, 2, 101, dtype=torch.int64, device="cuda")
    binding.sparsp_sharing_histogram(shape, mask, rank, 2, hist)
    assert int(hist.sum()) == 0
    assert refused == before + 1 and binding.sparsp_launch_count() == before + 2
    assert int((Q + 1).float().sum()) == 2 * H * d
    assert binding.sparsp_status(ws) == binding.SPARSP_OK
