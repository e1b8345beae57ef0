"""Which attention calls do without the launch that makes their items, seen from the number of launches: 64-token blocks up to
one an SM (more of them share Q tiles), 128-token blocks up to two, and a packed source only where every CTA has one item at
most, whoever owns the blocks."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    from paper_2609_32197_b200 import binding as b
    b.lib()
    return b


def _inputs(binding, b, H, NB, d=64):
    g = torch.Generator(device="cuda").manual_seed(H + NB)
    Q, K, V = (torch.randn(1, H, NB * b, d, generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    mask = torch.zeros(1, H, NB, (NB + 31) // 32, dtype=torch.int32, device="cuda")
    mask[..., 0] = 1
    return binding.make_shape(H, d, (1, 1, NB * b), 0, b), Q, K, V, mask


@pytest.mark.parametrize("b,per_sm", [(64, 1), (128, 2)])
@pytest.mark.parametrize("more", [0, 1])
def test_own_keys(binding, b, per_sm, more):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    shape, Q, K, V, mask = _inputs(binding, b, 1, per_sm * sms + more)
    ws = binding.make_workspace(shape, 1)
    O = torch.empty_like(Q)
    before = binding.sparsp_launch_count()
    binding.sparsp_sparse_attn_fwd(shape, Q, K, V, mask, 0.0, O, None, ws)
    assert binding.sparsp_launch_count() - before == 1 + more
    assert binding.sparsp_status(ws) == binding.SPARSP_OK


@pytest.mark.parametrize("b,per_item", [(64, 2), (128, 1)])
@pytest.mark.parametrize("more", [0, 1])
def test_packed(binding, b, per_item, more):
    sms, P = torch.cuda.get_device_properties(0).multi_processor_count, 4
    NB = per_item * sms + more
    shape, Q, K, V, mask = _inputs(binding, b, 1, NB)
    ws = binding.make_workspace(shape, P)
    rank = torch.zeros(NB, dtype=torch.int32, device="cuda")
    do = binding.alloc_demand_outputs(shape, P)
    binding.sparsp_demand_pack(shape, mask, rank, P, binding.SPARSP_PLAN_ONLY, None, None, do["union_mask"], do["cnt"],
                               do["seg_offset"], do["seg_total"], do["volume_bytes"], None, 0, None, ws)
    packed, O = torch.zeros(4 * b * 64, dtype=torch.uint8, device="cuda"), torch.empty_like(Q)
    before = binding.sparsp_launch_count()
    binding.sparsp_sparse_attn_fwd_packed(shape, Q, K, V, mask, rank, P, 0, do["union_mask"], do["seg_offset"],
                                          do["seg_total"], packed, packed.numel(), None, 0.0, O, None, ws)
    assert binding.sparsp_launch_count() - before == 1 + more
    assert binding.sparsp_status(ws) == binding.SPARSP_OK
