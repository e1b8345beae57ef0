"""Which calls do without a launch, seen from the number of launches.  Attention without the one that makes its items: 64-token blocks up to
one an SM (more of them share Q tiles), 128-token blocks up to two, and a packed source where a CTA has one item at most if the
consumer has its share of the blocks, and the items can be put in order if it has more.  The gather without the one that makes
the unions: up to 4096 mask words and four blocks a warp, or 2560 words and six blocks."""
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


@pytest.mark.parametrize("b,H,NB,P,launches", [
    # one item an SM (148) by an even share of the blocks, and one more
    (128, 1, 148, 1, 1), (128, 1, 149, 1, 2), (64, 1, 296, 1, 1), (64, 1, 297, 1, 2), (128, 4, 74, 2, 1), (128, 4, 76, 2, 2),
    # 1024 items if it owns all blocks, and more; half of that with more than 512 blocks a head
    (128, 8, 128, 8, 1), (128, 8, 129, 8, 2), (64, 4, 512, 8, 1), (64, 2, 513, 8, 2), (128, 1, 512, 8, 1),
    (128, 1, 513, 8, 2), (64, 1, 1024, 8, 1)])
def test_packed(binding, b, H, NB, P, launches):
    shape, Q, K, V, mask = _inputs(binding, b, H, NB)
    ws = binding.make_workspace(shape, P)
    rank = torch.zeros(NB, dtype=torch.int32, device="cuda")
    do = binding.alloc_demand_outputs(shape, P)
    binding.sparsp_demand_pack(shape, mask, rank, P, binding.SPARSP_PLAN_ONLY, None, None, do["union_mask"], do["cnt"],
                               do["seg_offset"], do["seg_total"], do["volume_bytes"], None, 0, None, ws)
    packed, O = torch.zeros(4 * b * 64, dtype=torch.uint8, device="cuda"), torch.empty_like(Q)
    before = binding.sparsp_launch_count()
    binding.sparsp_sparse_attn_fwd_packed(shape, Q, K, V, mask, rank, P, 0, do["union_mask"], do["seg_offset"],
                                          do["seg_total"], packed, packed.numel(), None, 0.0, O, None, ws)
    assert binding.sparsp_launch_count() - before == launches
    assert binding.sparsp_status(ws) == binding.SPARSP_OK


@pytest.mark.parametrize("H,NB,launches", [(4, 144, 1), (5, 118, 1), (5, 128, 1), (5, 129, 2), (13, 64, 1), (14, 64, 2),
                                           (1, 362, 2)])
def test_gather(binding, H, NB, launches):
    b, d, P = 128, 128, 3  # one warp copies a block
    shape, _, K, V, mask = _inputs(binding, b, H, NB, d)
    ws = binding.make_workspace(shape, P)
    rank = torch.arange(NB, dtype=torch.int32, device="cuda").remainder(P)
    do = binding.alloc_demand_outputs(shape, P)
    packed = torch.zeros(4 * b * d * H * P, dtype=torch.uint8, device="cuda")
    before = binding.sparsp_launch_count()
    binding.sparsp_demand_pack(shape, mask, rank, P, 0, K, V, do["union_mask"], do["cnt"], do["seg_offset"], do["seg_total"],
                               do["volume_bytes"], packed, packed.numel(), None, ws)
    assert binding.sparsp_launch_count() - before == launches
    assert binding.sparsp_status(ws) == binding.SPARSP_OK
