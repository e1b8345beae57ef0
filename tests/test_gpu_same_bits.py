"""A row's attention has the same bits whichever call it comes from: for lists of up to three tiles, whose rows take the first
tile's maximum as their reference in either call, a consumer that owns every block gets from a packed buffer what the call
over the sequence's own K and V returns."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    from paper_2609_32197_b200 import binding as b
    b.lib()
    return b


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("H,NB", [(3, 40), (30, 40)])  # with and without the launch that makes items
def test_source_of_the_tiles(binding, d, H, NB):
    b, P = 128, 2
    N = NB * b - 5
    g = torch.Generator(device="cuda").manual_seed(d + H)
    Q, K, V = (torch.randn(1, H, N, d, generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    # a block keeps itself, which a packed source takes first, and up to two of the blocks behind it
    n_keep = torch.randint(1, 4, (H, NB, 1), generator=g, device="cuda")
    behind = torch.arange(NB, device="cuda")[None] - torch.arange(NB, device="cuda")[:, None]
    kept = (behind >= 0) & (behind < n_keep)
    words = torch.zeros(1, H, NB, 2, dtype=torch.int64, device="cuda")
    for j in range(NB):
        words[0, :, :, j // 32] |= kept[..., j].long() << (j % 32)
    mask = torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32)
    rank = torch.ones(NB, dtype=torch.int32, device="cuda")
    shape = binding.make_shape(H, d, (1, 1, N), 0, b)
    ws = binding.make_workspace(shape, P)
    do = binding.alloc_demand_outputs(shape, P)
    binding.sparsp_demand_pack(shape, mask, rank, P, binding.SPARSP_PLAN_ONLY, None, None, do["union_mask"], do["cnt"],
                               do["seg_offset"], do["seg_total"], do["volume_bytes"], None, 0, None, ws)
    packed = torch.zeros(4 * b * d, dtype=torch.uint8, device="cuda")  # (nothing is remote)
    out = []
    for source in ("own", "packed"):
        O, lse = torch.full_like(Q, 5.0), torch.full((1, H, N), 5.0, device="cuda")
        if source == "own":
            binding.sparsp_sparse_attn_fwd(shape, Q, K, V, mask, 0.0, O, lse, ws)
        else:
            binding.sparsp_sparse_attn_fwd_packed(shape, Q, K, V, mask, rank, P, 1, do["union_mask"], do["seg_offset"],
                                                  do["seg_total"], packed, packed.numel(), None, 0.0, O, lse, ws)
        out.append((O.view(torch.int16), lse.view(torch.int32)))
    assert binding.sparsp_status(ws) == binding.SPARSP_OK
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
