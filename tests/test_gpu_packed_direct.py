"""Attention over a packed buffer with and without the launch that numbers items and places: both sides of the rule between
them (an item an SM if the consumer has its share of the blocks, 1024 if it has all of them), consumers that own nearly all, one
or none of the blocks, 64 ranks, batches, explicit slot bases, empty rows and heads, keys far out of range.  Foreign K and V are
not numbers; rows and their log-sum-exps against a masked softmax in 64 bits."""
import math

import pytest
import torch

import parity_util as pu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    from paper_2609_32197_b200 import binding as b
    b.lib()
    return b


@pytest.mark.parametrize("d,b", [(64, 64), (128, 64), (64, 128), (128, 128)])
@pytest.mark.parametrize("B,H,NB,P,owner", [(1, 1, 1, 1, "even"), (1, 2, 9, 3, "even"), (2, 3, 40, 4, "even"),
                                            (1, 8, 74, 2, "even"), (1, 9, 74, 2, "even"), (1, 16, 74, 2, "even"),
                                            (1, 17, 74, 2, "even"), (1, 30, 33, 8, "most"), (1, 4, 70, 64, "even"),
                                            (1, 6, 40, 4, "one"), (1, 6, 40, 4, "none")])
@pytest.mark.parametrize("bases,far", [(False, 1.0), (True, 60.0)])
def test_packed_rows(binding, d, b, B, H, NB, P, owner, bases, far):
    N, consumer = NB * b - 7, P // 2
    g = torch.Generator(device="cuda").manual_seed(H + NB + P + d + b)
    Q, K, V = (torch.randn(B, H, N, d, generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    Q[:, ::2] *= far  # every second head's scores leave the range that an item assumes
    rank = torch.randperm(NB, generator=g, device="cuda").remainder(P)
    if owner == "most":
        rank[torch.rand(NB, generator=g, device="cuda") < 0.9] = consumer
    elif owner in ("one", "none"):
        rank[rank == consumer] = consumer - 1
        if owner == "one":
            rank[5] = consumer
    rank = rank.to(torch.int32)
    kept = torch.rand(B, H, NB, NB, generator=g, device="cuda") < 0.2
    kept[:, :, 1::4] = False          # rows that keep nothing
    kept[:, 2::3] = False             # heads that do
    words = torch.zeros(B, H, NB, (NB + 31) // 32, dtype=torch.int64, device="cuda")
    for j in range(NB):
        words[..., j // 32] |= kept[..., j].long() << (j % 32)
    mask = words.to(torch.int32)
    shape = binding.make_shape(H, d, (1, 1, N), 0, b, batch=B)
    ws = binding.make_workspace(shape, P)
    do = binding.alloc_demand_outputs(shape, P)
    entry, room = 4 * b * d, B * P * H * NB + 2 * B * P
    packed = torch.zeros(room * entry, dtype=torch.uint8, device="cuda")
    base = None
    if bases:  # slots in descending order, each an odd number of tiles apart
        binding.sparsp_demand_pack(shape, mask, rank, P, binding.SPARSP_PLAN_ONLY, None, None, do["union_mask"], do["cnt"],
                                   do["seg_offset"], do["seg_total"], do["volume_bytes"], None, 0, None, ws)
        size = do["seg_total"].flatten() * entry + entry // 2
        base = (size.flip(0).cumsum(0).flip(0) - size).view(B, P).contiguous()
    binding.sparsp_demand_pack(shape, mask, rank, P, 0, K, V, do["union_mask"], do["cnt"], do["seg_offset"], do["seg_total"],
                               do["volume_bytes"], packed, packed.numel(), base, ws)
    mine = (rank == consumer).repeat_interleave(b)[:N]
    Kp, Vp = K.clone(), V.clone()
    Kp[:, :, ~mine], Vp[:, :, ~mine] = float("nan"), float("nan")
    O, lse = torch.full_like(Q, 5.0), torch.full((B, H, N), 5.0, device="cuda")
    binding.sparsp_sparse_attn_fwd_packed(shape, Q, Kp, Vp, mask, rank, P, consumer, do["union_mask"], do["seg_offset"],
                                          do["seg_total"], packed, packed.numel(), base, 0.0, O, lse, ws)
    assert binding.sparsp_status(ws) == binding.SPARSP_OK
    assert bool((O[:, :, ~mine] == 5.0).all()) and bool((lse[:, :, ~mine] == 5.0).all())
    for bb in range(B):
        for h in range(H):
            tokens = kept[bb, h].repeat_interleave(b, 0).repeat_interleave(b, 1)[:N, :N]
            s = (Q[bb, h].double() @ K[bb, h].double().T / math.sqrt(d)).masked_fill(~tokens, float("-inf"))
            live = mine & tokens.any(-1)
            want = torch.softmax(s[live], -1) @ V[bb, h].double()
            # bf16 output and bf16 probabilities, |V| up to 5
            assert live.sum() == 0 or (O[bb, h, live].double() - want).abs().max().item() <= pu.ATTN_MAX_ABS
            # sums of bf16 probabilities; an fp32 number of up to hundreds: eight units in the last place on top
            wl = torch.logsumexp(s[live], -1)
            assert bool(((lse[bb, h, live].double() - wl).abs() <= 2e-2 + wl.abs() * 2.0 ** -20).all())
            assert bool((O[bb, h, mine & ~live] == 0).all()) and bool((lse[bb, h, mine & ~live] == float("-inf")).all())


# consumers with far more than their share, whose items the CTAs put in order: as many as there is room for, one more, batches
@pytest.mark.parametrize("d,b", [(64, 64), (128, 64), (64, 128), (128, 128)])
@pytest.mark.parametrize("B,H,NB,P", [(1, 8, 60, 8), (1, 8, 64, 8), (2, 4, 64, 8), (1, 16, 64, 8), (1, 16, 65, 8), (1, 2, 200, 16),
                                      (3, 5, 34, 4), (1, 1, 480, 8), (1, 16, 128, 16)])
@pytest.mark.parametrize("far", [1.0, 60.0])
def test_more_than_its_share(binding, d, b, B, H, NB, P, far):
    if NB > 260 and b == 128:
        pytest.skip("64-bit scores of as many tokens")
    test_packed_rows(binding, d, b, B, H, NB, P, "most", False, far)
