"""Attention items of every length one behind the other: where an item ends, one warpgroup writes its rows while the other
one is at the next item, whose Q tile has taken a buffer of the K ring.  Lists of 1 to 11 tiles in random order, many items
to a CTA, odd and even numbers of entries and a ragged last block, against a masked softmax in 64 bits; K and V in place and
from a packed buffer; once more with the output in the place of the queries.  The log-sum-exps, which the same warpgroup writes
from the reference that its last tile was taken relative to, in all three; with a few heads whose scores leave the range."""
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
@pytest.mark.parametrize("longest", [1, 2, 3, 5, 11])
def test_items_of_every_length(binding, d, b, longest):
    H, NB, P, consumer = 48, 24, 2, 1
    N = NB * b - 5
    g = torch.Generator(device="cuda").manual_seed(d + b + longest)
    Q, K, V = (torch.randn(1, H, N, d, generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    Q[:, 5::11] *= 60.0
    # rows keep between one block and `longest` tiles of blocks
    n_keep = torch.randint(1, longest * (128 // b) + 1, (H, NB, 1), generator=g, device="cuda").clamp(max=NB)
    kept = torch.rand(H, NB, NB, generator=g, device="cuda").argsort(-1).argsort(-1) < n_keep
    words = (kept.long() << torch.arange(NB, device="cuda")).sum(-1, keepdim=True).to(torch.int32)
    rank_d = torch.arange(NB, dtype=torch.int32, device="cuda").remainder(P)
    shape = binding.make_shape(H, d, (1, 1, N), 0, b)
    ws = binding.make_workspace(shape, P)
    want, want_lse = torch.empty(H, N, d, dtype=torch.float64, device="cuda"), torch.empty(H, N, dtype=torch.float64, device="cuda")
    for h in range(H):
        s = Q[0, h].double() @ K[0, h].double().T / math.sqrt(d)
        s.masked_fill_(~kept[h].repeat_interleave(b, 0).repeat_interleave(b, 1)[:N, :N], float("-inf"))
        want[h] = torch.softmax(s, -1) @ V[0, h].double()
        want_lse[h] = torch.logsumexp(s, -1)

    def check(O, lse, rows):
        # bf16 output (2^-9 of values up to 5) and bf16 probabilities (2^-9 of their sum times |V| up to 5)
        assert (O[0].double() - want)[:, rows].abs().max().item() <= pu.ATTN_MAX_ABS
        # sums of bf16 probabilities; an fp32 number of up to hundreds: eight units in the last place on top
        assert bool(((lse[0].double() - want_lse).abs() <= 2e-2 + want_lse.abs() * 2.0 ** -20)[:, rows].all())
        assert binding.sparsp_status(ws) == binding.SPARSP_OK

    every = torch.ones(N, dtype=torch.bool, device="cuda")
    O, lse = torch.full_like(Q, 5.0), torch.zeros(1, H, N, device="cuda")
    binding.sparsp_sparse_attn_fwd(shape, Q, K, V, words, 0.0, O, lse, ws)
    check(O, lse, every)
    mine = rank_d.repeat_interleave(b)[:N] == consumer
    dm = pu.gpu_demand_pack(binding, shape, words, rank_d, P, 0, K, V, ws)
    part, part_lse = torch.full_like(Q, 5.0), torch.full((1, H, N), 5.0, device="cuda")
    binding.sparsp_sparse_attn_fwd_packed(shape, Q, K, V, words, rank_d, P, consumer, dm["union_mask"], dm["seg_offset"],
                                          dm["seg_total"], dm["packed"], dm["packed"].numel(), None, 0.0, part,
                                          part_lse, ws)
    check(part, part_lse, mine)
    assert bool((part[:, :, ~mine] == 5.0).all()) and bool((part_lse[:, :, ~mine] == 5.0).all())
    again, again_lse = Q.clone(), torch.zeros_like(lse)
    binding.sparsp_sparse_attn_fwd(shape, again, K, V, words, 0.0, again, again_lse, ws)
    assert torch.equal(again.view(torch.int16), O.view(torch.int16)) and torch.equal(again_lse, lse)
