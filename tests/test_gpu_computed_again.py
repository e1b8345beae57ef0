"""Items of one and two tiles that are computed again at once, because nothing else is left to do: every row keeps keys 150
log2 units below its reference, which the first pass gets wrong.  The rows of the second pass, which another warpgroup writes,
have to be the ones that stay: output and log-sum-exp against a masked softmax in 64 bits, the same bits in every call."""
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
@pytest.mark.parametrize("tiles", [1, 2])
@pytest.mark.parametrize("H,NB", [(2, 12), (8, 36), (40, 30)])  # one item a CTA, one or two, many
def test_short_items_computed_again(binding, d, b, tiles, H, NB):
    P, consumer, N = 2, 1, NB * b - 3
    g = torch.Generator(device="cuda").manual_seed(d + b + tiles + NB)
    Q, K, V = (torch.randn(1, H, N, d, generator=g, device="cuda") for _ in range(3))
    # channel 0 alone decides: a few keys at +50 log2 units, all others at -100, within about one unit
    unit = math.sqrt(d) / 1.4426950408889634
    high = torch.rand(1, H, N, generator=g, device="cuda") < 0.1
    Q, K = Q * 0.25, K * 0.25
    Q[..., 0] = 4.0
    K[..., 0] = torch.where(high, 50.0, -100.0) * unit / 4.0
    Q, K, V = (x.to(torch.bfloat16) for x in (Q, K, V))
    kept = torch.rand(H, NB, NB, generator=g, device="cuda").argsort(-1).argsort(-1) < tiles * (128 // b)
    words = torch.zeros(1, H, NB, (NB + 31) // 32, dtype=torch.int64, device="cuda")
    for j in range(NB):
        words[0, :, :, j // 32] |= kept[..., j].long() << (j % 32)
    mask = torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32)
    rank = torch.arange(NB, dtype=torch.int32, device="cuda").remainder(P)
    mine = rank.repeat_interleave(b)[:N] == consumer
    shape = binding.make_shape(H, d, (1, 1, N), 0, b)
    ws = binding.make_workspace(shape, P)
    dm = pu.gpu_demand_pack(binding, shape, mask, rank, P, 0, K, V, ws)
    want, want_lse = torch.empty(H, N, d, dtype=torch.float64, device="cuda"), torch.empty(H, N, dtype=torch.float64, device="cuda")
    for h in range(H):
        s = Q[0, h].double() @ K[0, h].double().T / math.sqrt(d)
        s.masked_fill_(~kept[h].repeat_interleave(b, 0).repeat_interleave(b, 1)[:N, :N], float("-inf"))
        want_lse[h] = torch.logsumexp(s, -1)
        want[h] = torch.softmax(s, -1) @ V[0, h].double()
    for packed in (False, True):
        rows = mine if packed else torch.ones_like(mine)
        first = None
        for _ in range(20):
            O, lse = torch.full_like(Q, 5.0), torch.full((1, H, N), 5.0, device="cuda")
            if packed:
                binding.sparsp_sparse_attn_fwd_packed(shape, Q, K, V, mask, rank, P, consumer, dm["union_mask"],
                                                      dm["seg_offset"], dm["seg_total"], dm["packed"], dm["packed"].numel(),
                                                      None, 0.0, O, lse, ws)
            else:
                binding.sparsp_sparse_attn_fwd(shape, Q, K, V, mask, 0.0, O, lse, ws)
            bits = torch.cat([O.view(torch.int16).flatten().int(), lse.view(torch.int32).flatten()])
            first = bits if first is None else first
            assert torch.equal(bits, first)
        assert binding.sparsp_status(ws) == binding.SPARSP_OK
        # bf16 output and bf16 probabilities, |V| up to 5; log-sum-exps of up to 110 in fp32 from sums of such probabilities
        assert (O[0].double() - want)[:, rows].abs().max().item() <= pu.ATTN_MAX_ABS
        assert (lse[0].double() - want_lse)[:, rows].abs().max().item() <= 2e-2
        assert bool((O[:, :, ~rows] == 5.0).all())
