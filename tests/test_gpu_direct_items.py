"""Attention calls of few query blocks, whose CTAs put the items in order for themselves: one and two an SM and one more than
that, rows of one to eight mask words, lists of every length in any order, rows and heads that keep nothing; and calls of many
blocks in few heads, whose items are put in order by counting.  Rows and their log-sum-exps against a masked softmax in 64
bits, also with scores that leave the range."""
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
@pytest.mark.parametrize("B,H,NB", [(1, 1, 1), (1, 4, 37), (1, 1, 149), (2, 2, 74), (1, 2, 148), (1, 11, 27), (1, 99, 3), (1, 1, 255),
                                    (1, 2, 260), (1, 1, 700)])
@pytest.mark.parametrize("far", [1.0, 60.0])
def test_few_items(binding, d, b, B, H, NB, far):
    if NB > 260 and b == 128:
        pytest.skip("64-bit scores of as many tokens")
    N = NB * b - 9 if NB > 1 else b
    g = torch.Generator(device="cuda").manual_seed(H + NB + d + b)
    Q, K, V = (torch.randn(B, H, N, d, generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    Q[:, ::2] *= far
    # between nothing and forty blocks a row; every fifth row and every seventh head keep nothing
    n_keep = torch.randint(0, min(NB, 40) + 1, (B, H, NB, 1), generator=g, device="cuda")
    n_keep[:, :, ::5] = 0 if NB > 4 else n_keep[:, :, ::5]
    n_keep[:, 6::7] = 0
    kept = torch.rand(B, H, NB, NB, generator=g, device="cuda").argsort(-1).argsort(-1) < n_keep
    words = torch.zeros(B, H, NB, (NB + 31) // 32, dtype=torch.int64, device="cuda")
    for j in range(NB):
        words[..., j // 32] |= kept[..., j].long() << (j % 32)
    shape = binding.make_shape(H, d, (1, 1, N), 0, b, batch=B)
    ws = binding.make_workspace(shape, 1)
    O, lse = torch.full_like(Q, 5.0), torch.full((B, H, N), 5.0, device="cuda")
    binding.sparsp_sparse_attn_fwd(shape, Q, K, V, words.to(torch.int32), 0.0, O, lse, ws)
    assert binding.sparsp_status(ws) == binding.SPARSP_OK
    for bb in range(B):
        for h in range(H):
            for r0 in range(0, N, 8192):  # rows at a time
                rows = slice(r0, min(N, r0 + 8192))
                tokens = kept[bb, h].repeat_interleave(b, 0)[rows].repeat_interleave(b, 1)[:, :N]
                s = (Q[bb, h, rows].double() @ K[bb, h].double().T / math.sqrt(d)).masked_fill(~tokens, float("-inf"))
                live = tokens.any(-1)
                want = torch.softmax(s, -1) @ V[bb, h].double()
                # bf16 output and bf16 probabilities, |V| up to 5
                assert not live.any() or (O[bb, h, rows].double() - want)[live].abs().max().item() <= pu.ATTN_MAX_ABS
                # sums of bf16 probabilities; an fp32 number of up to hundreds: eight units in the last place on top
                wl = torch.logsumexp(s, -1)[live]
                assert bool(((lse[bb, h, rows][live].double() - wl).abs() <= 2e-2 + wl.abs() * 2.0 ** -20).all())
                assert bool((O[bb, h, rows][~live] == 0).all()) and bool((lse[bb, h, rows][~live] == float("-inf")).all())
