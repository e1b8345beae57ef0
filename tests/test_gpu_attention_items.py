"""Attention over masks in which query blocks, and whole heads, keep nothing: such blocks are no work items, their rows are
cleared, and the items of more heads than a warp has lanes are found."""
import numpy as np
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
@pytest.mark.parametrize("layout", ["HND", "NHD"])
@pytest.mark.parametrize("H,live", [(1, "some"), (37, "some"), (70, "some"), (70, "last"), (37, "none")])
def test_rows_and_heads_that_keep_nothing(oracle_mod, binding, d, b, layout, H, live):
    NB, P, consumer = 9, 3, 1
    N = NB * b - 13
    rng = np.random.default_rng(H + d + b)
    Q, K, V = (torch.tensor(rng.standard_normal((H, N, d)) * 0.7).to(torch.bfloat16) for _ in range(3))
    M = rng.random((H, NB, NB)) < 0.4
    M[:, 2] = False                                   # a query block without any kept block in every head ...
    M[:, 7, :] = rng.random((H, 1)) < 0.3             # ... and one that keeps all or nothing
    M[rng.random(H) < 0.4] = False                    # whole heads
    if live == "last":
        M[:-1] = False
        M[-1, 3:6] = True
    if live == "none":
        M[:] = False
    words = np.zeros((H, NB, 1), np.uint32)
    for j in range(NB):
        words[:, :, 0] |= M[:, :, j].astype(np.uint32) << np.uint32(j)
    rank = np.array([j % P for j in range(NB)], np.int32)
    shape = binding.make_shape(H, d, (1, 1, N), 0, b, layout=layout)
    ws = binding.make_workspace(shape, P)
    Qd, Kd, Vd = (pu.to_layout(x, layout).cuda() for x in (Q, K, V))
    mask_d, rank_d = torch.as_tensor(words.view(np.int32)).cuda(), torch.as_tensor(rank).cuda()
    want, want_lse = oracle_mod.attn_all(Q, K, V, words, b)
    empty = torch.tensor(~M.any(-1)).repeat_interleave(b, 1)[:, :N]

    def check(O, lse, rows):
        got = pu.from_layout(O, layout).float().cpu()
        assert np.abs(got.numpy() - want)[:, rows].max() <= pu.ATTN_MAX_ABS
        assert bool((got[:, rows][empty[:, rows]] == 0).all())
        l = lse[0].cpu()
        assert bool((l[:, rows][empty[:, rows]] == float("-inf")).all())
        full = ~empty[:, rows]
        assert not bool(full.any()) or (l[:, rows][full] - torch.tensor(want_lse)[:, rows][full]).abs().max() < 2e-2

    # every rank's rows, K and V in place; outputs start as garbage
    O = torch.full_like(Qd, 5.0)
    lse = torch.full((1, H, N), 5.0, device="cuda")
    binding.sparsp_sparse_attn_fwd(shape, Qd, Kd, Vd, mask_d, 0.0, O, lse, ws)
    check(O, lse, torch.arange(N))
    # one rank's rows over its packed buffer; the other ranks' rows stay as they are
    dm = pu.gpu_demand_pack(binding, shape, mask_d, rank_d, P, 0, Kd, Vd, ws)
    packed = torch.nn.functional.pad(dm["packed"], (0, 4 * b * d))  # room for a tile even if nothing is packed
    O.fill_(5.0)
    lse.fill_(5.0)
    binding.sparsp_sparse_attn_fwd_packed(shape, Qd, Kd, Vd, mask_d, rank_d, P, consumer, dm["union_mask"],
                                          dm["seg_offset"], dm["seg_total"], packed, packed.numel(), None,
                                          0.0, O, lse, ws)
    mine = torch.as_tensor(rank).repeat_interleave(b)[:N] == consumer
    check(O, lse, torch.nonzero(mine)[:, 0])
    assert bool((pu.from_layout(O, layout).cpu()[:, ~mine] == 5.0).all()) and bool((lse[0].cpu()[:, ~mine] == 5.0).all())
    assert binding.sparsp_status(ws) == binding.SPARSP_OK


@pytest.mark.parametrize("d", [64, 128])
def test_stacked_blocks_of_a_packed_source_are_neighbours(binding, d):
    """64-token blocks: the rows of two neighbours in the consumer's list come out bit for bit the same whatever the
    consumer's other blocks keep, also where one of those keeps exactly what the first of the two keeps (the order in which
    a row meets its scores, and with it every rounding, depends on the block it is stacked with)."""
    H, NB, P, b = 2, 16, 2, 64
    N = NB * b
    rng = np.random.default_rng(d)
    Q, K, V = (torch.tensor(rng.standard_normal((1, H, N, d)) * s).to(torch.bfloat16).cuda() for s in (3.0, 1.0, 1.0))
    rank_d = torch.arange(NB, dtype=torch.int32).remainder(P).cuda()  # the consumer's list: blocks 0, 2, 4, ...
    shape = binding.make_shape(H, d, (1, 1, N), 0, b)
    ws = binding.make_workspace(shape, P)
    first, second = 0b0101010101010101, 0b0011001101100110  # half of the first's blocks, and others

    def rows_of_the_first_two(others):
        words = np.zeros((H, NB, 1), np.uint32)
        words[:, 0, 0], words[:, 2, 0] = first, second
        for pos in range(2, NB // 2):
            words[:, 2 * pos, 0] = others[pos]
        mask_d = torch.as_tensor(words.view(np.int32)).cuda()
        dm = pu.gpu_demand_pack(binding, shape, mask_d, rank_d, P, 0, K, V, ws)
        O, lse = torch.zeros_like(Q), torch.zeros(1, H, N, device="cuda")
        binding.sparsp_sparse_attn_fwd_packed(shape, Q, K, V, mask_d, rank_d, P, 0, dm["union_mask"], dm["seg_offset"],
                                              dm["seg_total"], dm["packed"], dm["packed"].numel(), None, 0.0, O, lse, ws)
        assert binding.sparsp_status(ws) == binding.SPARSP_OK
        mine = torch.cat([torch.arange(b), torch.arange(2 * b, 3 * b)]).cuda()
        return O[:, :, mine].view(torch.int16), lse[:, :, mine].view(torch.int32)

    apart = [1 << (2 * (pos % 2) + 1) for pos in range(NB // 2)]
    want = rows_of_the_first_two(apart)
    for twin in (2, 3, 4):
        got = rows_of_the_first_two(apart[:twin] + [first] + apart[twin + 1:])
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1]), twin
