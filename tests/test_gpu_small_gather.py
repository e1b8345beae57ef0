"""The gather that makes the unions for itself: both sides of the rules that choose it (4096 mask words; 6 blocks a warp), one
to 64 ranks, batches, own blocks packed or not, ranks that do not exist, a buffer that is too small.  Integers against the
planning call, bytes against the oracle."""
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


@pytest.mark.parametrize("B,H,NB,P,d,b", [(1, 1, 1, 1, 64, 64), (1, 2, 64, 4, 64, 64), (1, 32, 64, 3, 64, 64), (1, 33, 64, 3, 64, 64),
                                          (2, 5, 33, 7, 128, 64), (1, 2, 40, 64, 64, 128), (1, 37, 24, 2, 128, 128),
                                          (1, 37, 25, 2, 128, 128), (2, 3, 70, 8, 64, 64)])
@pytest.mark.parametrize("local", [0, 2])
@pytest.mark.parametrize("density", [0.0, 0.03, 0.4])
def test_small_gather(oracle_mod, binding, B, H, NB, P, d, b, local, density):
    N = NB * b - 11
    rng = np.random.default_rng(H + NB + P)
    K, V = (torch.tensor(rng.standard_normal((B, H, N, d))).to(torch.bfloat16) for _ in range(2))
    M = rng.random((B, H, NB, NB)) < density
    words = np.zeros((B, H, NB, (NB + 31) // 32), np.uint32)
    for j in range(NB):
        words[..., j // 32] |= M[..., j].astype(np.uint32) << np.uint32(j % 32)
    rank = (rng.permutation(NB) % P).astype(np.int32)
    shape = binding.make_shape(H, d, (1, 1, N), 0, b, batch=B)
    ws = binding.make_workspace(shape, P)
    mask_d, Kd, Vd = torch.as_tensor(words.view(np.int32)).cuda(), K.cuda(), V.cuda()
    entry = 4 * b * d

    def call(rank, room):
        rank_d = torch.as_tensor(rank).cuda()
        got, plan = binding.alloc_demand_outputs(shape, P), binding.alloc_demand_outputs(shape, P)
        for x in (*got.values(), *plan.values()):
            x.fill_(-7)
        buf = torch.full((room * entry + 64,), 0xAB, dtype=torch.uint8, device="cuda")
        binding.sparsp_demand_pack(shape, mask_d, rank_d, P, local, Kd, Vd, got["union_mask"], got["cnt"], got["seg_offset"],
                                   got["seg_total"], got["volume_bytes"], buf, room * entry, None, ws)
        binding.sparsp_demand_plan_noalloc(shape, mask_d, rank_d, P, local, plan["union_mask"], plan["cnt"],
                                           plan["seg_offset"], plan["seg_total"], plan["volume_bytes"])
        for k in plan:
            assert torch.equal(got[k], plan[k]), k
        return buf.cpu().numpy(), int(plan["seg_total"].sum())

    want = []
    for bb in range(B):
        ref = oracle_mod.demand(words[bb], rank, P, b, d, include_local=bool(local))
        want.append(oracle_mod.pack(K[bb], V[bb], ref["U"], rank, b, P, ref["total"], include_local=bool(local)))
    want = np.concatenate(want)
    n = want.size // entry
    for room in (n + 1, n):
        got, total = call(rank, room)
        assert total == n and binding.sparsp_status(ws) == binding.SPARSP_OK
        assert np.array_equal(got[:want.size], want) and (got[want.size:] == 0xAB).all()
    if n:  # the last entry does not fit
        got, _ = call(rank, n - 1)
        assert binding.sparsp_status(ws) == binding.SPARSP_ERR_CAPACITY
        assert np.array_equal(got[:want.size - entry], want[:want.size - entry]) and (got[want.size - entry:] == 0xAB).all()
    strange = rank.copy()
    strange[::3] = P + 5
    strange[::4] = -1
    call(strange, n + NB * H * B * P)
    assert binding.sparsp_status(ws) == binding.SPARSP_OK
