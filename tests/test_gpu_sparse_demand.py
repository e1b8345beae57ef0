"""Demand in few heads and blocks, or none: the gather hands out only blocks that anybody receives, and a segment's walk goes
straight to the heads that have entries.  And the gather at the edge of its shared memory, where the one by tables begins."""
import numpy as np
import pytest
import torch

import parity_util as pu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    from paper_2609_32197_b200 import binding as b
    return b


def _words(M):
    H, NB = M.shape[:2]
    words = np.zeros((H, NB, (NB + 31) // 32), np.uint32)
    for j in range(NB):
        words[:, :, j // 32] |= M[:, :, j].astype(np.uint32) << np.uint32(j % 32)
    return words


def _pack(oracle_mod, binding, M, P, rank, d, b, local, ragged=19):
    H, NB = M.shape[:2]
    N = NB * b - ragged
    rng = np.random.default_rng(NB + P)
    K, V = (torch.tensor(rng.standard_normal((H, N, d))).to(torch.bfloat16) for _ in range(2))
    words = _words(M)
    shape = binding.make_shape(H, d, (1, 1, N), 0, b)
    mask_d, rank_d = torch.as_tensor(words.view(np.int32)).cuda(), torch.as_tensor(rank).cuda()
    ws = binding.make_workspace(shape, P)
    K, V = K.cuda(), V.cuda()
    got = pu.gpu_demand_pack(binding, shape, mask_d, rank_d, P, binding.SPARSP_INCLUDE_LOCAL if local else 0, K, V, ws)
    ref = pu.check_demand(oracle_mod, binding, shape, words, rank, P, local, got)
    h, j = pu.oracle_entry_list(ref, rank, P, H, NB, local)
    pu.check_packed_full_on_device(K, V, b, got["packed"], h, j)
    assert binding.sparsp_status(ws) == binding.SPARSP_OK
    return K, V, shape, rank_d, ws, got


@pytest.mark.parametrize("what", ["nothing", "own blocks", "last block of the last head", "one head", "one in a word"])
@pytest.mark.parametrize("H,NB,P", [(5, 70, 3), (40, 33, 8), (1, 1000, 64), (3, 64, 1)])
@pytest.mark.parametrize("local", [False, True])
def test_only_what_is_wanted(oracle_mod, binding, what, H, NB, P, local):
    rank = (np.arange(NB) * P // NB).astype(np.int32)
    M = np.zeros((H, NB, NB), bool)
    if what == "own blocks":
        M[:, np.arange(NB), np.arange(NB)] = True
    elif what == "last block of the last head":
        M[-1, 0, -1] = True
    elif what == "one head":
        M[H // 2] = np.random.default_rng(1).random((NB, NB)) < 0.1
    elif what == "one in a word":
        M[:, :, 31::32] = True
    _pack(oracle_mod, binding, M, P, rank, 64, 64, local)


# words of shared memory behind the rings: H P^2 + 2 H Wd + P Wd + 2 = 7168 at 736 blocks (23 words), 7226 at 737, and the
# same sum for the longest rows: 6466 and 7554
@pytest.mark.parametrize("H,P,NB", [(2, 54, 736), (2, 54, 737), (5, 32, 1000), (6, 32, 1000)])
def test_edge_of_the_shared_memory(oracle_mod, binding, H, P, NB):
    rng = np.random.default_rng(NB)
    M = rng.random((H, NB, NB)) < 0.004
    _pack(oracle_mod, binding, M, P, (rng.permutation(NB) % P).astype(np.int32), 64, 64, False)


@pytest.mark.parametrize("heads", ["first", "last", "around a search step", "every other"])
@pytest.mark.parametrize("H,NB", [(1, 40), (33, 9), (70, 33), (1030, 5)])
def test_segments_of_few_heads(oracle_mod, binding, heads, H, NB):
    P, d, b = 3, 64, 64
    entry = 4 * b * d
    rng = np.random.default_rng(H)
    live = {"first": [0], "last": [H - 1], "around a search step": [h for h in (30, 31, 32, 33, 65, 1023, 1024) if h < H],
            "every other": list(range(1, H, 2))}[heads]
    M = np.zeros((H, NB, NB), bool)
    M[live] = rng.random((len(live), NB, NB)) < 0.5
    rank = (rng.permutation(NB) % P).astype(np.int32)
    K, V, shape, rank_d, ws, got = _pack(oracle_mod, binding, M, P, rank, d, b, False)
    cnt, seg, total = got["cnt"][0].cpu(), got["seg_offset"][0].cpu(), got["seg_total"][0].cpu()
    start = torch.cat([torch.zeros(1, dtype=torch.int64), total.cumsum(0)]) * entry
    for r in range(P):
        for p in range(P):
            n = int(cnt[r, p].sum())
            if p == r:
                continue
            first = int(start[r]) + int(seg[r, p, 0]) * entry
            slot = torch.full(((n + 1) * entry,), 0xEE, dtype=torch.uint8, device="cuda")
            binding.sparsp_pack_segment(shape, got["union_mask"], rank_d, P, r, p, got["cnt"], got["seg_offset"], K, V, slot,
                                        n * entry, ws)
            assert binding.sparsp_status(ws) == binding.SPARSP_OK
            assert torch.equal(slot[:n * entry], got["packed"][first:first + n * entry])
            assert bool((slot[n * entry:] == 0xEE).all())
