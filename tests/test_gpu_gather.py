"""The gather without tables, at the edge of the number of counts that it takes, and one producer's segments, which are
walked forwards for even and backwards for odd consumers."""
import numpy as np
import pytest
import torch

import parity_util as pu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    from paper_2609_32197_b200 import binding as b
    return b


def _case(binding, H, NB, P, d, b, density, seed):
    N = NB * b - 19
    rng = np.random.default_rng(seed)
    K, V = (torch.tensor(rng.standard_normal((H, N, d))).to(torch.bfloat16) for _ in range(2))
    M = rng.random((H, NB, NB)) < density
    M[1::5] = False  # heads that nobody selects from
    words = np.zeros((H, NB, (NB + 31) // 32), np.uint32)
    for j in range(NB):
        words[:, :, j // 32] |= M[:, :, j].astype(np.uint32) << np.uint32(j % 32)
    rank = (rng.permutation(NB) % P).astype(np.int32)
    shape = binding.make_shape(H, d, (1, 1, N), 0, b)
    return K, V, words, rank, shape, torch.as_tensor(words.view(np.int32)).cuda(), torch.as_tensor(rank).cuda()


@pytest.mark.parametrize("H,P", [(24, 16), (25, 16), (1, 64), (2, 64)])  # 6144 and 6400, 4096 and 8192 counts
@pytest.mark.parametrize("local", [False, True])
@pytest.mark.parametrize("bases", [False, True])
def test_edge_of_the_scan(oracle_mod, binding, H, P, local, bases):
    d, b, NB = 64, 64, 70
    K, V, words, rank, shape, mask_d, rank_d = _case(binding, H, NB, P, d, b, 0.1, H + P)
    ws = binding.make_workspace(shape, P)
    flags = binding.SPARSP_INCLUDE_LOCAL if local else 0
    got = pu.gpu_demand_pack(binding, shape, mask_d, rank_d, P, flags, K.cuda(), V.cuda(), ws)
    ref = pu.check_demand(oracle_mod, binding, shape, words, rank, P, local, got)
    want = oracle_mod.pack(K, V, ref["U"], rank, b, P, ref["total"], include_local=local)
    packed = got["packed"].cpu().numpy()
    assert np.array_equal(packed[:want.size], want) and (packed[want.size:] == 0xAB).all()
    if bases:  # consumers in descending order with a gap of one entry, the last of them cut off by the capacity
        entry = 4 * b * d
        total = np.asarray(ref["total"])
        base = np.zeros(P, np.int64)
        for r in range(P - 2, -1, -1):
            base[r] = base[r + 1] + (total[r + 1] + 1) * entry
        end = int(base[0] + total[0] * entry)
        room = end - (entry if total[0] > 0 else 0)
        buf = torch.full((end + entry,), 0xCD, dtype=torch.uint8, device="cuda")
        binding.sparsp_demand_pack(shape, mask_d, rank_d, P, flags, K.cuda(), V.cuda(), got["union_mask"], got["cnt"],
                                   got["seg_offset"], got["seg_total"], got["volume_bytes"], buf, room,
                                   torch.as_tensor(base).cuda(), ws)
        assert binding.sparsp_status(ws) == (binding.SPARSP_ERR_CAPACITY if total[0] > 0 else binding.SPARSP_OK)
        out, first = buf.cpu().numpy(), np.concatenate([[0], np.cumsum(total)]) * entry
        for r in range(P):
            n = int(total[r] * entry) - (entry if r == 0 and total[0] > 0 else 0)
            assert np.array_equal(out[base[r]:base[r] + n], want[first[r]:first[r] + n]), r
            assert (out[base[r] + n:base[r] + n + entry] == 0xCD).all(), r


@pytest.mark.parametrize("d,b,H,NB", [(64, 64, 7, 70), (128, 128, 40, 33), (64, 128, 1, 100), (128, 64, 33, 9)])
def test_segments_are_slices_of_the_packed_buffer(binding, d, b, H, NB):
    P, entry = 3, 4 * b * d
    K, V, _, _, shape, mask_d, rank_d = _case(binding, H, NB, P, d, b, 0.3, H)
    K, V = K.cuda(), V.cuda()
    ws = binding.make_workspace(shape, P)
    got = pu.gpu_demand_pack(binding, shape, mask_d, rank_d, P, 0, K, V, ws)
    cnt, seg, total = got["cnt"][0].cpu(), got["seg_offset"][0].cpu(), got["seg_total"][0].cpu()
    start = torch.cat([torch.zeros(1, dtype=torch.int64), total.cumsum(0)]) * entry
    for r in range(P):
        for p in range(P):
            if p == r:
                continue
            n = int(cnt[r, p].sum())
            first = int(start[r]) + int(seg[r, p, 0]) * entry
            want = got["packed"][first:first + n * entry]
            for cut in (0, 1):  # room for all entries, for all but one
                if n < cut:
                    continue
                room = (n - cut) * entry
                slot = torch.full(((n + 1) * entry,), 0xEE, dtype=torch.uint8, device="cuda")
                binding.sparsp_pack_segment(shape, got["union_mask"], rank_d, P, r, p, got["cnt"], got["seg_offset"], K, V,
                                            slot, room, ws)
                assert binding.sparsp_status(ws) == (binding.SPARSP_ERR_CAPACITY if cut else binding.SPARSP_OK)
                assert torch.equal(slot[:room], want[:room]) and bool((slot[room:] == 0xEE).all())
