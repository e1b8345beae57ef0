"""A plan does not depend on what the workspace holds: calls on a workspace of any contents, its header too, write the plan that
the call without a workspace returns.  Both sides of the rule that picks one launch (one to three heads a CTA and more, with
short and long rows; consumers x CTAs up to the number of multiprocessors and beyond), consumers without
blocks, ranks outside the range, own blocks packed or not."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    from paper_2609_32197_b200 import binding as b
    b.lib()
    return b


@pytest.mark.parametrize("B,P,H,NB", [(1, 1, 1, 1), (1, 2, 3, 33), (1, 4, 2, 64), (2, 9, 8, 70), (1, 18, 8, 90), (1, 19, 8, 90), (1, 5, 9, 100),
                                      (1, 18, 16, 40), (1, 8, 17, 929), (1, 8, 16, 1024), (1, 2, 16, 1024), (1, 2, 12, 600), (1, 8, 24, 929),
                                      (1, 11, 21, 130), (1, 2, 16, 500), (1, 4, 24, 384), (1, 2, 25, 64),
                                      (1, 37, 4, 96), (1, 64, 2, 200), (49, 3, 1, 20), (1, 2, 48, 300)])
@pytest.mark.parametrize("fill", [0, -1, 2])
def test_plan_on_any_workspace(binding, B, P, H, NB, fill):
    g = torch.Generator(device="cuda").manual_seed(B + P + H + NB)
    shape = binding.make_shape(H, 64, (1, 1, NB * 64), 0, 64, batch=B)
    ws = binding.make_workspace(shape, P)
    rank = torch.randint(0, P, (NB,), generator=g, device="cuda", dtype=torch.int32)
    rank[rank == P // 2] = 0    # a consumer that owns nothing
    rank[NB // 2::7] = P + 3    # blocks that nobody owns
    bits = torch.rand(B, H, NB, NB, generator=g, device="cuda") < 0.05
    words = torch.zeros(B, H, NB, (NB + 31) // 32, dtype=torch.int64, device="cuda")
    for j in range(NB):
        words[..., j // 32] |= bits[..., j].long() << (j % 32)
    mask = torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32)
    for local in (0, binding.SPARSP_INCLUDE_LOCAL):
        got, want = binding.alloc_demand_outputs(shape, P), binding.alloc_demand_outputs(shape, P)
        for x in (*got.values(), *want.values()):
            x.fill_(-7)
        ws[:1 << 20] = fill & 255
        for _ in range(2):
            binding.sparsp_demand_pack(shape, mask, rank, P, binding.SPARSP_PLAN_ONLY | local, None, None, got["union_mask"],
                                       got["cnt"], got["seg_offset"], got["seg_total"], got["volume_bytes"], None, 0, None, ws)
        binding.sparsp_demand_plan_noalloc(shape, mask, rank, P, local, want["union_mask"], want["cnt"], want["seg_offset"],
                                           want["seg_total"], want["volume_bytes"])
        torch.cuda.synchronize()
        for k in want:
            assert torch.equal(got[k], want[k]), (k, local)
