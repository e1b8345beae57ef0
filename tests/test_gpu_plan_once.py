"""Plans made in one launch, by a cluster of CTAs per consumer, against the two launches of the call that has no workspace: one to
three heads a CTA and more, few and many consumers, own blocks packed or not, and calls one behind the other on the same
workspace."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    from paper_2609_32197_b200 import binding as b
    b.lib()
    return b


@pytest.mark.parametrize("B,P,H,NB", [(1, 1, 1, 1), (1, 2, 3, 33), (2, 8, 5, 70), (1, 7, 70, 31), (1, 12, 12, 90), (1, 48, 3, 96), (1, 48, 12, 96), (3, 16, 3, 64), (1, 2, 74, 20), (1, 3, 50, 20),
                                      (7, 7, 2, 40), (1, 49, 3, 100), (1, 8, 24, 929), (2, 3, 200, 12)])
@pytest.mark.parametrize("local", [0, 2])
def test_plan_in_one_launch(binding, B, P, H, NB, local):
    g = torch.Generator(device="cuda").manual_seed(B + P + H + NB)
    shape = binding.make_shape(H, 64, (1, 1, NB * 64), 0, 64, batch=B)
    ws = binding.make_workspace(shape, P)
    rank = torch.randint(0, P, (NB,), generator=g, device="cuda", dtype=torch.int32)
    for density in (0.5, 0.02, 0.0, 1.0):
        bits = torch.rand(B, H, NB, NB, generator=g, device="cuda") < density
        words = torch.zeros(B, H, NB, (NB + 31) // 32, dtype=torch.int64, device="cuda")
        for j in range(NB):
            words[..., j // 32] |= bits[..., j].long() << (j % 32)
        mask = words.to(torch.int32)
        got, want = binding.alloc_demand_outputs(shape, P), binding.alloc_demand_outputs(shape, P)
        for x in (*got.values(), *want.values()):
            x.fill_(-7)
        for _ in range(2):
            binding.sparsp_demand_pack(shape, mask, rank, P, binding.SPARSP_PLAN_ONLY | local, None, None, got["union_mask"],
                                       got["cnt"], got["seg_offset"], got["seg_total"], got["volume_bytes"], None, 0, None, ws)
        binding.sparsp_demand_plan_noalloc(shape, mask, rank, P, local, want["union_mask"], want["cnt"], want["seg_offset"],
                                           want["seg_total"], want["volume_bytes"])
        assert binding.sparsp_status(ws) == binding.SPARSP_OK
        for k in want:
            assert torch.equal(got[k], want[k]), (k, density)
