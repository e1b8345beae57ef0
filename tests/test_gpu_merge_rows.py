"""The merge of two partial results where a thread's rows and a rank's list of blocks change form, and its rate."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    from paper_2609_32197_b200 import binding as b
    b.lib()
    return b


def _parts(H, N, d, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    O = [torch.randn(1, H, N, d, device="cuda", generator=g).to(torch.bfloat16) for _ in range(2)]
    lse = [torch.randn(1, H, N, device="cuda", generator=g) * 3 for _ in range(2)]
    lse[1][torch.rand(1, H, N, device="cuda", generator=g) < 0.2] = float("-inf")
    return O, lse


@pytest.mark.parametrize("d,b", [(64, 64), (128, 64), (64, 128), (128, 128)])
@pytest.mark.parametrize("NB,short", [(1, 0), (1, 63), (2, 31), (33, 32), (65, 1), (1024, 17)])
@pytest.mark.parametrize("in_place", [False, True])
def test_rows_of_a_rank_and_all_rows(binding, d, b, NB, short, in_place):
    """Against the formula in 64 bits: one rounding to bf16 (7 bits of fraction: half a unit is at most 2^-8 of the value),
    and weights from approximate exponentials and quotients in fp32 (2^-20) of terms of up to 8."""
    H, P, consumer, h0, h1 = 3, 3, 1, 1, 3
    N = NB * b - short
    shape = binding.make_shape(H, d, (1, 1, N), 0, b)
    rank = torch.randint(0, P, (NB,), generator=torch.Generator().manual_seed(NB), dtype=torch.int32).cuda()
    (Oa, Ob), (la, lb) = _parts(H, N, d, NB + d)
    w = torch.softmax(torch.stack([la, lb]).double(), 0)
    want = w[0, ..., None] * Oa.double() + w[1, ..., None] * Ob.double()
    want_lse = torch.logaddexp(la.double(), lb.double())
    for filtered in (True, False):
        A, lA = Oa.clone(), la.clone()
        O, lse = (A, lA) if in_place else (torch.full_like(Oa, 5.0), torch.full_like(la, 5.0))
        rest_O, rest_lse = O.clone(), lse.clone()
        if filtered:
            binding.sparsp_attn_merge_rows(shape, A, lA, Ob, lb, O, lse, rank, P, consumer, h0, h1)
            mine = torch.zeros(1, H, N, dtype=torch.bool, device="cuda")
            mine[:, h0:h1] = (rank == consumer).repeat_interleave(b)[:N]
        else:
            binding.sparsp_attn_merge(shape, A, lA, Ob, lb, O, lse)
            mine = torch.ones(1, H, N, dtype=torch.bool, device="cuda")
        assert torch.equal(O[~mine], rest_O[~mine]) and torch.equal(lse[~mine], rest_lse[~mine])
        err = (O[mine].double() - want[mine]).abs()
        assert bool((err <= want[mine].abs() * 2.0 ** -8 + 2.0 ** -17).all())
        assert bool(((lse[mine].double() - want_lse[mine]).abs() <= 1e-5).all())


@pytest.mark.parametrize("d,b,H,NB", [(64, 64, 48, 700), (128, 64, 24, 700), (128, 128, 24, 500)])
def test_rate_of_a_whole_merge(binding, d, b, H, NB):
    """It moves the bytes of an element-wise sum of two tensors into a third: 1.19, 1.18 and 1.11 times its time as measured,
    1.90, 1.40 and 1.34 times with a last wave of a quarter of the CTAs and loads of rows that do not exist (the limit is no
    more than what tells the last two shapes from noise)."""
    N = NB * b
    shape = binding.make_shape(H, d, (1, 1, N), 0, b)
    (Oa, Ob), (la, lb) = _parts(H, N, d, 1)
    O, lse = torch.zeros_like(Oa), torch.zeros_like(la)

    def best(f):
        times = []
        for _ in range(12):
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            start.record()
            f()
            end.record()
            torch.cuda.synchronize()
            times.append(start.elapsed_time(end))
        return min(times)

    merge = best(lambda: binding.sparsp_attn_merge(shape, Oa, la, Ob, lb, O, lse))
    add = best(lambda: torch.add(Oa, Ob, out=O))
    print("merge %.1f us, sum %.1f us: %.2f" % (merge * 1e3, add * 1e3, merge / add))
    assert merge < 1.3 * add
