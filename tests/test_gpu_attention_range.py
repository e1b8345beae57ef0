"""Rows whose first scores are out of the range that the attention kernel assumes take their running maximum, and items
whose scores leave it later are computed again.  Rows of all kinds among many items per CTA, the last items of the call among
them, against a masked softmax in 64 bits; the same bits whoever computes them; the output in the place of the queries; large
values; scores that are no numbers; rows that keep nothing.  And 64-token blocks where every one has an SM of its own, at the
edge of that rule."""
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


def _reference(Q, K, V, kept, b):
    """[H][N][d] in 64 bits: softmax over the keys of kept [H][NB][NB] blocks, and the log-sum-exp."""
    N, d = Q.shape[1:]
    O, lse = torch.empty_like(Q, dtype=torch.float64), torch.empty(Q.shape[:2], dtype=torch.float64, device="cuda")
    for h in range(Q.shape[0]):
        s = Q[h].double() @ K[h].double().T / math.sqrt(d)
        tokens = kept[h].repeat_interleave(b, 0).repeat_interleave(b, 1)[:N, :N]
        s.masked_fill_(~tokens, float("-inf"))
        lse[h] = torch.logsumexp(s, -1)
        O[h] = torch.exp(s - lse[h][:, None]) @ V[h].double()
    return O, lse


@pytest.mark.parametrize("d,b", [(64, 64), (128, 64), (64, 128), (128, 128)])
@pytest.mark.parametrize("large", ["some", "last", "all"])
@pytest.mark.parametrize("keep", [2, 9])  # lists of one to three and of four to nine tiles
def test_items_that_leave_the_range(binding, d, b, large, keep):
    H, NB = (24, 40) if b == 64 else (16, 32)
    N = NB * b - 9
    g = torch.Generator(device="cuda").manual_seed(d + b + keep)
    Q, K, V = (torch.randn(H, N, d, generator=g, device="cuda") for _ in range(3))
    # scores of a unit row spread over +-6 log2 units; times 40 over +-240 (far from 0, at times near the first tile's
    # maximum), times 400 over thousands
    block = torch.arange(N, device="cuda") // b
    factor = torch.ones(H, N, device="cuda")
    if large == "all":
        factor[:] = 40.0
    elif large == "last":
        factor[-1] = 40.0
    else:
        factor[3::7, :][:, block % 5 == 2] = 40.0
        factor[2::9, :][:, block % 11 == 3] = 400.0
        factor[5] = 3.0
    Q, K, V = (x.to(torch.bfloat16) for x in (Q * factor[..., None], K, V))
    kept = torch.rand(H, NB, NB, generator=g, device="cuda").argsort(-1).argsort(-1) < keep
    words = torch.zeros(H, NB, (NB + 31) // 32, dtype=torch.int64, device="cuda")
    for j in range(NB):
        words[:, :, j // 32] |= kept[:, :, j].long() << (j % 32)
    mask = torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32)[None].contiguous()
    want, want_lse = _reference(Q, K, V, kept, b)
    shape = binding.make_shape(H, d, (1, 1, N), 0, b)
    P = 3
    ws = binding.make_workspace(shape, P)

    def check(O, lse, rows):
        err = (O[0].double() - want)[:, rows].abs()
        assert err.max() <= pu.ATTN_MAX_ABS * max(1.0, float(want.abs().max()) / 4.0), float(err.max())
        # an fp32 number of up to thousands: eight units in the last place on top of the tolerance
        tol = 2e-2 + want_lse.abs() * 2.0 ** -20
        assert bool(((lse[0].double() - want_lse).abs() <= tol)[:, rows].all())

    O, lse = torch.full_like(Q, 7.0)[None], torch.full((1, H, N), 7.0, device="cuda")
    binding.sparsp_sparse_attn_fwd(shape, Q, K, V, mask, 0.0, O, lse, ws)
    assert binding.sparsp_status(ws) == binding.SPARSP_OK
    check(O, lse, torch.arange(N, device="cuda"))

    rank = torch.arange(NB, dtype=torch.int32, device="cuda").remainder(P)
    dm = pu.gpu_demand_pack(binding, shape, mask, rank, P, 0, K, V, ws)
    for consumer in (0, 2):
        O.fill_(7.0)
        lse.fill_(7.0)
        binding.sparsp_sparse_attn_fwd_packed(shape, Q, K, V, mask, rank, P, consumer, dm["union_mask"], dm["seg_offset"],
                                              dm["seg_total"], dm["packed"], dm["packed"].numel(), None, 0.0, O, lse, ws)
        assert binding.sparsp_status(ws) == binding.SPARSP_OK
        check(O, lse, torch.nonzero(rank.repeat_interleave(b)[:N] == consumer)[:, 0])


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("layout", ["HND", "NHD"])
@pytest.mark.parametrize("spare", [-1, 0, 1])
def test_as_many_blocks_as_multiprocessors(binding, d, layout, spare):
    sms, b, B = torch.cuda.get_device_properties(0).multi_processor_count, 64, 2
    H, NB = 1, (sms + 2 * spare) // B  # two batch items
    N = NB * b - 21
    g = torch.Generator(device="cuda").manual_seed(d + NB)
    Q, K, V = (torch.randn(B, N, d, generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    kept = torch.rand(B, NB, NB, generator=g, device="cuda") < 0.3
    kept[:, 5] = False                 # a block that keeps nothing
    kept[:, 7] = False
    kept[:, 7, NB - 1] = True          # the ragged block alone
    words = torch.zeros(B, H, NB, (NB + 31) // 32, dtype=torch.int64, device="cuda")
    for j in range(NB):
        words[:, 0, :, j // 32] |= kept[:, :, j].long() << (j % 32)
    mask = torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32).contiguous()
    want, want_lse = _reference(Q, K, V, kept, b)
    shape = binding.make_shape(H, d, (1, 1, N), 0, b, batch=B, layout=layout)
    ws = binding.make_workspace(shape, 2)
    q, k, v = ((x[:, None] if layout == "HND" else x[:, :, None]).contiguous() for x in (Q, K, V))
    O, lse = torch.full_like(q, 7.0), torch.full((B, H, N), 7.0, device="cuda")
    binding.sparsp_sparse_attn_fwd(shape, q, k, v, mask, 0.0, O, lse, ws)
    assert binding.sparsp_status(ws) == binding.SPARSP_OK
    rows = kept.any(-1).repeat_interleave(b, 1)[:, :N]
    out = O.reshape(B, N, d).double()
    assert (out - want)[rows].abs().max() <= pu.ATTN_MAX_ABS
    assert (lse[:, 0].double() - want_lse)[rows].abs().max() <= 2e-2
    assert bool((out[~rows] == 0).all()) and bool((lse[:, 0][~rows] == float("-inf")).all())


def _mask(kept):
    """[H][NB][NB] -> mask words [1][H][NB][Wd]."""
    words = torch.zeros(*kept.shape[:2], (kept.shape[2] + 31) // 32, dtype=torch.int64, device="cuda")
    for j in range(kept.shape[2]):
        words[:, :, j // 32] |= kept[:, :, j].long() << (j % 32)
    return torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32)[None].contiguous()


class _Calls:
    """The three calls that make an output, on [H][N][d] inputs in a layout: K / V source, packed, one hop of it."""

    def __init__(self, binding, kept, d, b, N, layout="HND", P=3, consumer=1):
        self.b, self.layout, self.P, self.consumer, self.N = binding, layout, P, consumer, N
        H, NB = kept.shape[:2]
        self.shape = binding.make_shape(H, d, (1, 1, N), 0, b, layout=layout)
        self.ws, self.mask = binding.make_workspace(self.shape, P), _mask(kept)
        self.rank = torch.arange(NB, dtype=torch.int32, device="cuda").remainder(P)
        self.mine = (self.rank == consumer).repeat_interleave(b)[:N]

    def place(self, x):
        return pu.to_layout(x, self.layout)

    def run(self, source, Q, K, V, scale=0.0, in_place=False):
        """O [H][N][d] and lse [H][N] as int16 / fp32; rows that a packed call leaves alone come back as 7."""
        bd, (q, k, v) = self.b, (self.place(x) for x in (Q, K, V))
        q = q.clone()
        O = q if in_place else torch.full_like(q, 7.0)
        lse = torch.full((1, Q.shape[0], self.N), 7.0, device="cuda")
        if source == "kv":
            bd.sparsp_sparse_attn_fwd(self.shape, q, k, v, self.mask, scale, O, lse, self.ws)
        else:
            mask = self.mask
            dm = pu.gpu_demand_pack(bd, self.shape, mask, self.rank, self.P, 0, k, v, self.ws)
            if source == "hop":
                mask = torch.empty_like(mask)
                bd.sparsp_hop_mask(self.shape, self.mask, self.rank, self.P, self.consumer, 0, mask)
            bd.sparsp_sparse_attn_fwd_packed(self.shape, q, k, v, mask, self.rank, self.P, self.consumer, dm["union_mask"],
                                             dm["seg_offset"], dm["seg_total"], dm["packed"], dm["packed"].numel(), None,
                                             scale, O, lse, self.ws)
        assert bd.sparsp_status(self.ws) == bd.SPARSP_OK
        return pu.from_layout(O, self.layout).contiguous(), lse[0]


def _same_bits(a, b):
    return torch.equal(a[0].view(torch.int16), b[0].view(torch.int16)) and torch.equal(a[1].view(torch.int32),
                                                                                       b[1].view(torch.int32))


def _mixed_heads(H, N, d, NB, b, seed):
    """Heads within the range, far out of it, and with single blocks of rows or keys that are."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    Q, K, V = (torch.randn(H, N, d, generator=g, device="cuda") for _ in range(3))
    block = torch.arange(N, device="cuda") // b
    Q[1::4] *= 40.0
    Q[2::5][:, block % 9 == 4] *= 300.0
    K[3::6][:, block % 13 == 6] *= 60.0
    return [x.to(torch.bfloat16) for x in (Q, K, V)], g


@pytest.mark.parametrize("d,b,layout", [(64, 64, "HND"), (128, 64, "NHD"), (64, 128, "NHD"), (128, 128, "HND")])
@pytest.mark.parametrize("source", ["kv", "packed", "hop"])
def test_a_row_does_not_depend_on_who_computes_it(binding, d, b, layout, source):
    """Many items per multiprocessor, some of which are computed again: a repeated call gives the same bits, and so does one
    with the heads in another order, in which other items meet in a CTA."""
    H, NB = 60, 60 if b == 64 else 45
    N = NB * b - 9
    (Q, K, V), g = _mixed_heads(H, N, d, NB, b, d + b)
    kept = torch.rand(H, NB, NB, generator=g, device="cuda") < 0.3
    kept[:, 4] = False
    first = _Calls(binding, kept, d, b, N, layout).run(source, Q, K, V)
    for _ in range(3):
        assert _same_bits(first, _Calls(binding, kept, d, b, N, layout).run(source, Q, K, V))
    order = torch.randperm(H, generator=g, device="cuda")
    other = _Calls(binding, kept[order], d, b, N, layout).run(source, Q[order], K[order], V[order])
    assert _same_bits((first[0][order], first[1][order]), other)


@pytest.mark.parametrize("d,b", [(64, 64), (128, 64), (64, 128), (128, 128)])
@pytest.mark.parametrize("source", ["kv", "packed", "hop"])
def test_output_may_take_the_place_of_the_queries(binding, d, b, source):
    H, NB = 20, 30
    N = NB * b - 9
    (Q, K, V), g = _mixed_heads(H, N, d, NB, b, 3 * d + b)
    kept = torch.rand(H, NB, NB, generator=g, device="cuda") < 0.3
    kept[:, 4] = False
    c = _Calls(binding, kept, d, b, N)
    apart, together = c.run(source, Q, K, V), c.run(source, Q, K, V, in_place=True)
    rows = c.mine if source != "kv" else torch.ones_like(c.mine)
    assert _same_bits((apart[0][:, rows], apart[1]), (together[0][:, rows], together[1]))


@pytest.mark.parametrize("d,b", [(64, 64), (128, 64), (64, 128), (128, 128)])
@pytest.mark.parametrize("source", ["kv", "packed", "hop"])
@pytest.mark.parametrize("most", [20.0, 90.0])
def test_large_values_of_v(binding, d, b, source, most):
    """Row sums up to 2^97 relative to a reference that is far too low, times |V| of 2^40: out of fp32, the result is not.
    A score is 0 but for one block's keys, whose score is `most` for every row (log2 units, softmax scale ln 2)."""
    H, NB = 4, 24
    N = NB * b - 9
    g = torch.Generator(device="cuda").manual_seed(d)
    Q, K = (torch.zeros(H, N, d, device="cuda") for _ in range(2))
    Q[..., 0] = 1.0
    block = torch.arange(N, device="cuda") // b
    K[:, block == 18, 0] = most
    V = torch.randn(H, N, d, generator=g, device="cuda") * 2.0 ** 40
    Q, K, V = (x.to(torch.bfloat16) for x in (Q, K, V))
    kept = torch.zeros(H, NB, NB, dtype=torch.bool, device="cuda")
    kept[:, :, ::3] = True  # rank 0's, block 18 among them, and a row's own
    kept[:, torch.arange(NB), torch.arange(NB)] = True
    c = _Calls(binding, kept, d, b, N)
    O, lse = c.run(source, Q, K, V, scale=math.log(2.0))
    s = Q.double() @ K.double().transpose(1, 2) * math.log(2.0)
    tokens = (kept & (c.rank == 0) if source == "hop" else kept).repeat_interleave(b, 1).repeat_interleave(b, 2)[:, :N, :N]
    s.masked_fill_(~tokens, float("-inf"))
    want = torch.softmax(s, -1) @ V.double()
    rows = c.mine if source != "kv" else torch.ones_like(c.mine)
    # weights and result are rounded to bf16: 2^-9 each, of values that are at most the largest |V|
    assert (O.double() - want)[:, rows].abs().max() <= 2.0 ** -8 * V.double().abs().max()
    assert (lse.double() - torch.logsumexp(s, -1))[:, rows].abs().max() <= 2e-2


@pytest.mark.parametrize("d,b", [(64, 64), (128, 64), (64, 128), (128, 128)])
@pytest.mark.parametrize("source", ["kv", "packed", "hop"])
@pytest.mark.parametrize("key", [0, 2, 63])  # by the special-function unit, by the polynomial, the last of a half tile
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_scores_that_are_no_numbers(binding, d, b, source, key, value):
    """A row that keeps a key whose score is NaN or +infinity is NaN throughout; all other rows are what they are."""
    H, NB = 8, 24
    N = NB * b - 9
    g = torch.Generator(device="cuda").manual_seed(d + b + key)
    Q, K, V = (torch.randn(H, N, d, generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    Q[..., 0] = 1.0  # (so that an infinite key gives every row the score +infinity)
    kept = torch.rand(H, NB, NB, generator=g, device="cuda") < 0.3
    c = _Calls(binding, kept, d, b, N)
    plain = c.run(source, Q, K, V)
    bad = 9  # a block of rank 0
    K[:, bad * b + key, 0] = value
    O, lse = c.run(source, Q, K, V)
    none = kept[:, :, bad].repeat_interleave(b, 1)[:, :N]
    rows = c.mine if source != "kv" else torch.ones_like(c.mine)
    assert bool(torch.isnan(O[none & rows]).all()) and bool(torch.isnan(lse[none & rows]).all())
    keep = ~none & rows
    # (another row of its item may have made the item be computed again: two roundings of the same result)
    assert (O.double() - plain[0].double())[keep].abs().max() <= 2 * pu.ATTN_MAX_ABS
    finite = keep & torch.isfinite(plain[1])
    assert bool(torch.isfinite(lse[finite]).all()) and (lse - plain[1])[finite].abs().max() <= 2e-2
    assert torch.equal(lse[keep & ~finite], plain[1][keep & ~finite])


@pytest.mark.parametrize("d,b", [(64, 64), (128, 128)])
@pytest.mark.parametrize("shift", [0, 8])
def test_rows_that_keep_nothing(binding, d, b, shift):
    """32-byte stores where the output begins on such a boundary, 16-byte ones where it does not."""
    H, NB = 6, 21
    N = NB * b - 9
    g = torch.Generator(device="cuda").manual_seed(d)
    Q, K, V = (torch.randn(H, N, d, generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    kept = torch.rand(H, NB, NB, generator=g, device="cuda") < 0.2
    kept[:, ::2] = False
    kept[:, -1] = False
    kept[2] = False
    shape = binding.make_shape(H, d, (1, 1, N), 0, b)
    ws = binding.make_workspace(shape, 1)
    buf = torch.full((Q.numel() + 16,), 7.0, dtype=torch.bfloat16, device="cuda")
    O, lse = buf[shift:shift + Q.numel()].view_as(Q), torch.full((1, H, N), 7.0, device="cuda")
    binding.sparsp_sparse_attn_fwd(shape, Q, K, V, _mask(kept), 0.0, O, lse, ws)
    assert binding.sparsp_status(ws) == binding.SPARSP_OK
    rows = kept.any(-1).repeat_interleave(b, 1)[:, :N]
    want, want_lse = _reference(Q, K, V, kept, b)
    assert bool((O[~rows] == 0).all()) and bool((lse[0][~rows] == float("-inf")).all())
    assert (O.double() - want)[rows].abs().max() <= pu.ATTN_MAX_ABS
    assert (lse[0].double() - want_lse)[rows].abs().max() <= 2e-2
    assert bool((buf[:shift] == 7.0).all()) and bool((buf[shift + Q.numel():] == 7.0).all())
