"""Calls between kernels of the caller's own: every launch takes its place while the one before it still runs, so each of
them has to wait for whatever writes its inputs, on its stream or behind an event of another one, and nothing that the
caller launches behind a call may come before it."""
import pytest
import torch

pytestmark = pytest.mark.gpu

H, NB, b, P, k = 6, 40, 64, 3, 9
N = NB * b - 11


@pytest.fixture(scope="module")
def binding():
    from paper_2609_32197_b200 import binding as b
    b.lib()
    return b


class _Layer:
    """Inputs, outputs and one method per call; every buffer of the library is the caller's."""

    def __init__(self, binding, d):
        self.binding, self.d = binding, d
        self.shape = binding.make_shape(H, d, (1, 1, N), 0, b)
        g = torch.Generator().manual_seed(d)
        self.src = [torch.randn(1, H, N, d, generator=g).to(torch.bfloat16).cuda() for _ in range(3)]
        self.rank_src = (torch.arange(NB, dtype=torch.int32) % P).cuda()
        self.Q, self.K, self.V = (torch.zeros_like(x) for x in self.src)
        self.rank = torch.zeros_like(self.rank_src)
        self.ws = binding.make_workspace(self.shape, P)
        self.mo = binding.alloc_mask_outputs(self.shape, k)
        self.do = binding.alloc_demand_outputs(self.shape, P)
        entry = 2 * b * d * 2
        self.packed = torch.zeros(H * NB * (P - 1) * entry, dtype=torch.uint8, device="cuda")
        self.O, self.part = torch.zeros_like(self.Q), torch.zeros_like(self.Q)
        self.lse, self.part_lse = (torch.zeros(1, H, N, device="cuda") for _ in range(2))
        self.hop = torch.zeros_like(self.mo["mask"])

    def arrive(self):
        """The inputs, written by kernels of the caller."""
        for x, y in zip((self.Q, self.K, self.V, self.rank), self.src + [self.rank_src]):
            x.copy_(y)

    def leave(self):
        """Kernels of the caller that overwrite the inputs."""
        for x in (self.Q, self.K, self.V):
            x.fill_(float("nan"))
        self.rank.fill_(P - 1)

    def calls(self):
        B, do, mo = self.binding, self.do, self.mo
        B.sparsp_block_mask(self.shape, self.Q, self.K, k, mo["mask"], mo["kv_list"], mo["kv_count"], None, None, self.ws)
        B.sparsp_demand_pack(self.shape, mo["mask"], self.rank, P, 0, self.K, self.V, do["union_mask"], do["cnt"],
                             do["seg_offset"], do["seg_total"], do["volume_bytes"], self.packed, self.packed.numel(), None,
                             self.ws)
        B.sparsp_sparse_attn_fwd(self.shape, self.Q, self.K, self.V, mo["mask"], 0.0, self.O, self.lse, self.ws)
        B.sparsp_hop_mask(self.shape, mo["mask"], self.rank, P, 1, 0, self.hop)
        B.sparsp_sparse_attn_fwd_packed(self.shape, self.Q, self.K, self.V, self.hop, self.rank, P, 1, do["union_mask"],
                                        do["seg_offset"], do["seg_total"], self.packed, self.packed.numel(), None, 0.0,
                                        self.part, self.part_lse, self.ws)
        B.sparsp_attn_merge_rows(self.shape, self.O, self.lse, self.part, self.part_lse, self.O, self.lse, self.rank, P, 1,
                                 0, H)

    def outputs(self):
        torch.cuda.synchronize()
        assert self.binding.sparsp_status(self.ws) == self.binding.SPARSP_OK
        out = {n: t.clone() for n, t in list(self.mo.items()) + list(self.do.items()) if t is not None}
        total = int(self.do["seg_total"].sum())
        out.update(packed=self.packed[:total * 2 * b * self.d * 2].clone(), O=self.O.clone(), lse=self.lse.clone(),
                   part=self.part.clone(), part_lse=self.part_lse.clone(), hop=self.hop.clone())
        for t in [self.O, self.lse, self.part, self.part_lse, self.hop, self.packed, *self.do.values(), *self.mo.values()]:
            if t is not None:
                t.zero_()
        torch.cuda.synchronize()
        return out


def _same(got, want):
    assert got.keys() == want.keys()
    for n in want:
        assert torch.equal(got[n].view(torch.uint8), want[n].view(torch.uint8)), n


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("where", ["same stream", "event"])
def test_calls_wait_for_the_callers_kernels_and_these_for_the_calls(binding, d, where):
    layer = _Layer(binding, d)
    layer.arrive()
    torch.cuda.synchronize()
    layer.calls()
    want = layer.outputs()
    compute = torch.cuda.Stream()
    writer = compute if where == "same stream" else torch.cuda.Stream()
    for late in (0, 200_000, 5_000_000):  # clocks that the writer is late by: up to some milliseconds
        layer.leave()
        torch.cuda.synchronize()
        arrived, done = torch.cuda.Event(), torch.cuda.Event()
        with torch.cuda.stream(writer):
            if late:
                torch.cuda._sleep(late)
            layer.arrive()
            arrived.record()
        with torch.cuda.stream(compute):
            compute.wait_event(arrived)
            layer.calls()
            done.record()
        with torch.cuda.stream(writer):
            writer.wait_event(done)
            layer.leave()
        _same(layer.outputs(), want)


@pytest.mark.parametrize("d", [64, 128])
def test_calls_behind_a_join_are_captured(binding, d):
    """The inputs come from two streams that join before the first call; they are overwritten on the other stream behind the last one.
    All of it is captured once and replayed."""
    layer = _Layer(binding, d)
    layer.arrive()
    torch.cuda.synchronize()
    layer.calls()
    want = layer.outputs()
    layer.leave()
    torch.cuda.synchronize()
    main, side = torch.cuda.Stream(), torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=main):
        begin, arrived, done, left = (torch.cuda.Event() for _ in range(4))
        begin.record()
        with torch.cuda.stream(side):
            side.wait_event(begin)
            for x, y in zip((layer.Q, layer.K), layer.src):
                x.copy_(y)
            arrived.record()
        layer.V.copy_(layer.src[2])
        layer.rank.copy_(layer.rank_src)
        main.wait_event(arrived)
        layer.calls()
        done.record()
        with torch.cuda.stream(side):
            side.wait_event(done)
            layer.leave()
            left.record()
        main.wait_event(left)
    for _ in range(2):
        graph.replay()
        _same(layer.outputs(), want)
