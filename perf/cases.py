"""The work that the performance of this library is judged by: one attention layer's calls over the range of shapes,
layouts, selection rules and rank counts that the library takes.

A case is a dict of plain values.  `kind` says which calls one pass makes, everything else describes the layer:

  layer     block mask -> demand + pack for all virtual ranks -> block-sparse attention (the step of bench.py);
            with pack = False the ranks are left out: mask -> attention, what a single-GPU user calls
  consumer  one rank's attention over the demand-routed exchange, everything already received: its own blocks, then
            hop by hop, chunk by chunk, attention on the remote blocks in place and the merge (exchange_driver.py)
  oneshot   one rank's attention over its whole received buffer in a single call
  producer  one rank's packing of the segments that its peers have selected, one per peer
  plan      demand and offsets only (what every rank derives once per attention call)

Inputs come from the repository's generator (positional structure plus noise: paper_2609_32197_b200/synth.py).
"""
import functools
import math

import torch

from paper_2609_32197_b200 import binding, synth


def _case(name, kind, heads, head_dim, grid, block, pct, ranks, *, n_text=0, topk=0, tau=0.0, batch=1, layout="HND",
          placement="contiguous", pack=True, lse=False, rank=0, chunks=1):
    return {"name": name, "kind": kind, "batch": batch, "heads": heads, "head_dim": head_dim, "grid_t": grid[0],
            "grid_h": grid[1], "grid_w": grid[2], "n_text": n_text, "block": block, "pct": pct, "topk": topk, "tau": tau,
            "layout": layout, "ranks": ranks, "placement": placement, "pack": pack, "lse": lse, "rank": rank,
            "chunks": chunks}


def listed():
    tiny, mid, cog, wan, hun = (synth.WORKLOADS[w] for w in ("tiny", "mid", "cog", "wan", "hunyuan"))
    return [
        # the smallest layer in use: launches and latency
        _case("layer-tiny", "layer", tiny.heads, 64, tiny.grid, 64, 0, 4, topk=16),
        # an ordinary layer, 64-token blocks
        _case("layer-mid", "layer", mid.heads, 128, mid.grid, 64, 15, 4),
        # head_dim 64, text tokens behind the video tokens, shuffled placement
        _case("layer-cog", "layer", cog.heads, 64, cog.grid, 64, 20, 8, n_text=cog.n_text, placement="shuffle"),
        # long video, 128-token blocks, the interval-periodic placement
        _case("layer-wan", "layer", wan.heads, 128, wan.grid, 128, 10, 8, placement="periodic"),
        # the longest sequence at its default sparsity, and the largest case of all: a quarter of the blocks kept
        _case("layer-hunyuan-10", "layer", hun.heads, 128, hun.grid, 128, 10, 8),
        _case("layer-hunyuan-25", "layer", hun.heads, 128, hun.grid, 128, 25, 8),
        # a batch of two odd-sized sequences in token-major layout, ragged last block, head_dim 64 with 128-token blocks
        _case("layer-ragged", "layer", 13, 64, (7, 23, 37), 128, 15, 3, n_text=77, batch=2, layout="NHD", lse=True),
        # single GPU, no ranks: threshold selection (rows keep different numbers of blocks), token-major layout
        _case("attn-cdf-mid", "layer", mid.heads, 128, mid.grid, 64, 0, 4, tau=0.9, layout="NHD", pack=False, lse=True),
        # one rank of eight on a node: hop-wise attention as the exchange runtime issues it, two chunks per hop
        _case("consumer-wan", "consumer", wan.heads, 128, wan.grid, 128, 10, 8, rank=3, chunks=2),
        # the same for a layer of 64-token blocks whose buffer has arrived as a whole
        _case("oneshot-mid", "oneshot", mid.heads, 128, mid.grid, 64, 15, 4, rank=1),
        # the producer's side of the exchange
        _case("producer-wan", "producer", wan.heads, 128, wan.grid, 128, 10, 8, rank=3),
        # the plan of an attention call alone
        _case("plan-hunyuan", "plan", hun.heads, 128, hun.grid, 128, 10, 8),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the same ranges: 1 thousand to 118 800 tokens, 1 to 48 heads, both head dims and block sizes,
    3 to 25 percent of the blocks (or a threshold of 0.8 to 0.95), 2 to 8 ranks."""
    kind = rng.choice(["layer", "layer", "layer", "layer", "consumer", "oneshot", "producer", "plan"])
    d, b = rng.choice([64, 128, 128]), rng.choice([64, 128])
    tokens = _log(rng, 1000, 60000 if b == 64 else 118800)
    t = min(33, max(1, int(_log(rng, 2, 33))))
    gh = max(4, int(math.sqrt(tokens / t) * rng.uniform(0.55, 1.0)))
    gw = max(4, int(tokens / (t * gh)))
    n_text = rng.choice([0, 0, rng.randint(1, 256)])
    ranks = rng.randint(2, 8)
    n = t * gh * gw + n_text
    pct = rng.randint(3, 25)
    tau = 0.0
    if kind == "layer" and rng.random() < 0.25:
        tau = round(rng.uniform(0.8, 0.95), 2)
    batch = rng.choice([1, 1, 1, 2])
    if kind in ("consumer", "oneshot", "producer"):
        batch = 1  # the exchange handles one batch item per call
    heads = max(1, int(_log(rng, 1.5, 49)))
    # no dearer than the largest listed case: 24 heads of 118 800 tokens at 25 percent
    cost = batch * heads * float(n) * n * (25 if tau else max(pct, 5)) * d
    most = 24 * 118800.0 * 118800 * 25 * 128 * 0.8
    heads = max(1, min(heads, int(heads * most / cost)))
    return _case("", kind, heads, d, (t, gh, gw), b, 0 if tau else pct, ranks, n_text=n_text, tau=tau, batch=batch,
                 layout=rng.choice(["HND", "HND", "NHD"]), placement=rng.choice(["contiguous", "periodic", "shuffle"]),
                 pack=rng.random() < 0.7, lse=rng.random() < 0.3, rank=rng.randrange(ranks), chunks=rng.randint(1, 3))


def _shape(case, heads=None):
    return binding.make_shape(heads or case["heads"], case["head_dim"], (case["grid_t"], case["grid_h"], case["grid_w"]),
                              case["n_text"], case["block"], batch=case["batch"], layout=case["layout"])


def _inputs(case, seed, heads):
    """Q, K, V in the case's layout on the GPU; batch items are further heads of the generator."""
    grid = (case["grid_t"], case["grid_h"], case["grid_w"])
    wl = synth.Workload("case", heads * case["batch"], case["head_dim"], grid, case["n_text"], case["block"], None, None,
                        case["ranks"], seed=seed)
    out = []
    for x in synth.make_qkv(wl, "cuda"):
        x = x.view(case["batch"], heads, *x.shape[1:])
        out.append(x.permute(0, 2, 1, 3).contiguous() if case["layout"] == "NHD" else x)
    return out


class _State:
    """What a user's program holds before the call: inputs, placement, output buffers, workspace."""

    def __init__(self, case, seed, heads=None):
        H = heads or case["heads"]
        self.case, self.P = case, case["ranks"]
        self.shape = _shape(case, H)
        g = self.geometry = binding.sparsp_geometry(self.shape)
        self.Q, self.K, self.V = _inputs(case, seed, H)
        if case["placement"] == "contiguous":
            rank = binding.sparsp_placement_contiguous(self.shape, self.P)
        elif case["placement"] == "periodic":
            rank = binding.sparsp_placement_periodic(self.shape, self.P)
        else:
            rank = synth.shuffled_placement(g.n_blocks, self.P, seed=1)
        self.rank_d = rank.cuda()
        self.ws = binding.make_workspace(self.shape, self.P)
        self.k = case["topk"] or binding.sparsp_resolve_topk(case["pct"], g.n_video_blocks)
        self.mo = binding.alloc_mask_outputs(self.shape, self.k, with_list=not case["tau"])
        if case["tau"]:
            self.mo["kv_count"] = torch.empty(case["batch"], H, g.n_blocks, dtype=torch.int32, device="cuda")
        self.do = binding.alloc_demand_outputs(self.shape, self.P)
        self.entry = 2 * case["block"] * case["head_dim"] * 2

    def mask(self):
        mo = self.mo
        if self.case["tau"]:
            binding.sparsp_block_mask_cdf(self.shape, self.Q, self.K, self.case["tau"], 0.0, mo["mask"], mo["kv_count"],
                                          None, None, self.ws)
        else:
            binding.sparsp_block_mask(self.shape, self.Q, self.K, self.k, mo["mask"], mo["kv_list"], mo["kv_count"], None,
                                      None, self.ws)

    def demand(self, flags, K=None, V=None, packed=None):
        do = self.do
        binding.sparsp_demand_pack(self.shape, self.mo["mask"], self.rank_d, self.P, flags, K, V, do["union_mask"],
                                   do["cnt"], do["seg_offset"], do["seg_total"], do["volume_bytes"], packed,
                                   packed.numel() * 8 if packed is not None else 0, None, self.ws)

    def segment(self, consumer, producer, dst):
        do = self.do
        binding.sparsp_pack_segment(self.shape, do["union_mask"], self.rank_d, self.P, consumer, producer, do["cnt"],
                                    do["seg_offset"], self.K, self.V, dst, dst.numel() * 8, self.ws)

    def entries(self, n):
        """A buffer of n packed entries (whole 8-byte words)."""
        return torch.zeros(max(int(n), 1) * self.entry // 8, dtype=torch.int64, device="cuda")


def prepare(case, seed):
    s = _State(case, seed)
    kind, P, r = case["kind"], s.P, case["rank"]
    s.O = torch.zeros_like(s.Q)
    s.lse = None
    if case["lse"] or kind in ("consumer", "oneshot"):
        s.lse = torch.full((case["batch"], case["heads"], s.geometry.n_tokens), float("-inf"), dtype=torch.float32,
                           device="cuda")
    if kind == "layer":
        if case["pack"]:
            # room for every block at every rank that does not own it, whatever the masks turn out to be
            s.packed = s.entries(case["batch"] * case["heads"] * s.geometry.n_blocks * (P - 1))
        return s
    s.mask()
    s.demand(binding.SPARSP_PLAN_ONLY)
    if kind == "plan":
        return s
    if kind == "producer":
        # one slot for every peer's segment: room for all of this rank's blocks
        room = case["heads"] * int((s.rank_d == r).sum())
        s.slots = [((r + u + 1) % P, s.entries(room)) for u in range(P - 1)]
        return s
    # this rank's receive buffer, filled by its peers
    cnt, seg = s.do["cnt"][0].cpu(), s.do["seg_offset"][0].cpu()
    s.recv = s.entries(s.do["seg_total"][0, r])
    for p in range(P):
        n, first = int(cnt[r, p].sum()), int(seg[r, p, 0])
        if p != r and n:
            s.segment(r, p, s.recv[first * s.entry // 8:(first + n) * s.entry // 8])
    s.base = torch.zeros(1, P, dtype=torch.int64, device="cuda")
    s.part, s.part_lse = torch.zeros_like(s.Q), torch.full_like(s.lse, float("-inf"))
    s.hop = torch.empty_like(s.mo["mask"])
    s.plan = [t for t in binding.sparsp_exchange_plan(s.shape, P, s.do["cnt"], s.do["seg_offset"], case["chunks"],
                                                      case["chunks"]) if t.consumer == r and t.n_entries]
    s.plan.sort(key=lambda t: (t.round, t.order))
    return s


def _packed_attention(s, mask, O, lse):
    do = s.do
    binding.sparsp_sparse_attn_fwd_packed(s.shape, s.Q, s.K, s.V, mask, s.rank_d, s.P, s.case["rank"], do["union_mask"],
                                          do["seg_offset"], do["seg_total"], s.recv, s.recv.numel() * 8, s.base, 0.0, O,
                                          lse, s.ws)


def run(s):
    kind, case = s.case["kind"], s.case
    if kind == "plan":
        s.demand(binding.SPARSP_PLAN_ONLY)
        return s.do
    if kind == "producer":
        for consumer, slot in s.slots:
            s.segment(consumer, case["rank"], slot)
        return [slot for _, slot in s.slots]
    if kind == "oneshot":
        _packed_attention(s, s.mo["mask"], s.O, s.lse)
        return {"O": s.O, "lse": s.lse}
    if kind == "consumer":
        r = case["rank"]
        binding.sparsp_hop_mask(s.shape, s.mo["mask"], s.rank_d, s.P, r, r, s.hop)
        binding.sparsp_sparse_attn_fwd(s.shape, s.Q, s.K, s.V, s.hop, 0.0, s.O, s.lse, s.ws)
        for t in s.plan:
            binding.sparsp_hop_chunk_mask(s.shape, s.mo["mask"], s.rank_d, s.P, r, t.producer, t.head_begin, t.head_end,
                                          s.hop)
            _packed_attention(s, s.hop, s.part, s.part_lse)
            binding.sparsp_attn_merge_rows(s.shape, s.O, s.lse, s.part, s.part_lse, s.O, s.lse, s.rank_d, s.P, r,
                                           t.head_begin, t.head_end)
        return {"O": s.O, "lse": s.lse}
    s.mask()
    out = {k: v for k, v in s.mo.items() if v is not None}
    if case["pack"]:
        s.demand(0, s.K, s.V, s.packed)
        out.update(s.do, packed=s.packed)
    binding.sparsp_sparse_attn_fwd(s.shape, s.Q, s.K, s.V, s.mo["mask"], 0.0, s.O, s.lse, s.ws)
    out["O"] = s.O
    if s.lse is not None:
        out["lse"] = s.lse
    return out


@functools.lru_cache(maxsize=None)
def _sample(items):
    """Per head, from the first heads of one seed: kept (query block, KV block) pairs over all rows and over the case's
    rank's rows, entries packed for all ranks, by and for the case's rank, and distinct tiles that its peers select."""
    case = dict(items)
    heads = min(case["heads"], 4)
    s = _State(case, 0, heads)
    s.mask()
    s.demand(binding.SPARSP_PLAN_ONLY)
    words = s.mo["mask"].view(torch.uint8).to(torch.int64)
    bits = sum((words >> i) & 1 for i in range(8)).sum(-1).double()  # [B][H][NB] kept blocks per row
    r, cnt = case["rank"], s.do["cnt"].double()
    off = ~torch.eye(s.P, dtype=torch.bool, device="cuda")
    n = 1.0 / heads  # per head, all batch items together
    return {"pairs": float(bits.sum()) * n, "rank_pairs": float(bits[..., s.rank_d == r].sum()) * n,
            "entries": float(cnt.sum(-1)[:, off].sum()) * n, "sent": float((cnt[:, :, r].sum() - cnt[:, r, r].sum())) * n,
            "received": float(s.do["seg_total"][:, r].sum()) * n, "rank_rows": float((s.rank_d == r).double().mean())}


def work(case):
    c = {k: v for k, v in case.items() if k != "name"}
    w = _sample(tuple(sorted(c.items())))
    g = binding.sparsp_geometry(_shape(case))
    H, BH, d, b, P = case["heads"], case["heads"] * case["batch"], case["head_dim"], case["block"], case["ranks"]
    tensor = BH * g.n_tokens * d * 2.0           # Q, K, V or O
    words = BH * g.n_blocks * g.n_words * 4.0    # a mask
    entry = 2.0 * b * d * 2
    fill = g.n_tokens / (g.n_blocks * float(b))  # a ragged last block
    plan = BH * P * g.n_words * 4.0 + BH * P * P * 12.0
    flops = 4.0 * d * b * b * H * fill * fill
    kind = case["kind"]
    if kind == "plan":
        return {"bytes": words + plan, "flops": 0.0}
    if kind == "producer":
        # its own K and V blocks are read once, every segment is written
        return {"bytes": 2 * tensor * w["rank_rows"] + w["sent"] * H * entry, "flops": 0.0}
    if kind in ("consumer", "oneshot"):
        mine = 4 * tensor * w["rank_rows"]       # its own Q, K, V, O
        return {"bytes": mine + w["received"] * H * entry + words, "flops": flops * w["rank_pairs"]}
    lists = BH * g.n_blocks * 4.0 + (0.0 if case["tau"] else w["pairs"] * H * 4.0)
    nbytes = 4 * tensor + words + lists + (BH * g.n_tokens * 4.0 if case["lse"] else 0.0)
    if case["pack"]:
        nbytes += w["entries"] * H * entry + plan
    # the scores of the selection: one product of pooled vectors per pair of blocks
    return {"bytes": nbytes, "flops": flops * w["pairs"] + 2.0 * d * BH * float(g.n_blocks) ** 2}


def tolerance(case):
    if case["kind"] in ("producer", "plan"):
        return "exact"
    # Masks, lists, counts, offsets and packed bytes are exact.  The attention output is bf16 from bf16 probabilities with
    # fp32 sums: 1.8e-3 to 2.2e-3 from the same attention in 64 bits (largest difference 0.043 of the root mean square);
    # hop by hop, with the running result rounded to bf16 after every merge, 4.2e-3 from the one-call result.
    return {"rel": 1.6e-2 if case["kind"] == "consumer" else 8e-3, "max": 0.15}


def _placement(case, n_blocks, n_video):
    """Rank of every block, as the library's placement functions define it."""
    P, j = case["ranks"], torch.arange(n_blocks, dtype=torch.int64)
    if case["placement"] == "contiguous":
        return j * P // n_blocks
    if case["placement"] == "shuffle":
        return synth.shuffled_placement(n_blocks, P, seed=1).long()
    first, frame = j * case["block"], case["grid_h"] * case["grid_w"]
    return torch.where(first >= n_video, j % P, P * (first % frame) // frame)


def _kept_blocks(case, q, k, n_cand):
    """Kept KV blocks [heads][NB][NB] of q, k [heads][NB][b][d] (zeros behind the last token): fp32 sums in token and
    channel order as the selection is defined, everything else in 64 bits."""
    NB, b, n = q.shape[1], case["block"], case["tokens"]
    count = torch.full((NB, 1), float(b), device=q.device)
    count[-1] = n - (NB - 1) * b

    def pooled(x):
        acc = torch.zeros_like(x[:, :, 0], dtype=torch.float32)
        for t in range(b):
            acc = acc + x[:, :, t].float()
        return (acc / count).double()

    pq, pk = pooled(q), pooled(k)
    score = torch.zeros(q.shape[0], NB, NB, dtype=torch.float32, device=q.device)
    for c in range(q.shape[-1]):
        score = (score.double() + pq[:, :, None, c] * pk[:, None, :, c]).float()
    score = score[:, :, :n_cand]
    kept = torch.ones(q.shape[0], NB, NB, dtype=torch.bool, device=q.device)
    top, order = torch.sort(score, dim=-1, descending=True, stable=True)
    if case["tau"]:
        scale = torch.tensor(1.0 / math.sqrt(q.shape[-1])) * torch.tensor(1.4426950408889634)
        weight = torch.floor(torch.exp2((top - top[..., :1]).double() * scale.double().item()) * 2.0 ** 26)
        mass = torch.cumsum(weight, -1)
        theta = torch.ceil(torch.tensor(case["tau"]).double().item() * mass[..., -1:])
        last = torch.argmax((mass >= theta).to(torch.uint8), -1, keepdim=True)
        kept[:, :, :n_cand] = score >= torch.gather(top, -1, last)
    else:
        topk = case["topk"] or max(1, (case["pct"] * n_cand + 99) // 100)
        kept[:, :, :n_cand] = False
        kept[:, :, :n_cand].scatter_(-1, order[..., :topk], True)
    return kept


def _attention(q, k, v, kept, tokens):
    """One head: q, k, v [NB][b][d], kept [NB][NB] -> output [NB][b][d] and log-sum-exp [NB][b], in 64 bits."""
    NB, b, d = q.shape
    O = torch.zeros(NB, b, d, dtype=torch.float64, device=q.device)
    lse = torch.full((NB, b), float("-inf"), dtype=torch.float64, device=q.device)
    k, v = k.double(), v.double()
    col = torch.arange(NB * b, device=q.device).view(NB, b) < tokens
    n_kept = kept.sum(-1)
    rows = torch.nonzero(n_kept, as_tuple=True)[0]
    rows = rows[torch.argsort(n_kept[rows])]  # rows of similar length together
    at = 0
    while at < rows.numel():
        most = int(n_kept[rows[min(at + 63, rows.numel() - 1)]])
        r = rows[at:at + max(1, min(64, (1 << 28) // (most * b * max(b, d))))]
        at += r.numel()
        live, block = torch.sort(kept[r].to(torch.uint8), dim=-1, descending=True, stable=True)
        live, block = live[:, :most].bool(), block[:, :most]
        s = torch.matmul(q[r].double(), k[block].flatten(1, 2).transpose(1, 2)) / math.sqrt(d)
        s.masked_fill_(~(live[..., None] & col[block]).flatten(1)[:, None], float("-inf"))
        lse[r] = torch.logsumexp(s, -1)
        O[r] = torch.matmul(torch.exp(s - lse[r][..., None]), v[block].flatten(1, 2))
    return O, lse


def exact(case, seed):
    """The attention output and its log-sum-exp in 64 bits; everything else that a pass returns is whole numbers or bytes."""
    kind, H, B, d, b = case["kind"], case["heads"], case["batch"], case["head_dim"], case["block"]
    if kind in ("producer", "plan"):
        return None
    n_video = case["grid_t"] * case["grid_h"] * case["grid_w"]
    n = n_video + case["n_text"]
    NB = (n + b - 1) // b
    n_cand = n_video // b if case["n_text"] else NB
    nhd = case["layout"] == "NHD"
    Q, K, V = _inputs(case, seed, H)
    mine = torch.ones(NB, dtype=torch.bool, device=Q.device)
    if kind != "layer":
        mine = (_placement(case, NB, n_video) == case["rank"]).to(Q.device)
    O = torch.zeros(Q.shape, dtype=torch.float64, device=Q.device)
    lse = torch.full((B, H, n), float("-inf"), dtype=torch.float64, device=Q.device)
    for bb in range(B):
        for h in range(H):
            q, k, v = ((x[bb, :, h] if nhd else x[bb, h]) for x in (Q, K, V))
            q, k, v = (torch.nn.functional.pad(x, (0, 0, 0, NB * b - n)).view(NB, b, d) for x in (q, k, v))
            kept = _kept_blocks(dict(case, tokens=n), q[None], k[None], n_cand)[0] & mine[:, None]
            o, l = _attention(q, k, v, kept, n)
            (O[bb, :, h] if nhd else O[bb, h]).copy_(o.flatten(0, 1)[:n])
            lse[bb, h] = l.flatten()[:n]
    return {"O": O, "lse": lse} if case["lse"] or kind != "layer" else {"O": O}
