"""The gather of packed tiles, source by source: a tile goes to every consumer that selected it."""
import numpy as np
import pytest
import torch

import parity_util as pu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    from paper_2609_32197_b200 import binding as b
    return b


@pytest.mark.parametrize("d,b", [(64, 64), (128, 64), (64, 128), (128, 128)])
@pytest.mark.parametrize("layout", ["HND", "NHD", "padded"])
@pytest.mark.parametrize("P,local", [(1, True), (3, False), (33, False), (64, True)])
def test_packed_bytes_and_plan(oracle_mod, binding, d, b, layout, P, local):
    """1 to 64 consumers per tile (more than a warp's lanes among them), a head that nobody selects from, a ragged last
    block, and token strides with and without a gap: all outputs equal the oracle's, byte for byte."""
    H, NB = 3, 37
    N = NB * b - 19
    rng = np.random.default_rng(100 * P + d + b)
    K = torch.tensor(rng.standard_normal((H, N, d))).to(torch.bfloat16)
    V = torch.tensor(rng.standard_normal((H, N, d))).to(torch.bfloat16)
    M = rng.random((H, NB, NB)) < 0.15
    M[1] = False
    words = np.zeros((H, NB, 2), np.uint32)
    for j in range(NB):
        words[:, :, j // 32] |= M[:, :, j].astype(np.uint32) << np.uint32(j % 32)
    rank = rng.permutation(np.arange(NB, dtype=np.int32) % P).astype(np.int32)
    shape = binding.make_shape(H, d, (1, 1, N), 0, b, layout="NHD" if layout == "NHD" else "HND")
    if layout == "padded":  # a gap of 24 elements behind every token, as in a slice of a wider tensor
        shape.stride_token, shape.stride_head = d + 24, N * (d + 24)
        Kd, Vd = (torch.nn.functional.pad(x, (0, 24), value=7.0).cuda() for x in (K, V))
    else:
        Kd, Vd = pu.to_layout(K, layout).cuda(), pu.to_layout(V, layout).cuda()
    ws = binding.make_workspace(shape, P)
    got = pu.gpu_demand_pack(binding, shape, torch.as_tensor(words.view(np.int32)).cuda(), torch.as_tensor(rank).cuda(), P,
                             binding.SPARSP_INCLUDE_LOCAL if local else 0, Kd, Vd, ws)
    ref = pu.check_demand(oracle_mod, binding, shape, words, rank, P, local, got)
    want = oracle_mod.pack(K, V, ref["U"], rank, b, P, ref["total"], include_local=local)
    packed = got["packed"].cpu().numpy()
    assert np.array_equal(packed[:want.size], want)
    assert (packed[want.size:] == 0xAB).all(), "bytes beyond the last entry were written"
    assert binding.sparsp_status(ws) == binding.SPARSP_OK
