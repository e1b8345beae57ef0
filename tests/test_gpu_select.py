"""Selection of blocks at the row lengths where the kernels change instance, with many equal scores and infinite ones; and
pooling on both sides of the size at which the kernel changes form."""
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


def _inputs(NB, b, d, seed, infinite):
    """Two heads; the blocks come in groups of five equal ones, so that thresholds fall inside runs of equal scores."""
    g = torch.Generator().manual_seed(seed)
    Q = torch.randn(2, NB * b, d, generator=g)
    K = torch.randn(2, (NB + 4) // 5, 1, b * d, generator=g).expand(-1, -1, 5, -1).reshape(2, -1, d)[:, :NB * b].clone()
    if infinite:  # one block scores +inf for half of the queries and -inf for the others
        Q[:, :, 0] = torch.where(torch.arange(NB * b) // b % 2 == 0, 1e30, -1e30)
        K[:, :, 0] = 1e-30
        K[:, 2 * b:3 * b, 0] = 1e30
    return Q.to(torch.bfloat16), K.to(torch.bfloat16)


@pytest.mark.parametrize("NB", [31, 128, 129, 256, 257, 384, 385, 512, 513, 640, 641, 768, 769, 1024])
@pytest.mark.parametrize("infinite", [False, True])
def test_topk_rows_of_every_instance(oracle_mod, binding, NB, infinite):
    b, d = 64, 64
    Q, K = _inputs(NB, b, d, NB, infinite)
    shape = binding.make_shape(2, d, (1, 1, NB * b - 3), 0, b)
    Q, K = Q[:, :NB * b - 3].contiguous(), K[:, :NB * b - 3].contiguous()
    ws = binding.make_workspace(shape, 1)
    Qd, Kd = Q.cuda(), K.cuda()
    for k in (1, 2, NB // 7 + 1, NB - 1, NB):
        pu.check_mask(oracle_mod, binding, shape, Q, K, Qd, Kd, k, 0, ws)


@pytest.mark.parametrize("NB", [31, 128, 129, 256, 257, 384, 385, 512, 513, 640, 641, 768, 769, 1024])
def test_threshold_rows_of_every_instance(oracle_mod, binding, NB):
    b, d = 64, 64
    Q, K = _inputs(NB, b, d, NB + 1, False)
    shape = binding.make_shape(2, d, (1, 1, NB * b), 0, b)
    ws = binding.make_workspace(shape, 1)
    g = binding.sparsp_geometry(shape)
    Qd, Kd = Q.cuda(), K.cuda()
    for tau, scale in ((1e-6, 0.0), (0.5, 40.0), (0.93, 3.0), (1.0, 0.0)):
        mask = torch.zeros(1, 2, NB, g.n_words, dtype=torch.int32, device="cuda")
        cnt = torch.zeros(1, 2, NB, dtype=torch.int32, device="cuda")
        binding.sparsp_block_mask_cdf(shape, Qd, Kd, tau, scale, mask, cnt, None, None, ws)
        ref = oracle_mod.block_mask_cdf(Q, K, b, tau, 0, scale)
        assert np.array_equal(pu.u32(mask[0]), ref["mask"]), (tau, scale)
        assert np.array_equal(cnt[0].cpu().numpy(), ref["kv_count"])


@pytest.mark.parametrize("NB", [31, 129, 257, 385, 513, 641, 769, 1024])
def test_threshold_rows_with_infinite_scores(oracle_mod, binding, NB):
    """Odd query blocks score one block -inf: the search starts at an infinite end.  Even ones score it +inf: no difference to
    that maximum is a number or finite, all weights are zero, and no block reaches the threshold."""
    b, d = 64, 64
    Q, K = _inputs(NB, b, d, NB + 2, True)
    shape = binding.make_shape(2, d, (1, 1, NB * b), 0, b)
    ws = binding.make_workspace(shape, 1)
    g = binding.sparsp_geometry(shape)
    Qd, Kd = Q.cuda(), K.cuda()
    for tau, scale in ((1e-6, 0.0), (0.5, 40.0), (0.93, 3.0), (1.0, 0.0)):
        mask = torch.zeros(1, 2, NB, g.n_words, dtype=torch.int32, device="cuda")
        cnt = torch.zeros(1, 2, NB, dtype=torch.int32, device="cuda")
        binding.sparsp_block_mask_cdf(shape, Qd, Kd, tau, scale, mask, cnt, None, None, ws)
        ref = oracle_mod.block_mask_cdf(Q, K, b, tau, 0, scale)
        got, count = pu.u32(mask[0]), cnt[0].cpu().numpy()
        assert np.array_equal(got[:, 1::2], ref["mask"][:, 1::2]), (tau, scale)
        assert np.array_equal(count[:, 1::2], ref["kv_count"][:, 1::2])
        assert not got[:, ::2].any() and not count[:, ::2].any()


@pytest.mark.parametrize("d,b", [(64, 64), (128, 128)])
@pytest.mark.parametrize("layout", ["HND", "NHD"])
def test_pool_at_the_change_of_form(oracle_mod, binding, d, b, layout):
    """2 * heads * blocks * d / 8 threads just below and just above 148 * 512, with a ragged last block."""
    NB = 37
    edge = 148 * 512 // (2 * NB * (d // 8))
    for H in (edge, edge + 1):
        N = NB * b - 21
        g = torch.Generator().manual_seed(H)
        Q, K = (torch.randn(H, N, d, generator=g).to(torch.bfloat16) for _ in range(2))
        shape = binding.make_shape(H, d, (1, 1, N), 0, b, layout=layout)
        ws = binding.make_workspace(shape, 1)
        got = pu.gpu_block_mask(binding, shape, pu.to_layout(Q, layout).cuda(), pu.to_layout(K, layout).cuda(), 5, ws)
        for name, x in (("pooled_q", Q), ("pooled_k", K)):
            assert np.array_equal(got[name][0].cpu().numpy().view(np.uint32), oracle_mod.pool(x, b).view(np.uint32)), name
