"""Scores and selection of rows of up to 128 blocks in one launch, and both sides of the rules that choose it and its rows per
CTA, against the oracle: masks, counts and lists to the bit, by top-k and by threshold."""
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


# heads x blocks: one block; a last word that is part full, full, and the first row too long; 4, 8 and 16 rows a CTA
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("H,NB", [(1, 1), (3, 31), (2, 33), (2, 127), (1, 128), (1, 129), (37, 16), (38, 16), (37, 64), (38, 64)])
def test_masks_of_short_rows(oracle_mod, binding, d, H, NB):
    b, n_text = 64, 5 if NB > 2 else 0
    N = NB * b - 3
    gen = torch.Generator().manual_seed(H + NB + d)
    Q, K = (torch.randn(H, N, d, generator=gen).to(torch.bfloat16) for _ in range(2))
    if NB > 4:
        K[:, 2 * b:3 * b] = K[:, :b]  # blocks of equal scores
    shape = binding.make_shape(H, d, (1, 1, N - n_text), n_text, b)
    g = binding.sparsp_geometry(shape)
    ws = binding.make_workspace(shape, 1)
    Qd, Kd = Q.cuda(), K.cuda()
    for k in sorted({1, max(1, g.n_video_blocks // 3), g.n_video_blocks}):
        pu.check_mask(oracle_mod, binding, shape, Q, K, Qd, Kd, k, n_text, ws)
    for tau in (0.4, 0.9):
        mask = torch.zeros(1, H, NB, g.n_words, dtype=torch.int32, device="cuda")
        count = torch.zeros(1, H, NB, dtype=torch.int32, device="cuda")
        binding.sparsp_block_mask_cdf(shape, Qd, Kd, tau, 0.0, mask, count, None, None, ws)
        ref = oracle_mod.block_mask_cdf(Q, K, b, tau, n_text)
        assert np.array_equal(pu.u32(mask[0]), ref["mask"]) and np.array_equal(count[0].cpu().numpy(), ref["kv_count"])
    assert binding.sparsp_status(ws) == binding.SPARSP_OK
