"""Pooled values against a sequential fp32 sum: sequences shorter than a block, a last block of one token up to a whole one,
batches, both layouts, and token strides with room behind a row."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    from paper_2609_32197_b200 import binding as b
    b.lib()
    return b


@pytest.mark.parametrize("d,b", [(64, 64), (128, 64), (64, 128), (128, 128)])
@pytest.mark.parametrize("layout,pad", [("HND", 0), ("HND", 8), ("NHD", 0), ("NHD", 24)])
@pytest.mark.parametrize("n", ["1", "b-1", "b", "b+1", "3*b+7"])
def test_pooled_values(binding, d, b, layout, pad, n):
    N, H, B = eval(n, {"b": b}), 3, 2
    rng = np.random.default_rng(N + d + b + pad)
    shape = binding.make_shape(H, d, (1, 1, N), 0, b, batch=B, layout=layout)
    row = d + pad
    if layout == "HND":
        dims, shape.stride_token, shape.stride_head, shape.stride_batch = (B, H, N, row), row, N * row, H * N * row
    else:
        dims, shape.stride_token, shape.stride_head, shape.stride_batch = (B, N, H, row), H * row, row, N * H * row
    X = [torch.tensor(rng.standard_normal(dims) * 4).to(torch.bfloat16) for _ in range(2)]
    for x in X:
        x[..., d:] = float("nan")  # behind a row: not the tensor's
    NB = (N + b - 1) // b
    mask = torch.zeros(B, H, NB, (NB + 31) // 32, dtype=torch.int32, device="cuda")
    pooled = [torch.full((B, H, NB, d), 7.0, device="cuda") for _ in range(2)]
    ws = binding.make_workspace(shape, 1)
    binding.sparsp_block_mask(shape, X[0].cuda(), X[1].cuda(), 1, mask, None, None, pooled[0], pooled[1], ws)
    assert binding.sparsp_status(ws) == binding.SPARSP_OK
    for x, got in zip(X, pooled):
        x = (x if layout == "HND" else x.permute(0, 2, 1, 3))[..., :d].float().numpy()
        for j in range(NB):
            rows = x[:, :, j * b:(j + 1) * b]
            acc = np.zeros((B, H, d), np.float32)
            for t in range(rows.shape[2]):
                acc = acc + rows[:, :, t]
            want = acc / np.float32(rows.shape[2])
            assert np.array_equal(got[:, :, j].cpu().numpy().view(np.int32), want.view(np.int32))
