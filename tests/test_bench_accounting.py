"""The figures that bench.py derives from masks and unions, against loops over their bits, and its functions' names."""
import builtins
import dis
import types

import numpy as np
import pytest
import torch

import bench


def _words(bits):
    """Bool [..., NB] -> int32 bit words [..., ceil(NB / 32)]."""
    NB = bits.shape[-1]
    out = np.zeros(bits.shape[:-1] + ((NB + 31) // 32,), np.uint32)
    for j in range(NB):
        out[..., j // 32] |= bits[..., j].astype(np.uint32) << np.uint32(j % 32)
    return torch.as_tensor(out.view(np.int32))


@pytest.mark.parametrize("B,P,H,NB", [(1, 1, 2, 5), (1, 4, 3, 32), (2, 3, 2, 71)])
def test_distinct_tiles(B, P, H, NB):
    rng = np.random.default_rng(NB)
    U, rank = rng.random((B, P, H, NB)) < 0.3, rng.integers(0, P, NB)
    want = sum(any(U[b, r, h, j] and rank[j] != r for r in range(P))
               for b in range(B) for h in range(H) for j in range(NB))
    assert bench.distinct_tiles(_words(U), torch.as_tensor(rank.astype(np.int32))) == want


@pytest.mark.parametrize("B,H,NB,b,N,d", [(1, 2, 5, 64, 5 * 64, 64), (2, 3, 40, 128, 40 * 128 - 77, 128)])
def test_kept_flops(B, H, NB, b, N, d):
    M = np.random.default_rng(NB).random((B, H, NB, NB)) < 0.4
    size = [min(b, N - j * b) for j in range(NB)]
    pairs = sum(size[i] * size[j] for _, _, i, j in zip(*np.nonzero(M)))
    flops, kept = bench.kept_flops_and_counts(_words(M), N, b, d)
    assert (flops, kept) == (4.0 * d * pairs, int(M.sum()))


def test_every_name_that_a_function_uses_exists():
    """A function that uses a module which only its neighbours import fails when it is called, on the GPU machine."""
    def globals_of(code):
        for i in dis.get_instructions(code):
            if i.opname in ("LOAD_GLOBAL", "LOAD_NAME"):
                yield i.argval
        for c in code.co_consts:
            if isinstance(c, types.CodeType):
                yield from globals_of(c)

    with open(bench.__file__) as f:
        code = compile(f.read(), bench.__file__, "exec")
    known = set(vars(bench)) | set(vars(builtins)) | {"__module__", "__qualname__", "__name__"}
    missing = {n for c in code.co_consts if isinstance(c, types.CodeType) for n in globals_of(c)} - known
    assert not missing, missing
