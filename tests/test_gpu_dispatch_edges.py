"""Sizes on both sides of the library's dispatch rules, where a kernel or a split changes. Tolerance 0 throughout: the
codec is lossless, so outputs equal the inputs or the oracle's bytes."""
import numpy as np
import pytest
import torch

from gpu_util import status_tensor, words_of

pytestmark = pytest.mark.gpu

DTYPES = {0: torch.bfloat16, 1: torch.float16, 2: torch.float32}
BITS = {0: torch.int16, 1: torch.int16, 2: torch.int32}


def _weights(count, dt, seed, std=0.02):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.randn(count, device="cuda", generator=gen) * std).to(DTYPES[dt])


@pytest.mark.parametrize("total_blocks", [17, 444, 1775, 1776, 1777])
def test_batched_decompress_chunk_lengths(total_blocks):
    """17 tensors (a ticketed list) around the number of blocks where chunks grow from one block to two."""
    import paper_2604_03298_b200 as enec
    blocks = [total_blocks // 17 + (1 if i < total_blocks % 17 else 0) for i in range(17)]
    srcs = [_weights(b * 16384 - (i * 977 if b > 1 else 0), 0, i) for i, b in enumerate(blocks)]
    status = status_tensor()
    streams = [enec.compress_tensor(s) for s in srcs]
    outs = [torch.zeros_like(s) for s in srcs]
    for _ in range(2):   # twice: the list's scratch is reused
        assert enec.enec_decompress_batched([(b, b.numel(), o, o.numel()) for b, o in zip(streams, outs)], 0, status) == 0
        assert int(status.item()) == 0
        for s, o in zip(srcs, outs):
            assert torch.equal(s.view(torch.int16), o.view(torch.int16))
            o.zero_()
