"""Calls that are refused, that fail on the device, or that carry nothing: what they answer and what they leave behind.
Tolerance 0 throughout: status words, stream bytes and lengths are compared as they are."""
import pytest
import torch

from gpu_util import status_tensor

pytestmark = pytest.mark.gpu

DTYPES = {0: torch.bfloat16, 1: torch.float16, 2: torch.float32}


def _weights(count, dt, seed, std=0.02):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.randn(count, device="cuda", generator=gen) * std).to(DTYPES[dt])


@pytest.mark.parametrize("dt", [0, 1, 2])
@pytest.mark.parametrize("tensors", [1, 16, 17, 40])
def test_batched_decompress_of_a_list_without_elements(dt, tensors):
    """Lists on both sides of the 16 tensors that travel in the launch parameters, none of which has a block to decode: their
    80-byte streams are accepted, and a damaged one among them is reported."""
    import paper_2604_03298_b200 as enec
    nothing = torch.empty(0, dtype=DTYPES[dt], device="cuda")
    out = torch.empty(16, dtype=DTYPES[dt], device="cuda")
    streams = [enec.compress_tensor(nothing).clone() for _ in range(tensors)]
    status = status_tensor()
    assert enec.enec_decompress_batched([(s, s.numel(), out, 0) for s in streams], dt, status) == 0
    assert int(status.item()) == 0
    streams[-1][0] = 0x58   # the magic
    assert enec.enec_decompress_batched([(s, s.numel(), out, 0) for s in streams], dt, status) == 0
    assert int(status.item()) == -4
