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


@pytest.mark.parametrize("dt", [0, 1, 2])
@pytest.mark.parametrize("count", [100, 5000, 16384 * 3, 16384 * 60 + 77, 16384 * 500 + 5003])
def test_given_parameters_that_lose_a_value_leave_no_stream(dt, count):
    """The output held a valid stream of the same size, the length word something else: neither may stand for the failed
    call's result. With and without a status word, the lost value in the first, a middle and the last block."""
    import paper_2604_03298_b200 as enec
    t = _weights(count, dt, count)
    least = 2e-3 if dt == 1 else 1e-6   # a range of exponents that does not need all bits: there are some to lose
    t = torch.where(t.abs() < least, torch.full_like(t, least), t)
    before = enec.compress_tensor(t)
    b, n, m = before[20:23].tolist()
    assert n < (5 if dt == 1 else 8)
    cap = enec.enec_max_compressed_size(dt, count)
    buf = torch.zeros(cap, dtype=torch.uint8, device="cuda")
    out = torch.empty_like(t)
    for at in {0, count // 2, count - 1}:
        for status in (status_tensor(), None):
            buf[:before.numel()] = before
            bad = t.clone()
            bad[at] = 3.0e4 if dt == 1 else 1.0e12   # the only value that (b, n) loses
            size, decoded = torch.full((1,), 77, dtype=torch.int64, device="cuda"), status_tensor()
            assert enec.enec_compress_with_params(bad, dt, count, b, n, m, buf, cap, size, status) == 0
            assert int(size.item()) == 0
            assert status is None or int(status.item()) == -5
            assert buf[:4].tolist() == [0, 0, 0, 0]
            assert enec.enec_decompress(buf, cap, dt, count, out, decoded) == 0
            assert int(decoded.item()) == -4


def test_checked_calls_while_the_stream_is_captured():
    """A checked compress call cannot be recorded: it is refused each time it is made and leaves the capture as it is, in a thread that
    has made checked calls before and in one that makes its first, after a call that failed and after one that did not."""
    import threading
    import paper_2604_03298_b200 as enec
    t = _weights(50000, 0, 3)
    stream = enec.compress_tensor(t)

    def work(said):
        x = torch.ones(8, device="cuda")
        for _ in range(2):
            graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.graph(graph, stream=side):
                for _ in range(3):
                    with pytest.raises(enec.EnecError) as err:
                        enec.compress_tensor(t)
                    said.append(err.value.status)
                y = x + 1
            graph.replay()
            torch.cuda.synchronize()
            said.append(bool((y == 2).all()))
            said.append(torch.equal(enec.compress_tensor(t), stream))   # and outside it works
            with pytest.raises(enec.EnecError):
                enec.compress_tensor(t, params=(100, 1, 1))               # loses exponents

    for place in ("here", "thread"):
        said = []
        if place == "here":
            work(said)
        else:
            th = threading.Thread(target=work, args=(said,))
            th.start()
            th.join()
        assert said == [-1, -1, -1, True, True] * 2, place
