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


def _compress_twice(enec, t, dt):
    """Two calls in a row (the second finds the scratch as the first left it); the stream, checked to be the same twice."""
    n = t.numel()
    cap = enec.enec_max_compressed_size(dt, n)
    got = []
    for _ in range(2):
        buf = torch.full((cap + 64,), 0xA5, dtype=torch.uint8, device="cuda")
        size, status = torch.zeros(1, dtype=torch.int64, device="cuda"), status_tensor()
        assert enec.enec_compress(t, dt, n, buf, cap, size, status) == 0
        assert int(status.item()) == 0
        assert bool((buf[cap:] == 0xA5).all()), "wrote behind the capacity"
        got.append(buf[:int(size.item())].cpu().numpy())
    assert np.array_equal(got[0], got[1])
    return got[0]


def _words(t, dt):
    return t.view(torch.int32).cpu().numpy().view(np.uint32) if dt == 2 else words_of(t)


@pytest.mark.parametrize("dt", [0, 1, 2])
@pytest.mark.parametrize("blocks", [1, 2, 127, 128, 129, 443, 444, 445, 704, 705, 1408, 1409])
@pytest.mark.parametrize("tail", [0, 37, 5003])
def test_compress_around_the_size_where_a_sample_is_taken(oracle, dt, blocks, tail):
    """Blocks of the tensor around 128 (the first-level sums), around the number of CTAs (444) and around 44 MB (704 blocks of
    fp32, 1408 of the others), from where on the parameters come from a sample, with a full, a short and an ordinary last
    block."""
    import paper_2604_03298_b200 as enec
    t = _weights(blocks * 16384 + tail, dt, blocks + tail)
    assert np.array_equal(_compress_twice(enec, t, dt), oracle.compress(_words(t, dt), dt))


@pytest.mark.parametrize("dt", [0, 1, 2])
@pytest.mark.parametrize("what", ["one zero", "one huge", "zero in the tail", "wider rest", "narrower rest", "sample too wide",
                                  "all wide", "constant"])
def test_compress_when_the_sample_misleads(oracle, dt, what):
    """2961 blocks, of which every twentieth is sampled. The stream has to be the one that the search on the whole tensor
    leads to."""
    import paper_2604_03298_b200 as enec
    blocks = 2961
    t = _weights(blocks * 16384 + 4000, dt, 7, 0.0002 if what == "one huge" else 0.02)
    t = torch.where(t == 0, torch.full_like(t, 0.001), t)
    if dt == 1:
        t = torch.where(t.abs() < 2e-3, torch.full_like(t, 2e-3), t)   # fp16: a narrow range of exponents otherwise
    body = t[:blocks * 16384].view(blocks, 16384)
    if what == "one zero":
        body[2641, 77] = 0
    elif what == "one huge":
        body[1, 16000] = 60000.0
    elif what == "zero in the tail":
        t[-3] = 0
    elif what == "wider rest":
        body[1::2] *= 3.0
        body[2::4] *= 0.4
    elif what == "narrower rest":
        body[1::20] = 0.02
        body[2::20] = 0.02
        body[3::4] = 0.02
    elif what == "sample too wide":
        body[0, 5] = 0
        body[2000, 6] = 3e4
    elif what == "all wide":
        bits = torch.randint(0, 1 << 15, (t.numel(),), device="cuda", generator=torch.Generator(device="cuda").manual_seed(3))
        t = (bits.to(torch.int32) << 16 if dt == 2 else bits.to(torch.int16)).view(DTYPES[dt])
    else:
        t = torch.full_like(t, 0.75)
    assert np.array_equal(_compress_twice(enec, t, dt), oracle.compress(_words(t, dt), dt))


@pytest.mark.parametrize("dt", [0, 1, 2])
def test_compress_batched_across_waves(oracle, dt):
    """A list whose tensors are counted and packed in several waves of 40 MB (one tensor is more than a wave), with tensors
    of one block, of a few elements, and with last blocks of every kind between them."""
    import paper_2604_03298_b200 as enec
    counts = [16384 * 1300 + 5, 16384 * 2, 100, 16384, 16385, 0, 16384 * 5 - 1, 2048, 16384 * 129, 37, 16384 * 400, 16384 * 500 + 60,
              16384 * 3, 5, 16384 * 7 + 8000]
    srcs = [_weights(c, dt, 70 + i, 0.02 * (1 + i % 4)) for i, c in enumerate(counts)]
    caps = [enec.enec_max_compressed_size(dt, c) for c in counts]
    for _ in range(2):   # twice: the call's scratch is reused
        bufs = [torch.full((c + 16,), 0xA5, dtype=torch.uint8, device="cuda") for c in caps]
        sizes, status = torch.zeros(len(counts), dtype=torch.int64, device="cuda"), status_tensor()
        assert enec.enec_compress_batched([(s, b, c, cap) for s, b, c, cap in zip(srcs, bufs, counts, caps)], dt, sizes, status) == 0
        assert int(status.item()) == 0
        for i, (b, n, cap) in enumerate(zip(bufs, sizes.tolist(), caps)):
            assert bool((b[cap:] == 0xA5).all())
            assert np.array_equal(b[:n].cpu().numpy(), oracle.compress(_words(srcs[i], dt), dt)), f"tensor {i}"


@pytest.mark.parametrize("dt", [0, 1, 2])
@pytest.mark.parametrize("count", [65, 127, 128, 4096, 8193, 16383, 16384 * 3 + 65, 16384 * 2 + 8192, 16384 * 2 + 16375])
@pytest.mark.parametrize("wide", [False, True])
def test_decompress_last_blocks(oracle, dt, count, wide):
    """Last blocks of 128 padded elements or more take a body of their own; `wide`: with more wide groups than the sixteen-byte
    form of the expanded records has room for."""
    import paper_2604_03298_b200 as enec
    t = _weights(count, dt, count, 0.02)
    if wide:   # one value in ten far below the others
        t = torch.where(torch.rand(count, device="cuda", generator=torch.Generator(device="cuda").manual_seed(5)) < 0.1, t / 64, t)
    w = _words(t, dt)
    stream = torch.from_numpy(oracle.compress(w, dt)).cuda()
    out = torch.full((count + 64,), 1.0, dtype=DTYPES[dt], device="cuda")
    status = status_tensor()
    assert enec.enec_decompress(stream, stream.numel(), dt, count, out, status) == 0
    assert int(status.item()) == 0
    assert torch.equal(out[:count].view(BITS[dt]), t.view(BITS[dt]))
    assert bool((out[count:] == 1.0).all()), "wrote behind the tensor"


@pytest.mark.parametrize("dt", [0, 1, 2])
@pytest.mark.parametrize("blocks", [0, 1, 2, 129, 445, 889])
@pytest.mark.parametrize("tail", [0, 37, 5003])
def test_compress_with_given_parameters(dt, blocks, tail):
    """The search's parameters given back lead to the search's stream (checked against the oracle elsewhere); parameters that
    lose a value, wherever it is, lead to an error and no stream length."""
    import paper_2604_03298_b200 as enec
    n = blocks * 16384 + tail
    if n == 0:
        return
    t = _weights(n, dt, blocks + tail)
    want = enec.compress_tensor(t)
    b, nn, m = want[20:23].tolist()
    assert torch.equal(enec.compress_tensor(t, params=(b, nn, m)), want)
    size, status = torch.full((1,), -1, dtype=torch.int64, device="cuda"), status_tensor()
    buf = torch.zeros(enec.enec_max_compressed_size(dt, n), dtype=torch.uint8, device="cuda")
    for at in {0, n // 2, n - 1}:
        bad = t.clone()
        bad[at] = 3.0e4                      # an exponent far above the others
        status.zero_()
        assert enec.enec_compress_with_params(bad, dt, n, b, 4, min(m, 4), buf, buf.numel(), size, status) == 0
        assert int(status.item()) == -5 and int(size.item()) == 0   # 0, not what the word held: no stream, no length
    wide = (b, 8 if dt != 1 else 5, m)       # any exponent survives the full width; the groups' form differs
    back = enec.decompress_tensor(enec.compress_tensor(t, params=wide), t.dtype, t.shape)
    assert torch.equal(back.view(BITS[dt]), t.view(BITS[dt]))


@pytest.mark.parametrize("dt", [0, 1, 2])
@pytest.mark.parametrize("blocks", [443, 444, 445, 887, 888, 889, 1331])
@pytest.mark.parametrize("tail", [0, 1, 5003])
def test_decompress_last_block_apart(dt, blocks, tail):
    """Sizes around multiples of the number of CTAs (three per SM), where a ragged last block gets a CTA of its own or not."""
    import paper_2604_03298_b200 as enec
    t = _weights(blocks * 16384 + tail, dt, blocks + tail)
    out = enec.decompress_tensor(enec.compress_tensor(t), t.dtype, t.shape)
    assert torch.equal(out.view(BITS[dt]), t.view(BITS[dt]))


def test_checked_calls_report_errors_and_recover():
    """compress_tensor / decompress_tensor read length and status from pinned host memory that the kernels write: an error is
    raised, and the next call on the thread starts clean; threads do not share the memory."""
    import threading
    import paper_2604_03298_b200 as enec
    t = _weights(16384 * 3 + 100, 0, 5)
    for _ in range(2):
        with pytest.raises(enec.EnecError) as err:
            enec.compress_tensor(t, params=(100, 1, 1))   # loses exponents
        assert err.value.status == -5
        s = enec.compress_tensor(t)
        assert torch.equal(enec.decompress_tensor(s, t.dtype, t.shape).view(torch.int16), t.view(torch.int16))
        bad = s.clone()
        bad[8] ^= 1                                      # another count in the header
        with pytest.raises(enec.EnecError) as err:
            enec.decompress_tensor(bad, t.dtype, t.shape)
        assert err.value.status == -4
    empty = enec.compress_tensor(t[:0])
    assert empty.numel() == 80 and enec.decompress_tensor(empty, t.dtype, (0,)).numel() == 0

    def work(seed, ok):
        x = _weights(16384 * 2 + seed, 0, seed)
        with torch.cuda.stream(torch.cuda.Stream()):
            x.record_stream(torch.cuda.current_stream())
            torch.cuda.current_stream().wait_stream(torch.cuda.default_stream())
            ok[seed] = all(torch.equal(enec.decompress_tensor(enec.compress_tensor(x), x.dtype, x.shape).view(torch.int16), x.view(torch.int16))
                           for _ in range(20))

    ok = {}
    threads = [threading.Thread(target=work, args=(i, ok)) for i in range(4)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert ok == {i: True for i in range(4)}


@pytest.mark.parametrize("low, high", [("100", ""), ("100", "150"), ("", "150")])
def test_the_environment_moves_the_split_forms_bounds(low, high):
    """ENEC_SPLIT_MIN_BLOCKS and ENEC_SPLIT_MAX_BLOCKS say for which sizes enec_compress takes three kernels; all other sizes, and
    given parameters of any size, take one. (Read once per process, hence the child.)"""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    child = f"""
import sys
sys.path.insert(0, {root!r})
import torch
import paper_2604_03298_b200 as enec
for blocks in (1, 99, 100, 149, 150, 300):
    t = (torch.randn(blocks * 16384, device="cuda", generator=torch.Generator(device="cuda").manual_seed(blocks)) * 0.02).bfloat16()
    before = enec.enec_launch_count()
    stream = enec.compress_tensor(t)
    searched = enec.enec_launch_count() - before
    assert torch.equal(enec.compress_tensor(t, params=stream[20:23].tolist()), stream)
    given = enec.enec_launch_count() - before - searched
    print(blocks, searched, given)
"""
    env = {k: v for k, v in os.environ.items() if not k.startswith("ENEC_")}
    env.update({k: v for k, v in (("ENEC_SPLIT_MIN_BLOCKS", low), ("ENEC_SPLIT_MAX_BLOCKS", high)) if v})
    res = subprocess.run([sys.executable, "-c", child], env=env, capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stderr[-2000:]
    want = {b: 3 if low and b >= 100 and (not high or b < 150) else 1 for b in (1, 99, 100, 149, 150, 300)}
    assert res.stdout.split("\n")[:-1] == [f"{b} {n} 1" for b, n in want.items()]


def _mislead(t, blocks, what):
    """Changes values of blocks that the sample (every (blocks // 148)-th, from the first on) does not hold."""
    step = blocks // 148
    body = t[:blocks * 16384].view(blocks, 16384)
    at = {"early": 1, "middle": blocks // 2 // step * step + 1, "late": (blocks - 2) // step * step + 1}
    if what in at:
        body[at[what], 77] = 0            # the pass ends there, the rest is counted, everything packed again
    else:
        for k in range(1, step):          # no value is lost, but the whole tensor has another (b, m)
            body[k::step] *= 3.0
    return t


@pytest.mark.parametrize("dt, blocks", [(0, 1409), (1, 1409), (2, 705)])
@pytest.mark.parametrize("tail", [0, 37, 5003])
@pytest.mark.parametrize("what", ["early", "middle", "late", "other parameters"])
def test_misled_samples_just_above_the_bound(oracle, dt, blocks, tail, what):
    """The smallest sizes of which a sample is taken."""
    import paper_2604_03298_b200 as enec
    least = 2e-3 if dt == 1 else 1e-6
    t = _weights(blocks * 16384 + tail, dt, 11)
    t = _mislead(torch.where(t.abs() < least, torch.full_like(t, least), t), blocks, what)
    assert np.array_equal(_compress_twice(enec, t, dt), oracle.compress(_words(t, dt), dt))


@pytest.mark.parametrize("what", ["early", "late", "other parameters"])
def test_misled_samples_with_second_level_sums(oracle, what):
    """More than 16384 blocks: the second pass has second-level sums of its own."""
    import paper_2604_03298_b200 as enec
    blocks = 16384 + 300
    t = _weights(blocks * 16384 + 100, 0, 12)
    t = _mislead(torch.where(t.abs() < 1e-6, torch.full_like(t, 1e-6), t), blocks, what)
    assert np.array_equal(_compress_twice(enec, t, 0), oracle.compress(_words(t, 0), 0))


def _sixteen_behind(t):
    """A copy of the tensor that starts 16 bytes behind a 32-byte boundary (torch's allocator never gives such an address)."""
    ahead = 16 // t.element_size()
    holder = torch.zeros(t.numel() + ahead, dtype=t.dtype, device="cuda")
    assert holder.data_ptr() % 32 == 0
    holder[ahead:].copy_(t)
    return holder[ahead:]


@pytest.mark.parametrize("dt", [0, 1, 2])
@pytest.mark.parametrize("full_width", [False, True])
@pytest.mark.parametrize("count", [16384, 8192 + 300, 16384 * 5, 16384 * 5 + 300, 16384 * 3 + 37, 16384 * 1409, 16384 * 1409 + 300])
def test_compress_inputs_sixteen_bytes_behind_a_32_byte_boundary(oracle, dt, full_width, count):
    """Such inputs take 16-byte loads, for bf16 and fp16 in a body of its own: with a search on the whole tensor and on a sample, with
    given parameters, and in a list beside inputs on a 32-byte boundary. full_width: an exact zero, so that n = E (for bf16 and fp32
    the form in which b + 2^(n-1) does not fit a byte)."""
    import paper_2604_03298_b200 as enec
    t = _weights(count, dt, count)
    t = torch.where(t.abs() < 2e-3, torch.full_like(t, 2e-3), t)
    if full_width:
        t[count // 2] = 0
    want = oracle.compress(_words(t, dt), dt)
    odd = _sixteen_behind(t)
    assert odd.data_ptr() % 32 == 16
    assert np.array_equal(_compress_twice(enec, odd, dt), want)
    assert np.array_equal(enec.compress_tensor(odd, params=want[20:23].tolist()).cpu().numpy(), want)
    srcs = [odd, t, odd]
    cap = enec.enec_max_compressed_size(dt, count)
    bufs = [torch.full((cap + 16,), 0xA5, dtype=torch.uint8, device="cuda") for _ in srcs]
    sizes, status = torch.zeros(len(srcs), dtype=torch.int64, device="cuda"), status_tensor()
    assert enec.enec_compress_batched([(s, b, count, cap) for s, b in zip(srcs, bufs)], dt, sizes, status) == 0
    assert int(status.item()) == 0
    for b, n in zip(bufs, sizes.tolist()):
        assert bool((b[cap:] == 0xA5).all())
        assert np.array_equal(b[:n].cpu().numpy(), want)


@pytest.mark.parametrize("dt, b, n, m", [(0, 120, 5, 3), (0, 120, 6, 3), (0, 120, 7, 3), (0, 127, 8, 3), (0, 127, 8, 1), (0, 120, 4, 3),
                                         (1, 14, 5, 4), (1, 14, 5, 3), (1, 14, 5, 2), (1, 14, 5, 1), (2, 120, 6, 3), (2, 127, 8, 1)])
def test_waiting_records_are_copied_to_any_offset(oracle, dt, b, n, m):
    """A block's packed records wait in 4096 bytes of shared memory and go to their offset in pieces of 16 bytes, with single halves
    (16 bits) before and behind them: blocks with no, few, many and all groups wide, with records that fill the 4096 bytes, fall just
    short of them or exceed them (those go straight to their place), at offsets of every remainder. Enough blocks that a CTA
    packs several and uses both of its places."""
    import paper_2604_03298_b200 as enec
    blocks, h = 1400, n - m
    rng = np.random.default_rng(100 * n + m + dt)
    fit = 2048 // h   # wide groups whose records fit
    wide = rng.choice([c for c in (0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 15, 250, fit - 1, fit, fit + 1, 1024) if c <= 1024], blocks)
    start = (np.cumsum(wide) - wide) * h   # in halves, from an address that is a multiple of 16 bytes
    waits = (wide <= fit) & (wide > 0)
    assert set((start[waits] % 8).tolist()) == (set(range(8)) if h % 8 % 2 else set(range(0, 8, 2 if h % 4 else 4)))
    assert h in (4, 7) or ((wide * h < (-start) % 8) & waits).any()   # records that end before the first aligned piece
    # every group holds b (stored as 0); a wide one also b + 1 (stored as 2^n - 1) and any below b
    is_wide = np.argsort(rng.random((blocks, 1024)), 1) < wide[:, None]
    x = np.full((blocks, 1024, 16), b, dtype=np.uint32)
    x[..., 5] += is_wide
    x[..., 11] = np.where(is_wide, b - rng.integers(0, 1 << (n - 1), is_wide.shape), b)
    x = x.reshape(-1)
    other = rng.integers(0, 1 << 32, x.size, dtype=np.uint32)   # sign and mantissa
    if dt == 2:
        w = x << 23 | (other & 0x807FFFFF)
    else:
        mant = 7 if dt == 0 else 10
        w = (x << mant | (other & (0x8000 | ((1 << mant) - 1)))).astype(np.uint16)
    t = torch.from_numpy(w.view(np.int32 if dt == 2 else np.int16)).cuda().view(DTYPES[dt])
    want = oracle.compress(w, dt, (b, n, m))
    assert want[32:36].view(np.uint32)[0] == wide.sum()   # the header's count of wide groups
    for _ in range(2):
        got = enec.compress_tensor(t, params=(b, n, m))
        assert np.array_equal(got.cpu().numpy(), want)


def test_where_a_ctas_shared_memory_begins():
    """The pack stage addresses its histogram by an AND-OR, which wants it on a multiple of its size; where it is not, sampled tensors
    are counted whole first (a waste that no stream shows). The kernels have no static shared memory, and dynamic shared memory
    begins where the layout in enec_fused.cuh takes it to begin."""
    import ctypes
    import os
    import re
    import paper_2604_03298_b200 as enec

    lib, runtime = enec.lib(), ctypes.CDLL("libcudart.so.12")
    for dt in range(3):
        for kernel, job in (("17enec_fused_kernel", "8FusedJob"), ("22enec_fused_list_kernel", "9FusedList")):
            attributes = (ctypes.c_size_t * 64)()   # cudaFuncAttributes begins with sharedSizeBytes
            stub = ctypes.cast(getattr(lib, f"_ZN4enec{kernel}ILi{dt}EEEvNS_{job}EPi"), ctypes.c_void_p)
            assert runtime.cudaFuncGetAttributes(attributes, stub) == 0
            assert attributes[0] == 0
    probe = torch.cuda._compile_kernel("""extern "C" __global__ void base(unsigned* out) {
        extern __shared__ __align__(128) unsigned char s[];
        if (threadIdx.x == 0) *out = (unsigned)__cvta_generic_to_shared(s);
    }""", "base")
    out = torch.zeros(1, dtype=torch.int32, device="cuda")
    probe(grid=(1, 1, 1), block=(32, 1, 1), args=[out], shared_mem=1024)
    text = open(os.path.join(os.path.dirname(enec.__file__), "csrc", "enec_fused.cuh")).read()
    place = int(re.search(r"kHistAt = (\d+);", text).group(1))
    for rows in (32, 64):   # of 32 counters
        assert (int(out.item()) + place) % (rows * 128) == 0
