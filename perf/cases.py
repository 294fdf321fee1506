"""What this codec is timed on: weight tensors compressed and decompressed through the package's entry points.

A case names its tensors (`set`), the direction (`op`), how the calls are made (`way`) and the values' type and
distribution. Sizes are those of `synth.config_specs` (a Llama-3-8B-shaped decoder layer, its embedding, one layer of
the MoE-shaped set, an OLMo-1B-shaped fp32 matrix, the heavy-tailed 4096 x 4096 tensors) and odd ones beside them.

  set "tensor"   one tensor of `elements` values
  set "layer"    a decoder layer: q, o (hidden x hidden), k, v (kv x hidden), gate, up, down (ffn x hidden), two norm vectors
  set "experts"  `experts` times gate, up, down (inter x hidden) and `vectors` vectors of `hidden` values

  way "one"      one enec_compress / enec_decompress call
  way "given"    one enec_compress_with_params call, with parameters found before (the offline tuned mode)
  way "each"     a call per tensor of the set, one after another on one stream (a checkpoint, tensor by tensor)
  way "batched"  one enec_compress_batched / enec_decompress_batched call for the set (many small tensors; layer prefetch)
  way "checked"  compress_tensor and decompress_tensor, which allocate and read the size and the status back

  op "roundtrip" compresses and decompresses again.
"""
import math

import torch

import paper_2604_03298_b200 as enec
from paper_2604_03298_b200 import synth

_DTYPES = {"bf16": (torch.bfloat16, enec.BF16, 2), "fp16": (torch.float16, enec.FP16, 2), "fp32": (torch.float32, enec.FP32, 4)}


def _case(name, op, way, dtype="bf16", dist="normal", std=0.02, outliers=False, zeros=False, **tensors):
    case = {"op": op, "way": way, "dtype": dtype, "dist": dist, "std": std, "outliers": outliers, "zeros": zeros, **tensors}
    return {"name": name, **case} if name else case


def _tensor(elements):
    return {"set": "tensor", "elements": elements}


def _layer(hidden, kv, ffn):
    return {"set": "layer", "hidden": hidden, "kv": kv, "ffn": ffn}


def _experts(experts, hidden, inter, vectors):
    return {"set": "experts", "experts": experts, "hidden": hidden, "inter": inter, "vectors": vectors}


def listed():
    return [
        # a norm vector: the smallest call of a checkpoint, 65 of the Llama set's 291 tensors; latency of one call
        _case("norm_compress", "compress", "one", std=0.05, **_tensor(4096)),
        _case("norm_decompress", "decompress", "one", std=0.05, **_tensor(4096)),
        # a k or v projection through the checked calls: a program that takes one tensor at a time and looks at the result
        _case("kv_roundtrip_checked", "roundtrip", "checked", **_tensor(1024 * 4096)),
        # a Llama-3-8B-shaped layer, tensor by tensor on one stream: writing and loading a checkpoint
        _case("layer_compress", "compress", "each", std=1 / 64, **_layer(4096, 1024, 14336)),
        _case("layer_decompress", "decompress", "each", std=1 / 64, **_layer(4096, 1024, 14336)),
        # its gate projection alone: one large call
        _case("gate_decompress", "decompress", "one", std=1 / 64, **_tensor(14336 * 4096)),
        # the embedding: the largest tensor, far beyond L2
        _case("embed_compress", "compress", "one", **_tensor(128256 * 4096)),
        # heavy-tailed fp16 with outliers and exact zeros: half of the groups are wide; once ragged
        _case("heavy_fp16_compress", "compress", "one", "fp16", "laplace", 0.03, outliers=True, **_tensor(4096 * 4096)),
        _case("heavy_fp16_decompress", "decompress", "one", "fp16", "student3", 0.03, outliers=True, **_tensor(4099 * 4093)),
        # an fp32 matrix of odd size, written and read back for a check
        _case("fp32_roundtrip", "roundtrip", "one", "fp32", **_tensor(8192 * 2048 + 1)),
        # one layer of a mixture of experts: many small tensors in one call
        _case("experts_compress", "compress", "batched", **_experts(8, 2048, 1408, 32)),
        _case("experts_decompress", "decompress", "batched", **_experts(8, 2048, 1408, 128)),
    ]


def _between(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    dtype = rng.choice(["bf16", "bf16", "bf16", "fp16", "fp32"])
    half = 2 if dtype == "fp32" else 1
    dist = rng.choice(["normal", "normal", "normal", "laplace", "student3"])
    kind = {"dtype": dtype, "dist": dist, "std": round(math.exp(rng.uniform(math.log(0.005), math.log(0.1))), 4),
            "outliers": dist != "normal" and rng.random() < 0.7,    # 1 % at 50 std, 0.5 % exact zeros
            "zeros": dist == "normal" and rng.random() < 0.15}      # the normal generator's rare exact zeros are left in
    op = rng.choice(["compress", "decompress"])
    way = rng.choice(["one", "one", "one", "each", "batched", "checked", "given"])
    if way in ("one", "given"):
        elements = _between(rng, 2048, 450_000_000 // half)
        if rng.random() < 0.5:
            elements = max(2048, elements & ~4095)
        return _case(None, "compress" if way == "given" else op, way, **kind, **_tensor(elements))
    if way == "checked":
        return _case(None, "roundtrip", way, **kind, **_tensor(_between(rng, 2048, 2 ** 25)))
    hidden = 64 * _between(rng, 12, 64 // half)
    if way == "each" or rng.random() < 0.5:
        return _case(None, op, way, **kind, **_layer(hidden, hidden // rng.choice([1, 2, 4]), int(hidden * rng.uniform(2.5, 4))))
    return _case(None, op, way, **kind, **_experts(rng.randint(4, 10), hidden, 8 * _between(rng, 48, 200), rng.randint(2, 28)))


def _counts(case):
    """(values, is a norm vector) of every tensor of the case."""
    if case["set"] == "tensor":
        return [(case["elements"], False)]
    h = case["hidden"]
    if case["set"] == "layer":
        return [(h * h, False), (case["kv"] * h, False), (case["kv"] * h, False), (h * h, False)] + \
               [(case["ffn"] * h, False)] * 3 + [(h, True)] * 2
    return [(case["inter"] * h, False)] * (3 * case["experts"]) + [(h, False)] * case["vectors"]


def _stream_bytes_per_value(case):
    # what the format needs: bf16 Gaussian weights 11.6 bits (ratio 1.38); exact zeros widen every exponent to n = E
    if case["dtype"] == "fp32":
        return 3.45
    return 1.757 if case["outliers"] else 1.45


def work(case):
    raw = sum(n for n, _ in _counts(case)) * _DTYPES[case["dtype"]][2]
    stream = int(sum(n for n, _ in _counts(case)) * _stream_bytes_per_value(case))
    return {"bytes": (raw + stream) * (2 if case["op"] == "roundtrip" else 1), "flops": 0}


def tolerance(case):
    return "exact"


def _values(case, index, count, norm, seed):
    """One tensor: the case's values, with their groups of 16 in an order and with signs that the seed draws. The length
    of a stream depends on the values group by group, so it is the same for every seed and a stream can be returned whole."""
    dtype = _DTYPES[case["dtype"]][0]
    spec = synth.TensorSpec("w", dtype, (count,), "normal" if norm else case["dist"], 1.0 if norm else 0.0,
                            0.05 if norm else case["std"], 9000 + index, case["outliers"] and not norm)
    t = synth.make_tensor(spec, "cuda", keep_zeros=case["zeros"])
    gen = torch.Generator(device="cuda").manual_seed(1000003 * seed + index)
    order = torch.randperm(count // 16, generator=gen, device="cuda")
    whole = count // 16 * 16
    t[:whole] = t[:whole].view(-1, 16)[order].view(-1)
    return torch.where(torch.rand(count, generator=gen, device="cuda") < 0.5, t, -t)


def prepare(case, seed):
    dtype, dt, _ = _DTYPES[case["dtype"]]
    raw = [_values(case, i, n, norm, seed) for i, (n, norm) in enumerate(_counts(case))]
    state = {"case": case, "raw": raw, "dt": dt}
    if case["way"] == "checked":
        return state
    caps = [enec.enec_max_compressed_size(dt, t.numel()) for t in raw]
    sizes = torch.zeros(len(raw), dtype=torch.int64, device="cuda")
    state["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    streams = [torch.zeros(c, dtype=torch.uint8, device="cuda") for c in caps]
    for i, t in enumerate(raw):
        if enec.enec_compress(t, dt, t.numel(), streams[i], caps[i], sizes[i:i + 1], state["status"]) != 0:
            raise RuntimeError("enec_compress")
    state["lengths"] = sizes.tolist()
    if case["op"] == "decompress":
        state["streams"] = [s[:n].clone() for s, n in zip(streams, state["lengths"])]
        state["out"] = torch.zeros(sum((t.numel() + 15) & ~15 for t in raw), dtype=dtype, device="cuda")
        state["outs"], at = [], 0
        for t in raw:
            state["outs"].append(state["out"][at:at + t.numel()])
            at += (t.numel() + 15) & ~15
        del state["raw"]
        if case["way"] == "batched":
            state["items"] = enec.make_batch([(s, o, o.numel(), s.numel()) for s, o in zip(state["streams"], state["outs"])])
        return state
    state["params"] = streams[0][20:23].tolist()
    for s in streams:
        s.zero_()
    state.update(streams=streams, caps=caps, sizes=sizes.zero_())
    if case["op"] == "roundtrip":
        state["outs"] = [torch.zeros_like(t) for t in raw]
    if case["way"] == "batched":
        state["items"] = enec.make_batch([(t, s, t.numel(), c) for t, s, c in zip(raw, streams, caps)])
    return state


def _must(status):
    if status != 0:
        raise RuntimeError(f"status {status}")


def run(s):
    case, dt, way = s["case"], s["dt"], s["case"]["way"]
    if way == "checked":
        t = s["raw"][0]
        stream = enec.compress_tensor(t)
        return {"stream": stream, "out": enec.decompress_tensor(stream, t.dtype, t.shape)}
    status = s["status"]
    if case["op"] == "decompress":
        if way == "batched":
            _must(enec.enec_decompress_batched(s["items"], dt, status))
        else:
            for stream, out in zip(s["streams"], s["outs"]):
                _must(enec.enec_decompress(stream, stream.numel(), dt, out.numel(), out, status))
        return {"out": s["out"], "status": status}
    if way == "batched":
        _must(enec.enec_compress_batched(s["items"], dt, s["sizes"], status))
    elif way == "given":
        t = s["raw"][0]
        _must(enec.enec_compress_with_params(t, dt, t.numel(), *s["params"], s["streams"][0], s["caps"][0], s["sizes"], status))
    else:
        for i, t in enumerate(s["raw"]):
            _must(enec.enec_compress(t, dt, t.numel(), s["streams"][i], s["caps"][i], s["sizes"][i:i + 1], status))
    got = {"sizes": s["sizes"], "status": status, "streams": [b[:n] for b, n in zip(s["streams"], s["lengths"])]}
    if case["op"] == "roundtrip":
        for stream, cap, out in zip(s["streams"], s["caps"], s["outs"]):
            _must(enec.enec_decompress(stream, cap, dt, out.numel(), out, status))
        got["outs"] = s["outs"]
    return got
