"""The work that users of this library have it do, as measurable cases.

Four kinds of pass, each through the public binding:

  encode    sentence embeddings: token ids + mask -> pooled, normalised rows.  The library's main path, in the
            two model shapes of the repository's configurations (6 x 384 with 12 heads of 32, 12 x 768 with
            12 heads of 64), from one query to a full throughput batch, from device buffers or from pinned
            host buffers (the end-to-end call)
  prefill   attention of a decoder layer over packed prompts: rotary q and k, causal or sliding-window mask,
            plain or grouped-query heads
  scaled    a Linear block on block-scaled FP8 / FP6 / FP4 weights with bf16 activations
  mx        a Linear block with both operands on the FP8 block-scaled grid: quantise the activations, multiply

Sequence lengths of a case are the quantiles of the uniform distribution over [lo, hi] in an order drawn from
the seed, so that every seed of a case is the same amount of work on other data.
"""
import math

import torch

import paper_2609_37916_b200 as rlx
from paper_2609_37916_b200 import binding

MODELS = {
    # layers, hidden, heads, feed-forward width
    "minilm": (6, 384, 12, 1536),
    "base": (12, 768, 12, 3072),
}
VOCAB, MAX_POS = 30522, 512
FORMATS = {
    # format word, code bits, largest finite magnitude code, packed nibbles
    "fp8_e4m3": (binding.FMT_FP8_E4M3, 8, 0x7E, False),
    "fp8_e5m2": (binding.FMT_FP8_E5M2, 8, 0x7B, False),
    "fp6_e2m3": (binding.FMT_FP6_E2M3, 6, 0x1F, False),
    "fp4_e2m1": (binding.FMT_FP4_E2M1, 4, 0x7, True),
}
CODE_BITS = {"fp8_e4m3": 8, "fp8_e5m2": 8, "fp6_e2m3": 8, "fp4_e2m1": 4}   # as stored
EPILOGUES = {"bias": binding.EPI_BIAS, "gelu": binding.EPI_BIAS_GELU, "residual": binding.EPI_BIAS_RESIDUAL}


def _encode(name, model, batch, seq, lo, hi, host=False, holes=False):
    return {"name": name, "op": "encode", "model": model, "batch": batch, "seq": seq, "lo": lo, "hi": hi, "host": host,
            "holes": holes}


def _prefill(name, batch, lo, hi, heads, kv_heads, dim, window, in_attention):
    return {"name": name, "op": "prefill", "batch": batch, "lo": lo, "hi": hi, "heads": heads, "kv_heads": kv_heads,
            "dim": dim, "window": window, "in_attention": in_attention}


def listed():
    return [
        # one search query, embedded from host buffers: what a lookup service does per request
        _encode("query_host_1x32", "minilm", 1, 32, 5, 31, host=True),
        # one passage, from device buffers: the repository's latency configuration
        _encode("passage_1x128", "minilm", 1, 128, 8, 128),
        # the headline batch, from device buffers (called in a loop) and end to end from pinned host buffers
        _encode("batch_32x128", "minilm", 32, 128, 8, 128),
        _encode("batch_host_32x128", "minilm", 32, 128, 8, 128, host=True),
        # an odd, fairly dense batch of a few thousand tokens with positions masked out inside the sequences
        _encode("ragged_61x203", "minilm", 61, 203, 40, 203, holes=True),
        # indexing a corpus: the repository's throughput configuration
        _encode("corpus_256x256", "minilm", 256, 256, 32, 256),
        # the larger encoder on a small batch and on long documents
        _encode("base_7x120", "base", 7, 120, 12, 120),
        _encode("base_64x512", "base", 64, 512, 64, 512),
        # prompts of a decoder layer with grouped-query heads, rotated in place first: the repository's causal workload
        _prefill("causal_gqa_16x4096", 16, 1024, 4096, 32, 8, 128, 0, False),
        # many shorter prompts, sliding window, rotation inside the attention (qkv stays as it is)
        _prefill("sliding_23x1500", 23, 100, 1500, 16, 16, 64, 512, True),
        # the larger encoder's feed-forward product on FP8 weights over a throughput batch, odd row count
        {"name": "scaled_fp8_32749", "op": "scaled", "rows": 32749, "n": 3072, "k": 768, "fmt": "fp8_e4m3",
         "epilogue": "gelu"},
        # the smaller encoder's feed-forward down product, both operands FP8, at its throughput batch
        {"name": "mx_36736", "op": "mx", "rows": 36736, "n": 384, "k": 1536, "fmt": "fp8_e4m3"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(("encode",) * 5 + ("prefill",) * 2 + ("scaled", "mx"))
    if op == "encode":
        model = rng.choice(("minilm", "minilm", "base"))
        seq = _log(rng, 16, 512)
        batch = _log(rng, 1, 256)
        batch = max(1, min(batch, (65536 if model == "minilm" else 18000) // seq))
        hi = seq if rng.random() < 0.7 else rng.randint(max(1, seq // 2), seq)
        lo = max(1, int(hi * rng.choice((0.0625, 0.125, 0.25, 0.5, 1.0))))
        c = _encode("", model, batch, seq, lo, hi, host=rng.random() < 0.3, holes=rng.random() < 0.2)
    elif op == "prefill":
        dim = rng.choice((32, 64, 64, 128))
        kv_heads = rng.choice((2, 4, 8))
        heads = kv_heads * rng.choice((1, 2, 4))
        hi = _log(rng, 64, 4096)
        lo = max(1, int(hi * rng.choice((0.1, 0.25, 1.0))))
        batch = max(1, min(_log(rng, 1, 64), 28000 // hi))
        window = 0 if rng.random() < 0.6 else _log(rng, 32, 1024)
        c = _prefill("", batch, lo, hi, heads, kv_heads, dim, window, rng.random() < 0.5)
    elif op == "scaled":
        width = rng.choice((384, 768, 1024))
        n, k = rng.choice(((3 * width, width), (width, width), (4 * width, width), (width, 4 * width)))
        fmt = rng.choice(sorted(FORMATS))
        c = {"op": op, "rows": _log(rng, 16, 32768), "n": n, "k": k, "fmt": fmt,
             "epilogue": rng.choice(sorted(EPILOGUES))}
    else:
        width = rng.choice((384, 768, 1024))
        n, k = rng.choice(((3 * width, width), (width, width), (4 * width, width), (width, 4 * width)))
        c = {"op": op, "rows": _log(rng, 64, 32768), "n": n, "k": k, "fmt": rng.choice(("fp8_e4m3", "fp8_e5m2"))}
    c.pop("name", None)
    return c


def _lengths(case):
    """The case's sequence lengths, before the seed puts them in order."""
    lo, hi, b = case["lo"], case["hi"], case["batch"]
    return [min(hi, lo + int((i + 0.5) / b * (hi - lo + 1))) for i in range(b)]


def _shuffled_lengths(case, seed):
    order = torch.randperm(case["batch"], generator=torch.Generator().manual_seed(seed)).tolist()
    lengths = _lengths(case)
    return [lengths[i] for i in order]


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _randn(g, *shape, scale=1.0, dtype=torch.bfloat16):
    return (torch.randn(*shape, device="cuda", generator=g) * scale).to(dtype)


def _prepare_encode(case, seed):
    layers, hidden, heads, ffn = MODELS[case["model"]]
    batch, seq = case["batch"], case["seq"]
    g = _generator(seed)
    f32 = torch.float32
    params = {
        "word_emb": _randn(g, VOCAB, hidden, scale=0.02), "pos_emb": _randn(g, MAX_POS, hidden, scale=0.02),
        "type_emb": _randn(g, 2, hidden, scale=0.02),
        "emb_ln_g": 1 + _randn(g, hidden, scale=0.1, dtype=f32), "emb_ln_b": _randn(g, hidden, scale=0.1, dtype=f32),
    }
    shapes = {"wqkv": (3 * hidden, hidden), "wo": (hidden, hidden), "w1": (ffn, hidden), "w2": (hidden, ffn)}
    biases = {"bqkv": 3 * hidden, "bo": hidden, "b1": ffn, "b2": hidden}
    stack = []
    for _ in range(layers):
        layer = {n: _randn(g, *s, scale=0.02) for n, s in shapes.items()}
        layer.update({n: _randn(g, s, scale=0.02, dtype=f32) for n, s in biases.items()})
        for n in ("ln1", "ln2"):
            layer[n + "_g"] = 1 + _randn(g, hidden, scale=0.1, dtype=f32)
            layer[n + "_b"] = _randn(g, hidden, scale=0.1, dtype=f32)
        stack.append(layer)
    ids = torch.randint(0, VOCAB, (batch, seq), generator=g, device="cuda", dtype=torch.int32)
    lengths = torch.tensor(_shuffled_lengths(case, seed), device="cuda")
    mask = torch.arange(seq, device="cuda")[None, :] < lengths[:, None]
    if case["holes"]:
        mask &= torch.rand(batch, seq, generator=g, device="cuda") >= 0.1
    mask = mask.to(torch.int32)
    out = torch.empty(batch, hidden, dtype=f32, device="cuda")
    enc = binding.Encoder(layers, hidden, heads, ffn, VOCAB, MAX_POS, max_batch=batch, max_seq=MAX_POS)
    state = {"encoder": enc, "weights": rlx.DeviceWeights(params, stack), "workspace": enc.alloc_workspace(batch, seq)}
    if case["host"]:
        ids, mask, out = (t.cpu().pin_memory() for t in (ids, mask, out))
    state.update(ids=ids, mask=mask, out=out)
    return state


def _prepare_prefill(case, seed):
    h, hkv, d = case["heads"], case["kv_heads"], case["dim"]
    lengths = torch.tensor(_shuffled_lengths(case, seed), dtype=torch.int32)
    start = torch.cumsum(lengths, 0, dtype=torch.int32) - lengths
    rows = int(lengths.sum())
    g = _generator(seed)
    return {"qkv": _randn(g, rows, (h + 2 * hkv) * d), "start": start.cuda(), "lengths": lengths.cuda(),
            "max_len": int(lengths.max()), "rope": rlx.rope_tables(case["hi"], d),
            "ctx": torch.zeros(rows, h * d, dtype=torch.bfloat16, device="cuda")}


def _prepare_scaled(case, seed):
    m, n, k = case["rows"], case["n"], case["k"]
    word, bits, largest, packed = FORMATS[case["fmt"]]
    g = _generator(seed)
    codes = torch.randint(0, largest + 1, (n, k), generator=g, device="cuda", dtype=torch.int32)
    codes |= torch.randint(0, 2, (n, k), generator=g, device="cuda", dtype=torch.int32) << (bits - 1)
    if packed:
        codes = codes[:, 0::2] | (codes[:, 1::2] << 4)
    return {"x": _randn(g, m, k), "codes": codes.to(torch.uint8).contiguous(),
            "scales": torch.randint(112, 120, (n, k // 32), generator=g, device="cuda", dtype=torch.int32).to(torch.uint8),
            "word": word, "bias": _randn(g, n, dtype=torch.float32),
            "residual": _randn(g, m, n) if case["epilogue"] == "residual" else None,
            "epilogue": EPILOGUES[case["epilogue"]],
            "scratch": torch.empty(n, k, dtype=torch.bfloat16, device="cuda"),
            "out": torch.empty(m, n, dtype=torch.bfloat16, device="cuda")}


def _prepare_mx(case, seed):
    m, n, k = case["rows"], case["n"], case["k"]
    word = FORMATS[case["fmt"]][0]
    g = _generator(seed)
    codes, scales = rlx.quantise_mx(_randn(g, n, k, scale=0.05), word)
    return {"x": _randn(g, m, k), "codes": codes, "scales": scales, "word": word, "bias": _randn(g, n, dtype=torch.float32),
            "out": torch.empty(m, n, dtype=torch.bfloat16, device="cuda")}


def prepare(case, seed):
    return {"case": case, **globals()["_prepare_" + case["op"]](case, seed)}


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "encode":
        forward = s["encoder"].forward_host if case["host"] else s["encoder"].forward
        return forward(s["ids"], s["mask"], s["weights"], s["out"], s["workspace"])
    if op == "prefill":
        rope, kind = s["rope"], binding.MASK_SLIDING_WINDOW if case["window"] else binding.MASK_CAUSAL
        if not case["in_attention"]:
            binding.qk_rope_bf16(s["qkv"], s["start"], s["lengths"], s["max_len"], case["heads"], rope,
                                 num_kv_heads=case["kv_heads"])
            rope = None
        ctx = rlx.attention_kind_bf16(s["qkv"], s["start"], s["lengths"], s["max_len"], case["heads"], kind,
                                      case["window"], rope, out=s["ctx"], num_kv_heads=case["kv_heads"])
        return {"ctx": ctx} if case["in_attention"] else {"ctx": ctx, "qkv": s["qkv"]}
    if op == "scaled":
        return rlx.scaled_matmul_bf16(s["x"], s["codes"], s["scales"], s["word"], s["bias"], s["residual"], s["epilogue"],
                                      w_scratch=s["scratch"], out=s["out"])
    codes, scales = rlx.quantise_mx(s["x"], s["word"])
    out = rlx.mx_matmul_bf16(codes, scales, s["word"], s["codes"], s["scales"], s["word"], bias=s["bias"], out=s["out"])
    return {"codes": codes, "scales": scales, "out": out}


def work(case):
    op = case["op"]
    if op == "encode":
        layers, hidden, _, ffn = MODELS[case["model"]]
        keep = 0.9 if case["holes"] else 1.0
        lengths = [keep * n for n in _lengths(case)]
        rows, pairs = sum(lengths), sum(n * n for n in lengths)
        weights = 2 * layers * (4 * hidden * hidden + 2 * hidden * ffn) + 4 * layers * (9 * hidden + ffn)
        tables = 2 * hidden * (min(rows, VOCAB) + min(case["seq"], MAX_POS) + 1)
        return {"bytes": weights + tables + 8 * case["batch"] * case["seq"] + 4 * case["batch"] * hidden,
                "flops": layers * (rows * (8 * hidden * hidden + 4 * hidden * ffn) + 4 * pairs * hidden)}
    if op == "prefill":
        h, hkv, d = case["heads"], case["kv_heads"], case["dim"]
        rows = sum(_lengths(case))
        pairs = 0
        for n in _lengths(case):
            w = min(case["window"] or n, n)
            pairs += w * (w + 1) // 2 + (n - w) * w
        moved = rows * (2 * h + 2 * hkv) * d
        if not case["in_attention"]:
            moved += rows * (h + hkv) * d          # the rotated q and k go back to memory: they are a result
        return {"bytes": 2 * moved, "flops": 4 * pairs * h * d}
    m, n, k = case["rows"], case["n"], case["k"]
    if op == "scaled":
        io = 2 * m * k + 2 * m * n * (2 if case["epilogue"] == "residual" else 1)
        return {"bytes": io + n * k * CODE_BITS[case["fmt"]] // 8 + n * k // 32 + 4 * n, "flops": 2 * m * n * k}
    return {"bytes": 2 * m * k + m * k + m * k // 32 + n * k + n * k // 32 + 4 * n + 2 * m * n, "flops": 2 * m * n * k}


def tolerance(case):
    # Four times the distance to the same pass in 64 bits, as measured: embeddings 1.3e-3 to 2.7e-3 (bf16 activations
    # through 6 or 12 layers), attention 2.9e-3 (bf16 probabilities and rotated keys), products 1.7e-3 (one rounding of
    # the result to bf16).  Codes and scale bytes of the quantiser are exact.
    return {"rel": {"encode": 1e-2, "prefill": 1.2e-2, "scaled": 7e-3, "mx": 7e-3}[case["op"]]}
