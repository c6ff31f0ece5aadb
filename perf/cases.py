"""What a program that serves video-LLM prompts with this library asks of it, as cases to measure.

A case is one of three kinds of work:

* ``answer``  one request batch: forget the last prompt, choose the protected tokens (p > 0), quantize the keys and
  values of every layer, then decode ``steps`` tokens (append, attention over the packed cache, flush of a full
  residual).  ``calls`` = "model": one library call per layer and tensor, the order in which a model reaches its
  layers; "all": one call for all layers, as a program does whose layers' tensors lie together.
* ``prompt``  the prefill alone: Eq. 7 scores from hidden states and the token selection (p > 0), then keys and
  values.  The outcome is the packed cache.
* ``shard``   one device's part of a decode step when a sequence is cut over ``parts`` devices: its own (maximum,
  sum, output) triples, then the merge of all devices' triples.

Shapes follow the workloads that this repository names (196 visual tokens a frame, 28 layers, 4 KV heads of 128
channels, 28 query heads; 8 to 1000 frames, batch 1 to 16), with ragged lengths in between.
"""
import math

import torch

import paper_2503_16257_b200 as P

D = 128
D_MODEL = 3584
OUTLIERS = 6            # planted key channels per head, as in the repository's workloads
_DEFAULTS = dict(kind="answer", layers=28, batch=1, h_kv=4, h_q=28, visual=0, p=0.0, dtype="fp16", out="fp32",
                 k_ratio=0.5, one_bit="fft", steps=0, calls="all", text=64, parts=1)


def _case(name, **kw):
    c = dict(_DEFAULTS, **kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call that the repository names: one layer, 8 frames; latency and launches count
        _case("tiny", layers=1, tokens=1632, visual=1568, steps=16),
        # 32 frames, one user, called by a model: 28 library calls per token
        _case("clip_by_layer", tokens=6400, visual=6272, steps=16, calls="model", out="fp16"),
        # the same clip with a fifth of its visual tokens protected, all layers in one call
        _case("clip_protected", tokens=6400, visual=6272, p=0.2, steps=64),
        # 64 frames in bfloat16, a ragged length, and an answer long enough to flush the residual once
        _case("video_bf16_flush", tokens=12819, visual=12544, dtype="bf16", out="bf16", steps=120),
        # 16 users with 64 frames each: the packed cache (1.6 GB) is far larger than L2
        _case("batch16", batch=16, tokens=12544, visual=12544, steps=32),
        # 16 users, protected tokens, called by a model layer by layer
        _case("batch16_protected_by_layer", batch=16, tokens=12544, visual=12544, p=0.2, steps=8, calls="model", out="fp16"),
        # 1000 frames on one device (a part of the layers): the longest sequence
        _case("frames1000_protected", layers=2, batch=4, tokens=196000, visual=196000, p=0.2, steps=16),
        # 1000 frames cut over eight devices: the work of one of them
        _case("frames1000_shard", kind="shard", batch=4, tokens=24500, visual=24500, steps=8, parts=8),
        # prefill of a few layers for 16 users, layer by layer
        _case("prompt_batch16", kind="prompt", layers=4, batch=16, tokens=12544, visual=12544, calls="model"),
        # prefill of one ragged clip with token scores and selection, layer by layer, bfloat16
        _case("prompt_clip_protected", kind="prompt", tokens=6307, visual=6174, p=0.2, dtype="bf16", text=128, calls="model"),
        # the paper's 1.75-bit keys (k = 0.75) with protected tokens, two users
        _case("keys175_protected", batch=2, tokens=6400, visual=6272, p=0.2, k_ratio=0.75, steps=16),
        # the paper's 1.25-bit keys (k = 0.25, plain one-bit code)
        _case("keys125_bf16", tokens=12800, visual=12544, dtype="bf16", out="bf16", k_ratio=0.25, one_bit="minmax", steps=16),
    ]


def draw(rng):
    log_int = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    while True:
        kind = rng.choice(["answer", "answer", "answer", "prompt", "shard"])
        layers, batch = rng.choice([1, 2, 4, 14, 28, 28]), rng.choice([1, 1, 2, 3, 4, 8, 16])
        tokens = log_int(256, 196000)
        h_kv, h_q = rng.choice([(4, 28), (4, 28), (4, 28), (8, 32), (2, 16)])
        k_ratio, one_bit = rng.choice([(0.5, "fft")] * 6 + [(0.25, "minmax"), (0.5, "minmax"), (0.75, "fft"), (0.75, "minmax"), (1.0, "fft")])
        p = rng.choice([0.0, 0.0, 0.1, 0.2, 0.3])
        visual = max(32, int(tokens * rng.uniform(0.8, 1.0))) // 32 * 32
        dtype = rng.choice(["fp16", "bf16"])
        case = _case(None, kind=kind, layers=layers, batch=batch, tokens=tokens, visual=min(visual, tokens // 32 * 32), p=p, h_kv=h_kv,
                     h_q=h_q, k_ratio=k_ratio, one_bit=one_bit, dtype=dtype, out=rng.choice(["fp32", dtype]), calls=rng.choice(["all", "model"]),
                     steps=0 if kind == "prompt" else log_int(4, 128), text=log_int(16, 256), parts=rng.choice([2, 4, 8]) if kind == "shard" else 1)
        slab_tokens = layers * batch * h_kv * tokens
        # no more than the largest listed case: its slabs' tokens, its bytes, and a few thousand calls
        if slab_tokens <= 28 * 16 * 4 * 12544 and work(case)["bytes"] <= 5e10 and case["steps"] * (layers if case["calls"] == "model" else 1) <= 1000:
            return case


# ---------------------------------------------------------------------------------------------------------------
# Bytes and operations
# ---------------------------------------------------------------------------------------------------------------
def _two_bit_channels(case):
    return int(round(case["k_ratio"] * D))


def _key_group_bytes(case):
    """32 tokens of keys: 2 bits per anomalous channel and 1 per normal one, a binary16 scale and zero point per
    2-bit channel, a scale (Eq. 5) or scale and zero point (plain code) per 1-bit channel."""
    n2 = _two_bit_channels(case)
    n1 = D - n2
    return (2 * n2 + n1) * 4 + 4 * n2 + (4 if case["one_bit"] == "minmax" else 2) * n1


def _packed_bytes(case, tokens_q, flushed):
    n_prot = int(case["p"] * case["visual"])
    ternary = (tokens_q - n_prot + 31) // 32 + 4 * flushed
    return (tokens_q // 32 + 4 * flushed) * _key_group_bytes(case) + ternary * (5376 / 5) + ((n_prot + 31) // 32) * 1536


def work(case):
    L, B, Hk, Hq, T, steps = (case[k] for k in ("layers", "batch", "h_kv", "h_q", "tokens", "steps"))
    slabs, tokens_q, res = L * B * Hk, T - T % 32, T % 32
    out_bytes = 4 if case["out"] == "fp32" else 2
    n_bytes = flops = 0.0
    if case["kind"] != "shard":
        n_bytes += slabs * (2 * T * D * 2 + _packed_bytes(case, tokens_q, 0) + 2 * res * D * 2)
        flops += slabs * tokens_q * 2 * D * 4
        if case["one_bit"] == "fft":
            n1 = D - _two_bit_channels(case)
            flops += slabs * tokens_q * 2.5 * n1 * (math.log2(n1) if n1 > 1 else 0)
    if case["kind"] == "prompt" and case["p"] > 0:
        n_bytes += B * (case["visual"] + case["text"]) * D_MODEL * 2 + B * case["visual"] * 8
        flops += 2.0 * B * (case["visual"] + case["text"]) * D_MODEL
    flushed = 0
    for _ in range(steps):
        io = L * B * Hq * D * (2 + out_bytes)
        if case["kind"] == "answer":
            res += 1
            io += slabs * 4 * D * 2                            # k_new and v_new read, and written to the residual
        n_bytes += slabs * (_packed_bytes(case, tokens_q, flushed) + 2 * res * D * 2) + io
        flops += 4.0 * L * B * Hq * D * (tokens_q + 128 * flushed + res)
        if case["kind"] == "shard":
            n_bytes += (case["parts"] + 1) * L * B * Hq * 130 * 4
        if res == 128:
            n_bytes += slabs * (2 * 128 * D * 2 + 4 * (_key_group_bytes(case) + 5376 / 5))
            flushed, res = flushed + 1, 0
    return {"bytes": n_bytes, "flops": flops}


def tolerance(case):
    # Outputs: the probabilities are rounded to binary16, and where the running maximum stands decides how.  The same
    # call cut into other runs of units differs by 1.7e-4 of the output (2-norm), at most 1.8e-3 of its rms; float64
    # over the dequantized cache by 1.7e-4.  Rounding the result to bfloat16 (2^-9) moves 6.9e-4 and one step, 7.8e-3.
    # Packed bytes: float32 sums in another order move 7e-5 of the spectrum scales (128 of 2227 bytes) by one step and
    # one sign bit in ten million.
    bf16 = case["out"] == "bf16"
    return {"rel": 2.8e-3 if bf16 else 7e-4, "max": 1.6e-2 if bf16 else 8e-3, "differ": 1e-5}


# ---------------------------------------------------------------------------------------------------------------
# State and pass
# ---------------------------------------------------------------------------------------------------------------
_TORCH = {"fp16": torch.float16, "bf16": torch.bfloat16, "fp32": torch.float32}
_VIDKV = {"fp16": P.VIDKV_F16, "bf16": P.VIDKV_BF16, "fp32": P.VIDKV_F32}


class _State:
    pass


def _key_affine(case, gen):
    """Per (KV head, channel) factor and offset: six channels of each head ten times as large and off centre."""
    scale, offset = torch.ones(case["h_kv"], D, device="cuda"), torch.zeros(case["h_kv"], D, device="cuda")
    ids = torch.rand(case["h_kv"], D, generator=gen, device="cuda").argsort(dim=1)[:, :OUTLIERS]
    return scale.scatter_(1, ids, 10.0), offset.scatter_(1, ids, 5.0)


def _keys(case, shape, affine, gen):
    x = torch.randn(shape, generator=gen, device="cuda")
    scale, offset = affine
    return x.mul_(scale[:, None, :]).add_(offset[:, None, :]).to(_TORCH[case["dtype"]])


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    L, B, Hk, Hq, T, steps = (case[k] for k in ("layers", "batch", "h_kv", "h_q", "tokens", "steps"))
    dtype = _TORCH[case["dtype"]]
    s = _State()
    s.case = case
    s.cache = P.VidKVCache(P.VidKVConfig(
        B=B, L=L, max_prefill_tokens=T, max_new_tokens=max(steps, 1), H_kv=Hk, H_q=Hq, p_ratio=case["p"], k_ratio=case["k_ratio"],
        key_1bit_mode=P.VIDKV_KEY1BIT_PLAIN_MINMAX if case["one_bit"] == "minmax" else P.VIDKV_KEY1BIT_FFT_SIGN,
        in_dtype=_VIDKV[case["dtype"]], out_dtype=_VIDKV[case["out"]]))
    affine = _key_affine(case, gen)
    s.K = torch.empty(L, B, Hk, T, D, dtype=dtype, device="cuda")
    s.V = torch.empty(L, B, Hk, T, D, dtype=dtype, device="cuda")
    for layer in range(L):
        for b in range(B):
            s.K[layer, b] = _keys(case, (Hk, T, D), affine, gen)
            s.V[layer, b] = torch.randn(Hk, T, D, generator=gen, device="cuda").to(dtype)
    s.saliency = s.x_v = s.x_t = None
    if case["p"] > 0:
        if case["kind"] == "prompt":
            s.x_v = torch.randn(B, case["visual"], D_MODEL, generator=gen, device="cuda", dtype=torch.float32).to(dtype)
            s.x_t = (torch.randn(B, case["text"], D_MODEL, generator=gen, device="cuda") + 0.5 * torch.randn(B, 1, D_MODEL, generator=gen, device="cuda")).to(dtype)
        else:
            s.saliency = torch.randn(B, case["visual"], generator=gen, device="cuda")
    if steps:
        s.q = torch.randn(steps, L, B, Hq, D, generator=gen, device="cuda").to(dtype)
        s.k_new = torch.stack([_keys(case, (L * B, Hk, 1, D), affine, gen).view(L, B, Hk, D) for _ in range(steps)])
        s.v_new = torch.randn(steps, L, B, Hk, D, generator=gen, device="cuda").to(dtype)
        s.out = torch.empty(steps, L, B, Hq, D, dtype=_TORCH[case["out"]], device="cuda")
        # what a model hands to the library in one step, layer by layer or all layers at once
        n = L if case["calls"] == "model" else 1
        s.args = [[(i * (L // n), L // n) + tuple(t[step].view(n, L // n, *t.shape[2:])[i] for t in (s.q, s.k_new, s.v_new, s.out))
                   for i in range(n)] for step in range(steps)]
    if case["kind"] == "shard":
        # the cache is filled once; the other devices' triples are what an all-gather would have brought
        _quantize(s)
        s.K = s.V = None
        s.partials = torch.randn(case["parts"], L, B, Hq, 130, generator=gen, device="cuda")
        s.partials[..., 1].abs_().mul_(T).add_(1.0)
        s.partials[..., 2:].mul_(T ** 0.5)
        s.own = s.partials[0]
        s.args = [[a[:3] + (s.own[a[0]:a[0] + a[1]],) for a in step] for step in s.args]
    return s


def _quantize(s):
    case, cache = s.case, s.cache
    cache.reset()
    if case["p"] > 0:
        saliency = s.saliency if s.saliency is not None else P.vidkv_saliency_scores(s.x_v, s.x_t)
        cache.select_tokens(saliency, 0, case["visual"], case["tokens"])
    if case["calls"] == "all":
        cache.quantize_keys_layers(0, s.K)
        cache.quantize_values_layers(0, s.V)
    else:
        for layer in range(case["layers"]):
            cache.quantize_keys(layer, s.K[layer])
            cache.quantize_values(layer, s.V[layer])


def run(s):
    case = s.case
    if case["kind"] == "shard":
        for step, calls in enumerate(s.args):
            for begin, n, q, own in calls:
                s.cache.decode_attention_partial(begin, n, q, None, None, own)
            P.vidkv_merge_partials(s.partials, s.out[step])
        return s.out, s.own
    _quantize(s)
    for calls in s.args if case["steps"] else ():
        for begin, n, q, k_new, v_new, out in calls:
            s.cache.decode_attention(begin, n, q, k_new, v_new, out)
    return (s.out, s.cache.cache) if case["steps"] else s.cache.cache
