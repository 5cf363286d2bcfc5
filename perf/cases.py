"""Cases by which the speed of the attention path is measured.

A case is one layer's worth of work as a training or inference program has it done, through the binding's
entry points: operand preparation, forward, row correction and gradient pass.  The shapes are those of
``workloads.WORKLOADS`` (the tiny problem, grouped queries at 4K and 8K tokens, head dims (192,128) and
(256,256), 64K tokens), of the sequence-shard driver, and generic ones between them; inputs follow the same
recipes as ``workloads`` (QK normalisation, outlier channels under rotary embedding, heavy-tailed channel
gains, plain normals), drawn on the GPU.

Fields of a case
  path      "step"     operands of Q, K, V, dO, forward, row correction, gradient pass
            "forward"  operands of Q, K, V in the orientations the forward reads, forward
            "shard"    the last `tokens` queries of a sequence of `keys` tokens against all its keys: own
                       tokens quantised, K / V assembled from the chunks (those of other ranks have arrived
                       quantised), forward, correction, gradient pass
  mode      "fp8", or "bf16" (the same kernels with BF16 operands)
  delta     "matched" or "stale" row correction
  producer  Q and K arrive ahead of rotary embedding, scale folding and key centering, which are fused
            into the quantiser
  tokens    queries (and keys, unless `keys` says otherwise); where it is no multiple of 128 the program
            pads every tensor to the next one, as the library asks for
"""
import math

import torch

from paper_2609_37852_b200 import binding as B
from paper_2609_37852_b200 import sequence_parallel as SP


def _case(name, path, batch, heads_q, heads_kv, tokens, d_qk, d_v, causal, recipe="plain", mode="fp8", delta="matched",
          producer=False, source="bf16", keys=0):
    case = dict(path=path, batch=batch, heads_q=heads_q, heads_kv=heads_kv, tokens=tokens, d_qk=d_qk, d_v=d_v, causal=causal,
                recipe=recipe, mode=mode, delta=delta, producer=producer, source=source, keys=keys)
    return dict(case, name=name) if name else case


def listed():
    return [
        # the smallest problem of the configuration list: FP32 tensors, one head, no mask; launches and host work
        _case("tiny_fp32", "step", 1, 1, 1, 256, 64, 64, False, "iid", source="fp32"),
        # a short training batch of small heads with the saved-output correction (the ablation without recomputation)
        _case("short_d64_stale", "step", 8, 12, 12, 1024, 64, 64, True, "qknorm", delta="stale"),
        # inference: prompts of about a thousand tokens that end anywhere
        _case("prefill_1k", "forward", 4, 16, 4, 1111, 128, 128, True, "outlier_rope"),
        # an encoder layer (no mask) on sequences whose length is no multiple of the tile
        _case("encoder_ragged", "step", 2, 16, 4, 1000, 128, 128, False, "qknorm"),
        # the training step of the 4K and 8K grouped-query configurations (the latter is the headline)
        _case("gqa4k", "step", 2, 16, 4, 4096, 128, 128, True, "qknorm"),
        _case("gqa8k", "step", 1, 32, 8, 8192, 128, 128, True, "outlier_rope"),
        # wide heads: the latent-attention shape and head dim 256
        _case("mla8k", "step", 1, 16, 16, 8192, 192, 128, True, "plain"),
        _case("gqa8k_d256", "step", 1, 8, 2, 8192, 256, 256, True, "plain"),
        # the BF16 reference mode of the 4K configuration
        _case("gqa4k_bf16", "step", 2, 16, 4, 4096, 128, 128, True, "qknorm", mode="bf16"),
        # a layer that leaves rotary embedding, scale folding and key centering to the quantiser
        _case("producer_4k", "step", 1, 16, 4, 4096, 128, 128, True, "plain", producer=True),
        # the last of four ranks of a 32K-token sequence
        _case("shard_32k", "shard", 1, 8, 2, 8192, 128, 128, True, "outlier_rope", keys=32768),
        # long context
        _case("long64k", "step", 1, 32, 8, 65536, 128, 128, True, "student_t"),
    ]


_HEADS = ((1, 1), (2, 2), (4, 1), (8, 2), (8, 8), (12, 12), (16, 4), (16, 16), (32, 8))
_DIMS = ((64, 64), (128, 128), (128, 128), (128, 128), (192, 128), (256, 256))
_MOST = 2.0e13          # executed multiply-adds of a drawn case: well below those of the 64K step


def _log_uniform(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    while True:
        path = rng.choices(("step", "forward", "shard"), (8, 3, 2))[0]
        heads_q, heads_kv = rng.choice(_HEADS)
        d_qk, d_v = rng.choice(_DIMS)
        batch = rng.choice((1, 1, 2, 3, 4, 8))
        tokens = _log_uniform(rng, 128, 24576)
        if path == "shard" or rng.random() < 0.4:
            tokens = -(-tokens // 128) * 128
        mode = "bf16" if path != "shard" and rng.random() < 0.2 else "fp8"
        producer = path == "step" and mode == "fp8" and rng.random() < 0.2
        if producer:                                   # the key mean is over the tokens handed over: whole tiles
            tokens = -(-tokens // 128) * 128
        delta = "stale" if path == "step" and rng.random() < 0.15 else "matched"
        causal = path == "shard" or rng.random() < 0.75
        recipe = "plain" if producer else rng.choice(("iid", "qknorm", "outlier_rope", "plain", "student_t"))
        source = "fp32" if path != "shard" and mode == "fp8" and not producer and delta == "matched" and rng.random() < 0.15 else "bf16"
        keys = tokens * rng.choice((2, 3, 4, 8)) if path == "shard" else 0
        case = _case(None, path, batch, heads_q, heads_kv, tokens, d_qk, d_v, causal, recipe, mode, delta, producer, source, keys)
        elements = batch * heads_q * (keys or tokens) * (d_qk + d_v)
        if work(case)["flops"] / 2 <= _MOST and elements <= 5e8:
            return case


# ----------------------------------------------------------------------------------------------- inputs

def _rope_tables(n, d, device):
    inv_freq = 10000.0 ** (-torch.arange(d // 2, dtype=torch.float32, device=device) / (d // 2))
    angle = torch.arange(n, dtype=torch.float32, device=device)[:, None] * inv_freq[None, :]
    return angle.cos().contiguous(), angle.sin().contiguous()


def _condition(x, recipe, g):
    """The input conditioning of `workloads` for Q and K."""
    heads, n, d = x.shape[1], x.shape[2], x.shape[3]
    if recipe == "qknorm":
        return x / torch.sqrt(x.pow(2).mean(dim=-1, keepdim=True) + 1e-6)
    if recipe == "outlier_rope":
        first4 = torch.rand((heads, d), generator=g, device=x.device).argsort(dim=-1)[:, :4]
        gain = torch.ones((heads, d), device=x.device).scatter_(1, first4, 20.0)
        x = x * gain[None, :, None, :]
        cos, sin = _rope_tables(n, d, x.device)
        a, b = x[..., :d // 2], x[..., d // 2:]
        return torch.cat([a * cos - b * sin, b * cos + a * sin], dim=-1)
    if recipe == "student_t":
        z = torch.randn((heads, d), generator=g, device=x.device)
        chi2 = torch.randn((heads, d, 3), generator=g, device=x.device).pow(2).sum(-1)
        return x * (z / torch.sqrt(chi2 / 3.0)).abs()[None, :, None, :]
    return x


def _inputs(case, seed, n_q, n_k):
    """Q, K, V, dO [B, H, n, d] on the GPU."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    b, dt = case["batch"], torch.bfloat16 if case["source"] == "bf16" else torch.float32
    out = []
    for i, (h, n, d) in enumerate(((case["heads_q"], n_q, case["d_qk"]), (case["heads_kv"], n_k, case["d_qk"]),
                                   (case["heads_kv"], n_k, case["d_v"]), (case["heads_q"], n_q, case["d_v"]))):
        x = torch.randn((b, h, n, d), generator=g, device="cuda")
        if i < 2:
            x = _condition(x, case["recipe"], g)
        if i == 1 and case["producer"]:
            x = x + 0.75                               # keys with a common mode, which centering takes out
        if i == 3:
            x = x * (1e-3 if case["recipe"] == "student_t" else 1.0 if case["recipe"] == "iid" else 1e-2)
        out.append(x.to(dt).contiguous())
    return out


def prepare(case, seed):
    path, bf16, tokens = case["path"], case["mode"] == "bf16", case["tokens"]
    b, hq, hkv, dqk, dv = case["batch"], case["heads_q"], case["heads_kv"], case["d_qk"], case["d_v"]
    padded = -(-tokens // 128) * 128
    keys = case["keys"] if path == "shard" else padded
    scale = 1.0 / math.sqrt(dqk)
    params = B.AttnParams(b, padded, hq, hkv, dqk, dv, case["causal"], 1.0 if case["producer"] else scale,
                          precision=B.ATTN_PREC_BF16 if bf16 else B.ATTN_PREC_MXFP8,
                          delta_mode=B.ATTN_DELTA_STALE if case["delta"] == "stale" else B.ATTN_DELTA_MATCHED,
                          seqlen_k=keys if path == "shard" else 0, q_start=keys - tokens if path == "shard" else 0,
                          keys_valid=tokens if tokens < padded else 0)
    s = dict(case=case, params=params, scale=scale, ws=B.new_workspace(B.ATTN_STATUS_WORKSPACE_BYTES, "cuda"))
    if path == "shard":
        # the whole sequence's tensors, cut into chunks; the chunks of the other ranks have been exchanged
        q, k, v, dO = _inputs(case, seed, tokens, keys)
        cut = lambda x, c: x[:, :, c * tokens:(c + 1) * tokens].contiguous()
        n = keys // tokens
        s["chunks"] = [[B.attn_fp8_quantize(cut(x, c)) for x in (k, v)] for c in range(n - 1)]
        s["src"] = [q, cut(k, n - 1), cut(v, n - 1), dO]
    else:
        s["src"] = _inputs(case, seed, tokens, tokens)
        if path == "forward":
            s["src"] = s["src"][:3]
    if case["producer"]:
        s["rope"] = _rope_tables(tokens, dqk, "cuda")
    # the operand buffers of the layer, kept from step to step (the fused producer makes its own)
    dims = ((hq, dqk), (hkv, dqk), (hkv, dv), (hq, dv))[:len(s["src"])]
    want = ((True, False), (True, False), (False, True)) if path == "forward" else ((True, True),) * 4
    s["operands"] = [_operand(bf16, case["source"], (b, h, padded, d), *w) for (h, d), w in zip(dims, want)]
    if case["producer"]:
        s["operands"] = s["operands"][2:]
    half = dict(dtype=torch.bfloat16, device="cuda")
    s["o"] = torch.empty((b, hq, padded, dv), **half)
    s["lse"] = torch.empty((b, hq, padded), dtype=torch.float32, device="cuda")
    if path != "forward":
        s["delta"] = torch.empty_like(s["lse"])
        s["grads"] = [torch.empty((b, hq, padded, dqk), **half), torch.empty((b, hkv, keys, dqk), **half),
                      torch.empty((b, hkv, keys, dv), **half)]
    return s


def _operand(bf16, source, shape, row, col):
    b, h, n, d = shape
    out = B.QTensor(shape=shape)
    if bf16:
        if row and source != "bf16":                   # a BF16 source is its own row operand
            out.row_codes = torch.empty((b, h, n, d), dtype=torch.bfloat16, device="cuda")
        if col:
            out.col_codes = torch.empty((b, h, d, n), dtype=torch.bfloat16, device="cuda")
        return out
    u8 = dict(dtype=torch.uint8, device="cuda")
    if row:
        out.row_codes, out.row_scales = torch.empty((b, h, n, d), **u8), torch.empty(B.attn_fp8_scale_bytes(b, h, n, d), **u8)
    if col:
        out.col_codes, out.col_scales = torch.empty((b, h, d, n), **u8), torch.empty(B.attn_fp8_scale_bytes(b, h, d, n), **u8)
    return out


# -------------------------------------------------------------------------------------------------- run

def run(s):
    case, params, ws, src, ops = s["case"], s["params"], s["ws"], s["src"], s["operands"]
    n = case["tokens"]
    if n % 128:
        src = [B.pad_tokens(x) for x in src]
    dO_bf16 = src[3] if case["delta"] == "stale" else None
    # operands
    if case["mode"] == "bf16":
        ops = [B.attn_fp8_prepare_bf16(x, want_row=case["path"] != "forward" or i < 2, out=t)
               for i, (x, t) in enumerate(zip(src, ops))]
    elif case["producer"]:
        cos, sin = s["rope"]
        q, _ = B.attn_fp8_quantize_fused(src[0], cos, sin, scale=s["scale"])
        k, _ = B.attn_fp8_quantize_fused(src[1], cos, sin, center=True)
        (v, dO), _ = B.attn_fp8_quantize_batch(src[2:], outs=ops, workspace=ws)
        ops = [q, k, v, dO]
    else:
        ops, _ = B.attn_fp8_quantize_batch(src, outs=ops, workspace=ws)
    q, k, v = ops[:3]
    if case["path"] == "shard":
        gather = lambda i, own, row: SP.concat_chunks([SP.only(c[i], row, not row) for c in s["chunks"]] + [SP.only(own, row, not row)])
        k_row, v_col = gather(0, k, True), gather(1, v, False)
        B.attn_fp8_fwd(params, q, k_row, v_col, o=s["o"], lse=s["lse"], workspace=ws)
        k, v = SP.merged(k_row, gather(0, k, False)), SP.merged(gather(1, v, True), v_col)
    else:
        B.attn_fp8_fwd(params, q, k, v, o=s["o"], lse=s["lse"], workspace=ws)
    # the rows of padded tokens are the caller's to ignore: a program goes on with the real ones
    real = lambda x: x[:, :, :n] if n % 128 else x
    if case["path"] == "forward":
        return {"o": real(s["o"]), "lse": real(s["lse"])}
    B.attn_fp8_bwd_delta(params, q, k, v, ops[3], s["lse"], dO_bf16=dO_bf16, o_bf16=s["o"], delta=s["delta"], workspace=ws)
    dq, dk, dv = s["grads"]
    B.attn_fp8_bwd(params, q, k, v, ops[3], s["lse"], s["delta"], dq=dq, dk=dk, dv=dv, workspace=ws)
    return {"o": real(s["o"]), "lse": real(s["lse"]), "delta": real(s["delta"]), "dq": real(dq), "dk": real(dk), "dv": real(dv)}


# ----------------------------------------------------------------------------------------- work, tolerance

def work(case):
    """Inputs read once, outputs written once; two products forward, and backward the two that the matched
    correction has to have finished over all keys before the first score gradient, then five (S, dP, dV, dK, dQ)."""
    b, hq, hkv, n, dqk, dv = (case[f] for f in ("batch", "heads_q", "heads_kv", "tokens", "d_qk", "d_v"))
    keys = case["keys"] or n
    pairs = b * hq * (n * keys - (n * (n - 1) // 2 if case["causal"] else 0))
    size = 2 if case["source"] == "bf16" else 4
    # own tokens (and, for a shard, the codes and scale bytes of the keys that came from elsewhere, both copies)
    reads = b * n * size * (hq * dqk + hkv * (dqk + dv)) + b * (keys - n) * hkv * (dqk + dv) * 2 * 33 // 32
    writes = b * hq * n * (2 * dv + 4)
    flops = 2 * pairs * (dqk + dv)
    if case["path"] != "forward":
        reads += b * n * size * hq * dv
        writes += b * hq * n * (2 * dqk + 4) + b * hkv * keys * 2 * (dqk + dv)
        flops += 2 * pairs * ((dqk + dv if case["delta"] == "matched" else 0) + 3 * dqk + 2 * dv)
    return {"bytes": reads + writes, "flops": flops}


def tolerance(case):
    """Probabilities and score gradients are quantised inside the kernels, so two correct implementations round
    single elements to neighbouring E4M3 (or BF16) values wherever their FP32 values differ in the last bits.
    Measured against the float64 oracle on 20 small cases of all recipes and modes: 2-norm at most 3.8e-4 of the
    outputs on diffuse scores and 2.8e-3 where outlier channels or heavy-tailed gains leave rows nearly one-hot
    (one element then carries its row), single values off by up to 0.06 and 0.7 of the larger of themselves and
    the root mean square.  Four times that, and 0.95 at most, for single values."""
    if case["recipe"] in ("outlier_rope", "student_t"):
        return {"rel": 1.1e-2, "max": 0.95}
    return {"rel": 1.6e-3, "max": 0.3}
