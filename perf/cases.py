"""What a user of the Set Block Decoding step has it do, as cases to time.

A case is one pass through the public entry points of
``paper_2509_04185_gb300``: a whole block step (block attention, LM head with
entropy and sampling, unmasking), one layer's attention, one LM-head call, or
the four linear layers of a transformer layer.  Step loops and linear layers
use the calls bound to fixed tensors (``prepare_*``), as a decode loop does;
single calls go through the plain functions with their outputs and workspaces
kept by the caller.
"""
import math

import torch

import paper_2509_04185_gb300 as sbd

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


# ------------------------------------------------------------------ cases

def _step(name=None, dtype="bf16", batch=1, k=16, q_heads=32, kv_heads=8, head_dim=128, len_lo=4096,
          len_hi=4096, hidden=4096, vocab=128256, dec_lo=1, dec_hi=1, noise="buffer", rule="eb", threshold=0.1):
    return dict(kind="step", name=name, dtype=dtype, batch=batch, k=k, q_heads=q_heads, kv_heads=kv_heads,
                head_dim=head_dim, len_lo=len_lo, len_hi=len_hi, hidden=hidden, vocab=vocab, dec_lo=dec_lo,
                dec_hi=dec_hi, noise=noise, rule=rule, threshold=threshold)


def _attn(name=None, dtype="bf16", batch=1, k=16, q_heads=32, kv_heads=8, head_dim=128, len_lo=4096,
          len_hi=4096, n_causal=0):
    return dict(kind="attn", name=name, dtype=dtype, batch=batch, k=k, q_heads=q_heads, kv_heads=kv_heads,
                head_dim=head_dim, len_lo=len_lo, len_hi=len_hi, n_causal=n_causal)


def _head(name=None, dtype="bf16", batch=1, k=16, hidden=4096, vocab=128256, dec_lo=0, dec_hi=0,
          noise="buffer", confidence=False):
    return dict(kind="head", name=name, dtype=dtype, batch=batch, k=k, hidden=hidden, vocab=vocab, dec_lo=dec_lo,
                dec_hi=dec_hi, noise=noise, confidence=confidence)


def _linear(name=None, rows=16, hidden=4096, q_heads=32, kv_heads=8, head_dim=128, ffn=14336):
    return dict(kind="linear", name=name, rows=rows, hidden=hidden, q_heads=q_heads, kv_heads=kv_heads,
                head_dim=head_dim, ffn=ffn)


def listed():
    return [
        # The smallest whole step: fp32, a few kilobytes, nothing but launches and latency.
        _step("step_tiny_f32", dtype="f32", k=4, q_heads=4, kv_heads=2, head_dim=64, len_lo=128, len_hi=128,
              hidden=256, vocab=512),
        # Plain next-token decoding (a block of one, greedy) of a small model with 64-wide heads.
        _step("step_small_ntp", batch=8, k=1, q_heads=32, kv_heads=8, head_dim=64, len_lo=200, len_hi=1999,
              hidden=2048, vocab=32003, dec_lo=0, dec_hi=0, noise="greedy"),
        # One user at Llama-3.1-8B shapes, the ordinary block of 16.
        _step("step_llama8b_b1_k16"),
        # A serving batch of uneven lengths, blocks half decoded.
        _step("step_ragged_b32_k8", batch=32, k=8, len_lo=512, len_hi=2048, dec_lo=1, dec_hi=7),
        # Long contexts, few users: one layer's attention over 32768 cached tokens.
        _attn("attn_long_b4_k16", batch=4, len_lo=32768, len_hi=32768),
        # The widest row tile (32 positions of 4 query heads a KV head) over a full batch.
        _attn("attn_wide_b16_k32", batch=16, k=32, len_lo=8192, len_hi=8192),
        # The first iteration of a block: 16 tokens of the last block enter the cache, uneven lengths.
        _attn("attn_first_b8_k32", batch=8, k=32, len_lo=500, len_hi=4001, n_causal=16),
        # Single-precision attention at full head counts, as a reference run of a model has it.
        _attn("attn_f32_b2_k8", dtype="f32", batch=2, k=8, len_lo=511, len_hi=2048),
        # The single-precision LM head of a small model with an odd vocabulary, probabilities asked for.
        _head("head_f32_small", dtype="f32", batch=2, k=16, hidden=2048, vocab=32003, dec_lo=1, dec_hi=7,
              confidence=True),
        # The start of 16 blocks of 32: every row masked, noise made in the kernel; the largest contraction.
        _head("head_philox_r512", batch=16, k=32, vocab=151936, noise="philox"),
        # The linear layers around the block step, one user (16 rows) and a full batch (512 rows).
        _linear("linear_8b_r16", rows=16),
        _linear("linear_8b_r512", rows=512),
    ]


def _spread(rng, lo, hi):
    """A whole number of [lo, hi], even over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _heads(rng):
    return rng.choice([(32, 8, 128), (32, 8, 64), (32, 4, 128), (16, 8, 128), (8, 8, 64), (12, 4, 128), (40, 8, 128)])


def _block(rng, group):
    return _spread(rng, 1, min(32, 128 // group))


def draw(rng):
    return {key: v for key, v in _draw(rng).items() if key != "name"}


def _draw(rng):
    kind = rng.choice(["step", "step", "attn", "attn", "first", "head", "head", "linear", "linear",
                       "step_f32", "attn_f32", "head_f32"])
    hq, hkv, d = _heads(rng)
    k = _block(rng, hq // hkv)
    noise = rng.choice(["buffer", "philox", "greedy"])
    if kind == "step":
        batch = _spread(rng, 1, min(64, 512 // k))
        hi = _spread(rng, 128, min(4096, 65536 // batch))
        lo = rng.randint(hi // 4, hi)
        dl = rng.randint(0, k - 1)
        return _step(batch=batch, k=k, q_heads=hq, kv_heads=hkv, head_dim=d, len_lo=lo, len_hi=hi,
                     hidden=64 * _spread(rng, 8, 64), vocab=_spread(rng, 8000, 128256), dec_lo=dl,
                     dec_hi=rng.randint(dl, k - 1), noise=noise, rule=rng.choice(["eb", "confidence", "factor"]),
                     threshold=rng.choice([0.01, 0.1, 0.35, 1.0]))
    if kind in ("attn", "first"):
        batch = _spread(rng, 1, 64)
        hi = _spread(rng, 64, min(32768, 131072 // batch))
        lo = rng.randint(hi // 4, hi)
        return _attn(batch=batch, k=k, q_heads=hq, kv_heads=hkv, head_dim=d, len_lo=lo, len_hi=hi,
                     n_causal=(k + 1) // 2 if kind == "first" else 0)
    if kind == "head":
        batch = _spread(rng, 1, 512 // k)
        dl = rng.randint(0, k - 1)
        return _head(batch=batch, k=k, hidden=64 * _spread(rng, 8, 64), vocab=_spread(rng, 8000, 151936), dec_lo=dl,
                     dec_hi=rng.randint(dl, k - 1), noise=noise, confidence=noise != "philox" and rng.random() < 0.5)
    if kind == "linear":
        hq, hkv, d = rng.choice([(32, 8, 128), (16, 8, 128), (12, 4, 128), (32, 8, 64)])
        return _linear(rows=_spread(rng, 1, 512), hidden=hq * d, q_heads=hq, kv_heads=hkv, head_dim=d,
                       ffn=64 * _spread(rng, 40, 224))
    # single precision: small models and short contexts
    batch = _spread(rng, 1, 4)
    hi = _spread(rng, 64, max(64, min(2048, 2 * 8 * 32 * 2048 // (batch * k * hq))))
    dl = rng.randint(0, k - 1)
    if kind == "attn_f32":
        return _attn(dtype="f32", batch=batch, k=k, q_heads=hq, kv_heads=hkv, head_dim=d,
                     len_lo=rng.randint(hi // 4, hi), len_hi=hi, n_causal=rng.choice([0, k // 2]))
    batch = min(batch, max(1, 32 // k))
    hidden, vocab = 4 * _spread(rng, 64, 512), _spread(rng, 500, 32003)
    if kind == "head_f32":
        return _head(dtype="f32", batch=batch, k=k, hidden=hidden, vocab=vocab, dec_lo=dl,
                     dec_hi=rng.randint(dl, k - 1), noise=noise, confidence=noise != "philox")
    return _step(dtype="f32", batch=batch, k=k, q_heads=hq, kv_heads=hkv, head_dim=d,
                 len_lo=rng.randint(hi // 4, hi), len_hi=hi, hidden=hidden, vocab=vocab, dec_lo=dl,
                 dec_hi=rng.randint(dl, k - 1), noise=noise, rule="eb", threshold=0.1)


# ------------------------------------------------------------------ inputs

class _Draws:
    """Tensors on the GPU, one stream of draws from one seed."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)

    def normal(self, *shape, dtype=torch.float32, std=1.0):
        if dtype == torch.float32:
            return torch.randn(shape, generator=self.g, device="cuda").mul_(std)
        out = torch.empty(shape, dtype=dtype, device="cuda")
        flat, step = out.view(-1), 1 << 26
        for at in range(0, flat.numel(), step):
            part = flat[at:at + step]
            part.copy_(torch.randn(part.numel(), generator=self.g, device="cuda").mul_(std))
        return out

    def uniform(self, *shape):
        return torch.rand(shape, generator=self.g, device="cuda")

    def whole(self, lo, hi, *shape):
        return torch.randint(lo, hi + 1, shape, generator=self.g, device="cuda", dtype=torch.int32)


def _attn_inputs(c, d):
    t, b, k = DTYPES[c["dtype"]], c["batch"], c["k"]
    hq, hkv, dim = c["q_heads"], c["kv_heads"], c["head_dim"]
    rows = c["len_hi"] + c.get("n_causal", 0)        # the cache's capacity
    s = {"lens": d.whole(c["len_lo"], c["len_hi"], b), "q": d.normal(b, k, hq, dim, dtype=t),
         "k_cache": d.normal(b, rows, hkv, dim, dtype=t), "v_cache": d.normal(b, rows, hkv, dim, dtype=t),
         "k_blk": d.normal(b, k, hkv, dim, dtype=t), "v_blk": d.normal(b, k, hkv, dim, dtype=t)}
    s["out"] = torch.empty_like(s["q"])
    return s


def _head_inputs(c, d):
    t, b, k, h, v = DTYPES[c["dtype"]], c["batch"], c["k"], c["hidden"], c["vocab"]
    # hidden rows of very different norms, so that some positions are certain and some are not
    scale = torch.exp(d.uniform(b, k, 1) * math.log(100.0) + math.log(0.1))
    n_dec = d.whole(c["dec_lo"], c["dec_hi"], b)
    rank = d.uniform(b, k).argsort(1).argsort(1)
    masked = (rank >= n_dec.view(b, 1)).to(torch.uint8)
    s = {"hidden": (d.normal(b, k, h) * scale).to(t), "w": d.normal(v, h, dtype=t, std=0.02),
         "masked": masked, "gumbel": None, "tau": 0.0 if c["noise"] == "greedy" else 1.0,
         "entropy": torch.empty(b, k, device="cuda"), "token": torch.empty(b, k, dtype=torch.int32, device="cuda"),
         "tokens": torch.where(masked.bool(), -1, d.whole(0, v - 1, b, k))}
    if c["noise"] == "buffer":
        s["gumbel"] = d.uniform(b, k, v).clamp_(1e-30, 1 - 2.0 ** -24).log_().neg_().log_().neg_()
    return s


def _workspace(size):
    return torch.empty(size, dtype=torch.uint8, device="cuda") if size else None


def _attn_workspace(s):
    import ctypes
    return _workspace(sbd.lib.sbd_block_attention_workspace_size(ctypes.byref(sbd.attn_desc(s["q"], s["k_cache"]))))


def _head_workspace(s):
    import ctypes
    return _workspace(sbd.lib.sbd_head_entropy_sample_workspace_size(ctypes.byref(sbd.head_desc(s["hidden"], s["w"]))))


def prepare(case, seed):
    d = _Draws(seed)
    s = {"case": case}
    if case["kind"] in ("step", "attn"):
        s.update(_attn_inputs(case, d))
        s["attn_ws"] = _attn_workspace(s)
    if case["kind"] in ("step", "head"):
        s.update(_head_inputs(case, d))
        s["head_ws"] = _head_workspace(s)
    if case["kind"] == "step":
        # tokens and masks of the blocks in one buffer, so that starting them again is one copy
        b, k = case["batch"], case["k"]
        at = (4 * b * k + 15) // 16 * 16
        s["block"] = torch.zeros(at + b * k, dtype=torch.uint8, device="cuda")
        bt, masked = s["block"][:4 * b * k].view(torch.int32).view(b, k), s["block"][at:].view(b, k)
        bt.copy_(s["tokens"])
        masked.copy_(s["masked"])
        s["start"], s["tokens"], s["masked"] = s["block"].clone(), bt, masked
        s["n"] = torch.empty(b, dtype=torch.int32, device="cuda")
        s["confidence"] = torch.empty(b, k, device="cuda")
        s["attend"] = sbd.prepare_block_attention(s["q"], s["k_cache"], s["v_cache"], s["lens"], s["k_blk"],
                                                  s["v_blk"], s["out"], s["attn_ws"])
        if case["rule"] == "eb":
            if case["noise"] == "philox":
                s["sample"] = sbd.prepare_head_entropy_sample_philox(
                    s["hidden"], s["w"], masked, seed, 7, s["tau"], s["entropy"], s["token"], s["head_ws"])
            else:
                s["sample"] = sbd.prepare_head_entropy_sample(
                    s["hidden"], s["w"], masked, s["gumbel"], s["tau"], s["entropy"], s["token"], s["head_ws"])
            s["select"] = sbd.prepare_eb_select(s["entropy"], s["token"], case["threshold"], masked, bt, s["n"])
    elif case["kind"] == "head":
        s["confidence"] = torch.empty_like(s["entropy"])
    elif case["kind"] == "linear":
        s["layers"], s["calls"] = [], []
        for rows, n_in, n_out in _layer_shapes(case):
            x = d.normal(rows, n_in, dtype=torch.bfloat16)
            w = d.normal(n_out, n_in, dtype=torch.bfloat16, std=0.02)
            y = torch.empty(rows, n_out, dtype=torch.bfloat16, device="cuda")
            s["layers"].append((x, w, y))
            s["calls"].append(sbd.prepare_linear(x, w, y))
    s["seed"] = seed
    return s


def _layer_shapes(c):
    """(rows, inputs, outputs) of a layer's query-key-value, output, gate-and-up and down projections."""
    r, h, q = c["rows"], c["hidden"], c["q_heads"] * c["head_dim"]
    return [(r, h, q + 2 * c["kv_heads"] * c["head_dim"]), (r, q, h), (r, h, 2 * c["ffn"]), (r, c["ffn"], h)]


# ------------------------------------------------------------------ one pass

_RULES = {"confidence": sbd.SBD_SELECT_EB_CONFIDENCE, "factor": sbd.SBD_SELECT_FACTOR}


def _run_head(c, s):
    if c["noise"] == "philox":
        return sbd.sbd_head_entropy_sample_philox(s["hidden"], s["w"], s["masked"], s["seed"], 7, s["tau"],
                                                  s["entropy"], s["token"], workspace=s["head_ws"])
    if c.get("confidence") or c.get("rule") in _RULES:
        return sbd.sbd_head_entropy_confidence_sample(s["hidden"], s["w"], s["masked"], s["gumbel"], s["tau"],
                                                      s["entropy"], s["confidence"], s["token"],
                                                      workspace=s["head_ws"])
    return sbd.sbd_head_entropy_sample(s["hidden"], s["w"], s["masked"], s["gumbel"], s["tau"], s["entropy"],
                                       s["token"], workspace=s["head_ws"])


def run(s):
    c = s["case"]
    if c["kind"] == "attn":
        if c["n_causal"]:
            sbd.sbd_block_attention_causal_prefix(s["q"], s["k_cache"], s["v_cache"], s["lens"], s["k_blk"],
                                                  s["v_blk"], c["n_causal"], s["out"], workspace=s["attn_ws"])
            return s["out"], s["k_cache"], s["v_cache"]
        return (sbd.sbd_block_attention(s["q"], s["k_cache"], s["v_cache"], s["lens"], s["k_blk"], s["v_blk"],
                                        s["out"], workspace=s["attn_ws"]),)
    if c["kind"] == "head":
        return _run_head(c, s)
    if c["kind"] == "linear":
        for call in s["calls"]:
            call()
        return tuple(y for _, _, y in s["layers"])
    s["block"].copy_(s["start"])
    s["attend"]()
    if c["rule"] == "eb":
        s["sample"]()
        s["select"]()
    else:
        if c["noise"] == "philox":       # the counter-based call has no confidences: the noise is written out first
            ids = torch.arange(c["batch"] * c["k"], dtype=torch.int32, device="cuda")
            s["gumbel"] = sbd.sbd_gumbel_philox(ids, c["vocab"], s["seed"], 7)
            s["gumbel"] = s["gumbel"].view(c["batch"], c["k"], c["vocab"])
        sbd.sbd_head_entropy_confidence_sample(s["hidden"], s["w"], s["masked"], s["gumbel"], s["tau"],
                                               s["entropy"], s["confidence"], s["token"], workspace=s["head_ws"])
        sbd.sbd_select(_RULES[c["rule"]], s["entropy"], s["confidence"], s["token"], c["threshold"], s["masked"],
                       s["tokens"], s["n"])
    return s["out"], s["entropy"], s["token"], s["masked"], s["tokens"], s["n"]


# ------------------------------------------------------------------ what a pass cannot do without

def _size(c):
    return 4 if c.get("dtype") == "f32" else 2


def _attn_work(c):
    b, k, hq, hkv, dim, e = c["batch"], c["k"], c["q_heads"], c["kv_heads"], c["head_dim"], _size(c)
    keys = (c["len_lo"] + c["len_hi"]) / 2
    moved = 2 * b * hkv * dim * e * (keys + k + c.get("n_causal", 0)) + 2 * b * k * hq * dim * e
    return moved, 4 * b * k * hq * dim * (keys + k)


def _head_work(c):
    b, k, h, v, e = c["batch"], c["k"], c["hidden"], c["vocab"], _size(c)
    rows = b * (k - (c["dec_lo"] + c["dec_hi"]) / 2)
    return v * h * e + rows * h * e + (4 * rows * v if c["noise"] == "buffer" else 0) + 9 * b * k, 2 * rows * v * h


def work(c):
    if c["kind"] == "linear":
        shapes = _layer_shapes(c)
        return {"bytes": sum(2 * (r * i + i * o + r * o) for r, i, o in shapes),
                "flops": sum(2 * r * i * o for r, i, o in shapes)}
    total = [0, 0]
    for part in ([_attn_work] if c["kind"] in ("step", "attn") else []) + \
            ([_head_work] if c["kind"] in ("step", "head") else []):
        total = [x + y for x, y in zip(total, part(c))]
    return {"bytes": total[0], "flops": total[1]}


# ------------------------------------------------------------------ how far off a correct answer may be

def tolerance(c):
    # About four times what a pass is off from its 64-bit values.  16-bit attention and linear outputs are
    # rounded to 8 bits of mantissa (and the probabilities before the second product): 2.3e-3 and 1.7e-3.
    # Entropies are 32-bit sums over the vocabulary, whatever the inputs' type (2e-6), and a confidence takes
    # the absolute error of its logit as a relative one (2e-5).  The share of tokens and masks is for ties.
    if c["kind"] == "head":
        return {"rel": 8e-5 if c["confidence"] else 1e-5, "max": 1e-3, "differ": 0.01}
    if c.get("dtype") == "f32":
        return {"rel": 1e-5, "max": 1e-3, "differ": 0.01}
    return {"rel": 1e-2, "max": 0.05, "differ": 0.01}


# ------------------------------------------------------------------ 64-bit values

def _exact_attn(c, s):
    f, k, nc = torch.float64, c["k"], c.get("n_causal", 0)
    group, out = c["q_heads"] // c["kv_heads"], torch.empty(s["q"].shape, dtype=torch.float64, device="cuda")
    at = torch.arange(k, device="cuda")
    seen = (at[None, :] <= at[:, None]) | (at[:, None] >= nc)          # block keys that a block row sees
    for b, n in enumerate(s["lens"].tolist()):
        keys = torch.cat([s["k_cache"][b, :n], s["k_blk"][b]]).to(f)     # [n + k, heads, dim]
        vals = torch.cat([s["v_cache"][b, :n], s["v_blk"][b]]).to(f)
        for h in range(c["kv_heads"]):
            q = s["q"][b, :, h * group:(h + 1) * group].to(f)            # [k, group, dim]
            z = torch.einsum("igd,nd->ign", q, keys[:, h]) / math.sqrt(c["head_dim"])
            z[:, :, n:].masked_fill_(~seen[:, None, :], -math.inf)
            out[b, :, h * group:(h + 1) * group] = torch.einsum("ign,nd->igd", torch.softmax(z, -1), vals[:, h])
    return out


def _exact_head(c, s):
    """(entropy, confidence) of the masked positions, from logits in 64 bits."""
    live = s["masked"].bool()
    x, v = s["hidden"][live].double(), c["vocab"]
    z = torch.cat([x @ s["w"][at:at + 8192].double().T for at in range(0, v, 8192)], 1)
    p = torch.log_softmax(z, 1)
    entropy = torch.full(live.shape, math.inf, dtype=torch.float64, device="cuda")
    confidence = torch.zeros(live.shape, dtype=torch.float64, device="cuda")
    entropy[live] = -(p.exp() * p).sum(1)
    confidence[live] = p.max(1).values.exp()
    return entropy, confidence


def exact(case, seed):
    s = prepare(case, seed)
    if case["kind"] == "linear":
        return tuple(torch.cat([x.double() @ w[at:at + 8192].double().T for at in range(0, w.shape[0], 8192)], 1)
                     for x, w, _ in s["layers"])
    if case["kind"] == "attn":
        out = (_exact_attn(case, s),)
        if case["n_causal"]:
            for cache, blk in ((s["k_cache"], s["k_blk"]), (s["v_cache"], s["v_blk"])):
                cache = cache.double()
                for b, n in enumerate(s["lens"].tolist()):
                    cache[b, n:n + case["n_causal"]] = blk[b, :case["n_causal"]].double()
                out += (cache,)
        return out
    entropy, confidence = _exact_head(case, s)
    if case["kind"] == "head":
        return (entropy, confidence, None) if case["confidence"] else (entropy, None)
    return _exact_attn(case, s), entropy, None, None, None, None
