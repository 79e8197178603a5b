"""The work that a user of this framework has it do, as cases that can be timed and compared.

Five kinds of case, all through the binding's public entry points:

  request       a whole dummy request on a fingerprint handle, as a profiling client sends it: prompt up, prefill,
                first tokens down, then one decode step per generated token with its input ids uploaded and its
                output ids read back, and the last step's logits.  The ids fed to the decode steps are fixed
                (as when two deployments are compared on one trace), so that a near-tie in one greedy choice does
                not change the work of the steps after it.
  linear        one weight-only linear (fp_op_linear): decode with m <= 64 rows, prefill with more.
  attn_decode   one query per sequence over a paged cache (fp_op_attention_decode), ragged context lengths,
                shuffled pages.
  attn_prefill  causal attention over the prompt (fp_op_attention_prefill), q read in place from the fused QKV
                rows, as the forward pass does.

Sizes are those of the repository's own workloads (tiny, 7B-, 13B- and 70B-shaped fingerprints and the 70B-block
sweep of batch 1-64 and context 128-4096) and odd ones between them.
"""
import math

import numpy as np
import torch

import paper_2501_13111_gb300 as fp

BF16, INT8, INT4 = fp.FP_W_BF16, fp.FP_W_INT8, fp.FP_W_INT4_G128
STORE, RESID, SWIGLU, F32 = fp.FP_EPI_STORE, fp.FP_EPI_RESID, fp.FP_EPI_SWIGLU, fp.FP_EPI_F32
PAGE = 16


def listed():
    return [
        # The smallest deployment: one 512-wide block, batch 1, 32-token prompt, 16 tokens.  All launches and latency.
        {"name": "request_tiny", "kind": "request", "layers": 1, "hidden": 512, "heads": 8, "kv_heads": 8, "hd": 64,
         "ffn": 1376, "vocab": 32000, "wq": BF16, "kvq": 0, "batch": 1, "prompt": 32, "steps": 16},
        # The 7B-shaped two-block fingerprint with its own configuration (int8 weights, batch 8, 512 + 100 tokens).
        {"name": "request_7b", "kind": "request", "layers": 2, "hidden": 4096, "heads": 32, "kv_heads": 32, "hd": 128,
         "ffn": 11008, "vocab": 32000, "wq": INT8, "kvq": 0, "batch": 8, "prompt": 512, "steps": 100},
        # Decode, batch 8, int8 weights: the 7B-shaped fused QKV projection.
        {"name": "dec_qkv_int8_b8", "kind": "linear", "wq": INT8, "epi": STORE, "m": 8, "n": 12288, "k": 4096},
        # Decode, batch 32, int4 weights: the 70B-shaped gate and up projections with SwiGLU, the largest matrix.
        {"name": "dec_gu_int4_b32", "kind": "linear", "wq": INT4, "epi": SWIGLU, "m": 32, "n": 57344, "k": 8192},
        # Decode, batch 16, int4 weights: the 13B-shaped down projection with its residual, few rows and a long K.
        {"name": "dec_down_int4_b16", "kind": "linear", "wq": INT4, "epi": RESID, "m": 16, "n": 5120, "k": 13824},
        # The LM head for one sequence: bf16 weights, fp32 logits.
        {"name": "dec_head_bf16_b1", "kind": "linear", "wq": BF16, "epi": F32, "m": 1, "n": 32000, "k": 4096},
        # Prefill of 8 x 512 tokens: the 7B-shaped gate and up projections, int8 weights.
        {"name": "pre_gu_int8_4096", "kind": "linear", "wq": INT8, "epi": SWIGLU, "m": 4096, "n": 22016, "k": 4096},
        # Prefill of one odd-length prompt: the 70B-shaped QKV projection, int4 weights.
        {"name": "pre_qkv_int4_1000", "kind": "linear", "wq": INT4, "epi": STORE, "m": 1000, "n": 10240, "k": 8192},
        # Decode attention, 70B-shaped grouped queries over an int8 cache, 32 sequences of up to 2148 tokens.
        {"name": "attn_dec_int8_b32", "kind": "attn_decode", "kvq": 1, "batch": 32, "heads": 64, "kv_heads": 8,
         "hd": 128, "context": 2148},
        # Decode attention, 7B-shaped, bf16 cache, 8 sequences of up to 612 tokens.
        {"name": "attn_dec_bf16_b8", "kind": "attn_decode", "kvq": 0, "batch": 8, "heads": 32, "kv_heads": 32,
         "hd": 128, "context": 612},
        # Prefill attention, 13B-shaped, bf16 cache, 8 prompts of 1024.
        {"name": "attn_pre_bf16_1024", "kind": "attn_prefill", "kvq": 0, "batch": 8, "heads": 40, "kv_heads": 40,
         "hd": 128, "prompt": 1024},
        # Prefill attention, 70B-shaped grouped queries over an int8 cache, 4 prompts of 2048.
        {"name": "attn_pre_int8_2048", "kind": "attn_prefill", "kvq": 1, "batch": 4, "heads": 64, "kv_heads": 8,
         "hd": 128, "prompt": 2048},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["request", "linear", "linear", "linear", "linear", "linear", "attn_decode", "attn_decode",
                       "attn_prefill", "attn_prefill"])
    if kind == "request":
        hd = rng.choice([64, 128])
        heads = rng.choice([8, 16, 24, 32])
        group = rng.choice([1, 1, 2, 4, 8])
        wq = rng.choice([BF16, INT8, INT4])
        hidden = 128 * rng.randint(4, 32)
        return {"kind": kind, "layers": rng.randint(1, 2), "hidden": hidden, "heads": heads, "kv_heads": heads // group,
                "hd": hd, "ffn": 128 * rng.randint(8, 86), "vocab": 32000, "wq": wq, "kvq": rng.randint(0, 1),
                "batch": _log(rng, 1, 8), "prompt": _log(rng, 16, 512), "steps": _log(rng, 8, 64)}
    if kind == "linear":
        wq = rng.choice([BF16, INT8, INT8, INT4, INT4])
        epi = rng.choice([STORE, RESID, SWIGLU, F32] if wq == BF16 else [STORE, RESID, SWIGLU])
        if rng.random() < 0.65:  # decode
            m = _log(rng, 1, 64)
            n, k = rng.choice([(12288, 4096), (4096, 4096), (22016, 4096), (4096, 11008), (15360, 5120), (5120, 5120),
                               (27648, 5120), (5120, 13824), (10240, 8192), (8192, 8192), (57344, 8192),
                               (8192, 28672), (32000, 4096),
                               (8 * _log(rng, 64, 4096), 128 * _log(rng, 4, 96))])
        else:
            m = _log(rng, 65, 4096)
            n, k = rng.choice([(12288, 4096), (4096, 4096), (22016, 4096), (4096, 11008), (15360, 5120), (5120, 5120),
                               (10240, 8192), (8192, 8192), (8 * _log(rng, 64, 2048), 128 * _log(rng, 4, 64))])
        return {"kind": kind, "wq": wq, "epi": epi, "m": m, "n": n, "k": k}
    heads, kv_heads = rng.choice([(32, 32), (40, 40), (64, 8), (64, 8), (32, 8), (16, 4), (8, 8)])
    if kind == "attn_decode":
        batch = _log(rng, 1, 64)
        context = _log(rng, 128, 4096)
        while batch * context * kv_heads > 32 * 2148 * 32:  # at most about a 1 GB cache
            context = max(128, context // 2)
            batch = max(1, batch * 3 // 4)
        return {"kind": kind, "kvq": rng.randint(0, 1), "batch": batch, "heads": heads, "kv_heads": kv_heads,
                "hd": 128, "context": context}
    prompt = _log(rng, 64, 4096)
    batch = _log(rng, 1, 8)
    while batch > 1 and batch * heads * prompt * prompt > 8 * 64 * 2048 * 2048:
        batch -= 1
    return {"kind": kind, "kvq": rng.randint(0, 1), "batch": batch, "heads": heads, "kv_heads": kv_heads, "hd": 128,
            "prompt": prompt}


# ------------------------------------------------------------------ helpers
def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFF)
    return g


def _randn(gen, *shape, scale=1.0):
    return (torch.randn(*shape, device="cuda", generator=gen) * scale).to(torch.bfloat16)


def _stream():
    return torch.cuda.current_stream().cuda_stream


def _opt(t):
    return None if t is None else t.data_ptr()


# ------------------------------------------------------------------ linear
def _linear_inputs(c, seed):
    m, n, k = c["m"], c["n"], c["k"]
    g = _gen(seed, 1)
    w = _randn(g, n, k, scale=0.02)  # the fingerprint's weight distribution
    x = _randn(g, m, k)              # RMS-normalised activations
    nout = n // 2 if c["epi"] == SWIGLU else n
    r = _randn(g, m, nout) if c["epi"] == RESID else None
    return w, x, r


def _linear_prepare(c, seed):
    m, n, k, wq, epi = c["m"], c["n"], c["k"], c["wq"], c["epi"]
    w, x, r = _linear_inputs(c, seed)
    s = {"c": c, "x": x, "r": r, "scales": None, "zeros": None}
    if wq == BF16:
        s["codes"] = w
    else:
        groups = k // 128
        s["codes"] = torch.empty(n * k if wq == INT8 else n * k // 2, dtype=torch.uint8, device="cuda")
        s["scales"] = torch.empty(n if wq == INT8 else n * groups, dtype=torch.bfloat16, device="cuda")
        s["zeros"] = torch.empty(n * groups, dtype=torch.bfloat16, device="cuda") if wq == INT4 else None
        fp.fp_op_quantize(wq, w.data_ptr(), n, k, s["codes"].data_ptr(), s["scales"].data_ptr(), _opt(s["zeros"]),
                          stream=_stream())
    nout = n // 2 if epi == SWIGLU else n
    s["y"] = torch.empty(m, nout, dtype=torch.float32 if epi == F32 else torch.bfloat16, device="cuda")
    s["ws_bytes"] = fp.fp_op_linear_workspace_bytes(wq, m, n, k)
    s["ws"] = torch.zeros(max(s["ws_bytes"], 16), dtype=torch.uint8, device="cuda")
    return s


def _linear_run(s):
    c = s["c"]
    fp.fp_op_linear(c["wq"], c["epi"], s["x"].data_ptr(), c["m"], c["n"], c["k"], s["codes"].data_ptr(),
                    _opt(s["scales"]), _opt(s["zeros"]), _opt(s["r"]), s["y"].data_ptr(), s["ws"].data_ptr(),
                    s["ws_bytes"], stream=_stream())
    return s["y"]


def _over(v, d):
    """The fp32 quotient v / d, rounded once (a division by a host number multiplies by its reciprocal)."""
    return v / torch.full_like(v, d)


def _bf16_up(v):
    """Smallest bf16 not below v (fp32, v >= 0), as fp32."""
    b = v.contiguous().view(torch.int32)
    return ((b + 0xFFFF) & ~0xFFFF).view(torch.float32)


def _dequantized(w, wq):
    """The weights the configuration's format holds, rows of fp64 (the definitions in fp.h)."""
    f = w.float()
    if wq == BF16:
        return f.double()
    if wq == INT8:
        s = _bf16_up(_over(f.abs().amax(1, keepdim=True), 127.0))
        q = torch.where(s > 0, torch.round(f / s), torch.zeros_like(f)).clamp(-127, 127)
        return q.double() * s.double()
    n, k = f.shape
    f = f.view(n, k // 128, 128)
    mn, mx = f.amin(2, keepdim=True).clamp(max=0), f.amax(2, keepdim=True).clamp(min=0)
    s = _bf16_up(_over(mx - mn, 15.0))
    z = torch.where(s > 0, torch.round(-mn / s), torch.zeros_like(s)).clamp(0, 15)
    q = torch.where(s > 0, torch.round(f / s) + z, torch.zeros_like(f)).clamp(0, 15)
    return ((q.double() - z.double()) * s.double()).view(n, k)


def _product(x, w, wq):
    """x W^T in fp64, a band of output columns at a time."""
    out = torch.empty(x.shape[0], w.shape[0], dtype=torch.float64, device="cuda")
    step = max(128, (1 << 26) // w.shape[1])
    for i in range(0, w.shape[0], step):
        out[:, i:i + step] = x.double() @ _dequantized(w[i:i + step], wq).T
    return out


def _linear_exact(c, seed):
    w, x, r = _linear_inputs(c, seed)
    y = _product(x, w, c["wq"])
    if c["epi"] == RESID:
        y = y + r.double()
    elif c["epi"] == SWIGLU:
        half = c["n"] // 2
        y = torch.nn.functional.silu(y[:, :half]) * y[:, half:]
    return y


def _linear_work(c):
    m, n, k, wq = c["m"], c["n"], c["k"], c["wq"]
    nout = n // 2 if c["epi"] == SWIGLU else n
    weights = 2 * n * k if wq == BF16 else n * k + 2 * n if wq == INT8 else n * k // 2 + 4 * n * (k // 128)
    act = 2 * m * k + (4 if c["epi"] == F32 else 2) * m * nout + (2 * m * nout if c["epi"] == RESID else 0)
    return {"bytes": weights + act, "flops": 2 * m * n * k}


# ------------------------------------------------------------------ paged cache
def _cache(c, tokens, seed):
    """Pools of normal keys and values in shuffled pages, and the page table."""
    b, hkv, hd = c["batch"], c["kv_heads"], c["hd"]
    pps = (tokens + PAGE - 1) // PAGE
    g = _gen(seed, 2)
    table = torch.randperm(b * pps, device="cuda", generator=g).to(torch.int32).view(b, pps)
    pools = []
    for _ in range(2):
        x = _randn(g, b * pps, hkv, PAGE, hd)
        if c["kvq"] == 0:
            pools.append((x, None))
        else:
            f = x.float()
            s = f.abs().amax(3) / 127.0
            pools.append((torch.round(f / s[..., None]).clamp(-127, 127).to(torch.int8), s))
    view = fp.fp_kv_view(c["kvq"], hkv, hd, PAGE, pps, b * pps, pools[0][0].data_ptr(), pools[1][0].data_ptr(),
                         _opt(pools[0][1]), _opt(pools[1][1]), table.data_ptr())
    return table, pools, view


def _sequence(pool, table, b, tokens):
    """Positions 0 .. tokens-1 of sequence b: [kv_heads, tokens, hd] fp64."""
    x, s = pool
    pages = table[b, :(tokens + PAGE - 1) // PAGE].long()
    v = x[pages].double()
    if s is not None:
        v = v * s[pages].double()[..., None]
    return v.permute(1, 0, 2, 3).reshape(x.shape[1], -1, x.shape[3])[:, :tokens]


# ------------------------------------------------------------------ decode attention
def _lens(c, seed):
    """Context lengths as a running batch has them: from a half to all of the longest."""
    r = np.random.RandomState(int(seed) % (1 << 31))
    lens = r.randint(c["context"] // 2, c["context"] + 1, c["batch"])
    lens[r.randint(c["batch"])] = c["context"]
    return np.maximum(lens, 1).astype(np.int32)


def _attn_decode_prepare(c, seed):
    table, pools, view = _cache(c, c["context"], seed)
    b, h, hd = c["batch"], c["heads"], c["hd"]
    ws_bytes = fp.fp_op_attention_decode_workspace_bytes(b, h, hd, c["context"])
    return {"c": c, "table": table, "pools": pools, "view": view, "ws_bytes": ws_bytes,
            "q": _randn(_gen(seed, 3), b, h * hd), "lens": torch.from_numpy(_lens(c, seed)).cuda(),
            "out": torch.empty(b, h * hd, dtype=torch.bfloat16, device="cuda"),
            "ws": torch.empty(max(16, ws_bytes), dtype=torch.uint8, device="cuda")}


def _attn_decode_run(s):
    c = s["c"]
    fp.fp_op_attention_decode(s["q"].data_ptr(), c["heads"] * c["hd"], c["batch"], c["heads"], s["view"],
                              s["lens"].data_ptr(), c["context"], s["out"].data_ptr(), s["ws"].data_ptr(),
                              s["ws_bytes"], stream=_stream())
    return s["out"]


def _attn_decode_exact(c, seed):
    table, pools, _ = _cache(c, c["context"], seed)
    b, h, hkv, hd = c["batch"], c["heads"], c["kv_heads"], c["hd"]
    q = _randn(_gen(seed, 3), b, h * hd).double().view(b, hkv, h // hkv, hd)
    out = torch.empty(b, h * hd, dtype=torch.float64, device="cuda")
    for i, n in enumerate(_lens(c, seed)):
        k, v = (_sequence(p, table, i, int(n)) for p in pools)
        p = torch.softmax(q[i] @ k.transpose(1, 2) / math.sqrt(hd), dim=-1)
        out[i] = (p @ v).reshape(-1)
    return out


def _attn_decode_work(c):
    tokens = c["batch"] * c["context"] * 3 // 4  # the mean length of the draw
    per = 2 * c["kv_heads"] * (2 * c["hd"] if c["kvq"] == 0 else c["hd"] + 4)
    return {"bytes": tokens * per + 4 * c["batch"] * c["heads"] * c["hd"],
            "flops": 4 * tokens * c["heads"] * c["hd"]}


# ------------------------------------------------------------------ prefill attention
def _attn_prefill_prepare(c, seed):
    table, pools, view = _cache(c, c["prompt"], seed)
    rows, width = c["batch"] * c["prompt"], (c["heads"] + 2 * c["kv_heads"]) * c["hd"]
    return {"c": c, "table": table, "pools": pools, "view": view, "qkv": _randn(_gen(seed, 4), rows, width),
            "out": torch.empty(rows, c["heads"] * c["hd"], dtype=torch.bfloat16, device="cuda")}


def _attn_prefill_run(s):
    c = s["c"]
    fp.fp_op_attention_prefill(s["qkv"].data_ptr(), s["qkv"].shape[1], c["batch"], c["prompt"], c["heads"], s["view"],
                               s["out"].data_ptr(), stream=_stream())
    return s["out"]


def _attn_prefill_exact(c, seed):
    table, pools, _ = _cache(c, c["prompt"], seed)
    b, s, h, hkv, hd = c["batch"], c["prompt"], c["heads"], c["kv_heads"], c["hd"]
    qkv = _randn(_gen(seed, 4), b * s, (h + 2 * hkv) * hd)
    q = qkv[:, :h * hd].view(b, s, hkv, h // hkv, hd)
    out = torch.empty(b, s, h, hd, dtype=torch.float64, device="cuda")
    later = torch.ones(s, s, dtype=torch.bool, device="cuda").triu(1)
    for i in range(b):
        k, v = (_sequence(p, table, i, s) for p in pools)
        for j in range(hkv):
            for t in range(h // hkv):
                x = q[i, :, j, t].double() @ k[j].T / math.sqrt(hd)
                out[i, :, j * (h // hkv) + t] = torch.softmax(x.masked_fill_(later, -math.inf), dim=-1) @ v[j]
    return out.view(b * s, h * hd)


def _attn_prefill_work(c):
    b, s, h, hkv, hd = c["batch"], c["prompt"], c["heads"], c["kv_heads"], c["hd"]
    per = 2 * hkv * (2 * hd if c["kvq"] == 0 else hd + 4)
    return {"bytes": b * s * (4 * h * hd + per), "flops": 2 * b * h * s * (s + 1) * hd}


# ------------------------------------------------------------------ whole requests
class _Handle:
    """A fingerprint handle that is destroyed with its state."""

    def __init__(self, h):
        self.h = h

    def __del__(self):
        fp.fp_destroy(self.h)


def _tensor_rows(c):
    """(tensor id, rows, columns) of a block's matrices."""
    d, q, kv, f = c["hidden"], c["heads"] * c["hd"], c["kv_heads"] * c["hd"], c["ffn"]
    return [(fp.FP_T_WQ, q, d), (fp.FP_T_WK, kv, d), (fp.FP_T_WV, kv, d), (fp.FP_T_WO, d, q), (fp.FP_T_WGATE, f, d),
            (fp.FP_T_WUP, f, d), (fp.FP_T_WDOWN, d, f)]


def _small(c):
    """A model whose own weights are uploaded (and which can be checked in 64 bits)."""
    return c["wq"] == BF16 and c["hidden"] <= 1024 and c["batch"] * c["prompt"] <= 1024


def _small_weights(c, seed):
    g = _gen(seed, 5)
    d, v = c["hidden"], c["vocab"]
    glob = {fp.FP_T_EMBED: _randn(g, v, d, scale=0.02), fp.FP_T_LM_HEAD: _randn(g, v, d, scale=0.02),
            fp.FP_T_FINAL_NORM: torch.ones(d, dtype=torch.bfloat16, device="cuda")}
    blocks = []
    for _ in range(c["layers"]):
        b = {t: _randn(g, n, k, scale=0.02) for t, n, k in _tensor_rows(c)}
        b[fp.FP_T_ATTN_NORM] = b[fp.FP_T_FFN_NORM] = torch.ones(d, dtype=torch.bfloat16, device="cuda")
        blocks.append(b)
    return glob, blocks


def _request_tokens(c, seed):
    r = np.random.RandomState(int(seed) % (1 << 31))
    return (r.randint(0, c["vocab"], (c["batch"], c["prompt"])).astype(np.int32),
            r.randint(0, c["vocab"], (c["steps"], c["batch"])).astype(np.int32))


def _request_prepare(c, seed):
    arch = dict(n_layers=c["layers"], hidden=c["hidden"], n_heads=c["heads"], n_kv_heads=c["kv_heads"],
                head_dim=c["hd"], ffn=c["ffn"], vocab=c["vocab"], rms_eps=1e-5, rope_base=1e4)
    small = _small(c)
    h = _Handle(fp.fp_create(arch, c["wq"], c["kvq"], c["batch"], c["prompt"] + c["steps"], seed=int(seed),
                             flags=fp.FP_FLAG_NO_INIT if small else 0))
    if small:
        glob, blocks = _small_weights(c, seed)
        for layer, tensors in enumerate([glob] + blocks):
            for t, w in tensors.items():
                fp.fp_set_weight(h.h, layer - 1, t, w.view(torch.int16).cpu().numpy().reshape(-1).view(np.uint16))
    prompt, forced = _request_tokens(c, seed)
    # the decode graph is captured on the first step of a handle, which a deployment pays once
    fp.fp_prefill(h.h, prompt)
    fp.fp_decode_step(h.h, forced[0])
    return {"c": c, "h": h, "prompt": prompt, "forced": forced, "out": np.empty(c["batch"], np.int32)}


def _request_run(s):
    c, h = s["c"], s["h"].h
    fp.fp_prefill(h, s["prompt"], out=s["out"])
    for tokens in s["forced"]:
        fp.fp_decode_step(h, tokens, out=s["out"])
    return fp.fp_get_tensor(h, fp.FP_G_LOGITS, dtype=np.float32).reshape(c["batch"], c["vocab"])


def _request_exact(c, seed):
    if not _small(c) or c["kvq"] != 0:
        return None
    glob, blocks = _small_weights(c, seed)
    prompt, forced = _request_tokens(c, seed)
    ids = torch.from_numpy(np.concatenate([prompt, forced.T], 1)).long().cuda()
    b, n = ids.shape
    h, hkv, hd = c["heads"], c["kv_heads"], c["hd"]
    ang = torch.arange(n, device="cuda", dtype=torch.float64)[:, None] * (
        1e4 ** (-torch.arange(hd // 2, device="cuda", dtype=torch.float64) * 2 / hd))
    cos, sin = ang.cos(), ang.sin()

    def norm(x, gain):
        return x / torch.sqrt((x * x).mean(-1, keepdim=True) + 1e-5) * gain.double()

    def rope(x):  # [b, heads, n, hd], pairs (i, i + hd/2)
        lo, hi = x[..., :hd // 2], x[..., hd // 2:]
        return torch.cat([lo * cos - hi * sin, hi * cos + lo * sin], -1)

    later = torch.ones(n, n, dtype=torch.bool, device="cuda").triu(1)
    x = glob[fp.FP_T_EMBED][ids].double()
    for w in blocks:
        y = norm(x, w[fp.FP_T_ATTN_NORM])
        q, k, v = ((y @ w[t].double().T).view(b, n, -1, hd).transpose(1, 2)
                   for t in (fp.FP_T_WQ, fp.FP_T_WK, fp.FP_T_WV))
        k, v = (t.repeat_interleave(h // hkv, 1) for t in (rope(k), v))
        p = torch.softmax((rope(q) @ k.transpose(2, 3) / math.sqrt(hd)).masked_fill(later, -math.inf), -1)
        x = x + (p @ v).transpose(1, 2).reshape(b, n, -1) @ w[fp.FP_T_WO].double().T
        y = norm(x, w[fp.FP_T_FFN_NORM])
        a = torch.nn.functional.silu(y @ w[fp.FP_T_WGATE].double().T) * (y @ w[fp.FP_T_WUP].double().T)
        x = x + a @ w[fp.FP_T_WDOWN].double().T
    return norm(x[:, -1], glob[fp.FP_T_FINAL_NORM]) @ glob[fp.FP_T_LM_HEAD].double().T


def _request_work(c):
    params = sum(n * k for _, n, k in _tensor_rows(c))
    groups = sum(n * (k // 128) for _, n, k in _tensor_rows(c))
    rows = sum(n for _, n, _ in _tensor_rows(c))
    wbytes = 2 * params if c["wq"] == BF16 else params + 2 * rows if c["wq"] == INT8 else params // 2 + 4 * groups
    head = 2 * c["vocab"] * c["hidden"]
    b, s, n = c["batch"], c["prompt"], c["steps"]
    per = 2 * c["kv_heads"] * (2 * c["hd"] if c["kvq"] == 0 else c["hd"] + 4)
    cached = sum(s + i + 1 for i in range(n))
    qk = 2 * c["heads"] * c["hd"]
    return {"bytes": (n + 1) * (c["layers"] * wbytes + head) + c["layers"] * b * per * (cached + 2 * s),
            "flops": c["layers"] * (2 * params * b * (s + n) + b * qk * (s * (s + 1) + 2 * cached)) + (n + 1) * b * head}


# ------------------------------------------------------------------ the file's interface
_KINDS = {
    "request": (_request_prepare, _request_run, _request_work, _request_exact),
    "linear": (_linear_prepare, _linear_run, _linear_work, _linear_exact),
    "attn_decode": (_attn_decode_prepare, _attn_decode_run, _attn_decode_work, _attn_decode_exact),
    "attn_prefill": (_attn_prefill_prepare, _attn_prefill_run, _attn_prefill_work, _attn_prefill_exact),
}


def prepare(case, seed):
    return _KINDS[case["kind"]][0](case, seed)


def run(state):
    return _KINDS[state["c"]["kind"]][1](state)


def work(case):
    return _KINDS[case["kind"]][2](case)


def exact(case, seed):
    return _KINDS[case["kind"]][3](case, seed)


def tolerance(case):
    """About four times what was measured against `exact` (its rounding to bf16 is 1.7e-3 of the result by itself)."""
    if case["kind"] == "request":  # two bf16 blocks and their caches: 5e-3 against 64 bits, 4e-3 from run to run
        return {"rel": 2e-2, "max": 1.5e-1}
    if case["kind"] == "linear":
        if case["epi"] == F32:  # bf16 products summed in fp32, no rounding of the result
            return {"rel": 5e-5, "max": 2e-4}
        # int4 weights may be rounded to bf16 after their zero point and scale are applied
        return {"rel": 1e-2, "max": 8e-2} if case["wq"] == INT4 else {"rel": 7e-3, "max": 2e-2}
    return {"rel": 8e-3, "max": 1e-1}  # probabilities rounded to 16 bits before the second product
