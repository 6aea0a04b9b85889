"""What this library's users have it do, as cases that can be timed and compared.

Four kinds of work, each through the public binding and with the buffers that a
serving or training program keeps between calls:

  decode  one token per sequence appended to the cache and attended to
          (tk_attn_decode_append): every step of text generation.
  prompt  a new prompt stored in the cache (tk_kv_append) and attended to
          (tk_attn_prefill): the first pass of every request.
  chunk   a piece of a prompt after cached tokens (tk_attn_prefill_cached):
          chunked prefill, a further turn of a conversation.
  train   forward with row logsumexp and gradients (tk_attn_forward,
          tk_attn_backward): one attention layer of a training step.

Shapes are those of the repository's workloads (a GPT-2-small layer, a 7B MHA
layer, a Mistral-shaped GQA layer) or generic.  Inputs are N(0, 1) rounded to
bf16; query heads are of different sharpness (N(0, 1) logits up to a standard
deviation of 2.5), as trained heads are.
"""

import math

import torch

from paper_2603_04427_gb300 import binding as tk

DEV = "cuda"
BF16_PEAK, HBM = 1.9e15, 6.8e12    # for the cost of a drawn case only


def _case(name, kind, batch, h_q, h_kv, r, d_v, new, lo=0, hi=0, page=0, keys="bf16", out="bf16",
          causal=True):
    """`new` tokens per sequence after lo..hi cached ones (uniform; the same for all if equal)."""
    return dict(name=name, kind=kind, batch=batch, h_q=h_q, h_kv=h_kv, r=r, d_v=d_v, new=new, lo=lo,
                hi=hi, page=page, keys=keys, out=out, causal=causal)


def listed():
    return [
        # one layer of a GPT-2-small step, one user: nothing but latency
        _case("decode_gpt2_b1_ctx270", "decode", 1, 12, 12, 16, 64, 1, 270, 270, out="f32"),
        # a small server's step: short ragged conversations, 4-bit keys, 16-token pages
        _case("decode_int4_b24_ragged_p16", "decode", 24, 32, 8, 64, 128, 1, 60, 2500, page=16,
              keys="int4"),
        # the Mistral-shaped GQA step at full batch, contiguous cache
        _case("decode_gqa_b16_ctx4095", "decode", 16, 32, 8, 32, 128, 1, 4095, 4095, out="f32"),
        # long documents: four contexts of 64K to 128K tokens in 64-token pages
        _case("decode_paged_b4_64k_128k", "decode", 4, 32, 8, 32, 128, 1, 65536, 131000, page=64,
              out="f32"),
        # throughput serving: a large batch over int8 keys
        _case("decode_int8_b64_8k_16k", "decode", 64, 32, 8, 32, 128, 1, 8000, 16383, keys="int8",
              out="f32"),
        # a short prompt of a small model
        _case("prompt_gpt2_s256", "prompt", 1, 12, 12, 16, 64, 256, out="f32"),
        # an ordinary prompt of one user, odd length, GQA
        _case("prompt_gqa_b1_s1531", "prompt", 1, 32, 8, 32, 128, 1531),
        # the 7B-shaped long prompt
        _case("prompt_mha7b_b2_s8192", "prompt", 2, 32, 32, 32, 128, 8192),
        # a further turn: a few hundred tokens after a long ragged paged context
        _case("chunk_paged_b2_s500_after_8k", "chunk", 2, 32, 8, 32, 128, 500, 6000, 9000, page=64),
        # chunked prefill of a long prompt over int8 keys
        _case("chunk_int8_b2_s4096_after_4096", "chunk", 2, 32, 32, 32, 128, 4096, 4096, 4096,
              keys="int8"),
        # training, small model: GPT-2-small layer with thin keys, odd sequence length
        _case("train_gpt2_b8_s1000", "train", 8, 12, 12, 16, 64, 1000),
        # training, the 7B shape at a 4K context
        _case("train_mha7b_b2_s4096", "train", 2, 32, 32, 32, 128, 4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(c):
    w = work(c)
    return max(w["bytes"] / HBM, w["flops"] / BF16_PEAK)


def draw(rng):
    """Another case of these ranges; odd sizes come by themselves."""
    most = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(("decode", "prompt", "chunk", "train"))
        h_q, h_kv = rng.choice(((12, 12), (32, 32), (32, 8), (32, 8), (16, 2), (16, 8)))
        d_v = rng.choice((64, 128, 128))
        r = rng.choice((16, 32, 32, 64, d_v))
        keys = rng.choice(("bf16", "bf16", "int8", "int4")) if kind in ("decode", "chunk") else "bf16"
        page = rng.choice((0, 0, 16, 64, 128)) if kind in ("decode", "chunk") else 0
        if keys == "int4":
            r = max(r, 32)
        out = "bf16" if kind == "train" else rng.choice(("bf16", "f32"))
        causal = kind == "chunk" or kind == "decode" or rng.random() < 0.8
        batch = _log_int(rng, 1, 96 if kind == "decode" else 8)
        lo = hi = 0
        if kind == "decode":
            new = 1
            lo = _log_int(rng, 16, 60000)
            hi = lo if rng.random() < 0.4 else int(lo * rng.uniform(1.2, 4.0))
        elif kind == "chunk":
            new = _log_int(rng, 16, 4096)
            lo = _log_int(rng, 64, 24000)
            hi = lo if rng.random() < 0.4 else int(lo * rng.uniform(1.1, 2.0))
        else:
            new = _log_int(rng, 64, 8192 if kind == "prompt" else 4096)
        c = _case("", kind, batch, h_q, h_kv, r, d_v, new, lo, hi, page, keys, out, causal)
        del c["name"]
        if _cost(c) <= most:
            return c


# ------------------------------------------------------------------ inputs (plain torch)

def _lens(c):
    """Cached tokens of every sequence; part of the case, the same for every seed."""
    n = c["batch"]
    if c["hi"] <= c["lo"]:
        return [c["lo"]] * n
    g = torch.Generator().manual_seed(977 + c["lo"] + c["hi"])
    return [int(x) for x in torch.randint(c["lo"], c["hi"] + 1, (n,), generator=g)]


def _randn(shape, g):
    return torch.randn(shape, generator=g, device=DEV, dtype=torch.float32)


def _quantise(k, keys):
    """Symmetric per-token codes and fp32 scales; int4 packed two per byte, even element low."""
    top = 127.0 if keys == "int8" else 7.0
    scale = k.abs().amax(-1) / top
    code = torch.where(scale[..., None] > 0, (k / scale[..., None]).round().clamp(-top, top),
                       torch.zeros((), device=k.device)).to(torch.int8)
    return code, scale


def _stored_keys(k, keys):
    """What a cache of this format stores for keys k (bf16): (k buffer, scales or None)."""
    if keys == "bf16":
        return k, None
    code, scale = _quantise(k.float(), keys)
    if keys == "int4":
        u = code.view(torch.uint8)
        code = (u[..., 0::2] & 15) | ((u[..., 1::2] & 15) << 4)
    return code, scale


def _inputs(c, seed):
    """Queries, new keys and values and, for decode and chunk, the cache's content."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    B, hq, hkv, r, dv, n = (c[x] for x in ("batch", "h_q", "h_kv", "r", "d_v", "new"))
    sharp = 1.0 + 0.5 * (torch.arange(hq, device=DEV) % 4).float()
    x = dict(q=(_randn((B, hq, n, r), g) * sharp[None, :, None, None]).bfloat16(),
             k=_randn((B, hkv, n, r), g).bfloat16(), v=_randn((B, hkv, n, dv), g).bfloat16())
    if c["kind"] == "train":
        x["d_out"] = _randn((B, hq, n, dv), g).bfloat16()
    if c["kind"] in ("prompt", "train"):
        return x
    lens = _lens(c)
    cap = -(-(max(lens) + n) // 16) * 16
    if c["page"]:
        p = c["page"]
        need = [-(-(t + n) // p) for t in lens]
        pages = torch.randperm(sum(need), generator=torch.Generator().manual_seed(int(seed)))
        table = torch.zeros((B, max(need)), dtype=torch.int32)
        at = 0
        for b, m in enumerate(need):
            table[b, :m] = pages[at:at + m].int()
            at += m
        x["table"], lead = table.to(DEV), (sum(need), hkv, p)
    else:
        lead = (B, hkv, cap)
    x["lens"], x["lead"], x["cap"] = lens, lead, cap
    # in pieces: a cache may be gigabytes, and fp32 copies of it would be several times that
    k_buf = s_buf = None
    x["v_cache"] = torch.empty(lead + (dv,), dtype=torch.bfloat16, device=DEV)
    step = max(1, (1 << 28) // (hkv * lead[2] * max(r, dv)))
    for i in range(0, lead[0], step):
        m = min(step, lead[0] - i)
        kk, ss = _stored_keys(_randn((m,) + lead[1:] + (r,), g).bfloat16(), c["keys"])
        if k_buf is None:
            k_buf = torch.empty(lead + (kk.shape[-1],), dtype=kk.dtype, device=DEV)
            s_buf = torch.empty(lead, device=DEV) if ss is not None else None
        k_buf[i:i + m] = kk
        if ss is not None:
            s_buf[i:i + m] = ss
        x["v_cache"][i:i + m] = _randn((m,) + lead[1:] + (dv,), g)
    x["k_cache"], x["k_scale"] = k_buf, s_buf
    return x


# ------------------------------------------------------------------ the program's side

def prepare(case, seed):
    c, x = case, _inputs(case, seed)
    B, hq, hkv, r, dv, n = (c[f] for f in ("batch", "h_q", "h_kv", "r", "d_v", "new"))
    s = dict(kind=c["kind"], causal=bool(c["causal"]))
    dt = torch.float32 if c["out"] == "f32" else torch.bfloat16
    if c["kind"] == "train":
        s.update(x, out=torch.empty((B, hq, n, dv), dtype=dt, device=DEV),
                 lse=torch.empty((B, hq, n), device=DEV), dq=torch.empty((B, hq, n, r), device=DEV),
                 dk=torch.empty((B, hkv, n, r), device=DEV), dv=torch.empty((B, hkv, n, dv), device=DEV),
                 ws=torch.empty(tk.load_library().tk_backward_workspace_size(B, hq, n),
                                dtype=torch.uint8, device=DEV))
        return s
    s["out"] = torch.empty((B, hq, n, dv) if c["kind"] != "decode" else (B, hq, dv), dtype=dt, device=DEV)
    if c["kind"] == "prompt":
        cache = tk.ThinKeyCache.allocate(B, hq, hkv, r, dv, capacity=-(-n // 16) * 16)
        s.update(x, cache=cache, lens=torch.zeros(B, dtype=torch.int32, device=DEV))
        return s
    quant = dict(k_int8=c["keys"] == "int8", k_int4=c["keys"] == "int4")
    if c["page"]:
        cache = tk.ThinKeyCache.allocate(B, hq, hkv, r, dv, page_size=c["page"], num_pages=x["lead"][0],
                                         page_table=x["table"], **quant)
    else:
        cache = tk.ThinKeyCache.allocate(B, hq, hkv, r, dv, capacity=x["cap"], **quant)
    cache.k, cache.v = x["k_cache"], x["v_cache"]
    if x["k_scale"] is not None:
        cache.k_scale = x["k_scale"]
    s.update(cache=cache, bound=max(x["lens"]) + n,
             lens=torch.tensor(x["lens"], dtype=torch.int32, device=DEV))
    if c["kind"] == "decode":
        s.update(q=x["q"][:, :, 0].contiguous(), k=x["k"][:, :, 0].contiguous(),
                 v=x["v"][:, :, 0].contiguous(), ws=tk.decode_workspace(cache.desc, s["bound"]))
    else:
        s.update(q=x["q"], k=x["k"], v=x["v"], ws=tk.prefill_cached_workspace(cache, s["bound"]))
    return s


def run(s):
    kind = s["kind"]
    if kind == "train":
        tk.tk_attn_forward(s["q"], s["k"], s["v"], s["out"], s["lse"], causal=s["causal"])
        tk.tk_attn_backward(s["q"], s["k"], s["v"], s["out"], s["d_out"], s["lse"], s["dq"], s["dk"],
                            s["dv"], workspace=s["ws"], causal=s["causal"])
        return {"out": s["out"], "lse": s["lse"], "dq": s["dq"], "dk": s["dk"], "dv": s["dv"]}
    c = s["cache"]
    if kind == "decode":
        tk.tk_attn_decode_append(c, s["q"], s["k"], s["v"], s["lens"], s["bound"], s["out"], s["ws"])
    elif kind == "prompt":
        tk.tk_kv_append(c, s["k"], s["v"], s["lens"])
        tk.tk_attn_prefill(s["q"], s["k"], s["v"], s["out"], causal=s["causal"])
    else:
        tk.tk_attn_prefill_cached(c, s["q"], s["k"], s["v"], s["lens"], s["bound"], s["out"],
                                  causal=s["causal"], workspace=s["ws"])
    # the cache is updated state
    return {"out": s["out"], "k_cache": c.k, "v_cache": c.v, "k_scale": c.k_scale}


# ------------------------------------------------------------------ what it cannot do without

def work(case):
    c = case
    B, hq, hkv, r, dv, n = (c[f] for f in ("batch", "h_q", "h_kv", "r", "d_v", "new"))
    ob = 4 if c["out"] == "f32" else 2
    kb = {"bf16": 2 * r, "int8": r + 4, "int4": r // 2 + 4}[c["keys"]]
    qo = B * hq * n * (2 * r + ob * dv)
    new = B * hkv * n * (2 * r + 2 * dv)
    if c["kind"] in ("prompt", "train"):
        pairs = B * hq * (n * (n + 1) // 2 if c["causal"] else n * n)
        if c["kind"] == "prompt":
            return {"bytes": qo + 2 * new, "flops": 2 * pairs * (r + dv)}
        # q, k, v, d_out read once, out, lse and the fp32 gradients written once
        grads = 4 * (B * hq * n * r + B * hkv * n * (r + dv))
        return {"bytes": qo + new + 4 * B * hq * n + 2 * B * hq * n * dv + grads,
                "flops": 2 * pairs * (r + dv) + 2 * pairs * (3 * r + 2 * dv)}
    lens = _lens(c)
    cached = sum(lens) * hkv * (kb + 2 * dv)
    pairs = hq * sum(t * n + n * (n + 1) // 2 for t in lens)
    return {"bytes": cached + new + B * hkv * n * (kb + 2 * dv) + qo, "flops": 2 * pairs * (r + dv)}


def tolerance(case):
    # The softmax weights enter the second product as bf16 (2^-9 each, errors that average out over
    # the keys): 0.4e-3 to 0.9e-3 of the result's norm against 64 bits, 1.6e-3 to 2.3e-3 once the
    # result is rounded to bf16, up to 2.8e-3 for gradients (two such roundings); all measured.
    # Another order of the same sums rounds other weights: about four times that.  Single values
    # may be a bf16 unit or two (2^-7) apart.
    if case["kind"] == "train":
        return {"rel": 1e-2, "max": 0.1}
    return {"rel": 4e-3 if case["out"] == "f32" else 8e-3, "max": 0.1}


# ------------------------------------------------------------------ the same in 64 bits

def _context(c, x, b):
    """Keys [Hkv, t, r] and values of sequence b after the new tokens are stored, in fp64."""
    t, n = x["lens"][b], c["new"]
    if c["page"]:
        pages = x["table"][b, :-(-t // c["page"])].long()
        rows = lambda a: a[pages].transpose(0, 1).reshape((c["h_kv"], -1) + a.shape[3:])[:, :t]  # noqa: E731
    else:
        rows = lambda a: a[b, :, :t]  # noqa: E731
    new, new_s = _stored_keys(x["k"][b], c["keys"])
    k = torch.cat((rows(x["k_cache"]), new), 1)
    v = torch.cat((rows(x["v_cache"]), x["v"][b]), 1).double()
    if c["keys"] == "bf16":
        return k.double(), v
    if c["keys"] == "int4":
        k = torch.stack((k & 15, k >> 4), -1).reshape(k.shape[:-1] + (c["r"],)).to(torch.int16)
        k = torch.where(k > 7, k - 16, k)
    scale = torch.cat((rows(x["k_scale"]), new_s), 1)
    return k.double() * scale.double()[..., None], v


def _scores(q, k, r, shift):
    """Masked scores of q [n, r] against k [t, r]; shift: query i sees keys 0 .. shift + i (None: all)."""
    s = q @ k.T / math.sqrt(r)
    if shift is not None:
        i = torch.arange(q.shape[0], device=DEV)[:, None] + shift
        s.masked_fill_(torch.arange(k.shape[0], device=DEV)[None, :] > i, -math.inf)
    return s


def exact(case, seed):
    c, x = case, _inputs(case, seed)
    B, hq, hkv, r, dv, n = (c[f] for f in ("batch", "h_q", "h_kv", "r", "d_v", "new"))
    G = hq // hkv
    out = torch.empty((B, hq, n, dv), dtype=torch.float64, device=DEV)
    f64 = dict(dtype=torch.float64, device=DEV)
    if c["kind"] == "train":
        lse = torch.empty((B, hq, n), **f64)
        dq, dk, dval = (torch.zeros((B, h, n, w), **f64) for h, w in ((hq, r), (hkv, r), (hkv, dv)))
    for b in range(B):
        if c["kind"] in ("decode", "chunk"):
            kk, vv = _context(c, x, b)
            shift = x["lens"][b] if c["causal"] else None
        else:
            kk, vv, shift = x["k"][b].double(), x["v"][b].double(), 0 if c["causal"] else None
        for h in range(hq):
            q, k, v = x["q"][b, h].double(), kk[h // G], vv[h // G]
            s = _scores(q, k, r, shift)
            m = torch.logsumexp(s, 1)
            p = s.sub_(m[:, None]).exp_()
            out[b, h] = p @ v
            if c["kind"] == "train":
                lse[b, h] = m
                do = x["d_out"][b, h].double()
                ds = p * (do @ v.T - (do * out[b, h]).sum(1, keepdim=True)) / math.sqrt(r)
                dq[b, h] = ds @ k
                dk[b, h // G] += ds.T @ q
                dval[b, h // G] += p.T @ do
    if c["kind"] == "train":
        return {"out": out, "lse": lse, "dq": dq, "dk": dk, "dv": dval}
    # the cache holds inputs and codes: nothing computed in floating point but the scales
    return {"out": out[:, :, 0] if c["kind"] == "decode" else out, "k_cache": None, "v_cache": None,
            "k_scale": None}
