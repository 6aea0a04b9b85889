"""Prefill of few query tiles: the kv tiles of a pair split over a cluster.

Launches with at most half as many query tile pairs as SMs, and at least ten kv
tiles, split a pair's kv tiles over 2, 4 or 8 CTAs, which merge through
distributed shared memory.  Covered:
every split, shares without a tile for query tile A or for any (causal pairs
early in the sequence), rows that a share sees nothing of (contexts that end
off a tile boundary), every output type, key format, r / d_v staging layout,
and that the result is the unsplit kernel's (tk_attn_forward's) but for the
rounding of the softmax weights.  The split of each case (on 152 SMs) is asserted.
"""

import math

import pytest
import torch

from _helpers import f64, parity, parity_bf16, require_gpu
from _split import prefill_pairs, rules, sms, tiles
from oracle import attention as oa
from oracle import cache as oc
from paper_2603_04427_gb300 import binding as tb
from paper_2603_04427_gb300 import inputs

pytestmark = pytest.mark.gpu


def _assert_split(B, hq, S, tokens, split):
    require_gpu()
    if sms() == 152:
        assert rules().prefill_cluster(prefill_pairs(B, hq, S), tiles(tokens), 152) == split


@pytest.mark.parametrize("B,hq,hkv,S,r,dv,bf16,causal,split", [
    (1, 4, 4, 1281, 32, 128, False, True, 2),    # 24 pairs, 11 kv tiles
    (1, 2, 1, 1700, 16, 64, True, True, 4),      # 14 kv tiles
    (1, 1, 1, 3100, 64, 128, False, True, 8),    # 25 kv tiles
    (1, 1, 1, 4097, 32, 128, True, True, 8),     # 33 kv tiles
    (1, 2, 2, 1300, 128, 128, False, False, 2),  # full attention
    (1, 1, 1, 1921, 128, 64, False, False, 4),   # a last query tile of one row
])
def test_prefill_split(B, hq, hkv, S, r, dv, bf16, causal, split):
    _assert_split(B, hq, S, S, split)
    q = inputs.normal_bf16((B, hq, S, r), 91, device="cuda")
    k = inputs.normal_bf16((B, hkv, S, r), 92, device="cuda")
    v = inputs.normal_bf16((B, hkv, S, dv), 93, device="cuda")
    out = torch.full((B, hq, S, dv), float("nan"), device="cuda", dtype=torch.bfloat16 if bf16 else torch.float32)
    tb.tk_attn_prefill(q, k, v, out, causal=causal)
    assert tb.tk_get_device_error() == 0
    ref = oa.attention_prefill(f64(q), f64(k), f64(v), 1 / math.sqrt(r), causal=causal)
    (parity_bf16 if bf16 else parity)(f64(out), ref, what=f"split prefill S={S} r={r} d_v={dv}")
    whole, lse = torch.empty((B, hq, S, dv), device="cuda"), torch.empty((B, hq, S), device="cuda")
    tb.tk_attn_forward(q, k, v, whole, lse, causal=causal)
    (parity_bf16 if bf16 else parity)(f64(out), f64(whole), what=f"split against unsplit S={S} r={r} d_v={dv}")


@pytest.mark.parametrize("hq,hkv,S,lens,r,dv,page,keys,split", [
    (4, 2, 23, [3001, 1], 32, 128, 0, "bf16", 8),     # one query tile; the second sequence not split
    (4, 1, 130, [2000, 777], 64, 64, 16, "bf16", 4),  # two tiles, the second of two rows
    (2, 2, 300, [1111], 32, 128, 64, "int8", 4),      # hi + lo keys
    (2, 1, 200, [1500], 128, 128, 0, "int4", 4),      # scales in the softmax
    (8, 2, 256, [130, 1200], 16, 128, 128, "bf16", 4),
])
def test_chunk_split(hq, hkv, S, lens, r, dv, page, keys, split):
    _assert_split(len(lens), hq, S, max(lens) + S, split)
    B, L = len(lens), max(lens) + S
    cap = (L + 15) // 16 * 16
    kw = dict(k_int8=keys == "int8", k_int4=keys == "int4")
    if page:
        table, n = inputs.paged_layout([x + S for x in lens], page, seed=95)
        cache = tb.ThinKeyCache.allocate(B, hq, hkv, r, dv, page_size=page, num_pages=n, page_table=table, **kw)
    else:
        cache = tb.ThinKeyCache.allocate(B, hq, hkv, r, dv, capacity=cap, **kw)
    k = inputs.normal_bf16((B, hkv, L, r), 96, device="cuda")
    v = inputs.normal_bf16((B, hkv, L, dv), 97, device="cuda")
    q = inputs.normal_bf16((B, hq, S, r), 98, device="cuda")
    zero = torch.zeros(B, dtype=torch.int32, device="cuda")
    sl = torch.tensor(lens, dtype=torch.int32, device="cuda")
    kn = torch.stack([k[b, :, n:n + S] for b, n in enumerate(lens)])
    vn = torch.stack([v[b, :, n:n + S] for b, n in enumerate(lens)])
    if not page:
        tb.tk_kv_append(cache, k[:, :, :max(lens)].contiguous(), v[:, :, :max(lens)].contiguous(), zero)
    else:   # sequence by sequence: only its own tokens have pages
        for b, n in enumerate(lens):
            one = tb.ThinKeyCache(type(cache.desc).from_buffer_copy(cache.desc), cache.k, cache.v, cache.k_scale,
                                  cache.page_table[b:b + 1].contiguous())
            one.desc.batch = 1
            tb.tk_kv_append(one, k[b:b + 1, :, :n].contiguous(), v[b:b + 1, :, :n].contiguous(), zero[:1])
    out = torch.full((B, hq, S, dv), float("nan"), device="cuda")
    tb.tk_attn_prefill_cached(cache, q, kn, vn, sl, L, out)
    assert tb.tk_get_device_error() == 0
    kq = f64(k)
    if keys == "int8":
        code, scale = oc.quantize_int8_per_token(kq)
        kq = code * scale[..., None].astype(float)
    elif keys == "int4":
        code, scale = oc.quantize_int4_per_token(kq)
        kq = code * scale[..., None].astype(float)
    G = hq // hkv
    for b, n in enumerate(lens):
        for h in range(hq):
            ref = oa.attention_head(f64(q[b, h]), kq[b, h // G, :n + S], f64(v[b, h // G, :n + S]),
                                    1 / math.sqrt(r), causal_offset=n)
            parity(f64(out[b, h]), ref, what=f"split chunk b={b} h={h} {keys} r={r} page={page}")


@pytest.mark.parametrize("where", ["share", "diagonal", "value"])
def test_a_nan_is_not_lost_in_the_merge(where):
    """Rows that see a NaN key or value are NaN whichever CTA of the cluster sees it, and only those.

    S = 3100, one head: 13 pairs of query tiles over clusters of 8 CTAs, so the first pair's
    two kv tiles lie in CTAs 3 and 7: of CTA 7's keys row 128 sees key 128 alone.  A value
    whose weight underflows to 0 is NaN times 0 in one CTA's sums, so it is in the merge.
    """
    require_gpu()
    S, r, dv = 3100, 32, 64
    q = inputs.normal_bf16((1, 1, S, r), 101, device="cuda")
    k = inputs.normal_bf16((1, 1, S, r), 102, device="cuda")
    v = inputs.normal_bf16((1, 1, S, dv), 103, device="cuda")
    if where == "share":
        first = 128
        k[0, 0, first] = float("nan")
    elif where == "diagonal":
        first = 2943     # the last row of a tile
        k[0, 0, first, 3] = float("nan")
    else:
        # keys 0 .. 127 score 400 below the others: e^-400 is 0 in fp32
        first = 0
        q[..., 0], k[..., 0], k[0, 0, :128, 0] = 40.0, 10.0, -46.5
        v[0, 0, 5] = float("nan")
    out = torch.empty((1, 1, S, dv), device="cuda")
    tb.tk_attn_prefill(q, k, v, out)
    assert tb.tk_get_device_error() == 0
    bad = torch.isnan(out[0, 0]).any(1)
    assert bad[first:].all(), f"rows {torch.nonzero(~bad[first:])[:4].flatten().tolist()} past {first} are finite"
    assert not bad[:first].any()


@pytest.mark.parametrize("B,hq,hkv,S,lens,r,dv,page,keys,shares", [
    (1, 4, 2, 300, [500], 32, 128, 0, "bf16", 1),         # one CTA of eight has work
    (1, 4, 2, 300, [0], 32, 128, 0, "bf16", 1),           # the plain prefill
    (1, 2, 1, 2000, [0], 16, 64, 0, "bf16", 4),           # the plain prefill, split itself
    (1, 4, 4, 200, [1400], 64, 64, 64, "bf16", 4),        # four of eight
    (2, 8, 2, 130, [3000, 77], 32, 128, 16, "int8", 8),   # eight beside one, in one launch
    (1, 4, 1, 100, [600], 128, 128, 0, "int4", 1),
])
def test_the_bound_does_not_change_the_result(B, hq, hkv, S, lens, r, dv, page, keys, shares):
    """A loose max_seq_len launches clusters of up to eight CTAs over short contexts: each
    sequence is split by its own length, so the bits are those of a tight bound (and, for an
    empty cache, of the plain prefill)."""
    tight, loose = max(lens) + S, 16384
    _assert_split(B, hq, S, tight, shares)
    _assert_split(B, hq, S, loose, 8)
    g = dict(device="cuda")
    kw = dict(k_int8=keys == "int8", k_int4=keys == "int4")
    if page:
        table, n = inputs.paged_layout([loose] * B, page, seed=111)
        cache = tb.ThinKeyCache.allocate(B, hq, hkv, r, dv, page_size=page, num_pages=n, page_table=table, **kw)
    else:
        cache = tb.ThinKeyCache.allocate(B, hq, hkv, r, dv, capacity=loose, **kw)
    L = max(lens)
    q, k, v = (inputs.normal_bf16(s, 112 + i, **g) for i, s in enumerate(
        ((B, hq, S, r), (B, hkv, L + S, r), (B, hkv, L + S, dv))))
    kn, vn = k[:, :, L:].contiguous(), v[:, :, L:].contiguous()
    if L:
        tb.tk_kv_append(cache, k[:, :, :L].contiguous(), v[:, :, :L].contiguous(),
                        torch.zeros(B, dtype=torch.int32, **g))
    sl = torch.tensor(lens, dtype=torch.int32, **g)
    outs = []
    for bound in (tight, 4096, loose):
        out = torch.full((B, hq, S, dv), float("nan"), **g)
        tb.tk_attn_prefill_cached(cache, q, kn, vn, sl, bound, out)
        assert tb.tk_get_device_error() == 0
        outs.append(out)
    if L == 0:
        out = torch.full((B, hq, S, dv), float("nan"), **g)
        tb.tk_attn_prefill(q, kn, vn, out)
        outs.append(out)
    assert torch.isfinite(outs[0]).all()
    for out in outs[1:]:
        assert torch.equal(outs[0], out)
