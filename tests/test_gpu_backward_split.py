"""Backward by the number of CTAs per key tile (csrc/split.h: backward_split, tile order).

Split: the CTAs of a cluster share a key tile's query tiles and add up dK and dV
through distributed shared memory.  Covered: clusters of 2, 4 and 8, CTAs without a
tile (the last key tiles of a causal sequence), a ragged last key tile, every (r, d_v)
layout of the partial results, and launches of more CTAs than SMs.  dK and dV are
summed in a fixed order: two calls agree bit for bit.

Not split: one CTA per key tile, what large launches use.  Covered: every (r, d_v),
causal and full, groups of query heads, and both CTA orders.

The split of each case (on 152 SMs) is asserted.
"""

import math

import pytest
import torch

from _helpers import f64, require_gpu
from _split import rules, sms
from oracle import attention as oa
from test_gpu_backward import _case, _grad_parity

pytestmark = pytest.mark.gpu


def _assert_split(B, hq, hkv, S, causal, split):
    require_gpu()
    if sms() == 152:
        assert rules().backward_split(B, hq, hkv, S, causal, 152) == split


def _check(case, kv_heads, r, causal, what):
    """The gradients of these (sequence, kv head) pairs against the oracle."""
    q, k, v, do, lse, dq, dk, dvv = case
    G = q.shape[1] // k.shape[1]
    for b, g in kv_heads:
        one, grp = (slice(b, b + 1), slice(g, g + 1)), (slice(b, b + 1), slice(g * G, (g + 1) * G))
        rq, rk, rv = oa.attention_backward(f64(q[grp]), f64(k[one]), f64(v[one]), f64(do[grp]), 1 / math.sqrt(r),
                                           causal)
        for got, ref, name in ((dq[grp], rq, "dq"), (dk[one], rk, "dk"), (dvv[one], rv, "dv")):
            _grad_parity(f64(got), ref, f"{name} b={b} g={g} {what}")


@pytest.mark.parametrize("B,hq,hkv,S,r,dv,causal,split", [
    (1, 8, 1, 300, 32, 128, True, 8),      # 3 key tiles, 24 query tiles of the first
    (1, 1, 1, 1921, 16, 64, True, 8),      # 16 key tiles, the last with one query tile: CTAs without tiles
    (1, 16, 2, 138, 64, 128, True, 8),     # 4 key tiles, the second of ten keys
    (1, 8, 1, 257, 128, 128, True, 8),
    (1, 4, 1, 1000, 64, 64, False, 8),     # 8 key tiles, 32 query tiles each
    (2, 8, 1, 260, 16, 128, True, 8),
    (1, 8, 2, 520, 128, 64, True, 8),
    (1, 4, 4, 1030, 32, 64, True, 4),      # 36 key tiles
    (1, 32, 8, 528, 32, 128, True, 4),     # 40 key tiles, 160 CTAs on 152 SMs
    (2, 4, 2, 300, 128, 128, False, 2),
    (8, 16, 4, 140, 64, 64, True, 2),      # 64 key tiles
    (8, 32, 4, 520, 32, 128, False, 2),    # 160 key tiles, 320 CTAs
])
def test_backward_split(B, hq, hkv, S, r, dv, causal, split):
    _assert_split(B, hq, hkv, S, causal, split)
    case = _case(B, hq, hkv, S, r, dv, causal, seed=61)
    again = _case(B, hq, hkv, S, r, dv, causal, seed=61)
    assert torch.equal(case[6], again[6]) and torch.equal(case[7], again[7])
    pairs = [(b, g) for b in range(B) for g in range(hkv)]
    _check(case, pairs if len(pairs) <= 8 else [pairs[0], pairs[-1]], r, causal, f"{hq}/{hkv} S={S} r={r} d_v={dv}")


@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("r,dv", [(r, dv) for r in (16, 32, 64, 128) for dv in (64, 128)])
def test_backward_one_cta_per_key_tile(r, dv, causal):
    """B=4, 16/16 heads, S=300: 192 key tiles, the last of 44 keys."""
    _assert_split(4, 16, 16, 300, causal, 1)
    case = _case(4, 16, 16, 300, r, dv, causal, seed=200 + r + dv)
    _check(case, [(0, 0), (1, 9), (3, 15)], r, causal, f"r={r} d_v={dv} causal={causal}")


@pytest.mark.parametrize("r,dv", [(16, 64), (64, 64), (64, 128), (128, 128)])
def test_backward_one_cta_per_key_tile_of_a_group(r, dv):
    """B=8, 16/8 heads: two query heads per kv head."""
    _assert_split(8, 16, 8, 300, True, 1)
    case = _case(8, 16, 8, 300, r, dv, True, seed=300 + r + dv)
    _check(case, [(0, 0), (7, 7)], r, True, f"G=2 r={r} d_v={dv}")


@pytest.mark.parametrize("r,causal", [(32, True), (64, False)])
def test_backward_head_by_head(r, causal):
    """Q and dO of 32 heads and 2 sequences of 2700 tokens exceed the part of L2 that the key
    tile order is for: the CTAs go head by head."""
    B, H, S, dv = 2, 32, 2700, 128
    _assert_split(B, H, H, S, causal, 1)
    assert not rules().backward_tile_major(B, H, S, r, dv) and rules().backward_tile_major(4, 16, 300, 128, 128)
    case = _case(B, H, H, S, r, dv, causal, seed=400 + r)
    _check(case, [(0, 1), (1, 31)], r, causal, f"S={S} r={r}")
