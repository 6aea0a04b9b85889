"""Backward of few key tiles: a key tile's query tiles shared by a cluster.

Launches with at most half as many key tiles as SMs split a key tile's query
tiles over 2, 4 or 8 CTAs, which add up dK and dV through distributed shared
memory.  Covered: every split, CTAs without a tile (the last key tiles of a
causal sequence), a ragged last key tile, and every (r, d_v) layout of the
partial results.  dK and dV are summed in a fixed order: two calls agree bit
for bit.
"""

import math

import pytest
import torch

from _helpers import f64, require_gpu
from oracle import attention as oa
from test_gpu_backward import _case, _grad_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,hq,hkv,S,r,dv,causal", [
    (1, 8, 1, 300, 32, 128, True),      # 3 key tiles, 24 tiles of the first: split 4
    (1, 1, 1, 1921, 16, 64, True),      # 16 key tiles, the last with one tile: split 4, CTAs without tiles
    (1, 16, 2, 138, 64, 128, True),     # 4 key tiles, the second of ten keys
    (1, 8, 1, 257, 128, 128, True),
    (1, 4, 1, 1000, 64, 64, False),     # 8 key tiles, 32 tiles each: split 8
    (2, 8, 1, 260, 16, 128, True),
    (1, 8, 2, 520, 128, 64, True),
    (1, 4, 4, 1030, 32, 64, True),      # 36 key tiles: split 2
])
def test_backward_split(B, hq, hkv, S, r, dv, causal):
    require_gpu()
    q, k, v, do, lse, dq, dk, dvv = _case(B, hq, hkv, S, r, dv, causal, seed=61)
    again = _case(B, hq, hkv, S, r, dv, causal, seed=61)
    assert torch.equal(dk, again[6]) and torch.equal(dvv, again[7])
    rq, rk, rv = oa.attention_backward(f64(q), f64(k), f64(v), f64(do), 1 / math.sqrt(r), causal)
    for got, ref, what in ((dq, rq, "dq"), (dk, rk, "dk"), (dvv, rv, "dv")):
        _grad_parity(f64(got), ref, f"{what} {hq}/{hkv} S={S} r={r} d_v={dv}")
