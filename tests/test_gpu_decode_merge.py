"""Decode over pairs whose partials many CTAs share, and over caches of small pages.

A (sequence, kv head) pair is split over CTAs in slices of about four 64-token
chunks.  Its partials are merged by one warp (few) or by five (many); both
sides of that line and every layout of a lane's pieces (G * d_v from 64 to
1024) are covered, with an output of either type.  Pages of 16 and 32 tokens
put several boxes into one chunk, whose column blocks (two of them for r = 128
bf16 keys and d_v = 128) are laid out per box.
"""

import math

import pytest
import torch

from _helpers import f64, parity, parity_bf16, require_gpu
from oracle import attention as oa
from paper_2603_04427_gb300 import binding as tb
from paper_2603_04427_gb300 import inputs

pytestmark = pytest.mark.gpu

# (h_q, h_kv, r, d_v, lengths, page_size, bf16 output)
CASES = [
    (8, 8, 16, 64, [5000], 0, False),         # G * d_v = 64: 20 partials
    (4, 4, 32, 64, [64 * 17], 0, False),      # one-chunk slices, 17 partials
    (8, 4, 32, 64, [4990, 1], 0, True),       # 128
    (8, 4, 64, 128, [7001], 0, False),        # 256
    (16, 4, 32, 128, [7000, 65], 0, True),    # 512
    (16, 4, 128, 128, [7000, 3], 16, False),
    (16, 2, 64, 128, [9000, 640], 0, False),  # 1024
    (8, 1, 128, 128, [9001], 32, True),
    (12, 12, 16, 64, [270, 33], 16, False),   # few partials, ragged last page
    (8, 2, 64, 128, [129, 47, 500], 32, False),
]


@pytest.mark.parametrize("hq,hkv,r,dv,lens,page,bf16", CASES)
def test_merge_and_small_pages(hq, hkv, r, dv, lens, page, bf16):
    require_gpu()
    B, cap = len(lens), (max(lens) + 15) // 16 * 16
    kn = inputs.normal_bf16((B, hkv, cap, r), 81, device="cuda")
    vn = inputs.normal_bf16((B, hkv, cap, dv), 82, device="cuda")
    if page:
        table, n_pages = inputs.paged_layout(lens, page, seed=83)
        cache = tb.ThinKeyCache.allocate(B, hq, hkv, r, dv, page_size=page, num_pages=n_pages, page_table=table)
        for b, n in enumerate(lens):   # only what the context holds; the rest stays NaN
            for t in range(0, n, page):
                m, pg = min(page, n - t), int(table[b, t // page])
                cache.k[pg].fill_(float("nan")), cache.v[pg].fill_(float("nan"))
                cache.k[pg, :, :m], cache.v[pg, :, :m] = kn[b, :, t:t + m], vn[b, :, t:t + m]
    else:
        cache = tb.ThinKeyCache.allocate(B, hq, hkv, r, dv, capacity=cap, fill=float("nan"))
        for b, n in enumerate(lens):
            cache.k[b, :, :n], cache.v[b, :, :n] = kn[b, :, :n], vn[b, :, :n]
    q = inputs.normal_bf16((B, hq, r), 84, device="cuda")
    sl = torch.tensor(lens, dtype=torch.int32, device="cuda")
    ws = tb.decode_workspace(cache.desc, max(lens))
    outs = []
    for _ in range(2):   # the second call finds the counters as the first left them
        out = torch.full((B, hq, dv), float("nan"), device="cuda",
                         dtype=torch.bfloat16 if bf16 else torch.float32)
        tb.tk_attn_decode(cache, q, sl, max(lens), out, ws)
        outs.append(out)
    assert tb.tk_get_device_error() == 0
    assert torch.equal(outs[0], outs[1])
    ref = oa.attention_decode(f64(q), f64(kn), f64(vn), lens, 1 / math.sqrt(r))
    (parity_bf16 if bf16 else parity)(f64(outs[0]), ref, what=f"decode {hq}/{hkv} r={r} d_v={dv} {lens}")
