"""The native argument checks (csrc/py_binding.cpp) and the Python checks behind them.

On the CPU: whatever is not the plain case is left to the Python checks, which
raise.  On the GPU: both routes make the same call, and arguments that the
Python checks refuse are refused with the native route in front of them.
"""

import torch
import pytest

from _helpers import require_gpu
from paper_2603_04427_gb300 import binding as tb
from paper_2603_04427_gb300 import build as tbuild

B, HQ, HKV, R, DV, S, CAP = 2, 4, 2, 32, 64, 40, 96


class NoNative:
    """Every call is left to the Python checks."""

    def __getattr__(self, name):
        return lambda *a: None


def _args(device):
    g = torch.Generator(device=device).manual_seed(7)

    def bf(*s):
        return torch.randn(s, generator=g, device=device).bfloat16()

    cache = tb.ThinKeyCache.allocate(B, HQ, HKV, R, DV, capacity=CAP, k_int8=True, device=device)
    cache.k.random_(-127, 128, generator=g)
    cache.v.normal_(generator=g)
    cache.k_scale.uniform_(0.01, 0.03, generator=g)
    lens = torch.tensor([9, 30], dtype=torch.int32, device=device)
    q, k, v, do = bf(B, HQ, S, R), bf(B, HKV, S, R), bf(B, HKV, S, DV), bf(B, HQ, S, DV)
    q1, k1, v1 = bf(B, HQ, R), bf(B, HKV, R), bf(B, HKV, DV)
    f = dict(device=device)
    out, outb, out1 = torch.zeros(B, HQ, S, DV, **f), do.clone(), torch.zeros(B, HQ, DV, **f)
    lse, dq = torch.zeros(B, HQ, S, **f), torch.zeros(B, HQ, S, R, **f)
    dk, dv = torch.zeros(B, HKV, S, R, **f), torch.zeros(B, HKV, S, DV, **f)
    ws = torch.zeros(8 << 20, dtype=torch.uint8, device=device)
    return {
        "kv_append": (tb.tk_kv_append, [cache, k, v, lens], [cache.k, cache.v, cache.k_scale]),
        "decode": (tb.tk_attn_decode, [cache, q1, lens, CAP, out1, ws], [out1]),
        "decode_noalloc": (tb.tk_attn_decode_noalloc, [cache, q1, lens, CAP, out1], [out1]),
        "decode_append": (tb.tk_attn_decode_append, [cache, q1, k1, v1, lens, CAP, out1, ws],
                          [out1, cache.k, cache.v, cache.k_scale]),
        "prefill": (tb.tk_attn_prefill, [q, k, v, out], [out]),
        "forward": (tb.tk_attn_forward, [q, k, v, outb, lse], [outb, lse]),
        "backward": (tb.tk_attn_backward, [q, k, v, outb, do, lse, dq, dk, dv, ws], [dk, dv]),
        "prefill_cached": (tb.tk_attn_prefill_cached, [cache, q, k, v, lens, CAP, out],
                           [out, cache.k, cache.v]),
    }


NAMES = ("kv_append", "decode", "decode_noalloc", "decode_append", "prefill", "forward", "backward",
         "prefill_cached")


@pytest.mark.parametrize("name", NAMES)
def test_host_tensors_are_left_to_the_python_checks(name):
    tbuild.build()
    fn, args, _ = _args("cpu")[name]
    assert getattr(tb._fast(), name)(*args) is None          # too few arguments as well
    with pytest.raises(ValueError, match="CUDA tensor"):
        fn(*args)


def test_a_module_built_for_another_torch_is_rebuilt_and_not_loaded(monkeypatch):
    """_tkpy.so is compiled against torch's C++ tensors: after a change of torch (or of Python) it
    counts as out of date and is refused, where its accessors could read another layout.  The C
    library, which needs neither, still loads and is not built again."""
    tbuild.build()
    assert tbuild.up_to_date()
    monkeypatch.setattr(tbuild, "py_tag", lambda: "another")
    assert not tbuild.up_to_date() and tbuild.lib_up_to_date()
    monkeypatch.setattr(tb, "_native", None)
    monkeypatch.setattr(tb, "_lib", None)
    assert tb.tk_status_string(tb.TK_OK) == "TK_OK"
    with pytest.raises(RuntimeError, match="not built for this Python and torch"):
        tb._fast()


@pytest.mark.gpu
@pytest.mark.parametrize("name", NAMES)
def test_both_routes_make_the_same_call(name, monkeypatch):
    require_gpu()
    got = []
    for native in (True, False):
        fn, args, outs = _args("cuda")[name]
        if not native:
            monkeypatch.setattr(tb, "_native", NoNative())
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        kw = {} if name == "kv_append" else {"scale": 0.3}
        if name == "prefill_cached":
            kw["workspace"] = tb.prefill_cached_workspace(args[0], CAP)
        fn(*args, stream=stream, **kw)
        torch.cuda.synchronize()
        assert tb.tk_get_device_error() == 0
        got.append(outs)
    for a, b in zip(*got):
        assert torch.equal(a, b)
        assert a.float().abs().sum() > 0


@pytest.mark.gpu
@pytest.mark.parametrize("name", NAMES)
def test_what_the_python_checks_refuse_is_refused(name):
    require_gpu()
    fn, args, _ = _args("cuda")[name]
    for i, t in enumerate(args):
        if not isinstance(t, torch.Tensor):
            continue
        bad = [t.double(), t.cpu()]
        # (sequence lengths and workspaces have no shape to check)
        if t.dtype in (torch.bfloat16, torch.float32):
            bad += [t.transpose(0, 1), t[..., :-1].contiguous()]
        for x in bad:
            with pytest.raises((TypeError, ValueError)):
                fn(*args[:i], x, *args[i + 1:])
    torch.cuda.synchronize()
    assert tb.tk_get_device_error() == 0
