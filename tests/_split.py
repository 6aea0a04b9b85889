"""The launchers' split rules (csrc/split.h), compiled with the host compiler and called here."""

import ctypes
import functools
import os
import subprocess
import tempfile

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_04427_gb300",
                    "csrc")
SOURCE = """
#include "split.h"
extern "C" int prefill_shares(long long kv_tiles, int most) { return tk::prefill_shares(kv_tiles, most); }
extern "C" int prefill_cluster(long long pairs, long long kv_tiles, int num_sms) {
  return tk::prefill_cluster(pairs, kv_tiles, num_sms);
}
extern "C" int backward_split(int batch, int h_q, int h_kv, int seq, int causal, int num_sms) {
  return tk::backward_split(batch, h_q, h_kv, seq, causal != 0, num_sms);
}
extern "C" int backward_tile_major(int batch, int h_q, int seq, int r, int d_v) {
  return tk::backward_tile_major(batch, h_q, seq, r, d_v);
}
"""


@functools.lru_cache(maxsize=1)
def rules():
    with tempfile.TemporaryDirectory() as d:
        src, lib = os.path.join(d, "rules.cpp"), os.path.join(d, "rules.so")
        with open(src, "w") as f:
            f.write(SOURCE)
        subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I", CSRC, src, "-o", lib], check=True)
        L = ctypes.CDLL(lib)
    L.prefill_shares.argtypes = [ctypes.c_longlong, ctypes.c_int]
    L.prefill_cluster.argtypes = [ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int]
    return L


def sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


def tiles(n):
    """128-row tiles of n rows."""
    return -(-n // 128)


def prefill_pairs(B, hq, S):
    return B * hq * -(-tiles(S) // 2)
