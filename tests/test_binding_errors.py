"""Tensors without memory of their own (under tracing, under vmap) and a missing device end in a Python exception, never in
the end of the process: the calls run in a process of their own."""
import subprocess
import sys

import pytest
import torch

PROLOGUE = """
import torch
import paper_2405_03917_b200 as cq
from torch._subclasses.fake_tensor import FakeTensorMode
D, C, B, H, CAP = 128, 8, 8, 2, 16

def args(make):
    half = lambda *s: make(*s, dtype=torch.float16)
    byte = lambda n: make(n, dtype=torch.uint8)
    book = make(H, D // C, 256, C, dtype=torch.float32)
    lens = make(1, dtype=torch.int32)
    out = make(1, H, D, dtype=torch.float32)
    codes = byte(100000), byte(100000)
    return half, book, lens, out, codes, byte(1 << 20)

def calls(make):
    half, cb, sl, out, (kc, vc), ws = args(make)
    rope = make(CAP, D // 2, dtype=torch.float32)
    return {
        "encode": lambda: cq.cq_encode(half(1, 4, H, D), cb, C, B, kc, CAP),
        "encode_kv": lambda: cq.cq_encode_kv(half(1, 4, H, D), half(1, 4, H, D), cb, cb, C, B, kc, vc, CAP),
        "decode_attn": lambda: cq.cq_decode_attn(half(1, H, D), kc, vc, cb, cb, sl, 0.1, C, B, CAP, out, ws),
        "decode_attn_rope": lambda: cq.cq_decode_attn_rope(half(1, H, D), kc, vc, cb, cb, sl, rope, rope, 0.1, C, B, CAP, out=out, workspace=ws),
        "prefill_attn": lambda: cq.cq_prefill_attn(half(1, 1, H, D), kc, vc, cb, cb, sl, 0.1, C, B, CAP, make(1, 1, H, D, dtype=torch.float32)),
        "decode_step": lambda: cq.cq_decode_step(half(1, H, D), half(1, H, D), half(1, H, D), sl, kc, vc, cb, cb, 0.1, C, B, CAP, out, ws),
    }
"""

FAKE = PROLOGUE + """
with FakeTensorMode():
    make = lambda *s, dtype: torch.empty(*s, dtype=dtype, device="cuda")
    for name, call in calls(make).items():
        try:
            call()
        except Exception as e:
            print("raised", name, flush=True)
"""

VMAP = PROLOGUE + """
x = torch.randn(3, 1, 4, H, D, device="cuda").half()
make = lambda *s, dtype: torch.zeros(*s, dtype=dtype, device="cuda")
half, cb, sl, out, (kc, vc), ws = args(make)
try:
    torch.vmap(lambda x: cq.cq_encode(x, cb, C, B, kc, CAP))(x)
except Exception as e:
    print("raised", type(e).__name__)
"""


def run(code):
    return subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)


@pytest.mark.skipif(torch.cuda.is_available(), reason="the current stream is there: no error to raise")
def test_no_device_raises():
    r = run(FAKE)
    names = ["encode", "encode_kv", "decode_attn", "decode_attn_rope", "prefill_attn", "decode_step"]
    assert r.returncode == 0 and r.stdout.split("\n")[:-1] == ["raised " + n for n in names], (r.returncode, r.stdout, r.stderr[-500:])


@pytest.mark.gpu
def test_vmap_raises():
    r = run(VMAP)
    assert r.returncode == 0 and r.stdout.startswith("raised"), (r.returncode, r.stdout, r.stderr[-500:])
