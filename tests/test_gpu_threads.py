"""Calls of the Python binding let other Python threads run while they wait inside the CUDA runtime."""
import threading
import time

import pytest
import torch

import paper_2405_03917_b200 as cq

pytestmark = pytest.mark.gpu

D, C, B, H = 128, 8, 8, 1


def calls():
    """name -> a call of one launch or more on small buffers."""
    dev = "cuda"
    G = D // C
    cap = 64
    x = torch.randn(1, 1, H, D, device=dev).half()
    q = torch.randn(1, H, D, device=dev).half()
    q4 = q.view(1, 1, H, D)
    cb = torch.randn(H, G, 1 << B, C, device=dev)
    kc, vc = (torch.zeros(cq.cq_codes_bytes(1, cap, H, D, C, B), dtype=torch.uint8, device=dev) for _ in range(2))
    sl = torch.full((1,), 8, dtype=torch.int32, device=dev)
    out, out4 = torch.empty(1, H, D, device=dev), torch.empty(1, 1, H, D, device=dev)
    ws = torch.empty(cq.cq_decode_step_workspace_bytes(1, H, H, D, C, B, cap), dtype=torch.uint8, device=dev)
    rope = torch.ones(cap, D // 2, device=dev)
    return {
        "encode": lambda: cq.cq_encode(x, cb, C, B, kc, cap),
        "encode_kv": lambda: cq.cq_encode_kv(x, x, cb, cb, C, B, kc, vc, cap),
        "decode_attn": lambda: cq.cq_decode_attn(q, kc, vc, cb, cb, sl, 0.1, C, B, cap, out, ws),
        "decode_attn_rope": lambda: cq.cq_decode_attn_rope(q, kc, vc, cb, cb, sl, rope, rope, 0.1, C, B, cap, out=out, workspace=ws),
        "prefill_attn": lambda: cq.cq_prefill_attn(q4, kc, vc, cb, cb, sl, 0.1, C, B, cap, out4),
        "decode_step": lambda: cq.cq_decode_step(q, x[0], x[0], sl, kc, vc, cb, cb, 0.1, C, B, cap, out, ws),
    }


@pytest.mark.parametrize("name", ["encode", "encode_kv", "decode_attn", "decode_attn_rope", "prefill_attn", "decode_step"])
def test_full_launch_queue_stops_no_other_thread(name):
    call = calls()[name]
    call()
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    times = []

    def work():
        with torch.cuda.stream(stream):
            for _ in range(4000):                     # more than the launch queue takes: the later calls wait for it
                t = time.perf_counter()
                call()
                times.append(time.perf_counter() - t)

    with torch.cuda.stream(stream):
        torch.cuda._sleep(1_500_000_000)              # keeps the stream busy for three quarters of a second or so
    th = threading.Thread(target=work)
    gap, last = 0.0, time.perf_counter()              # (the first calls may fill the queue before this thread runs again)
    th.start()
    while th.is_alive():
        now = time.perf_counter()
        gap, last = max(gap, now - last), now
        time.sleep(0.001)
    gap = max(gap, time.perf_counter() - last)
    th.join()
    torch.cuda.synchronize()
    longest = max(times)
    assert longest > 0.2, f"the launch queue took every call at once (longest {longest:.3f} s): the test needs more of them"
    assert gap < 0.5 * longest, f"another thread stood still for {gap:.3f} s while a call waited {longest:.3f} s"
