"""Decode steps whose kernel ahead of the attention appends the tokens and, for few queries, builds the tables of all sequences
(cq_decode_tables.cu), against cq_encode_kv and cq_decode_attn, whose CTAs build their tables: the entries are the same sums in
the same order, so the results agree as two calls do."""
import mmap

import numpy as np
import pytest
import torch

import paper_2405_03917_b200 as cq

pytestmark = pytest.mark.gpu
DEV = "cuda"
SPREAD = 2e-6          # two calls of one kernel differ by no more (the weight unit depends on warp timing)


def make(c, b, n_seq, n_q, n_kv, D, cap, seed):
    g = torch.Generator().manual_seed(seed)
    books = [torch.randn(n_kv, D // c, 1 << b, c, generator=g).to(DEV) for _ in range(2)]
    x = [torch.randn(n_seq, cap, n_kv, D, generator=g).half().to(DEV) for _ in range(2)]
    codes = [torch.zeros(cq.cq_codes_bytes(n_seq, cap, n_kv, D, c, b), dtype=torch.uint8, device=DEV) for _ in range(2)]
    for i in range(2):
        cq.cq_encode(x[i], books[i], c, b, codes[i], cap)
    q = torch.randn(n_seq, n_q, D, generator=g).half().to(DEV)
    new = [torch.randn(n_seq, n_kv, D, generator=g).half().to(DEV) for _ in range(2)]
    return q, codes, books, new


def lengths(n_seq, cap):
    # empty, one token, both sides of a block's end, a warp's share, one below capacity, capacity
    edge = [0, 1, 15, 16, 17, min(cap, 129), cap - 1, cap]
    return torch.tensor([edge[(i * 5) % 8] if i % 3 else (i * 37) % (cap + 1) for i in range(n_seq)], dtype=torch.int32, device=DEV)


def close(got, want):
    got, want = got.double().cpu().numpy(), want.double().cpu().numpy()
    assert np.abs(got - want).max() <= SPREAD * max(1.0, np.abs(want).max())


# (c, b, n_seq, query heads, KV heads): tables ahead (at most 2^17 entries) and not, every width of a CTA, one vector per warp
# of the append up to more than one warp's share (16), more queries of a KV head than a CTA of the tables takes (32)
SHAPES = [(2, 8, 4, 3, 3), (2, 8, 33, 4, 2), (4, 8, 1, 1, 1), (4, 8, 5, 3, 3), (4, 8, 7, 8, 2), (4, 8, 37, 2, 2), (8, 8, 1, 1, 1), (8, 8, 9, 6, 1),
          (8, 8, 34, 1, 1), (8, 8, 34, 4, 2), (8, 8, 17, 8, 2), (8, 10, 4, 2, 2), (8, 10, 6, 8, 2), (8, 10, 15, 1, 1)]


@pytest.mark.parametrize("scale", [None, 40.0])          # 40: entries beyond what a half holds, the tables are scaled
@pytest.mark.parametrize("c,b,n_seq,n_q,n_kv", SHAPES)
def test_step(c, b, n_seq, n_q, n_kv, scale):
    cap, D = 700, 128
    q, codes, books, new = make(c, b, n_seq, n_q, n_kv, D, cap, 3 * c + b + n_seq)
    if scale:
        q = q * 64
    scale = scale or D ** -0.5
    lens = lengths(n_seq, cap)
    ref = [x.clone() for x in codes]
    cq.cq_encode_kv(new[0][:, None].contiguous(), new[1][:, None].contiguous(), *books, c, b, *ref, cap, seq_offsets=lens)
    want = cq.cq_decode_attn(q, *ref, *books, torch.clamp(lens + 1, max=cap), scale, c, b, cap)
    got = cq.cq_decode_step(q, *new, lens, *codes, *books, scale, c, b, cap)
    assert torch.equal(codes[0], ref[0]) and torch.equal(codes[1], ref[1])
    close(got, want)


@pytest.mark.parametrize("n_q", [1, 4])
def test_contexts_split_over_ctas(n_q):
    c, b, n_seq, D, cap = 8, 8, 4, 128, 9000
    q, codes, books, new = make(c, b, n_seq, n_q, 1, D, cap, 1)
    lens = torch.tensor([9000, 0, 4096, 2047], dtype=torch.int32, device=DEV)
    ref = [x.clone() for x in codes]
    cq.cq_encode_kv(new[0][:, None].contiguous(), new[1][:, None].contiguous(), *books, c, b, *ref, cap, seq_offsets=lens)
    want = cq.cq_decode_attn(q, *ref, *books, torch.clamp(lens + 1, max=cap), D ** -0.5, c, b, cap)
    got = cq.cq_decode_step(q, *new, lens, *codes, *books, D ** -0.5, c, b, cap)
    assert torch.equal(codes[0], ref[0]) and torch.equal(codes[1], ref[1])
    close(got, want)


@pytest.mark.parametrize("c,b", [(4, 8), (8, 10)])
def test_a_workspace_without_room_for_tables(c, b):
    n_seq, D, cap = 4, 128, 300
    q, codes, books, new = make(c, b, n_seq, 2, 2, D, cap, 2)
    lens = lengths(n_seq, cap)
    full = cq.cq_decode_step_workspace_bytes(n_seq, 2, 2, D, c, b, cap)
    assert full > n_seq * 2 * (D // c) * (1 << b) * 4
    ws = torch.empty(full - 256, dtype=torch.uint8, device=DEV)
    other = [x.clone() for x in codes]
    want = cq.cq_decode_step(q, *new, lens, *other, *books, D ** -0.5, c, b, cap)
    got = cq.cq_decode_step(q, *new, lens, *codes, *books, D ** -0.5, c, b, cap, workspace=ws)
    assert torch.equal(codes[0], other[0]) and torch.equal(codes[1], other[1])
    close(got, want)


def back_to_back(c, b, n_seq, n_q, n_kv, cap, steps):
    """Steps with no launch of anything else between them, so that each kernel may start before the one ahead has ended, against the
    same steps with a wait between them.  One workspace, caches that are carried on, another query and other new tokens each time."""
    D = 128
    _, codes, books, _ = make(c, b, n_seq, n_q, n_kv, D, cap, c + b + n_seq)
    g = torch.Generator().manual_seed(n_seq)
    q = torch.randn(steps, n_seq, n_q, D, generator=g).half().to(DEV)
    new = torch.randn(2, steps, n_seq, n_kv, D, generator=g).half().to(DEV)
    lens = torch.clamp(lengths(n_seq, cap), max=cap - steps) + torch.arange(steps, dtype=torch.int32, device=DEV)[:, None]
    ws = torch.empty(cq.cq_decode_step_workspace_bytes(n_seq, n_q, n_kv, D, c, b, cap), dtype=torch.uint8, device=DEV)

    def run(wait):
        kv = [x.clone() for x in codes]
        out = torch.zeros(steps, n_seq, n_q, D, device=DEV)
        args = [(q[i], new[0, i], new[1, i], lens[i], *kv, *books, D ** -0.5, c, b, cap, out[i], ws) for i in range(steps)]
        torch.cuda.synchronize()
        for a in args:
            cq.cq_decode_step(*a)
            if wait:
                torch.cuda.synchronize()
        return out, kv
    (w, kw), (a, ka) = run(True), run(False)
    assert torch.equal(ka[0], kw[0]) and torch.equal(ka[1], kw[1])
    close(a, w)


# tables ahead; the append ahead alone, with the attention launched at its end (an SM to each CTA) and at its start (an SM to each CTA of
# both; several waves; one CTA fills an SM); split contexts with a merge, with tables and without;
# CQ-8c10b with tables and with an append of its own
@pytest.mark.parametrize("c,b,n_seq,n_q,n_kv,cap", [(4, 8, 3, 2, 2, 64), (8, 8, 1, 1, 1, 1024), (8, 8, 8, 8, 8, 300), (8, 8, 8, 6, 2, 300), (4, 8, 12, 32, 32, 200), (2, 8, 9, 8, 8, 120),
                                                    (8, 8, 4, 1, 1, 9000), (8, 8, 3, 16, 16, 9000), (8, 10, 4, 2, 2, 200), (8, 10, 8, 16, 16, 200)])
def test_steps_right_behind_one_another(c, b, n_seq, n_q, n_kv, cap):
    back_to_back(c, b, n_seq, n_q, n_kv, cap, 12)


@pytest.mark.parametrize("c,b,n_seq,n_q,n_kv", [(8, 8, 3, 8, 2), (4, 8, 2, 3, 3), (4, 8, 3, 24, 24), (8, 10, 2, 2, 1), (4, 4, 2, 2, 2)])
@pytest.mark.parametrize("how", ["pinned", "one block", "off by two bytes", "pageable", "pageable result"])
def test_host_buffers(c, b, n_seq, n_q, n_kv, how):
    # pinned buffers are read and written by kernels (16 bytes at a time where they are aligned), others are copied
    D, cap = 128, 200
    q, codes, books, new = make(c, b, n_seq, n_q, n_kv, D, cap, 9 + c)
    lens = torch.arange(5, 5 + 60 * n_seq, 60, dtype=torch.int32)
    other = [x.clone() for x in codes]
    want = cq.cq_decode_step(q, *new, lens.to(DEV), *other, *books, D ** -0.5, c, b, cap)
    parts = [q, *new]
    skip = 1 if how == "off by two bytes" else 0
    pin = (lambda t: t) if how == "pageable" else (lambda t: t.pin_memory())
    if how == "pinned":
        host = [pin(p.cpu()) for p in parts]
    else:
        block = pin(torch.empty(sum(p.numel() for p in parts) + skip, dtype=torch.float16))
        host, at = [], skip
        for p in parts:
            host.append(block[at:at + p.numel()].view(p.shape).copy_(p.cpu()))
            at += p.numel()
    out = torch.empty(n_seq, n_q, D) if "pageable" in how else torch.empty(n_seq, n_q, D).pin_memory()
    ws = torch.empty(cq.cq_decode_step_host_workspace_bytes(n_seq, n_q, n_kv, D, c, b, cap), dtype=torch.uint8, device=DEV)
    got = cq.cq_decode_step_host(*host, pin(lens), *codes, *books, D ** -0.5, c, b, cap, out, ws)
    assert torch.equal(codes[0], other[0]) and torch.equal(codes[1], other[1])
    close(got, want)


@pytest.mark.parametrize("c,b,n_seq,n_q,n_kv", [(4, 8, 4, 4, 4), (8, 8, 2, 32, 8), (8, 8, 16, 8, 8), (8, 10, 16, 2, 1)])
def test_host_buffers_side_by_side(c, b, n_seq, n_q, n_kv):
    # pinned memory of three registrations that lie back to back (whole pages each): not one copy
    D, cap = 128, 200
    q, codes, books, new = make(c, b, n_seq, n_q, n_kv, D, cap, 5 + c)
    lens = torch.arange(5, 5 + 10 * n_seq, 10, dtype=torch.int32)
    other = [x.clone() for x in codes]
    want = cq.cq_decode_step(q, *new, lens.to(DEV), *other, *books, D ** -0.5, c, b, cap)
    parts = [q, *new]
    block = torch.frombuffer(mmap.mmap(-1, sum(2 * p.numel() for p in parts)), dtype=torch.float16)
    rt, registered, host, at = torch.cuda.cudart(), [], [], 0
    out = torch.empty(n_seq, n_q, D).pin_memory()
    ws = torch.empty(cq.cq_decode_step_host_workspace_bytes(n_seq, n_q, n_kv, D, c, b, cap), dtype=torch.uint8, device=DEV)
    try:
        for p in parts:
            host.append(block[at:at + p.numel()].view(p.shape).copy_(p.cpu()))
            at += p.numel()
            assert host[-1].data_ptr() % mmap.PAGESIZE == 0 and 2 * p.numel() % mmap.PAGESIZE == 0
            assert int(rt.cudaHostRegister(host[-1].data_ptr(), 2 * p.numel(), 0)) == 0
            registered.append(host[-1].data_ptr())
        got = cq.cq_decode_step_host(*host, lens.pin_memory(), *codes, *books, D ** -0.5, c, b, cap, out, ws)
    finally:
        for ptr in registered:
            assert int(rt.cudaHostUnregister(ptr)) == 0
    assert torch.equal(codes[0], other[0]) and torch.equal(codes[1], other[1])
    close(got, want)


@pytest.mark.parametrize("part", ["q", "k_new", "v_new", "out"])
def test_host_buffers_of_which_only_the_beginning_is_pinned(part):
    # one page of two or more is registered: no kernel reaches the rest, the buffers are copied (or the copy is refused)
    c, b, n_seq, n_q, n_kv, D, cap = 8, 8, 4, 8, 8, 128, 200
    q, codes, books, new = make(c, b, n_seq, n_q, n_kv, D, cap, 31)
    lens = torch.arange(5, 5 + 10 * n_seq, 10, dtype=torch.int32)
    other = [x.clone() for x in codes]
    want = cq.cq_decode_step(q, *new, lens.to(DEV), *other, *books, D ** -0.5, c, b, cap)
    host = {"q": q.cpu(), "k_new": new[0].cpu(), "v_new": new[1].cpu(), "out": torch.empty(n_seq, n_q, D)}
    size = host[part].numel() * host[part].element_size()
    assert size >= 2 * mmap.PAGESIZE
    block = torch.frombuffer(mmap.mmap(-1, size), dtype=host[part].dtype).view(host[part].shape)
    block.copy_(host[part])
    host = {name: block if name == part else x.pin_memory() for name, x in host.items()}
    ws = torch.empty(cq.cq_decode_step_host_workspace_bytes(n_seq, n_q, n_kv, D, c, b, cap), dtype=torch.uint8, device=DEV)
    rt = torch.cuda.cudart()
    assert int(rt.cudaHostRegister(block.data_ptr(), mmap.PAGESIZE, 0)) == 0
    try:
        got = cq.cq_decode_step_host(host["q"], host["k_new"], host["v_new"], lens.pin_memory(), *codes, *books, D ** -0.5, c, b, cap,
                                     host["out"], ws)
        close(got, want)
    except cq.CQError:
        cq.lib().cudaGetLastError()              # (the refused copy's: torch would report it at its next launch)
    finally:
        torch.cuda.synchronize()
        assert int(rt.cudaHostUnregister(block.data_ptr())) == 0


@pytest.mark.parametrize("n_seq,cap", [(2, 64), (20, 64), (3, 9000), (14, 9000)])
def test_steps_with_the_append_inside_right_behind_one_another(n_seq, cap):
    # decode_pair_kernel lets the next kernel go ahead at its start or at its epilogue, by its CTAs (16, 160; 96 and 448 of split
    # contexts)
    back_to_back(8, 8, n_seq, 32, 8, cap, 8)
