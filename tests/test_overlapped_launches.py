"""Kernels that may be launched ahead of the end of the kernel before them (programmatic stream serialisation) wait for
that end before they read memory: whatever lies ahead in the stream - a k-means update that writes the codebooks, a
caller's kernel - may still be writing.  Checked on the source, and on the GPU for codebooks made right before their use."""
import os
import re

import pytest
import torch

import paper_2405_03917_b200 as cq

CSRC = os.path.join(os.path.dirname(cq.__file__), "csrc")
WAIT = "griddepcontrol.wait"


def kernels():
    """(file, name, text from the parameter list to the end of the file) of every kernel"""
    for f in sorted(os.listdir(CSRC)):
        if f.endswith(".cu"):
            text = open(os.path.join(CSRC, f)).read()
            for m in re.finditer(r"__global__ void(?:\s+__launch_bounds__\((?:[^()]|\([^()]*\))*\))?\s+(\w+)\(", text):
                yield f, m.group(1), text[m.end():]


def early_launches():
    """names of the kernels that are launched with an overlapped_config"""
    names = set()
    for f in os.listdir(CSRC):
        if not f.endswith(".cu"):
            continue
        text = open(os.path.join(CSRC, f)).read()
        for body in re.split(r"\n}\n", text):                  # function by function
            if "= overlapped_config(" in body:
                names |= set(re.findall(r"cudaLaunchKernelEx\(&cfg, (\w+_kernel)\b", body)) | set(re.findall(r"go\((\w+_kernel)\b", body))
    return names


def test_every_early_launch_is_of_a_kernel_that_waits():
    waiting = {name for _, name, text in kernels() if WAIT in text.split("__global__")[0]}
    early = early_launches()
    assert early, "no early launches found: the search no longer fits the source"
    assert early <= waiting
    assert waiting <= early


@pytest.mark.parametrize("file,name,text", [k for k in kernels() if WAIT in k[2].split("__global__")[0]], ids=lambda v: v if isinstance(v, str) and len(v) < 40 else "")
def test_nothing_is_read_before_the_wait(file, name, text):
    depth, end = 1, 0
    while depth:                                                # the end of the parameter list
        depth += {"(": 1, ")": -1}.get(text[end], 0)
        end += 1
    pointers = re.findall(r"\*\s*(?:__restrict__\s+)?(\w+)", text[:end])
    ahead = re.sub(r"//[^\n]*", "", text[end:text.index(WAIT)])
    assert "*reinterpret_cast<const" not in ahead and "ld.global" not in ahead and "__ldg" not in ahead, ahead
    grown = set(pointers)
    for var, expr in re.findall(r"\*\s*(?:__restrict__\s+)?(\w+) = ([^;]*);", ahead):       # pointers made from them
        if any(re.search(rf"\b{p}\b", expr) for p in grown):
            grown.add(var)
    for p in grown:
        assert not re.search(rf"\b{p}\s*\[", ahead), f"{file}: {name} reads {p} ahead of its wait"


@pytest.mark.parametrize("name", ["merge_kernel", "decode_rope_tuned_kernel", "encode_tc_kernel", "encode_few_kernel"])
def test_lets_nothing_go_ahead(name):
    # the CTAs of a kernel launched beside these kernels' are placed unevenly over the SMs, and stay there
    (body,) = [text.split("__global__")[0] for _, kernel, text in kernels() if kernel == name]
    assert WAIT in body and "griddepcontrol.launch_dependents" not in body.split("\ncudaError_t")[0]


D = 128


@pytest.mark.gpu
@pytest.mark.parametrize("c,b", [(2, 8), (4, 9), (8, 10)])
def test_codebooks_written_right_ahead_of_an_append(c, b):
    g = torch.Generator().manual_seed(c + b)
    h, n = 8, 32
    x = torch.randn(1, n, h, D, generator=g).half().cuda()
    books = torch.randn(6, h, D // c, 1 << b, c, generator=g).cuda()
    size = cq.cq_codes_bytes(1, n, h, D, c, b)
    cb = torch.empty_like(books[0])
    want = torch.zeros(6, size, dtype=torch.uint8, device="cuda")
    got = torch.zeros_like(want)
    for i in range(6):
        cq.cq_encode(x, books[i].contiguous(), c, b, want[i], n, variant=1)
    torch.cuda.synchronize()
    for i in range(6):
        torch.mul(books[i], 1.0, out=cb)
        cq.cq_encode(x, cb, c, b, got[i], n)
    assert torch.equal(got, want)


@pytest.mark.gpu
@pytest.mark.parametrize("c", [2, 4, 8])
def test_iterations_over_few_vectors_follow_their_codebooks(c):
    # every assignment reads the codebooks that the update right ahead of it has written
    g = torch.Generator().manual_seed(c)
    x = torch.randn(32, 4, D, generator=g).half().cuda()
    first = torch.randn(4, D // c, 256, c, generator=g).cuda()

    def iterate(wait):
        books = [first]
        for _ in range(4):
            if wait:
                torch.cuda.synchronize()
            books.append(cq.cq_lloyd_step(x, None, books[-1], c, 8)[0])
        return books

    want = iterate(True)
    assert not torch.equal(want[2], want[1])                   # the second iteration still moves centroids
    for a, b in zip(iterate(False), want):
        assert torch.allclose(a, b, rtol=1e-5, atol=1e-6)      # sums of at most 32 fp16 values in fp32, in any order
