"""A wait of the tensor-core prefill kernel that runs out is visible in the result: the rows it held up are NaN, nothing
hangs, and the device is usable afterwards.  The kernel is compiled here once more, from the same source, with waits of
no polls at all, which all run out at once."""
import ctypes
import os
import shutil
import subprocess

import pytest
import torch

import paper_2405_03917_b200 as cq
from paper_2405_03917_b200 import build

pytestmark = pytest.mark.gpu

WRAPPER = """
#include "cq_prefill.cu"
cudaError_t cq::ensure_dynamic_smem(const void* func, int bytes, int)
{
    return cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}
extern "C" int prefill_no_polls(const void* q, const void* kc, const void* vc, const float* kcb, const float* vcb, const int* lens,
                                float scale, int n_seq, int n_q, int hq, int hkv, int c, long long cap, float* out, void* stream)
{
    cq::Shape sh{};
    sh.n_seq = n_seq; sh.max_tokens = cap; sh.n_blocks = (cap + cq::kTokenBlock - 1) / cq::kTokenBlock;
    sh.n_q_heads = hq; sh.n_kv_heads = hkv; sh.head_dim = 128; sh.c = c; sh.b = 8;
    sh.G = 128 / c; sh.K = 256; sh.R = hq / hkv; sh.hb = 0; sh.block_bytes = sh.G * 16;
    if (!cq::prefill_mma_supported(sh)) return -1;
    return cq::launch_prefill((const __half*)q, (const uint8_t*)kc, (const uint8_t*)vc, kcb, vcb, lens, scale, sh, n_q, out, false,
                              (cudaStream_t)stream);
}
"""


@pytest.fixture(scope="module")
def no_polls(tmp_path_factory):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc on this machine")
    d = tmp_path_factory.mktemp("prefill")
    src, so = d / "no_polls.cu", d / "no_polls.so"
    src.write_text(WRAPPER)
    subprocess.check_call([nvcc, *build.NVCC_FLAGS, "-DCQ_PREFILL_POLLS=0", "-I" + build.CSRC, "-shared", "-Xlinker", "-Bsymbolic", "-o", str(so), str(src)])
    return ctypes.CDLL(str(so)).prefill_no_polls


@pytest.mark.parametrize("c,n_q,hq,hkv,lens", [(8, 40, 8, 2, [300, 17]), (4, 3, 2, 2, [64]), (2, 130, 4, 4, [500, 130])])
def test_rows_of_a_wait_that_ran_out_are_nan(no_polls, c, n_q, hq, hkv, lens):
    D, n, cap = 128, len(lens), max(lens)
    g = torch.Generator().manual_seed(c)
    q = torch.randn(n, n_q, hq, D, generator=g).half().cuda()
    cb = torch.randn(hkv, D // c, 256, c, generator=g).cuda()
    codes = torch.randint(0, 256, (cq.cq_codes_bytes(n, cap, hkv, D, c, 8),), generator=g, dtype=torch.uint8).cuda()
    sl = torch.tensor(lens, dtype=torch.int32, device="cuda")
    want = cq.cq_prefill_attn(q, codes, codes, cb, cb, sl, 0.1, c, 8, cap)
    out = torch.zeros_like(want)
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    st = no_polls(ptr(q), ptr(codes), ptr(codes), ptr(cb), ptr(cb), ptr(sl), ctypes.c_float(0.1), n, n_q, hq, hkv, c,
                  ctypes.c_longlong(cap), ptr(out), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    torch.cuda.synchronize()
    rows_per_cta = 256 // (hq // hkv)
    for s, length in enumerate(lens):
        for first in range(0, n_q, rows_per_cta):
            last = min(first + rows_per_cta, n_q) - 1
            block = out[s, first:last + 1]
            if length - n_q + last < 0:                  # nothing to attend in all of the CTA: it waits for nothing
                assert (block == 0).all()
            else:
                assert torch.isnan(block).all()
    # the library itself is unharmed
    assert torch.equal(cq.cq_prefill_attn(q, codes, codes, cb, cb, sl, 0.1, c, 8, cap), want)
