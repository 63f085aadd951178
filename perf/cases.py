"""Timed cases of the CQ library: the calls that a serving or a calibration program makes.

A case is a dict of plain values:

    path       "step"       cq_decode_step: append the new token's codes, attend over the cache
               "host_step"  cq_decode_step_host: the same from pinned host buffers
               "attention"  cq_decode_attn: attention over a cache that is complete
               "rope"       cq_decode_attn_rope: attention over codes of keys taken before RoPE
               "prefill"    cq_prefill_attn: causal attention of a prompt chunk over the cache
               "encode"     cq_encode_kv: key and value vectors of a prompt into the cache
               "learn"      cq_learn_centroids: centroids of one calibration tensor
    c, b       channels per group and bits per code ("CQ-<c>c<b>b"); head_dim: channels per head
    n_seq, n_q_heads, n_kv_heads
    min_len, max_len   context lengths: spread evenly over [min_len, max_len], dealt out by the seed
    capacity   tokens that a sequence's cache has room for
    n_new      new tokens per sequence (prefill, encode); encode appends them at ragged positions
    n_vec, n_iters, weighted   calibration vectors, k-means iterations, Eq. 6 instead of Eq. 5

Inputs follow the library's synthetic recipe: x = A z + mu + 0.1 eps per head, low rank, keys with four
outlier channels (mean +8, std x5), fp16; codebooks are further draws of the same source, queries N(0, 1).
Caches hold the codes that cq_encode gives for such vectors.
"""
from __future__ import annotations

import math

import torch

import paper_2405_03917_b200 as cq

DEV = "cuda"


def _decode(name, path, c, b, n_seq, n_q, n_kv, min_len, max_len, capacity, head_dim=128, **more):
    return dict(name=name, path=path, c=c, b=b, head_dim=head_dim, n_seq=n_seq, n_q_heads=n_q, n_kv_heads=n_kv,
                min_len=min_len, max_len=max_len, capacity=capacity, **more)


def listed():
    return [
        # the smallest call: one sequence, one head (configuration 0); launch and host cost
        _decode("step_8c8b_one_head", "step", 8, 8, 1, 1, 1, 1024, 1024, 1024),
        # a decode step of a Llama-2-7B-shaped layer at 2 bits per channel (configuration 1)
        _decode("step_4c8b_mha", "step", 4, 8, 16, 32, 32, 4096, 4096, 4096),
        # a decode step of a Mistral-7B-shaped GQA layer at 1 bit per channel, the headline (configuration 2)
        _decode("step_8c8b_gqa", "step", 8, 8, 64, 32, 8, 16384, 16384, 16384),
        # one layer of the Llama-2-13B-shaped step, long ragged contexts, the largest cache (configuration 4)
        _decode("step_8c8b_mha_ragged", "step", 8, 8, 32, 40, 40, 8192, 32768, 32768),
        # the paper's best quantiser near one bit: codes wider than a byte
        _decode("step_8c10b_mha", "step", 8, 10, 16, 32, 32, 8192, 8192, 8192),
        # one interactive user with a long conversation, driven from host memory, cache partly filled
        _decode("host_step_8c8b_gqa_one_user", "host_step", 8, 8, 1, 32, 8, 20011, 20011, 32768),
        # a model with 64-channel heads, mixed short and long conversations
        _decode("attention_4c8b_head64_ragged", "attention", 4, 8, 12, 32, 8, 301, 4001, 4096, head_dim=64),
        # encoding whole prompts at 4 bits per channel, the largest encode (configuration 3)
        _decode("encode_2c8b_prompts", "encode", 2, 8, 8, 32, 32, 0, 0, 8192, n_new=8192),
        # a scheduler's chunk: a few sequences, an odd number of tokens, appended at ragged positions
        _decode("encode_8c8b_chunk", "encode", 8, 8, 5, 32, 8, 17, 1500, 2048, n_new=333),
        # attention of a prompt chunk over an 8192-token cache, Mistral-7B-shaped GQA layer
        _decode("prefill_8c8b_gqa", "prefill", 8, 8, 4, 32, 8, 8192, 8192, 8192, n_new=2048),
        # decode attention where the cache holds keys from before RoPE, as the paper quantises them
        _decode("rope_4c8b_mha", "rope", 4, 8, 16, 32, 32, 4096, 4096, 4096),
        # learning the centroids of one Llama-2-7B-shaped key tensor with the paper's calibration size (16 x 2048
        # tokens), weights (Eq. 6) and 100 iterations; the largest call
        dict(name="learn_8c8b", path="learn", c=8, b=8, head_dim=128, n_kv_heads=32, n_vec=32768, n_iters=100, weighted=True),
    ]


def _log(rng, lo, hi):
    """An integer in [lo, hi], uniform over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# (tokens x sequences x heads x groups) that the largest listed case of a path goes through: what a drawn one may cost
_MOST_CODES = {"step": 16 * 20480 * 32 * 40, "host_step": 16 * 16384 * 64 * 8, "rope": 32 * 4096 * 16 * 32}


def draw(rng):
    path = rng.choice(["step", "step", "step", "host_step", "attention", "encode", "prefill", "rope", "learn"])
    if path == "learn":
        return dict(path=path, c=rng.choice([4, 8]), b=8, head_dim=128, n_kv_heads=_log(rng, 1, 32),
                    n_vec=_log(rng, 1000, 32768), n_iters=rng.randint(5, 100), weighted=rng.random() < 0.5)
    if path == "encode":
        c, b = rng.choice([(2, 8), (4, 8), (8, 8), (8, 10)])
        n_kv = rng.choice([1, 8, 32, 40])
        n_seq = _log(rng, 1, 64)
        most = (8 * 8192 * 32 // (8 if b > 8 else 1)) // (n_seq * n_kv)
        n_new = _log(rng, 1, min(8192, most))
        first = _log(rng, 1, 4096)
        return _drawn(path, c, b, n_seq, n_kv, n_kv, 0, first, first + n_new, n_new=n_new)
    if path == "prefill":
        n_q, n_kv = rng.choice([(32, 8), (32, 32), (8, 8)])
        n_seq = _log(rng, 1, 4)
        n_new = _log(rng, 16, 2048)
        last = _log(rng, n_new, 8192)
        first = rng.randint(n_new, last)
        return _drawn(path, rng.choice([2, 4, 8]), 8, n_seq, n_q, n_kv, first, last, last, n_new=n_new)
    head_dim = 128
    if path == "attention":
        head_dim = 64
        c, b = rng.choice([(4, 8), (8, 8)])
        n_q, n_kv = rng.choice([(32, 8), (12, 12)])
        n_seq, last = _log(rng, 1, 12), _log(rng, 64, 4096)
    else:
        c, b = rng.choice([(4, 8), (8, 8)] if path == "rope" else [(2, 8), (4, 8), (8, 8), (8, 10)])
        n_q, n_kv = rng.choice([(32, 32), (32, 8), (40, 40), (8, 1), (1, 1)])
        n_seq = _log(rng, 1, 64)
        most = _MOST_CODES[path] // (n_seq * (n_q if path == "rope" or b > 8 else n_kv) * (head_dim // c))
        last = min(_log(rng, 64, 32768), most)
    first = rng.choice([last, rng.randint(max(1, last // 4), last)])
    room = rng.choice([last, min(32768, 2 * last)])
    return _drawn(path, c, b, n_seq, n_q, n_kv, first, last, room, head_dim=head_dim)


def _drawn(*shape, **more):
    case = _decode("", *shape, **more)
    del case["name"]
    return case


# ------------------------------------------------------------------------------------------ inputs

class _Source:
    """Key or value vectors of every head of a layer."""

    def __init__(self, gen, n_heads, head_dim, outliers):
        rank = head_dim // 4
        self.gen, self.n_heads, self.head_dim, self.rank = gen, n_heads, head_dim, rank
        self.A = torch.randn(n_heads, rank, head_dim, generator=gen, device=DEV) / rank ** 0.5
        self.mu = 0.5 * torch.randn(n_heads, 1, head_dim, generator=gen, device=DEV)
        self.gain = torch.ones(n_heads, 1, head_dim, device=DEV)
        self.shift = torch.zeros(n_heads, 1, head_dim, device=DEV)
        if outliers:
            at = torch.rand(n_heads, 1, head_dim, generator=gen, device=DEV).argsort(-1)[..., :4]
            self.gain.scatter_(-1, at, 5.0)
            self.shift.scatter_(-1, at, 8.0)

    def draw(self, n):
        """n fp32 vectors of every head: (n_heads, n, head_dim)."""
        z = torch.randn(self.n_heads, n, self.rank, generator=self.gen, device=DEV)
        x = torch.randn(self.n_heads, n, self.head_dim, generator=self.gen, device=DEV).mul_(0.1)
        return x.baddbmm_(z, self.A).mul_(self.gain).add_(self.mu + self.shift)

    def tokens(self, n_seq, n):
        """fp16 (n_seq, n, n_heads, head_dim)."""
        x = self.draw(n_seq * n).view(self.n_heads, n_seq, n, self.head_dim)
        return x.permute(1, 2, 0, 3).to(torch.float16, memory_format=torch.contiguous_format)

    def codebook(self, c, b):
        x = self.draw(1 << b).view(self.n_heads, 1 << b, self.head_dim // c, c)
        return x.permute(0, 2, 1, 3).contiguous()


def _lengths(case, gen, extra=0):
    """The case's lengths, the same ones for every seed, dealt out to the sequences by the seed."""
    n, lo, hi = case["n_seq"], case["min_len"], case["max_len"]
    lens = [hi - (hi - lo) * i // max(1, n - 1) + extra for i in range(n)]
    deal = torch.rand(n, generator=gen, device=DEV).argsort().cpu()
    return torch.tensor(lens, dtype=torch.int32)[deal].contiguous()


def _cache(case, src, cb):
    """A code buffer whose every position holds the code of a vector of the source."""
    n_seq, cap, n_kv, D, c, b = (case[k] for k in ("n_seq", "capacity", "n_kv_heads", "head_dim", "c", "b"))
    codes = torch.zeros(cq.cq_codes_bytes(n_seq, cap, n_kv, D, c, b), dtype=torch.uint8, device=DEV)
    per_seq = codes.numel() // n_seq
    run = max(1, min(n_seq, (1 << 22) // (cap * n_kv)))
    for s in range(0, n_seq, run):
        n = min(run, n_seq - s)
        # the sequences lie one after the other
        cq.cq_encode(src.tokens(n, cap), cb, c, b, codes[s * per_seq:(s + n) * per_seq], cap)
    return codes


def prepare(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    D, c, b, n_kv, path = case["head_dim"], case["c"], case["b"], case["n_kv_heads"], case["path"]
    G = D // c
    k_src, v_src = _Source(gen, n_kv, D, True), _Source(gen, n_kv, D, False)
    st = dict(case)
    if path == "learn":
        n = case["n_vec"]
        st["x"] = k_src.tokens(1, n)[0]
        # stand-ins for the squared gradients of Eq. 6
        st["weights"] = torch.randn(n, n_kv, G, generator=gen, device=DEV).square_() if case["weighted"] else None
        st["uniforms"] = torch.rand(n_kv, G, 1 << b, generator=gen, device=DEV, dtype=torch.float64)
        return st

    st["k_cb"], st["v_cb"] = k_src.codebook(c, b), v_src.codebook(c, b)
    n_seq, cap, n_q = case["n_seq"], case["capacity"], case["n_q_heads"]
    if path == "encode":
        st["k"], st["v"] = k_src.tokens(n_seq, case["n_new"]), v_src.tokens(n_seq, case["n_new"])
        nbytes = cq.cq_codes_bytes(n_seq, cap, n_kv, D, c, b)
        st["k_codes"], st["v_codes"] = (torch.zeros(nbytes, dtype=torch.uint8, device=DEV) for _ in range(2))
        st["offsets"] = _lengths(case, gen).to(DEV) if case["max_len"] else None
        return st

    st["k_codes"], st["v_codes"] = _cache(case, k_src, st["k_cb"]), _cache(case, v_src, st["v_cb"])
    st["scale"] = D ** -0.5
    if path == "prefill":
        st["q"] = torch.randn(n_seq, case["n_new"], n_q, D, generator=gen, device=DEV).to(torch.float16)
        st["lens"] = _lengths(case, gen).to(DEV)
        st["out"] = torch.empty(st["q"].shape, dtype=torch.float32, device=DEV)
        return st

    st["q"] = torch.randn(n_seq, n_q, D, generator=gen, device=DEV).to(torch.float16)
    st["out"] = torch.empty(n_seq, n_q, D, dtype=torch.float32, device=DEV)
    shape = (n_seq, n_q, n_kv, D, c, b, cap)
    if path in ("step", "host_step"):
        st["lens"] = _lengths(case, gen, extra=-1).to(DEV)            # cached before the step; it appends one more
        st["k_new"], st["v_new"] = k_src.tokens(n_seq, 1)[:, 0].contiguous(), v_src.tokens(n_seq, 1)[:, 0].contiguous()
        size = cq.cq_decode_step_workspace_bytes if path == "step" else cq.cq_decode_step_host_workspace_bytes
        st["workspace"] = torch.empty(max(256, size(*shape)), dtype=torch.uint8, device=DEV)
        if path == "host_step":
            # query, key and value back to back in one pinned block
            parts = [st[k] for k in ("q", "k_new", "v_new")]
            block = torch.empty(sum(p.numel() for p in parts), dtype=torch.float16).pin_memory()
            for key, p, at in zip(("q", "k_new", "v_new"), parts, (0, parts[0].numel(), parts[0].numel() + parts[1].numel())):
                st[key] = block[at:at + p.numel()].view(p.shape).copy_(p.cpu())
            st["lens"] = st["lens"].cpu().pin_memory()
            st["out"] = torch.empty(n_seq, n_q, D, dtype=torch.float32).pin_memory()
        return st

    st["lens"] = _lengths(case, gen).to(DEV)
    st["workspace"] = torch.empty(max(256, cq.cq_decode_attn_workspace_bytes(*shape)), dtype=torch.uint8, device=DEV)
    if path == "rope":
        angle = torch.arange(cap, dtype=torch.float64, device=DEV)[:, None] * \
            (10000.0 ** (-torch.arange(D // 2, dtype=torch.float64, device=DEV) / (D // 2)))[None, :]
        st["cos"], st["sin"] = torch.cos(angle).float().contiguous(), torch.sin(angle).float().contiguous()
    return st


# ------------------------------------------------------------------------------------------ one pass

def run(st):
    path, c, b = st["path"], st["c"], st["b"]
    if path == "step":
        out = cq.cq_decode_step(st["q"], st["k_new"], st["v_new"], st["lens"], st["k_codes"], st["v_codes"], st["k_cb"], st["v_cb"],
                                st["scale"], c, b, st["capacity"], out=st["out"], workspace=st["workspace"])
        return out, st["k_codes"], st["v_codes"]
    if path == "host_step":
        out = cq.cq_decode_step_host(st["q"], st["k_new"], st["v_new"], st["lens"], st["k_codes"], st["v_codes"], st["k_cb"],
                                     st["v_cb"], st["scale"], c, b, st["capacity"], st["out"], st["workspace"])
        return out, st["k_codes"], st["v_codes"]
    if path == "attention":
        return cq.cq_decode_attn(st["q"], st["k_codes"], st["v_codes"], st["k_cb"], st["v_cb"], st["lens"], st["scale"], c, b,
                                 st["capacity"], out=st["out"], workspace=st["workspace"])
    if path == "rope":
        return cq.cq_decode_attn_rope(st["q"], st["k_codes"], st["v_codes"], st["k_cb"], st["v_cb"], st["lens"], st["cos"],
                                      st["sin"], st["scale"], c, b, st["capacity"], out=st["out"], workspace=st["workspace"])
    if path == "prefill":
        return cq.cq_prefill_attn(st["q"], st["k_codes"], st["v_codes"], st["k_cb"], st["v_cb"], st["lens"], st["scale"], c, b,
                                  st["capacity"], out=st["out"])
    if path == "encode":
        cq.cq_encode_kv(st["k"], st["v"], st["k_cb"], st["v_cb"], c, b, st["k_codes"], st["v_codes"], st["capacity"],
                        seq_offsets=st["offsets"])
        return st["k_codes"], st["v_codes"]
    return cq.cq_learn_centroids(st["x"], st["weights"], st["uniforms"], c, b, st["n_iters"])


# ------------------------------------------------------------------------------------------ what a pass takes

def work(case):
    """Bytes: every input that the call has to read once, every output once.  Flops: the contractions that the
    definition asks for; decode scores and sums count in their table form (one addition per group and side)."""
    D, c, b, n_kv, path = case["head_dim"], case["c"], case["b"], case["n_kv_heads"], case["path"]
    G, K = D // c, 1 << b
    code = (16 + 2 * max(0, b - 8)) / 16 if b > 8 else 1                    # bytes of one code
    books = n_kv * G * K * c * 4
    if path == "learn":
        n = case["n_vec"]
        return {"bytes": n * n_kv * (2 * D + (4 * G if case["weighted"] else 0)) + n_kv * G * K * 8 + books + n_kv * G * 8,
                "flops": n * n_kv * D * K * (3 + 2 * case["n_iters"])}
    n_seq, n_q = case["n_seq"], case["n_q_heads"]
    if path == "encode":
        vectors = 2 * n_seq * case["n_new"] * n_kv
        return {"bytes": vectors * (2 * D + G * code) + 2 * books, "flops": vectors * 2 * D * K}
    n, lo, hi = n_seq, case["min_len"], case["max_len"]
    lens = [hi - (hi - lo) * i // max(1, n - 1) for i in range(n)]
    tokens = sum(lens)
    bytes_ = 2 * tokens * n_kv * G * code + 2 * books
    if path == "prefill":
        m = case["n_new"]
        keys = sum(m * (length - m) + m * (m + 1) // 2 for length in lens)
        return {"bytes": bytes_ + n_seq * m * n_q * D * 6, "flops": 4 * keys * n_q * D}
    bytes_ += n_seq * n_q * D * 6
    flops = 2 * tokens * n_q * G + 4 * n_seq * n_q * D * K
    if path in ("step", "host_step"):
        bytes_ += n_seq * n_kv * (4 * D + 2 * G * code)
        flops += n_seq * n_kv * 6 * D * K
    if path == "rope":
        bytes_ += 2 * max(lens) * (D // 2) * 4
        flops = tokens * (n_kv * 3 * D + n_q * (2 * D + G)) + 2 * n_seq * n_q * D * K
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """Codes are whole numbers and stay the same.  Attention results are fp32 sums; where the path itself computes in
    fewer bits (keys and values from fp16 centroids in prefill and in front of RoPE), what those leave.  Learning:
    fp32 sums decide which of two equally near centroids a vector moves to, and the iterations carry that on."""
    path = case["path"]
    if path == "encode":
        return "exact"
    if path == "learn":
        return {"rel": 1e-2, "max": 0.9}
    if path in ("prefill", "rope"):
        return {"rel": 5e-4, "max": 0.01}
    return {"rel": 1e-5}
