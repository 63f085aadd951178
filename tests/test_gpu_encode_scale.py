"""Codes do not depend on the magnitude of the data: every encode kernel against the generic one, bit for bit, on
inputs and codebooks scaled by powers of two (channels of standard deviation 64 down to 2^-20), on vectors far outside
the codebook, and on codebooks that fp16 operands cannot carry."""
import pytest
import torch

import paper_2405_03917_b200 as cq

pytestmark = pytest.mark.gpu

D = 128
VARIANTS = [0, 2, 4]


def encode(x, cb, c, b, variant):
    n, h = x.shape[1], x.shape[2]
    codes = torch.zeros(cq.cq_codes_bytes(1, n, h, D, c, b), dtype=torch.uint8, device="cuda")
    cq.cq_encode(x, cb, c, b, codes, n, variant=variant)
    return codes


def draw(seed, n, h, c, b):
    g = torch.Generator().manual_seed(seed)
    x = torch.randn(1, n, h, D, generator=g)
    cb = torch.randn(h, D // c, 1 << b, c, generator=g)
    return x, cb


def check(x, cb, c, b, what):
    x, cb = x.to(torch.float16).cuda().contiguous(), cb.float().cuda().contiguous()
    want = encode(x, cb, c, b, 1)
    for variant in VARIANTS:
        if variant == 4 and b != 8:
            continue
        differ = int((encode(x, cb, c, b, variant) != want).sum())
        assert differ == 0, f"{what}, variant {variant}: {differ} of {want.numel()} bytes differ"


@pytest.mark.parametrize("b", [8, 9, 10])
@pytest.mark.parametrize("c", [2, 4, 8])
def test_codes_at_every_scale(c, b):
    x, cb = draw(100 * c + b, 1500, 2, c, b)
    for e in (6, 0, -5, -8, -11, -13, -16, -20):
        check(x * 2.0 ** e, cb * 2.0 ** e, c, b, f"scale 2^{e}")


@pytest.mark.parametrize("c", [2, 4, 8])
def test_codes_of_groups_of_different_scale(c):
    # every group of a head has its own magnitude, vectors and codebook alike
    x, cb = draw(7 + c, 700, 3, c, 8)
    s = 2.0 ** (torch.arange(D // c) % 17 - 12.0)
    check(x * s.repeat_interleave(c), cb * s[None, :, None, None], c, 8, "scale per group")


@pytest.mark.parametrize("c", [2, 4, 8])
def test_codes_of_vectors_outside_the_codebook(c):
    # up to 2^15 times as far out as any centroid: the scaled squares overflow fp16
    x, cb = draw(17 + c, 700, 2, c, 8)
    far = 2.0 ** (torch.arange(700) % 16.0)
    check(x * far[None, :, None, None] * 2.0 ** -6, cb * 2.0 ** -6, c, 8, "vectors far out")


@pytest.mark.parametrize("c", [2, 4, 8])
def test_codes_of_codebooks_fp16_cannot_carry(c):
    x, cb = draw(27 + c, 700, 2, c, 8)
    G = D // c
    cb[:, 0] = 0.0                       # nothing but zeros
    cb[:, 1] *= 1e-30                    # squares vanish
    cb[:, 2, 17] = 3e5                   # one centroid beyond fp16
    cb[:, 3, 255] = 250.0                # its square nearly is
    cb[:, 4 % G, 1:] = cb[:, 4 % G, :1]  # equal centroids: the lowest index
    cb[:, 5 % G, 128:] = cb[:, 5 % G, :128]
    cb[:, 6 % G] *= 2.0 ** -11
    cb[:, 6 % G, 3] = 8.0                # one large centroid among small ones
    check(x, cb, c, 8, "odd codebooks")
    check(x * 2.0 ** -11, cb, c, 8, "odd codebooks, small vectors")


def test_codes_of_the_plane_kernel_at_every_scale():
    # enough vectors for the kernel that looks up the centroids near a point of the plane
    x, cb = draw(5, 100000, 1, 2, 8)
    for e in (0, -8, -14, -20):
        check(x * 2.0 ** e, cb * 2.0 ** e, 2, 8, f"scale 2^{e}")
