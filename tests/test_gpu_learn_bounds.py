"""Iterations of cq_learn_centroids that skip vectors whose nearest centroid cannot have changed (cq_learn_assign.cu) against
iterations that evaluate every vector (cq_lloyd_step)."""
import pytest
import torch

import paper_2405_03917_b200 as cq

pytestmark = pytest.mark.gpu
DEV = "cuda"
D = 128


def vectors(n, heads, seed, scale=1.0):
    g = torch.Generator().manual_seed(seed)
    A = torch.randn(heads, 32, D, generator=g) / 32 ** 0.5
    x = torch.einsum("nhr,hrd->nhd", torch.randn(n, heads, 32, generator=g), A) + 0.1 * torch.randn(n, heads, D, generator=g)
    x = x + 0.5 * torch.randn(heads, D, generator=g)
    x[..., ::31] = 8 + 5 * x[..., ::31]
    return (scale * x).half().contiguous().to(DEV), g


def learn(x, w, u, c, iters):
    return cq.cq_learn_centroids(x, w, u, c, 8, iters)


def plain(x, w, u, c, iters):
    cb, obj = cq.cq_kmeanspp_init(x, w, u, c, 8), None
    for _ in range(iters):
        cb, obj = cq.cq_lloyd_step(x, w, cb, c, 8)
    return cb, obj


def check_next_iteration(x, w, u, c, k):
    """Iteration k + 1 is the full evaluation of the codebooks after k iterations; returns how many centroids it changes.  Both sides
    give every vector to the same centroid (near ties are evaluated exactly by both), so centroids of m members differ by the
    additions of cq_lloyd_step's fp32 sums only: m roundings at most of w x and of w, each 2^-24 of their sum, and one in each
    result."""
    n, heads, _ = x.shape
    G = D // c
    a = learn(x, w, u, c, k)[0] if k else cq.cq_kmeanspp_init(x, w, u, c, 8)
    got, og = learn(x, w, u, c, k + 1)
    want, ow = cq.cq_lloyd_step(x, w, a, c, 8)
    buf = torch.zeros(cq.cq_codes_bytes(1, n, heads, D, c, 8), dtype=torch.uint8, device=DEV)
    cq.cq_encode(x.view(1, n, heads, D), a, c, 8, buf, n)
    codes = cq.cq_codes_to_rowmajor(buf, 1, n, heads, D, c, 8).view(n, heads * G).long()
    members = torch.bincount((codes + 256 * torch.arange(heads * G, device=DEV)).flatten(), minlength=heads * G * 256).view(heads, G, 256)
    top = x.float().abs().view(n, heads, G, c).amax(dim=(0, 3))                          # per problem
    off = (got - want).abs().amax(-1) > (2 * members + 2) * 2.0 ** -24 * top[..., None]
    assert not off.any(), (k, off.nonzero()[:5])
    assert torch.allclose(og, ow, rtol=1e-5)
    return (got != a).any(-1).sum()


# one tile and less, a tile's end, many CTAs to a problem (with few problems a CTA takes 128 or 256 vectors), blocks of 16 that are not whole
@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("c,n,heads", [(8, 300, 2), (8, 1024, 1), (8, 4097, 1), (4, 333, 2), (4, 2047, 1), (4, 9001, 1)])
def test_the_first_iterations_are_those_of_full_evaluation(c, n, heads, weighted):
    x, g = vectors(n, heads, c + n)
    w = torch.randn(n, heads, D // c, generator=g).square().to(DEV) if weighted else None
    u = torch.rand(heads, D // c, 256, generator=g, dtype=torch.float64).to(DEV)
    for k in (0, 1, 4):
        check_next_iteration(x, w, u, c, k)


# Problems enough that a CTA takes 4096 vectors, 32 steps of 128, and lists them in two rounds; the last CTA of a problem has 904 (5000
# vectors), 1807 (9999), or the range's last block of 16 is not whole (4090).  30: most vectors are skipped; 31: and are again.
@pytest.mark.parametrize("c,n,heads,weighted", [(4, 5000, 32, True), (4, 5000, 32, False), (8, 9999, 32, True), (8, 4090, 80, False)])
def test_iterations_of_large_calls_are_those_of_full_evaluation(c, n, heads, weighted):
    x, g = vectors(n, heads, c + n)
    w = torch.randn(n, heads, D // c, generator=g).square().to(DEV) if weighted else None
    u = torch.rand(heads, D // c, 256, generator=g, dtype=torch.float64).to(DEV)
    moved = [check_next_iteration(x, w, u, c, k) for k in (0, 1, 2, 5, 12, 30, 31)]
    assert 0 < moved[-1] < moved[1]
    assert torch.equal(learn(x, w, u, c, 32)[0], learn(x, w, u, c, 32)[0])                           # whole-number sums: no order of additions shows


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -9])
@pytest.mark.parametrize("c,n,heads,weighted", [(8, 700, 2, True), (8, 1500, 1, False), (4, 900, 1, True), (4, 600, 2, False)])
def test_what_has_converged_is_a_fixed_point_of_full_evaluation(c, n, heads, weighted, scale):
    # few vectors to a centroid converge within some twenty iterations; a vector wrongly skipped would move a centroid now
    x, g = vectors(n, heads, 7 * c + n, scale)
    w = torch.rand(n, heads, D // c, generator=g).add(0.1).to(DEV) if weighted else None
    u = torch.rand(heads, D // c, 256, generator=g, dtype=torch.float64).to(DEV)
    a, _ = learn(x, w, u, c, 80)
    b, _ = cq.cq_lloyd_step(x, w, a, c, 8)
    assert (a - b).abs().amax() <= 1e-5 * a.abs().amax()
    again, _ = learn(x, w, u, c, 80)
    assert torch.equal(a, again)                       # whole-number sums: no order of additions shows


@pytest.mark.parametrize("c", [4, 8])
def test_weights_over_many_orders_of_magnitude(c):
    n = 1000
    x, g = vectors(n, 1, c)
    w = torch.pow(10.0, -12 * torch.rand(n, 1, D // c, generator=g)).to(DEV)
    w[::7] = 0
    u = torch.rand(1, D // c, 256, generator=g, dtype=torch.float64).to(DEV)
    for k in (0, 2):
        check_next_iteration(x, w, u, c, k)


# Some vectors weigh up to 2^-120 of the others.  The heavy ones are drawn first and are fewer than the centroids, so that light
# ones become centres too and centroids have light members only.  2^-40: ruled out by the smallest weight; 2^-60 and less: sums
# formed anew, 2^-95 and less: the fixed-point sums would hold less than fp32 ones, or nothing.  (200 vectors: fewer than
# centroids, whose rest stays empty; 5000: two CTAs to a problem)
@pytest.mark.parametrize("light", [2.0 ** -40, 2.0 ** -60, 2.0 ** -95, 2.0 ** -120])
@pytest.mark.parametrize("c,n", [(8, 900), (4, 900), (8, 200), (4, 5000)])
def test_centroids_with_light_members_only(c, n, light):
    x, g = vectors(n, 1, 5 * c + n)
    w = torch.rand(n, 1, D // c, generator=g).add(0.5)
    w *= torch.where(torch.arange(n) % (n // 100) == 0, 1.0, light)[:, None, None]
    w[3] = 0
    w = w.to(DEV)
    u = torch.rand(1, D // c, 256, generator=g, dtype=torch.float64).to(DEV)
    for k in (0, 2):
        moved = check_next_iteration(x, w, u, c, k)
        if n > 256 and k == 0:
            assert moved > 0.2 * D // c * 256                      # centroids of light vectors have moved, not only heavy ones


@pytest.mark.parametrize("what", ["inf", "nan", "negative weight", "infinite weight"])
def test_problems_without_bounds(what):
    # the problem that holds the value is evaluated in full; the others keep their result
    n, c, heads = 500, 8, 2
    x, g = vectors(n, heads, 3)
    w = torch.rand(n, heads, D // c, generator=g).add(0.1).to(DEV)
    u = torch.rand(heads, D // c, 256, generator=g, dtype=torch.float64).to(DEV)
    good, _ = learn(x, w, u, c, 4)
    if what in ("inf", "nan"):
        x[17, 1, 8 * 3 + 2] = float(what)
    else:
        w[17, 1, 3] = -0.5 if what == "negative weight" else float("inf")
    got, _ = learn(x, w, u, c, 4)
    keep = torch.ones(heads, D // c, dtype=torch.bool)
    keep[1, 3] = False
    assert torch.equal(got[keep.to(DEV)], good[keep.to(DEV)])
    if what == "negative weight":
        want, _ = plain(x, w, u, c, 4)
        assert torch.allclose(got[1, 3], want[1, 3], rtol=1e-4, atol=1e-4)
